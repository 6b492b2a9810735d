"""Performance cases: what a user of the library has it do, from one step of a
large job to a long recorded run.

A case names a kind of call and its sizes.  d is [T][R][S], T steps of R ranks
with S stages, int64 nanoseconds; W is the window length in steps.

  label     sf_label_windows: labels of a recorded run, with wall times, roles
            and missing-rank counts where `wall` is set
  step      the whole analysis with lead-rank credit: window median, evidence
            pass, top-k suspects, gates
  route     routing only: window aggregation with lead-rank credit, top-k
  frontier  per-step frontier and the size of its tie set
  lag       cross-rank lag, delta-lag and gap per step
  report    the comparison summaries of a report: baselines, raw rank spread,
            window sums of lag and gap
  groups    a gathered (rank-major) run turned into steps, then the frontier
            inside node groups and reporting-group sums
  stream    gathered windows in pinned host memory, streamed through the whole
            analysis; the host-to-device copy is part of it
"""
import math
import random

import torch

from paper_2606_06751_gb300 import stagefrontier as sf

MS = 1e6  # nanoseconds
CELLS = 1 << 24  # records handled at a time when inputs or exact results are made


def listed():
    return [
        # a small job's run, labelled with all of its metadata: launches and host calls
        dict(name="label_small", kind="label", T=1000, R=8, S=6, W=100, wall=True),
        # one step of a large job, looked at as it ends: the smallest call there is
        dict(name="frontier_one_step", kind="frontier", T=1, R=8192, S=8),
        # one window of a large job, analysed as it closes
        dict(name="step_live_window", kind="step", T=100, R=8192, S=8, W=100, k=5),
        # long recorded runs of a data-parallel, a sharded and a very wide job
        dict(name="step_ddp", kind="step", T=100000, R=128, S=8, W=1000, k=2),
        dict(name="step_fsdp", kind="step", T=50000, R=1024, S=10, W=500, k=5, tail=True),
        dict(name="step_wide", kind="step", T=20000, R=8192, S=8, W=1000, k=5),
        # sizes that are no multiple of anything, and a partial last window
        dict(name="step_ragged", kind="step", T=13421, R=1000, S=5, W=1000, k=5),
        # routing over many fine stages on few ranks
        dict(name="route_fine", kind="route", T=131072, R=64, S=16, W=1000, k=5),
        # localisation evidence on a wide job
        dict(name="lag_wide", kind="lag", T=4000, R=8192, S=8),
        # the summaries that a report sets beside the frontier
        dict(name="report_fsdp", kind="report", T=10000, R=1024, S=10, W=500, tail=True),
        # node groups of a wide job whose windows came from a gather
        dict(name="groups_wide", kind="groups", T=2000, R=8192, S=8, W=1000),
        # gathered windows that arrive in host memory
        dict(name="stream_fsdp", kind="stream", T=2000, R=1024, S=10, W=500, k=5, tail=True),
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["label", "step", "step", "route", "frontier", "lag", "report", "groups", "stream"])
    S = rng.choice([4, 6, 8, 8, 10, 16, rng.randint(1, 24)])
    R = _between(rng, 8, 32768)
    if rng.random() < 0.5:  # half of the jobs have whole nodes
        R = max(8, R // 8 * 8)
    most = {"stream": 1 << 24, "label": 1 << 26}.get(kind, 1 << 27)
    least = 1 if kind == "frontier" else 20  # steps
    T = _between(rng, max(50000, least * R * S), most) // (R * S)
    case = dict(kind=kind, T=T, R=R, S=S)
    if kind not in ("frontier", "lag"):
        case["W"] = min(T, rng.choice([100, 500, 1000, _between(rng, 20, 1000)]))
    if kind in ("step", "route", "stream"):
        case["k"] = rng.choice([2, 5, 5, 10])
    if kind == "label":
        case["wall"] = rng.random() < 0.5
    if rng.random() < 0.3:
        case["tail"] = True
    return case


# ---------------------------------------------------------------- inputs


def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _telemetry(case, seed):
    """d[T][R][S] of a synchronous trainer: lognormal stage work around seeded
    stage medians of 1 to 100 ms; at two collectives every rank waits for the
    last one; a stalled (rank, stage) in 1 % of the windows, one node 10 % slower
    over an eighth of the run, and with `tail` heavy-tailed (step, rank) cells."""
    T, R, S = case["T"], case["R"], case["S"]
    dev, rnd = _device(), random.Random(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    median = torch.tensor([MS * 100.0 ** rnd.random() for _ in range(S)], dtype=torch.float64, device=dev)
    W = case.get("W", 1000)
    nW = -(-T // W)
    stalls = [(w * W, rnd.randrange(R), rnd.randrange(S), int(rnd.uniform(5, 50) * MS))
              for w in sorted(rnd.sample(range(nW), max(1, round(0.01 * nW))))]
    per = max(1, R // 64)
    node = rnd.randrange(0, R - per + 1)
    slow_at = rnd.randrange(T)
    slow_end = slow_at + max(1, T // 8)
    d = torch.empty((T, R, S), dtype=torch.int64, device=dev)
    n = max(1, CELLS // (R * S))
    for t0 in range(0, T, n):
        t1 = min(T, t0 + n)
        x = torch.randn((t1 - t0, R, S), generator=gen, device=dev).double().mul_(0.1).exp_().mul_(median)
        if case.get("tail"):
            u = torch.rand((t1 - t0, R, 1), generator=gen, device=dev)
            x.mul_(torch.where(u < 0.005, (u / 0.005).clamp_(1e-6, 1.0).pow_(-1.0 / 3.0), 1.0).double())
        a, b = max(slow_at, t0), min(slow_end, t1)
        if a < b:
            x[a - t0:b - t0, node:node + per] *= 1.1
        v = x.round_().long()
        for begin, r, s, extra in stalls:
            a, b = max(begin, t0), min(begin + W, t1)
            if a < b:
                v[a - t0:b - t0, r, s] += extra
        since, left = 0, 0  # the first stage after the last collective, and each rank's time since its release
        for q in sorted({S // 2, S - 1}):
            arrive = left + v[:, :, since:q].sum(2)
            left = v[:, :, q].clone()
            v[:, :, q] += arrive.amax(1, keepdim=True) - arrive
            since = q + 1
        d[t0:t1] = v
    return d


def _groups(R, S):
    """Ranks to node groups of 128 ranks (larger ones where that would be too many)."""
    per = max(128, -(-R * S // 4000))
    return torch.arange(R, dtype=torch.int32) // per, -(-R // per)


def _gathered(d, W):
    """The windows' rank-major [R][n][S] blocks, one after another."""
    return torch.cat([d[t:t + W].transpose(0, 1).reshape(-1) for t in range(0, d.shape[0], W)])


def prepare(case, seed):
    kind, T, R, S, W = case["kind"], case["T"], case["R"], case["S"], case.get("W")
    dev = _device()
    d = _telemetry(case, seed)
    st = dict(case=case, d=d, status=sf.new_status(dev))
    if kind == "label":
        st["workspace"] = torch.empty(sf.workspace_size(T, R, S, W), dtype=torch.uint8, device=dev)
        if case.get("wall"):
            gen = torch.Generator(device=dev).manual_seed(seed + 1)
            extra = 0.02 * torch.rand((T, R), generator=gen, device=dev).double()
            total = d.sum(2)
            st["wall"] = total + (total.double() * extra).long()
            st["role"] = torch.zeros(R, dtype=torch.int32, device=dev)
            st["missing"] = torch.zeros(-(-T // W), dtype=torch.int32, device=dev)
    elif kind in ("lag", "report"):
        st["workspace"] = sf.rank_workspace(T, R, S, dev)
    elif kind == "groups":
        group, st["G"] = _groups(R, S)
        st["group"] = group.to(dev)
        st["gathered"] = _gathered(d, W)
        st["d"] = torch.empty_like(d)
        st["stage_group"] = [0 if s < S // 2 else 1 for s in range(S)]
    elif kind == "stream":
        host = torch.empty(T * R * S, dtype=torch.int64, pin_memory=True)
        host.copy_(_gathered(d, W))
        del st["d"]
        st["host"] = host
        chunk = W * max(1, min(-(-T // W), (1 << 23) // max(1, R * S * W)))
        st["chunk"] = chunk
        st["buffers"] = sf.StreamBuffers(T, R, S, W, case["k"], chunk, dev, gathered=True)
        st["copy_stream"] = torch.cuda.Stream(dev)
    return st


# ---------------------------------------------------------------- one pass


def run(state):
    case, status = state["case"], state["status"]
    kind, T, R, S, W = case["kind"], case["T"], case["R"], case["S"], case.get("W")
    d = state.get("d")
    if kind == "label":
        return vars(sf.sf_label_windows(d, W, role=state.get("role"), missing=state.get("missing"),
                                        wall=state.get("wall"), workspace=state["workspace"], status=status))
    if kind == "step":
        m = sf.sf_window_median(d, W, status=status)
        ev = sf.sf_direct_gain(d, W, m, lead_credit=True, status=status)
        top = sf.sf_topk_suspects(ev.X, ev.E, case["k"])
        lab = sf.sf_label_gates(T, R, S, W, ev)
        return dict(median=m, evidence=vars(ev), top=vars(top), labels=vars(lab), status=status)
    if kind == "route":
        win = sf.sf_window_aggregate(d, W, status=status)
        return dict(windows=vars(win), top=vars(sf.sf_topk_suspects(win.X, win.E, case["k"])), status=status)
    if kind == "frontier":
        f = sf.sf_frontier(d, status=status)
        return dict(frontier=vars(f), ties=sf.sf_frontier_ties(d, a=f.a, status=status), status=status)
    if kind == "lag":
        return dict(lag=vars(sf.sf_rank_lag(d, workspace=state["workspace"], status=status)), status=status)
    if kind == "report":
        base = sf.sf_window_baselines(d, W, status=status)
        spread = sf.sf_raw_spread(d, W, workspace=state["workspace"], status=status)
        lag, gap = sf.sf_rank_lag_windows(d, W, workspace=state["workspace"], status=status)
        return dict(M=base.M, SUM=base.SUM.view(torch.int64), SLOW=base.SLOW, RANK0=base.RANK0, spread=spread,
                    lag=lag, gap=gap, status=status)
    if kind == "groups":
        sf.sf_gathered_to_steps(state["gathered"], T, R, S, W, dst=d)
        win = sf.sf_group_aggregate(d, state["group"], state["G"], W, status=status)
        per_stage = win.X.view(-1, S)
        return dict(d=d, X=win.X, D=win.D, reported=sf.sf_stage_group_sum(per_stage, state["stage_group"], 2),
                    status=status)
    state["copy_stream"].wait_stream(torch.cuda.current_stream())  # the last pass may still read the staging buffers
    return vars(sf.sf_stream_gathered_windows(state["host"], T, R, S, W, case["k"], state["chunk"],
                                              bufs=state["buffers"], status=status,
                                              copy_stream=state["copy_stream"]))


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    kind, T, R, S, W = case["kind"], case["T"], case["R"], case["S"], case.get("W")
    nW = -(-T // W) if W else 0
    k = case.get("k", 0)
    cells = T * R * S
    labels = nW * (12 + 16 * S)  # label, two masks, shares and gains
    top = nW * k * 28
    out = {
        "label": labels + nW * 8 * (2 * S + 1) + (T * R * 8 + R * 4 + nW * 4 if case.get("wall") else 0),
        "step": nW * R * S * 20 + nW * 8 * (2 * S + 1) + T + top + labels + nW * 8,
        "route": nW * R * S * 12 + nW * 8 * (S + 1) + T + top,
        "frontier": T * (S * 16 + 8),
        "lag": T * S * 24,
        "report": nW * S * 64,
        "groups": cells * 8,
        "stream": nW * R * S * 12 + nW * 8 * (2 * S + 1) + nW * k * 20 + labels,
    }[kind]
    if kind == "groups":
        G = _groups(R, S)[1]
        out += R * 4 + nW * G * (S + 1) * 8 + nW * G * 16
    return {"bytes": cells * 8 + out, "flops": 2 * cells}


def tolerance(case):
    # whole numbers throughout; shares and gains are one IEEE division of two of them
    return "exact"


# ---------------------------------------------------------------- the same in plain torch, 64 bits


def _spans(case, W=None):
    """Step ranges of a bounded size, none across a window's end."""
    T, n = case["T"], max(1, CELLS // (case["R"] * case["S"]))
    W = W or T
    for w0 in range(0, T, W):
        end = min(T, w0 + W)
        for t0 in range(w0, end, n):
            yield w0 // W, t0, min(end, t0 + n)


def _step_frontier(P):
    """F, lowest attaining rank and increments, each [n][S], of the prefixes P [n][R][S]."""
    R = P.shape[1]
    key = ((P << 16) | (65535 - torch.arange(R, device=P.device).view(1, R, 1))).amax(1)
    F = key >> 16
    return F, 65535 - (key & 65535), torch.diff(F, dim=1, prepend=torch.zeros_like(F[:, :1]))


def _windows(case, d, m=None):
    """Sums per window: X, D, E, C, the leading stage per step, and with the
    window medians m the gain numerators Y and the leaders' confidence."""
    T, R, S, W = case["T"], case["R"], case["S"], case["W"]
    nW, dev = -(-T // W), d.device
    X = torch.zeros((nW, S), dtype=torch.int64, device=dev)
    Y, D = torch.zeros_like(X), torch.zeros(nW, dtype=torch.int64, device=dev)
    E = torch.zeros((nW, S, R), dtype=torch.int64, device=dev)
    C = torch.zeros((nW, S, R), dtype=torch.int32, device=dev)
    lead_stage = torch.empty(T, dtype=torch.uint8, device=dev)
    stage = 31 - torch.arange(S, device=dev)
    for w, t0, t1 in _spans(case, W):
        P = d[t0:t1].cumsum(2)
        F, lead, a = _step_frontier(P)
        X[w] += a.sum(0)
        D[w] += F[:, -1].sum()
        E[w].scatter_add_(1, lead.t().contiguous(), a.t().contiguous())
        C[w].scatter_add_(1, lead.t().contiguous(), torch.ones_like(lead.t(), dtype=torch.int32).contiguous())
        key = ((a << 5) | stage).amax(1)
        best = 31 - (key & 31)
        if m is not None:
            cut = (d[t0:t1] - m[w]).clamp_(min=0)
            Y[w] += (F[:, -1:] - (P[:, :, -1:] - cut).amax(1)).sum(0)
            second = a.scatter(1, best.view(-1, 1), 0).amax(1)
            best = best + 128 * ((F[:, -1] > 0) & (((key >> 5) - second) * 20 >= F[:, -1])).long()
        lead_stage[t0:t1] = best.to(torch.uint8)
    return X, Y, D, E, C, lead_stage


def _medians(case, d):
    T, R, S, W = case["T"], case["R"], case["S"], case["W"]
    m = torch.empty((-(-T // W), R * S), dtype=torch.int64, device=d.device)
    for w in range(m.shape[0]):
        rows = d[w * W:(w + 1) * W].view(-1, R * S)
        n = max(1, CELLS // rows.shape[0])
        for c in range(0, R * S, n):
            m[w, c:c + n] = rows[:, c:c + n].sort(0).values[(rows.shape[0] - 1) // 2]
    return m.view(-1, R, S)


def _ratio(X, D):
    return torch.where(D.view(-1, 1) > 0, X.double() / D.double().view(-1, 1), 0.0)


def _order_statistics(v):
    """Maximum, lower median and second largest over the ranks of v [n][R][S]."""
    v = v.sort(1).values
    R = v.shape[1]
    return v[:, -1], v[:, (R - 1) // 2], v[:, max(0, R - 2)]


def _top(X, E, k):
    """The k largest stages by X and (stage, rank) pairs by E; value 0 is no suspect."""
    nW, S = X.shape
    R = E.shape[2]

    def largest(V):
        v, at = V.sort(dim=1, descending=True, stable=True)
        v = torch.nn.functional.pad(v, (0, max(0, k - v.shape[1])))[:, :k]
        at = torch.nn.functional.pad(at, (0, max(0, k - at.shape[1])))[:, :k]
        return v, torch.where(v > 0, at, -1)

    sv, si = largest(X)
    pv, pi = largest(E.view(nW, S * R))
    pair = torch.stack([torch.where(pi >= 0, pi // R, -1), torch.where(pi >= 0, pi % R, -1)], 2)
    return si.to(torch.int32), sv, pair.to(torch.int32), pv


def exact(case, seed):
    """The outputs of run() without the label decisions, which are no computed numbers."""
    kind, T, R, S, W = case["kind"], case["T"], case["R"], case["S"], case.get("W")
    d = _telemetry(case, seed)
    dev = d.device
    if kind in ("label", "step", "stream"):
        m = _medians(case, d)
        X, Y, D, E, C, lead_stage = _windows(case, d, m)
        share, gain = _ratio(X, D), _ratio(Y, D)
        if kind == "label":
            return dict(share=share, gain=gain, X=X, Y=Y, D=D)
        si, sv, pi, pv = _top(X, E, case["k"])
        if kind == "stream":
            return dict(X=X, Y=Y, D=D, E=E, C=C, top_stage=si, top_pair=pi, top_pair_value=pv, share=share, gain=gain)
        return dict(median=m, evidence=dict(X=X, Y=Y, D=D, E=E, C=C, step_lead=lead_stage),
                    top=dict(stage=si, stage_value=sv, pair=pi, pair_value=pv), labels=dict(share=share, gain=gain))
    if kind == "route":
        X, _, D, E, C, lead_stage = _windows(case, d)
        si, sv, pi, pv = _top(X, E, case["k"])
        return dict(windows=dict(X=X, D=D, E=E, C=C, step_lead=lead_stage),
                    top=dict(stage=si, stage_value=sv, pair=pi, pair_value=pv))
    if kind == "frontier":
        a = torch.empty((T, S), dtype=torch.int64, device=dev)
        lead, ties = torch.empty_like(a, dtype=torch.int32), torch.empty_like(a, dtype=torch.int32)
        for _, t0, t1 in _spans(case):
            P = d[t0:t1].cumsum(2)
            F, at, a[t0:t1] = _step_frontier(P)
            lead[t0:t1] = at.to(torch.int32)
            ties[t0:t1] = (P == F[:, None]).sum(1).to(torch.int32)
        return dict(frontier=dict(a=a, lead=lead, makespan=a.sum(1)), ties=ties)
    if kind == "lag":
        L = torch.empty((T, S), dtype=torch.int64, device=dev)
        G = torch.empty_like(L)
        for _, t0, t1 in _spans(case):
            top, mid, second = _order_statistics(d[t0:t1].cumsum(2))
            L[t0:t1], G[t0:t1] = top - mid, top - second
        return dict(lag=dict(L=L, dL=torch.diff(L, dim=1, prepend=torch.zeros_like(L[:, :1])), G=G))
    nW = -(-T // W)
    if kind == "report":
        M, total, slow, rank0, spread, lag, gap = (torch.zeros((nW, S), dtype=torch.int64, device=dev) for _ in range(7))
        for w, t0, t1 in _spans(case, W):
            v = d[t0:t1]
            P = v.cumsum(2)
            key = ((P[:, :, -1] << 16) | (65535 - torch.arange(R, device=dev))).amax(1)
            at = (65535 - (key & 65535)).view(-1, 1, 1).expand(-1, 1, S)
            top, mid, _ = _order_statistics(v)
            M[w] += top.sum(0)
            spread[w] += (top - mid).sum(0)
            total[w] += v.sum((0, 1))
            slow[w] += v.gather(1, at).sum((0, 1))
            rank0[w] += v[:, 0].sum(0)
            top, mid, second = _order_statistics(P)
            lag[w] += (top - mid).sum(0)
            gap[w] += (top - second).sum(0)
        return dict(M=M, SUM=torch.stack([total, torch.zeros_like(total)], 2), SLOW=slow, RANK0=rank0, spread=spread,
                    lag=lag, gap=gap)
    group, G = _groups(R, S)
    group = group.long().to(dev)
    X = torch.zeros((nW, G, S), dtype=torch.int64, device=dev)
    D = torch.zeros((nW, G), dtype=torch.int64, device=dev)
    for w, t0, t1 in _spans(case, W):
        P = d[t0:t1].cumsum(2)
        for g in range(G):
            F = P[:, group == g].amax(1)
            X[w, g] += torch.diff(F, dim=1, prepend=torch.zeros_like(F[:, :1])).sum(0)
            D[w, g] += F[:, -1].sum()
    first = X[..., :S // 2].sum(2)
    reported = torch.stack([first, X.sum(2) - first], 2).view(-1, 2)
    return dict(d=d, X=X, D=D, reported=reported)
