"""The kernels' bookkeeping, run on the host: the headers that the kernels use,
compiled with the host compiler and driven by a restatement of what surrounds them."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_06751_gb300", "csrc")


def run_host(tmp_path, source, *args):
    src, exe = tmp_path / "logic.cpp", tmp_path / "logic"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe), *map(str, args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


# rank_step_kernel's search of one column: a first bracket from the lanes' minima and
# maxima, histogram rounds, the last 32 keys ranked by counting
SEARCH = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "sf_bracket.h"
using sf::KeyBracket;

// Whether the search finds the kth smallest of x; B < A: no bracket from the lanes.
static bool search(const std::vector<uint32_t>& x, uint32_t kth, uint32_t A, uint32_t B, uint32_t& ans) {
  const uint32_t lo = *std::min_element(x.begin(), x.end()), hi = *std::max_element(x.begin(), x.end());
  if (A > B) A = lo, B = hi;
  KeyBracket br = KeyBracket::between(A, B);
  uint32_t rem = kth;
  ans = lo;
  bool first = true;
  for (int round = 0; lo != hi; ++round) {
    if (round == sf::kBracketRounds) return false;  // the kernel's limit
    const int sh = br.shift();
    if ((br.span >> sh) > 255) return false;  // more bins than there are
    std::vector<uint32_t> hist(256, 0);
    uint32_t below = 0, upto = 0;
    for (uint32_t k : x) {
      if (br.has(k)) hist[((k - br.lo) >> sh) & 255u]++;
      else if (k < br.lo) below++;
      upto += k <= br.last();
    }
    if (first) {
      first = false;
      if (kth < below || kth >= upto) {
        if (kth < below) br = KeyBracket::between(lo, br.lo - 1);
        else br = KeyBracket::between(br.last() + 1, hi), rem = kth - upto;
        continue;
      }
      rem = kth - below;
    }
    uint32_t digit = 0;
    while (digit < 256 && rem >= hist[digit]) rem -= hist[digit++];
    if (digit == 256) return false;
    const uint32_t kept = hist[digit];
    br.narrow(digit);
    ans = br.lo;
    if (sh == 0) return true;
    if (kept <= 32) {
      std::vector<uint32_t> c;
      for (uint32_t k : x)
        if (br.has(k)) c.push_back(k);
      if (c.size() != kept) return false;  // the kernel holds 32
      std::sort(c.begin(), c.end());
      ans = c[rem];
      return true;
    }
  }
  return true;
}

int main() {
  std::mt19937_64 g(1);
  auto in = [&](uint64_t a, uint64_t b) { return static_cast<uint32_t>(a + g() % (b - a + 1)); };
  const uint64_t top = 0xffffffffull;
  for (int n = 0; n < 20000; ++n) {
    const int R = in(1, 600) * (n % 8 ? 1 : 16);
    std::vector<uint32_t> x(R);
    const int kind = n % 5, bits = in(0, 32);
    for (uint32_t& k : x) {
      const bool far = in(0, 99) < 25;  // the ranks that were not the last
      if (kind == 0) k = far ? in(2500000000ull, 3500000000ull) : in(top - (1u << 23), top - (1u << 20));
      else if (kind == 1) k = far ? in(0, top) : in(top - (1ull << std::min(bits, 31)), top);
      else if (kind == 2) k = far ? in(0, 1u << 20) : top - in(0, 40);
      else if (kind == 3) k = in(0, (1ull << bits) - 1);
      else k = in(0, 3) * 0x55555555u;
    }
    const uint32_t kth = (R - 1) / 2;
    std::vector<uint32_t> sorted = x;
    std::sort(sorted.begin(), sorted.end());
    uint32_t A = 0, B = top;
    const int lanes = std::max(1, R / 16);  // each stands for 16 keys
    for (int l = 0; l < lanes; ++l) {
      uint32_t mn = top, mx = 0;
      for (int i = l; i < R; i += lanes) mn = std::min(mn, x[i]), mx = std::max(mx, x[i]);
      A = std::max(A, mn);
      B = std::min(B, mx);
    }
    uint32_t ans;
    if (!search(x, kth, A, B, ans) || ans != sorted[kth]) {
      std::printf("case %d: kind %d, %d keys\n", n, kind, R);
      return 1;
    }
  }
  return 0;
}
"""


def test_bracket_search(tmp_path):
    run_host(tmp_path, SEARCH)


# the tiled evidence pass's resident medians: one producer per warp group (the first
# also copies the windows' medians), ring stages per group, a CTA's range of steps, every
# thread's next action taken in any order
SLOTS = r"""
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>
#include "sf_median_slots.h"
using namespace sf;

struct Barrier {  // an mbarrier: `count` arrivals to a phase
  int count, left, phase = 0;
  explicit Barrier(int n) : count(n), left(n) {}
  void arrive() {
    if (--left == 0) left = count, ++phase;
  }
  bool done(uint32_t parity) const { return (phase & 1u) != parity; }
};

struct Run {
  int n, offset, W, G, gw, slots, tiles, stages;  // steps, place of the first in its window, groups of gw warps
  int last;
  std::mt19937 g;
  MedianPlace place;
  std::vector<Barrier> full, done;
  int held[2] = {-1, -1};                          // window whose medians a slot holds
  std::vector<int> issued;                         // tiles of each group copied so far
  struct Warp { MedianWalk walk; int step, tile = 0, phase = 0, done = 0; };
  std::vector<Warp> warps;
  std::vector<std::vector<int>> at_step_end;       // arrivals of a group's warps per step
  struct Producer { int step, tile = 0, part = 0, next = 0; };
  std::vector<Producer> prods;
  bool wrong = false;

  Run(int n, int offset, int W, int G, int gw, int slots, int tiles, int stages, unsigned seed)
      : n(n), offset(offset), W(W), G(G), gw(gw), slots(slots), tiles(tiles), stages(stages),
        last((offset + n - 1) / W), g(seed), place{slots}, full(2, Barrier(1)), done(2, Barrier(G * gw)), issued(G, 0),
        at_step_end(G, std::vector<int>(n + G, 0)) {
    for (int w = 0; w < G * gw; ++w) warps.push_back({MedianWalk(), w / gw});
    for (int q = 0; q < G; ++q) prods.push_back({q});
  }
  int window(int t) const { return (offset + t) / W; }
  int consumed(int q) const {  // tiles every warp of the group is done with
    int c = 1 << 30;
    for (int w = q * gw; w < (q + 1) * gw; ++w) c = std::min(c, (warps[w].step - q) / G * tiles + warps[w].tile);
    return c;
  }
  // One action of producer q; false if it waits or is through.
  bool produce(int q) {
    Producer& p = prods[q];
    if (p.step >= n) return false;
    if (p.part != 1) {  // the windows up to the step's, after its tiles up to the round's
      const int upto = window(p.part == 0 ? p.step : std::min(p.step + G, n) - 1);
      if (q != 0 || p.next > upto) {
        if (p.part == 0) p.part = 1;
        else p.part = 0, p.step += G;
        return true;
      }
      const uint32_t s = place.slot(p.next);
      if (!done[s].done(place.parity(p.next) ^ 1u)) return false;
      held[s] = p.next++;
      full[s].arrive();
      return true;
    }
    if (p.tile == tiles) {
      p.tile = 0;
      p.part = 2;
      return true;
    }
    if (issued[q] - consumed(q) >= stages) return false;
    ++issued[q];
    ++p.tile;
    return true;
  }
  // The warp's walk up to the first wait that holds it; false until it is through.
  // (The walk starts over from its first action each time, so those done are counted.)
  template <typename F>
  bool walk(Warp& c, F f) {
    const MedianWalk from = c.walk;
    int k = 0;
    bool held_up = false;
    f([&](int i) { if (!held_up && k++ == c.done) done[place.slot(i)].arrive(), ++c.done; },
      [&](int i) {
        if (held_up || k++ < c.done) return;
        if (full[place.slot(i)].done(place.parity(i))) ++c.done;
        else held_up = true;
      });
    if (held_up) c.walk = from;
    else c.done = 0;
    return !held_up;
  }
  bool consume(int w) {
    Warp& c = warps[w];
    const int q = w / gw;
    if (c.step >= n) {
      if (c.phase == 4) return false;
      if (!walk(c, [&](auto arrive, auto wait) { c.walk.leave(last, slots, arrive, wait); })) return false;
      c.phase = 4;
      return true;
    }
    const int i = window(c.step);
    if (c.phase == 0) {
      if (!walk(c, [&](auto arrive, auto wait) { c.walk.enter(i, arrive, wait); })) return false;
      c.phase = 2;
      return true;
    }
    if (c.phase == 2) {  // a tile, read beside the medians
      if (issued[q] <= (c.step - q) / G * tiles + c.tile) return false;
      wrong |= held[place.slot(i)] != i;
      if (++c.tile == tiles) {
        c.phase = 3;
        ++at_step_end[q][c.step];
      }
      return true;
    }
    wrong |= c.walk.at != i;
    if (at_step_end[q][c.step] < gw) return false;
    c.step += G;
    c.tile = c.phase = 0;
    return true;
  }
  // Whether every thread came to its end and read its own windows' medians.
  bool go() {
    const int N = G * gw + G;
    std::vector<double> weight(N);  // some threads slow
    for (double& x : weight) x = g() % 3 ? 1.0 : 0.02;
    const int slow = g() % (2 * G);  // or a whole group
    for (int w = 0; slow < G && w < gw; ++w) weight[slow * gw + w] = 0.02;
    std::discrete_distribution<int> pick(weight.begin(), weight.end());
    auto step = [&](int a) { return a < G * gw ? consume(a) : produce(a - G * gw); };
    for (;;) {
      bool moved = false;
      for (int k = 0; k < 4 * N; ++k) moved |= step(pick(g));
      if (wrong) return false;
      if (moved) continue;
      for (int a = 0; a < N; ++a) moved |= step(a);
      if (!moved) break;
    }
    for (const Warp& c : warps)
      if (c.step < n || c.phase != 4) return false;
    for (const Producer& p : prods)
      if (p.step < n) return false;
    return !wrong;
  }
};

int main() {
  std::mt19937 g(7);
  for (int k = 0; k < 6000; ++k) {
    const int slots = 1 + g() % 2, G = 1 << g() % 3, gw = (g() % 2 ? 12 : 8) / G, W = 16 + g() % 20;
    int n = 1 + g() % 90, offset = g() % W;
    if (g() % 2) {  // a range that ends within a round of steps after a window's start
      const int windows = 1 + g() % 3;
      n = windows * W - offset + 1 + g() % G;
    }
    Run r(n, offset, W, G, gw, slots, 1 + g() % 4, 2 + g() % 2, g());
    if (!r.go()) {
      std::printf("steps %d of windows of %d from %d, %d groups of %d warps, %d slots\n", n, W, offset, G, gw, slots);
      return 1;
    }
  }
  return 0;
}
"""


def test_median_slots(tmp_path):
    run_host(tmp_path, SLOTS)
