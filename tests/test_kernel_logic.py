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
