"""The gathers of the narrow direct convolution read no byte outside their tensors, and the right bytes:
csrc/wino_narrow_rows.cuh compiled for the host, with loads that check their addresses."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#define __device__
#define __forceinline__ inline
static const int8_t* g_at; static long g_size; static long g_bad;
template <typename T> T __ldg(const T* p) {
  const int8_t* b = reinterpret_cast<const int8_t*>(p);
  if (b < g_at || b + sizeof(T) > g_at + g_size || reinterpret_cast<uintptr_t>(p) % sizeof(T)) { ++g_bad; return T(0); }
  T v; std::memcpy(&v, p, sizeof(T)); return v;
}
static uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) {
  return (uint32_t)(((((uint64_t)hi) << 32) | lo) >> (s & 31));
}
#include "wino_narrow_rows.cuh"

static int8_t* tensor(long n) {
  int8_t* p = static_cast<int8_t*>(aligned_alloc(16, (n + 31) / 16 * 16));
  for (long i = 0; i < n; ++i) p[i] = (int8_t)(i * 37 + 11);
  g_at = p; g_size = n;
  return p;
}
static long g_wrong;
template <int C> void check(const uint32_t (&r)[3][3], int a, int e, int want) {
  if ((uint8_t)(r[a][e / 4] >> (8 * (e % 4))) != (uint8_t)want) ++g_wrong;
}
// TAIL as the launcher chooses it: for both tensors if either needs it
template <int C, bool TAIL> void windows() {
  for (int N = 1; N <= 2; ++N) for (int H = 1; H <= 4; ++H) for (int W = 1; W <= 7; ++W) for (int st = 1; st <= 2; ++st) {
    if (!TAIL && wino::narrow_has_tail((long)N * H * W * C)) continue;
    int8_t* x = tensor((long)N * H * W * C);
    for (int n = 0; n < N; ++n) for (int h = 0; h < H; h += st) for (int w = 0; w < W; w += st) {
      uint32_t r[3][3];
      wino::narrow_window<C, TAIL>(x, N, H, W, n, h - 1, w - 1, 0x05050505u, r);
      for (int a = 0; a < 3; ++a) for (int e = 0; e < 3 * C; ++e) {
        const int hh = h - 1 + a, ww = w - 1 + e / C;
        const bool in = hh >= 0 && hh < H && ww >= 0 && ww < W;
        check<C>(r, a, e, in ? x[(((long)n * H + hh) * W + ww) * C + e % C] : 5);
      }
    }
    free(x);
  }
  for (int K = 1; K <= 9; ++K) {
    if (!TAIL && wino::narrow_has_tail((long)K * 9 * C)) continue;
    int8_t* w = tensor((long)K * 9 * C);
    for (int k = 0; k < K + 2; ++k) {
      uint32_t r[3][3];
      wino::narrow_filter<C, TAIL>(w, K, k, r);
      for (int a = 0; a < 3; ++a) for (int e = 0; e < 3 * C; ++e)
        check<C>(r, a, e, k < K ? w[((long)k * 3 + a) * 3 * C + e] : 0);
    }
    free(w);
  }
}
int main() {
  windows<1, false>(); windows<2, false>(); windows<3, false>(); windows<4, false>();
  windows<1, true>(); windows<2, true>(); windows<3, true>(); windows<4, true>();
  std::printf("%ld %ld\n", g_bad, g_wrong);
}
"""


def test_no_byte_outside_the_tensors(tmp_path):
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-I",
                           os.path.join(ROOT, "paper_2002_10711_b200", "csrc"), str(src), "-o", str(exe)])
    bad, wrong = map(int, subprocess.check_output([str(exe)]).split())
    assert bad == 0, f"{bad} loads outside a tensor"
    assert wrong == 0, f"{wrong} wrong bytes"
