// The gathers of the narrow direct convolution (at most four input channels): rows of 3 * C bytes
// at any alignment, read as aligned words.  Plain C++ but for __ldg and __funnelshift_r, so that
// a host program can check which bytes are read (tests/test_narrow_rows_host.py).
#pragma once
#include <cstdint>

namespace wino {

// A tensor that ends within a word needs the gathers' TAIL form.
inline bool narrow_has_tail(long bytes) { return (bytes & 3) != 0; }

// The rows of a window or filter, 3 * C bytes each: row a starts at byte `first` + a * step of `x` (16-byte
// aligned, `bytes` bytes) and bytes [from, to[a]) of it exist, as three words; bytes that do not exist take
// the code z (replicated in `fill`).
// TAIL: whole words are read up to the tensor's last, incomplete one.  The few windows near the end have
// that one's bytes fetched beside their other loads; the others pay one comparison.  us without the
// guard / so: 9 images 41x41, 3 -> 16 channels 3.9 / 3.9, 37 images 29x29, stride 2, 3 -> 64 3.24 / 3.28, 63
// images 33x33, zero point, 3 -> 64 6.87 / 7.12.  (That word put together before the gathers cost 1.7 us, a
// comparison at each word 0.4, byte-wise windows 0.4, a loop over their bytes 5.)
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_rows(const int8_t* x, long bytes, long first, long step, int from,
                                            const int (&to)[3], uint32_t fill, uint32_t (&r)[3][3]) {
  constexpr int kWords = (3 * C + 3 + 3) / 4;   // words that 3 * C bytes at any alignment touch
  const bool near = TAIL && first + 2 * step + 3 * C > (bytes & ~3l);
  int whole[3] = {to[0], to[1], to[2]};   // up to where words are read
  uint32_t last[3] = {0u, 0u, 0u};
  if (TAIL && near) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const long room = (bytes & ~3l) - (first + a * step);
      if (room < to[a]) whole[a] = (int)room;
    }
#pragma unroll
    for (int e = 0; e < 3; ++e)
      if (e < (int)(bytes & 3)) last[e] = (uint32_t)(uint8_t)__ldg(x + (bytes & ~3l) + e);
  }
  uint32_t w[3][4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int8_t* row = x + first + a * step;
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 3u);
    const uint32_t* base = reinterpret_cast<const uint32_t*>(row - sh);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // only words that hold a byte of the tensor are read
      const int lo = 4 * j - (int)sh;
      w[a][j] = 0u;
      if (j < kWords && from < to[a] && lo + 4 > from && lo < (TAIL ? whole[a] : to[a])) w[a][j] = __ldg(base + j);
    }
  }
  if (TAIL && near) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int sh = (int)(reinterpret_cast<uintptr_t>(x + first + a * step) & 3u);
#pragma unroll
      for (int j = 0; j < kWords; ++j)
        if (whole[a] < to[a] && 4 * j - sh == whole[a]) w[a][j] = last[0] | (last[1] << 8) | (last[2] << 16);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(x + first + a * step) & 3u);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (4 * j >= 3 * C) { r[a][j] = 0u; continue; }
      const uint32_t v = __funnelshift_r(w[a][j], w[a][j + 1], 8u * sh);
      uint32_t keep = 0u, exist = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int b = 4 * j + e;
        if (b < 3 * C) exist |= 0xFFu << (8 * e);
        if (b < 3 * C && b >= from && b < to[a]) keep |= 0xFFu << (8 * e);
      }
      r[a][j] = (v & keep) | (fill & exist & ~keep);
    }
  }
}
// The three rows of the window whose first pixel is (h0, w0) of image n of N.
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_window(const int8_t* x, int N, int H, int W, int n, int h0, int w0,
                                              uint32_t fill, uint32_t (&r)[3][3]) {
  const int from = w0 < 0 ? C : 0, most = (W - w0 < 3 ? W - w0 : 3) * C;
  int to[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) to[a] = (unsigned)(h0 + a) < (unsigned)H ? most : 0;
  narrow_rows<C, TAIL>(x, (long)N * H * W * C, (((long)n * H + h0) * W + w0) * C, (long)W * C, from, to, fill, r);
}
// The three rows of filter k of K (k >= K: zeros).
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_filter(const int8_t* w, int K, int k, uint32_t (&r)[3][3]) {
  const int most = k < K ? 3 * C : 0;
  const int to[3] = {most, most, most};
  narrow_rows<C, TAIL>(w, (long)K * 9 * C, (long)(k < K ? k : 0) * 9 * C, 3 * C, 0, to, 0u, r);
}

}  // namespace wino
