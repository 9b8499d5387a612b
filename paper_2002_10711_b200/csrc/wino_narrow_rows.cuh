// The gathers of the narrow direct convolution (at most four input channels): rows of 3 * C bytes
// at any alignment, read as aligned words.  Plain C++ but for __ldg and __funnelshift_r, so that
// a host program can check which bytes are read (tests/test_narrow_rows_host.py).
#pragma once
#include <cstdint>

namespace wino {

// The end of a tensor of `bytes` bytes, 4-byte aligned: where its last, incomplete word lies, and
// its bytes.  Only a tensor with such a word needs the gathers' TAIL form (narrow_has_tail), which
// costs them a comparison a word (9 images 41x41, 3 -> 16 channels: 3.9 -> 4.3 us).  Bytes put together
// before the gathers, byte-wise loads in the windows concerned, or a loop there were slower (5.6, 4.4, 9 us).
struct NarrowEnd {
  const uint32_t* at;
  uint32_t byte[3];   // put together where they are needed: nothing waits for them before
};
inline bool narrow_has_tail(long bytes) { return (bytes & 3) != 0; }
__device__ __forceinline__ NarrowEnd narrow_end(const int8_t* x, long bytes) {
  NarrowEnd end;
  const int8_t* last = x + (bytes & ~3l);
  end.at = reinterpret_cast<const uint32_t*>(last);
#pragma unroll
  for (int e = 0; e < 3; ++e) end.byte[e] = e < (int)(bytes & 3) ? (uint32_t)(uint8_t)__ldg(last + e) : 0u;
  return end;
}
// The rows of a window or filter, 3 * C bytes each: row a is at `at` + a * step and bytes [from, to[a])
// of it exist, as three words; bytes that do not exist take the code z (replicated in `fill`).  All
// loads of whole words come first.
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_rows(const int8_t* at, long step, int from, const int (&to)[3], uint32_t fill,
                                            const NarrowEnd& end, uint32_t (&r)[3][3]) {
  constexpr int kWords = (3 * C + 3 + 3) / 4;   // words that 3 * C bytes at any alignment touch
  uint32_t w[3][4];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int8_t* row = at + a * step;
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 3u);
    const uint32_t* base = reinterpret_cast<const uint32_t*>(row - sh);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // only words that hold a byte of the tensor are read
      const int lo = 4 * j - (int)sh;
      w[a][j] = 0u;
      if (j < kWords && from < to[a] && lo + 4 > from && lo < to[a] && !(TAIL && base + j == end.at))
        w[a][j] = __ldg(base + j);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int8_t* row = at + a * step;
    const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 3u);
    if (TAIL) {
      const uint32_t* base = reinterpret_cast<const uint32_t*>(row - sh);
      const uint32_t last = end.byte[0] | (end.byte[1] << 8) | (end.byte[2] << 16);
#pragma unroll
      for (int j = 0; j < kWords; ++j)
        if (base + j == end.at) w[a][j] = last;
    }
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
// The three rows of the window whose first pixel is (h0, w0) of image n.
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_window(const int8_t* x, int H, int W, int n, int h0, int w0, uint32_t fill,
                                              const NarrowEnd& end, uint32_t (&r)[3][3]) {
  const int from = w0 < 0 ? C : 0, most = (W - w0 < 3 ? W - w0 : 3) * C;
  int to[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) to[a] = (unsigned)(h0 + a) < (unsigned)H ? most : 0;
  narrow_rows<C, TAIL>(x + (((long)n * H + h0) * W + w0) * C, (long)W * C, from, to, fill, end, r);
}
// The three rows of filter k of K (k >= K: zeros).
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_filter(const int8_t* w, int K, int k, const NarrowEnd& end,
                                              uint32_t (&r)[3][3]) {
  const int most = k < K ? 3 * C : 0;
  const int to[3] = {most, most, most};
  narrow_rows<C, TAIL>(w + (long)(k < K ? k : 0) * 9 * C, 3 * C, 0, to, 0u, end, r);
}

}  // namespace wino
