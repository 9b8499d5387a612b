// The gathers of the narrow direct convolution (at most four input channels): rows of 3 * C bytes
// at any alignment, read as aligned words.  Plain C++ but for __ldg and __funnelshift_r, so that
// a host program can check which bytes are read (tests/test_narrow_rows_host.py).
#pragma once
#include <cstdint>

namespace wino {

// The end of a tensor of `bytes` bytes, 4-byte aligned: where its last, incomplete word lies, and
// its bytes.  Only a tensor with such a word needs the gathers' TAIL form (narrow_has_tail), which
// costs them a comparison a word.
struct NarrowEnd {
  const uint32_t* at;
  uint32_t word;
};
inline bool narrow_has_tail(long bytes) { return (bytes & 3) != 0; }
__device__ __forceinline__ NarrowEnd narrow_end(const int8_t* x, long bytes) {
  NarrowEnd end;
  const int8_t* last = x + (bytes & ~3l);
  end.at = reinterpret_cast<const uint32_t*>(last);
  end.word = 0u;
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (e < (int)(bytes & 3)) end.word |= (uint32_t)(uint8_t)__ldg(last + e) << (8 * e);
  return end;
}
// A row of 3 * C bytes at `at`, of which bytes [from, to) exist, as three words; bytes that do not
// exist take the code z (replicated in `fill`).
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_row(const int8_t* at, int from, int to, uint32_t fill, const NarrowEnd& end,
                                           uint32_t (&r)[3]) {
  const uint32_t sh = (uint32_t)(reinterpret_cast<uintptr_t>(at) & 3u);
  const uint32_t* base = reinterpret_cast<const uint32_t*>(at - sh);
  constexpr int kWords = (3 * C + 3 + 3) / 4;   // words that 3 * C bytes at any alignment touch
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < kWords; ++j) {
    // only words that hold a byte of the image are read
    const int lo = 4 * j - (int)sh;
    if (from < to && lo + 4 > from && lo < to) w[j] = TAIL && base + j == end.at ? end.word : __ldg(base + j);
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (4 * j >= 3 * C) { r[j] = 0u; continue; }
    uint32_t v = __funnelshift_r(w[j], j + 1 < kWords ? w[j + 1] : 0u, 8u * sh);
    uint32_t keep = 0u, exist = 0u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int b = 4 * j + e;
      if (b < 3 * C) exist |= 0xFFu << (8 * e);
      if (b < 3 * C && b >= from && b < to) keep |= 0xFFu << (8 * e);
    }
    r[j] = (v & keep) | (fill & exist & ~keep);
  }
}
// The three rows of the window whose first pixel is (h0, w0) of image n.
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_window(const int8_t* x, int H, int W, int n, int h0, int w0, uint32_t fill,
                                              const NarrowEnd& end, uint32_t (&r)[3][3]) {
  const int from = w0 < 0 ? C : 0, to = (W - w0 < 3 ? W - w0 : 3) * C;
  const int8_t* xp = x + (((long)n * H + h0) * W + w0) * C;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const bool in = (unsigned)(h0 + a) < (unsigned)H;
    narrow_row<C, TAIL>(xp + (long)a * W * C, in ? from : 0, in ? to : 0, fill, end, r[a]);
  }
}
// The three rows of filter k of K (k >= K: zeros).
template <int C, bool TAIL>
__device__ __forceinline__ void narrow_filter(const int8_t* w, int K, int k, const NarrowEnd& end,
                                              uint32_t (&r)[3][3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
    narrow_row<C, TAIL>(w + (long)(k < K ? k : 0) * 9 * C + a * 3 * C, 0, k < K ? 3 * C : 0, 0u, end, r[a]);
}

}  // namespace wino
