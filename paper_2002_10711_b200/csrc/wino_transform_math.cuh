// Transform arithmetic shared by every kernel that applies B^T d B or A^T m A
// (paper: Eq. 1): the two-sided transforms as fused-multiply-add chains in the
// contract's order, with compile-time Cook-Toom constants (zero entries vanish)
// and the factored exact forms for F4.
//
// Transform modes:
//   kDense  : matrices are data (learnt "flex" transforms); every entry is used.
//   kDensePair: the same for two channels, with the entries read as pairs.
//   kSparse : the built-in Cook-Toom matrices as compile-time constants.
//   kExact  : Cook-Toom matrices on integer codes where every intermediate is
//             exactly representable (input stage for m = 2, 4, 6; output stage on
//             int8 codes for m = 2, 4 and, for m = 6, all of it but six of the 36
//             pixels), so any summation order gives the same bits; shared
//             sub-expressions are factored out.
#pragma once
#include "wino_f32x2.cuh"

namespace wino {

enum { kDense = 0, kSparse = 1, kExact = 2, kDensePair = 3 };

template <int CPT> struct Pack;
template <> struct Pack<1> { typedef uint8_t type; };
template <> struct Pack<2> { typedef uint16_t type; };
template <> struct Pack<4> { typedef uint32_t type; };

__device__ __forceinline__ uint32_t insert_byte(uint32_t word, uint32_t bits, int ch) {
  const uint32_t sel = ch == 0 ? 0x3214u : ch == 1 ? 0x3240u : ch == 2 ? 0x3410u : 0x4210u;
  return __byte_perm(word, bits, sel);
}

// 1-D B^T, factored (exact mode only: every intermediate is a multiple of 1/16 below 2^20,
// so the order of the sums does not change the bits).
__device__ __forceinline__ void bt_exact(const float (&d)[4], float (&r)[4]) {
  r[0] = __fsub_rn(d[0], d[2]);
  r[1] = __fadd_rn(d[1], d[2]);
  r[2] = __fsub_rn(d[2], d[1]);
  r[3] = __fsub_rn(d[3], d[1]);
}
__device__ __forceinline__ void bt_exact(const float (&d)[8], float (&r)[8]) {
  const float e1 = __fmaf_rn(4.25f, d[4], -__fadd_rn(d[2], d[6]));
  const float o1 = __fmaf_rn(4.25f, d[3], -__fadd_rn(d[1], d[5]));
  const float e2 = __fmaf_rn(0.25f, d[2], __fmaf_rn(-1.25f, d[4], d[6]));
  const float o2 = __fmaf_rn(0.5f, d[1], __fmaf_rn(-2.5f, d[3], __fmul_rn(2.0f, d[5])));
  const float e3 = __fmaf_rn(4.0f, d[2], __fmaf_rn(-5.0f, d[4], d[6]));
  const float o3 = __fmaf_rn(2.0f, d[1], __fmaf_rn(-2.5f, d[3], __fmul_rn(0.5f, d[5])));
  r[0] = __fmaf_rn(5.25f, __fsub_rn(d[4], d[2]), __fsub_rn(d[0], d[6]));
  r[1] = __fadd_rn(e1, o1);
  r[2] = __fsub_rn(e1, o1);
  r[3] = __fadd_rn(e2, o2);
  r[4] = __fsub_rn(e2, o2);
  r[5] = __fadd_rn(e3, o3);
  r[6] = __fsub_rn(e3, o3);
  r[7] = __fmaf_rn(5.25f, __fsub_rn(d[3], d[5]), __fsub_rn(d[7], d[1]));
}
__device__ __forceinline__ void bt_exact(const float (&d)[6], float (&r)[6]) {
  const float t1 = __fsub_rn(d[3], d[1]);
  const float t2 = __fsub_rn(d[4], d[2]);
  const float u = __fmaf_rn(4.0f, d[2], -d[4]);
  const float v = __fmaf_rn(4.0f, d[1], -d[3]);
  r[0] = __fmaf_rn(4.0f, d[0], __fmaf_rn(-5.0f, d[2], d[4]));
  r[1] = __fadd_rn(u, v);
  r[2] = __fsub_rn(u, v);
  r[3] = __fmaf_rn(2.0f, t1, t2);
  r[4] = __fmaf_rn(-2.0f, t1, t2);
  r[5] = __fmaf_rn(4.0f, d[1], __fmaf_rn(-5.0f, d[3], d[5]));
}
// The same for a pair of values, with row 1 NEGATED: packed instructions take no operand
// negation, and every other row comes out with the same operation count.  (B^T d) B of such
// passes has the sign pair_sign(i) * pair_sign(j) at (i, j), which the quantizer's multiplier
// absorbs (rounding half to even is symmetric).
template <int T_>
__device__ __forceinline__ constexpr bool pair_negated(int i) { return T_ >= 6 && i == 1; }
__device__ __forceinline__ void bt_exact(const F2 (&d)[4], F2 (&r)[4]) {
  r[0] = v_sub(d[0], d[2]);
  r[1] = v_add(d[1], d[2]);
  r[2] = v_sub(d[2], d[1]);
  r[3] = v_sub(d[3], d[1]);
}
__device__ __forceinline__ void bt_exact(const F2 (&d)[6], F2 (&r)[6]) {
  const F2 t1 = v_sub(d[3], d[1]);
  const F2 t2 = v_sub(d[4], d[2]);
  const F2 u = v_fma(-4.0f, d[2], d[4]);
  const F2 v = v_fma(-4.0f, d[1], d[3]);
  r[0] = v_fma(4.0f, d[0], v_fma(-5.0f, d[2], d[4]));
  r[1] = v_add(u, v);
  r[2] = v_sub(v, u);
  r[3] = v_fma(2.0f, t1, t2);
  r[4] = v_fma(-2.0f, t1, t2);
  r[5] = v_fma(4.0f, d[1], v_fma(-5.0f, d[3], d[5]));
}
__device__ __forceinline__ void bt_exact(const F2 (&d)[8], F2 (&r)[8]) {
  const F2 e1 = v_fma(-4.25f, d[4], v_add(d[2], d[6]));
  const F2 o1 = v_fma(-4.25f, d[3], v_add(d[1], d[5]));
  const F2 e2 = v_fma(0.25f, d[2], v_fma(-1.25f, d[4], d[6]));
  const F2 o2 = v_fma(0.5f, d[1], v_fma(-2.5f, d[3], v_add(d[5], d[5])));
  const F2 e3 = v_fma(4.0f, d[2], v_fma(-5.0f, d[4], d[6]));
  const F2 o3 = v_fma(2.0f, d[1], v_fma(-2.5f, d[3], v_mul(0.5f, d[5])));
  r[0] = v_fma(5.25f, v_sub(d[4], d[2]), v_sub(d[0], d[6]));
  r[1] = v_add(e1, o1);
  r[2] = v_sub(o1, e1);
  r[3] = v_add(e2, o2);
  r[4] = v_sub(e2, o2);
  r[5] = v_add(e3, o3);
  r[6] = v_sub(e3, o3);
  r[7] = v_fma(5.25f, v_sub(d[3], d[5]), v_sub(d[7], d[1]));
}
// 1-D A^T, factored (exact mode only: integer codes in, integers below 2^24 throughout).
template <typename V>
__device__ __forceinline__ void at_exact(const V (&m)[4], V (&y)[2]) {
  y[0] = v_add(v_add(m[0], m[1]), m[2]);
  y[1] = v_add(v_sub(m[1], m[2]), m[3]);
}
template <typename V>
__device__ __forceinline__ void at_exact(const V (&m)[6], V (&y)[4]) {
  const V a = v_add(m[1], m[2]);
  const V b = v_sub(m[1], m[2]);
  const V c = v_add(m[3], m[4]);
  const V d = v_sub(m[3], m[4]);
  y[0] = v_add(v_add(m[0], a), c);
  y[1] = v_fma(2.0f, d, b);
  y[2] = v_fma(4.0f, c, a);
  y[3] = v_add(v_fma(8.0f, d, b), m[5]);
}
// 1-D A^T of F6 for the R = m A pass (COL < 0) and for column COL of the A^T R pass.  On codes of
// magnitude at most 128 the first pass is exact: multiples of 1/32 below 128 * 67.1.  Column b of R
// consists of multiples of 2^-b below 128 r_b, and row a of A^T R of multiples of 2^-(a+b) below
// 128 r_a r_b, with r = 7, 7, 10.5, 18.25, 34.125, 67.0625 the absolute row sums of A^T; that is exact,
// whatever the order, while 128 r_a r_b 2^(a+b) <= 2^24, i.e. for all (a, b) but (4,4), (3,5), (4,5),
// (5,5) and their mirror images, whose rows are the ordered chains.
__device__ constexpr bool at6_ordered(int a, int b) { return (a >= 4 && b >= 4) || (a >= 3 && b >= 5) || (a >= 5 && b >= 3); }
template <int COL, typename V>
__device__ __forceinline__ void at6_exact(const V (&m)[8], V (&y)[6]) {
  const V s1 = v_add(m[1], m[2]), d1 = v_sub(m[1], m[2]);     // the first two links of every chain
  const V s2 = v_add(m[3], m[4]), d2 = v_sub(m[3], m[4]);
  const V s3 = v_add(m[5], m[6]), d3 = v_sub(m[5], m[6]);
  y[0] = v_add(v_add(v_add(m[0], s1), s2), s3);
  y[1] = v_fma(0.5f, d3, v_fma(2.0f, d2, d1));
  y[2] = v_fma(0.25f, s3, v_fma(4.0f, s2, s1));
  if constexpr (at6_ordered(3, COL)) y[3] = v_fma(-0.125f, m[6], v_fma(0.125f, m[5], v_fma(-8.0f, m[4], v_fma(8.0f, m[3], d1))));
  else y[3] = v_fma(0.125f, d3, v_fma(8.0f, d2, d1));
  if constexpr (at6_ordered(4, COL)) y[4] = v_fma(0.0625f, m[6], v_fma(0.0625f, m[5], v_fma(16.0f, m[4], v_fma(16.0f, m[3], s1))));
  else y[4] = v_fma(0.0625f, s3, v_fma(16.0f, s2, s1));
  if constexpr (at6_ordered(5, COL))
    y[5] = v_add(v_fma(-0.03125f, m[6], v_fma(0.03125f, m[5], v_fma(-32.0f, m[4], v_fma(32.0f, m[3], d1)))), m[7]);
  else
    y[5] = v_add(v_fma(0.03125f, d3, v_fma(32.0f, d2, d1)), m[7]);
}
__device__ __forceinline__ float v_zero(float) { return 0.0f; }
__device__ __forceinline__ F2 v_zero(F2) { return f2_both(0.0f); }
// One step of a fused-multiply-add chain; with a compile-time zero coefficient
// the step disappears (the chain's value is unchanged by it).
template <bool STD, typename V>
__device__ __forceinline__ V chain(F2 coef, V x, V acc) { return v_fma(coef, x, acc); }
template <bool STD, typename V>
__device__ __forceinline__ V chain(float coef, V x, V acc) {
  if constexpr (STD) {
    if (coef == 0.0f) return acc;
  }
  return v_fma(coef, x, acc);
}

// Entries of B^T and A^T: floats, or pairs as they lie in Params.
template <int M, int MODE>
__device__ __forceinline__ auto bt_coef(const Params& p, int i, int k) {
  if constexpr (MODE == kDensePair) {
    return F2{*reinterpret_cast<const unsigned long long*>(p.BT_pair + 2 * (i * (M + 2) + k))};
  } else {
    return Mat<M, MODE != kDense>::bt(p, i, k);
  }
}
template <int M, int MODE>
__device__ __forceinline__ auto at_coef(const Params& p, int i, int k) {
  if constexpr (MODE == kDensePair) {
    return F2{*reinterpret_cast<const unsigned long long*>(p.AT_pair + 2 * (i * (M + 2) + k))};
  } else {
    return Mat<M, MODE != kDense>::at(p, i, k);
  }
}

// V = (B^T d) B for one channel, or for a pair of channels (VT = F2; kExact: with the signs of
// pair_negated).  d is given column-wise through `col(l, out)`.
template <int M, int MODE, typename VT, typename ColFn>
__device__ __forceinline__ void input_transform_2d(const Params& p, ColFn col,
                                                   VT (&V)[(M + 2) * (M + 2)]) {
  constexpr int T_ = M + 2;
  constexpr bool STD = MODE == kSparse || MODE == kExact;
  VT P[T_][T_];
#pragma unroll
  for (int l = 0; l < T_; ++l) {
    VT dcol[T_];
    col(l, dcol);
    if constexpr (MODE == kExact) {
      VT r[T_];
      bt_exact(dcol, r);
#pragma unroll
      for (int i = 0; i < T_; ++i) P[i][l] = r[i];
    } else {
#pragma unroll
      for (int i = 0; i < T_; ++i) {
        VT acc = v_zero(VT());
#pragma unroll
        for (int k = 0; k < T_; ++k) acc = chain<STD>(bt_coef<M, MODE>(p, i, k), dcol[k], acc);
        P[i][l] = acc;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < T_; ++i) {
    if constexpr (MODE == kExact) {
      VT r[T_];
      bt_exact(P[i], r);
#pragma unroll
      for (int j = 0; j < T_; ++j) V[i * T_ + j] = r[j];
    } else {
#pragma unroll
      for (int j = 0; j < T_; ++j) {
        VT acc = v_zero(VT());
#pragma unroll
        for (int l = 0; l < T_; ++l) acc = chain<STD>(bt_coef<M, MODE>(p, j, l), P[i][l], acc);
        V[i * T_ + j] = acc;
      }
    }
  }
}

// y = A^T v, one 1-D pass of the output transform: COL < 0 the first, else column COL of the second.
template <int M, int MODE, int COL, typename VT>
__device__ __forceinline__ void at_pass(const Params& p, const VT (&v)[M + 2], VT (&y)[M]) {
  constexpr int T_ = M + 2;
  constexpr bool STD = MODE == kSparse || MODE == kExact;
  if constexpr (MODE == kExact && M == 6) {
    at6_exact<COL>(v, y);
  } else if constexpr (MODE == kExact) {
    at_exact(v, y);
  } else {
#pragma unroll
    for (int r = 0; r < M; ++r) {
      VT acc = v_zero(VT());
#pragma unroll
      for (int j = 0; j < T_; ++j) acc = chain<STD>(at_coef<M, MODE>(p, r, j), v[j], acc);
      y[r] = acc;
    }
  }
}

template <int M, int MODE, int COL, typename VT>
__device__ __forceinline__ void output_columns(const Params& p, const VT (&R)[M + 2][M], VT (&Y)[M * M]) {
  VT c[M + 2], y[M];
#pragma unroll
  for (int i = 0; i < M + 2; ++i) c[i] = R[i][COL];
  at_pass<M, MODE, COL>(p, c, y);
#pragma unroll
  for (int ip = 0; ip < M; ++ip) Y[ip * M + COL] = y[ip];
  if constexpr (COL + 1 < M) output_columns<M, MODE, COL + 1>(p, R, Y);
}
// Y = A^T (m A) for one channel or a pair of them: right factor first.  m row-wise via `row(i, out)`.
template <int M, int MODE, typename VT, typename RowFn>
__device__ __forceinline__ void output_transform_2d(const Params& p, RowFn row,
                                                    VT (&Y)[M * M]) {
  constexpr int T_ = M + 2;
  VT R[T_][M];
#pragma unroll
  for (int i = 0; i < T_; ++i) {
    VT mrow[T_];
    row(i, mrow);
    at_pass<M, MODE, -1>(p, mrow, R[i]);
  }
  output_columns<M, MODE, 0>(p, R, Y);
}

}  // namespace wino
