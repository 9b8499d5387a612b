// Two fp32 values in one 64-bit register pair, for the packed fp32 instructions of sm_100
// (add / fma on f32x2), and the quantizer on such pairs.
//
// Why: the transforms and quantizers are bound by instruction issue and by the ALU pipe.
// Measured on B200, issue cycles per warp instruction and scheduler: packed fma / add 2.05
// (two results), scalar fma / add 1.25, integer add 1.3 (either pipe); prmt, lop3, min, max,
// the 16x2 integer min / max, int-to-float and the saturating pack 2.05 each, all on the ALU
// pipe, which the packed fp32 instructions leave free (a packed fma and a prmt together: 2.3 to
// 2.5).  So the arithmetic goes in pairs on the fp32 pipe, and the quantizer's clamp, which in
// fp32 costs two ALU instructions a code, is done on two 16-bit codes per instruction.
#pragma once
#include "wino_common.cuh"

namespace wino {

struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2_make(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F2 f2_bits(uint32_t lo, uint32_t hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ F2 f2_both(float a) { return f2_make(a, a); }
__device__ __forceinline__ void f2_split(F2 a, uint32_t& lo, uint32_t& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(a.v));
}

// The operations of the transforms, for one value and for a pair.
__device__ __forceinline__ float v_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float v_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float v_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float v_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ F2 v_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 v_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 v_fma(float a, F2 b, F2 c) { return v_fma(f2_both(a), b, c); }
__device__ __forceinline__ F2 v_sub(F2 a, F2 b) {   // a - b, rounded once
  return v_fma(f2_both(-1.0f), b, a);
}
__device__ __forceinline__ F2 v_mul(float a, F2 b) {
  F2 r;
  const F2 aa = f2_both(a);
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(aa.v), "l"(b.v));
  return r;
}

// Codes of the quantizer in 16-bit lanes.  r holds kMagic + n for two rounded products n; the
// caller has made sure that |n| < 2^15, so the low halves are the n in two's complement.
__device__ __forceinline__ uint32_t f2_low_halves(F2 r) {
  uint32_t lo, hi;
  f2_split(r, lo, hi);
  return __byte_perm(lo, hi, 0x5410u);
}
__device__ __forceinline__ uint32_t clamp_s16x2(uint32_t a, uint32_t lo, uint32_t hi) {
  uint32_t t, r;
  asm("max.s16x2 %0, %1, %2;" : "=r"(t) : "r"(a), "r"(lo));
  asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(t), "r"(hi));
  return r;
}
__device__ __forceinline__ uint32_t s16x2_both(int v) { return ((uint32_t)v & 0xFFFFu) * 0x00010001u; }

// round_half_even(v * mult) of a pair, clamped, as 16-bit lanes (|v * mult| < 2^15).
__device__ __forceinline__ uint32_t quant_s16x2(F2 v, F2 mult, F2 magic, uint32_t lo, uint32_t hi) {
  return clamp_s16x2(f2_low_halves(v_fma(v, mult, magic)), lo, hi);
}

// The same for the accumulators of a product, where the ALU pipe has nothing else to do and is the
// limit: the 16-bit lanes are n + 2^15, unsigned, and a multiply-add on the fp32 pipe joins them
// instead of a prmt.  With the sums
//   r0 = kMagic + 2^15 + n0:  bits 0x4B400000 + (n0 + 2^15),
//   r1 = kMagic + (2^15 - 0x4B40) + n1 (both offsets are even, so ties round as without them)
// the word 2^16 r1 + r0 has n0 + 2^15 below and (r1 mod 2^16) + 0x4B40 = n1 + 2^15 above, without carries
// for |n| < 2^15.  The clamped lanes' low bytes are the codes.  Sixteen warps, 32 columns each from tensor
// memory, beside 64-column products: 777 cycles a round with prmt and signed lanes, 675 so.
__device__ __forceinline__ F2 u16x2_magic() { return f2_make(kMagic + 32768.0f, kMagic + (32768.0f - 19264.0f)); }
__device__ __forceinline__ uint32_t u16x2_both(int v) { return (uint32_t)(v + 32768) * 0x00010001u; }
__device__ __forceinline__ uint32_t quant_u16x2(F2 v, F2 mult, F2 magic, uint32_t lo, uint32_t hi) {
  uint32_t r0, r1, t, r;
  f2_split(v_fma(v, mult, magic), r0, r1);
  asm("mad.lo.u32 %0, %1, 65536, %2;" : "=r"(t) : "r"(r1), "r"(r0));
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(t), "r"(lo));
  asm("min.u16x2 %0, %1, %2;" : "=r"(t) : "r"(r), "r"(hi));
  return t;
}
// Two int32 values as floats; SMALL (|value| <= 2^22): by adding kMagic's bits and taking kMagic off
// again, which is no conversion on the ALU pipe but more instructions.  Half a quantizer's values
// that way: 652 cycles in the measurement above; all of them 770.
template <bool SMALL>
__device__ __forceinline__ F2 f2_from_ints(uint32_t a, uint32_t b) {
  if constexpr (SMALL) return v_add(f2_bits(a + kMagicBits, b + kMagicBits), f2_both(-kMagic));
  else return f2_make(__int2float_rn((int)a), __int2float_rn((int)b));
}
// 32 int32 values of one row -> 32 codes in eight words (|value * mult| < 2^15; |value| < 2^24, SMALL:
// <= 2^22).  U16: unsigned lanes, with magic, lo, hi from u16x2_magic and u16x2_both; else signed ones
// (f2_both(kMagic), s16x2_both), which are the faster where something else loads the fp32 pipe (F6
// input transform, whose two products are joined by a multiply-add a value: 14.5 us against 14.7).
template <bool U16, bool SMALL>
__device__ __forceinline__ void quant32_fits16(const uint32_t (&v)[32], F2 mult, F2 magic, uint32_t lo, uint32_t hi,
                                               uint32_t (&w)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const F2 v0 = f2_from_ints<SMALL>(v[4 * q], v[4 * q + 1]), v1 = f2_from_ints<false>(v[4 * q + 2], v[4 * q + 3]);
    if constexpr (U16)
      w[q] = __byte_perm(quant_u16x2(v0, mult, magic, lo, hi), quant_u16x2(v1, mult, magic, lo, hi), 0x6420u);
    else
      w[q] = __byte_perm(quant_s16x2(v0, mult, magic, lo, hi), quant_s16x2(v1, mult, magic, lo, hi), 0x6420u);
  }
}
// 32 bytes of a row, of which `left` (a positive multiple of 16) exist; wide: 32-byte aligned.
__device__ __forceinline__ void store_row32(int8_t* dst, const uint32_t (&w)[8], bool wide, int left) {
  if (wide) {   // the whole sector in one request
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
  } else {
    uint4* d = reinterpret_cast<uint4*>(dst);
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    if (left > 16) d[1] = make_uint4(w[4], w[5], w[6], w[7]);
  }
}

}  // namespace wino
