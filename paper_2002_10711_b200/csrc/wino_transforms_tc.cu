// Input and output transforms of the Winograd-aware layer on the tensor cores (paper: Eq. 1,
// stages 1 and 4 of Fig. 2), for the Cook-Toom matrices.
//
// B^T d B and A^T m A are linear maps of a patch, so per channel they are one matrix-vector
// product with the Kronecker matrix,
//     V[xi] = sum_ab (B^T (x) B^T)[xi][ab] d[ab],   Y[pq] = sum_xi (A^T (x) A^T)[pq][xi] m[xi],
// and on integer codes every value is an integer (F6: a multiple of 1/16) far below 2^24, so the
// int32 result of an int8 tensor-core product has the bits of the fp32 chains of the arithmetic
// contract (the A^T of F6 is not exact: its output transform stays on the ALUs).
//
// What bounds a transform of a large layer is the number of issue slots a code costs.
// Transforming on the ALUs takes 10 to 14 for F4; here the product leaves the tensor cores as
// int32 and a code costs 4.2: conversion 1, half a packed fma (two slots), the clamp on 16-bit
// lanes 1, packing 0.75 (on the input side of F2 and F4 half of it as multiply-adds, off the ALU
// pipe), its share of a 32-column tensor-memory load and of a 32-byte store.  To
// have it so, the product is laid out with (tile, position) as its rows and channels as its
// columns: a thread then holds 32 consecutive channels of one row of V_q (of one pixel of y).
//     A operand  constant, K-major: the Kronecker matrix of several tiles, block diagonal,
//                128 rows = 3 tiles x 36 positions (F4), 8 x 16 (F2), 2 x 64 (F6);
//                for y 8 tiles x 16 pixels (F4), 32 x 4 (F2).  Most of it is zero; the products
//                are a quarter to a half of the epilogue's time all the same.
//     B operand  the patches (the block of m_q) as TMA delivers them: a row of 64 or 128 channel
//                bytes per K index, swizzled, "MN-major".
// F6: 16 B^T (x) B^T has entries up to 441, split as 16 * hi + lo, two products.
//
// Persistent blocks, 704 threads on the input side and 672 on the output side: warps 0-3 load, warp 4
// issues the products, on the input side every other unit's and warp 5 the rest (a unit's waits, products
// and commits took a single warp 500 cycles, which held up the 64-channel units: 32x32, batch 256, F4 17.4 us
// with one warp, 15.6 with two, 15.3 with four, where 128-channel ones lost 0.1; the output side, of larger
// units, lost 0 to 0.3 with a second one, 0.05 to 0.1 with an idle warp), sixteen epilogue
// warps; warp w reads tensor-memory lanes 32 * (w % 4) and takes every fourth 32-column chunk.
// Stores go out directly, as 32-byte pieces of lines that other warps complete: exchanging rows
// between warps to store whole lines cost 6 to 30 % (barriers), a staging tile with TMA stores
// 0 to 16 %; the ALU pipe (60 % busy before packing left it in part: 64 channels, 32x32, F4, batch 256, 9.98 M
// warp instructions for 75.5 M codes, 53 % of the issue slots) and the latency of the few warps are what is left.
// Four load warps for the input side: a unit is two to eight boxes of short rows, and one warp
// issuing them (1200 cycles a unit) held everything else up.
#include <vector>

#include "wino_f32x2.cuh"
#include "wino_launch.h"
#include "wino_ptx.cuh"

namespace wino {

namespace {

// Warps of the two kernels: loads, products (two warps on the input side), epilogue.
constexpr int kXtLoadWarps = 4, kXtMmaWarp = 4, kXtEpiWarps = 16;
constexpr int kXiEpi0 = kXtMmaWarp + 2, kXiThreads = 32 * (kXiEpi0 + kXtEpiWarps);
constexpr int kXoEpi0 = kXtMmaWarp + 1, kXoThreads = 32 * (kXoEpi0 + kXtEpiWarps);

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// MN-major tile of CH-byte rows (one row per K index) with the CH-byte swizzle: 8-row groups of
// 8 * CH bytes along K.  N = CH elements is exactly one row.
template <int CH>
__device__ __forceinline__ uint64_t desc_mn(uint32_t smem_addr) {
  constexpr uint64_t group = CH * 8 / 16, layout = CH == 128 ? 2 : 4;
  return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | (group << 16) | (group << 32) | (1ull << 46) | (layout << 61);
}
// D int32, A and B signed 8-bit, A K-major, B MN-major (bit 16).
__host__ __device__ constexpr uint32_t idesc_i8_b_mn(int M, int N) {
  return (2u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Geometry of the two products.
template <int M> struct InGeom {
  static constexpr int T_ = M + 2, R = T_ * T_;                   // rows (positions) per tile
  static constexpr int TP = M == 2 ? 8 : M == 4 ? 3 : 2;          // tiles per unit
  static constexpr int KP = M == 4 ? 40 : R;                      // K indices per tile: whole 8-row groups
  static constexpr int NA = M == 6 ? 2 : 1;                       // products (high and low part)
};
template <int M> struct OutGeom {
  static constexpr int T2 = (M + 2) * (M + 2), PX = M * M;
  static constexpr int TP = 128 / PX;                             // 32 (F2), 8 (F4)
  static constexpr int K = T2 * TP, KB = (K + 127) / 128;         // K index = xi * TP + tile
};

// Shared memory: A operand, load slots, barriers; 1024-byte aligned.
template <int A_BYTES, int SLOT_BYTES, int SLOTS>
struct XtSmem {
  static constexpr uint32_t kBytes = A_BYTES + SLOTS * SLOT_BYTES + 256;
  uint32_t a, slot, tail, bar_a, bar_full, bar_empty, bar_acc_full, bar_acc_empty, tmem_slot, abort_slot;
  __device__ explicit XtSmem(uint32_t base) {
    a = base;
    slot = a + A_BYTES;
    bar_full = slot + SLOTS * SLOT_BYTES;
    bar_empty = bar_full + 8 * SLOTS;
    bar_acc_full = bar_empty + 8 * SLOTS;    // up to 4
    bar_acc_empty = bar_acc_full + 32;
    bar_a = bar_acc_empty + 32;
    tmem_slot = bar_a + 8;
    abort_slot = tmem_slot + 4;
    tail = base + kBytes;
  }
};

// The part that both kernels share: barriers, tensor memory.
template <typename L, int SLOTS, int NBUF>
__device__ __forceinline__ void xt_setup(const L& s, volatile uint32_t* abort_p, int warp, int columns,
                                         uint32_t acc_arrivals) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < SLOTS; ++i) {
      mbar_init(s.bar_full + 8u * i, 1);
      mbar_init(s.bar_empty + 8u * i, 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(s.bar_acc_full + 8u * b, 1);
      mbar_init(s.bar_acc_empty + 8u * b, acc_arrivals);
    }
    mbar_init(s.bar_a, 1);
    *abort_p = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kXtMmaWarp) tmem_alloc(s.tmem_slot, (uint32_t)columns);
}

// The MMA warps' loop: for each of `n_my` units one accumulator of NA products of KSTEPS steps, the
// units dealt out in turn (NM divides the numbers of slots and of accumulators, so that each of
// those always belongs to the same warp and no warp can fall a phase behind on its barrier).
template <typename L, int SLOTS, int NBUF, int NM, int NA, int KSTEPS, int CH, int A_ONE, int SLOT_BYTES>
__device__ __forceinline__ void xt_mma_loop(const L& s, int n_my, int which, uint32_t tmem_base,
                                            volatile uint32_t* abort_p) {
  static_assert(SLOTS % NM == 0 && NBUF % NM == 0, "a slot and an accumulator belong to one MMA warp");
  const bool leader = elect_one();
  const uint32_t idesc = idesc_i8_b_mn(128, CH);
  const uint64_t da = make_desc_sw128(s.a), db0 = desc_mn<CH>(s.slot);
  bool ok = __all_sync(0xffffffffu, mbar_wait<false>(s.bar_a, 0u, abort_p));
  int sl = which, b = which;
  uint32_t ph = 0, aph = 0;
  for (int i = which; i < n_my && ok; i += NM) {
    ok = __all_sync(0xffffffffu, mbar_wait<false>(s.bar_acc_empty + 8u * b, aph ^ 1u, abort_p)) &&
         __all_sync(0xffffffffu, mbar_wait<false>(s.bar_full + 8u * sl, ph, abort_p));
    if (!ok) break;
    tc_fence_after();
    const uint64_t db = db0 + (uint64_t)(sl * (SLOT_BYTES >> 4));
    if (leader) {
#pragma unroll
      for (int na = 0; na < NA; ++na)
#pragma unroll
        for (int ks = 0; ks < KSTEPS; ++ks)
          mma_i8(tmem_base + (uint32_t)((b * NA + na) * CH),
                 da + (uint64_t)(na * (A_ONE >> 4) + (ks >> 2) * 1024 + (ks & 3) * 2), db + (uint64_t)(ks * 2 * CH),
                 idesc, ks != 0 ? 1u : 0u);
      mma_commit(s.bar_empty + 8u * sl);
      mma_commit(s.bar_acc_full + 8u * b);
    }
    __syncwarp();
    if ((sl += NM) >= SLOTS) { sl = which; ph ^= 1u; }
    if ((b += NM) >= NBUF) { b = which; aph ^= 1u; }
  }
  if (!ok) *abort_p = 1u;
}

// ---------------------------------------------------------------------------
// Input transform.  x [N][H][W][C] -> V_q [t*t][T][C].  Unit = (TP tiles, CH channels), the
// channel chunk varying fastest; rows of the product: tiles fastest, as in V_q.  Z: the input has
// a zero point.  TMA fills what lies outside the image with the code 0, so the product is that of
// x itself, and z_x times the sum of the in-image matrix entries of the row's position is taken
// off it.
// ---------------------------------------------------------------------------
template <int M, int CH, bool Z>
__global__ void __launch_bounds__(kXiThreads, 1)
k_input_transform_tc(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap mapX,
                     const uint8_t* __restrict__ a_image, int8_t* __restrict__ Vq, int* __restrict__ status,
                     const uint8_t* __restrict__ l2_hint, uint32_t l2_hint_bytes) {
  using G = InGeom<M>;
  constexpr int R = G::R, TP = G::TP, NA = G::NA;
  constexpr int kSlots = CH == 128 ? 4 : 8, kSlot = 128 * CH, kA = NA * 16384;
  constexpr int kBuf = NA * CH <= 128 ? 4 : 2, kCols = kBuf * NA * CH, kColChunks = CH / 32;
  using L = XtSmem<kA, kSlot, kSlots>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const L s(base);
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  volatile uint32_t* abort_p = reinterpret_cast<volatile uint32_t*>(gen + (s.abort_slot - base));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cchunks = (p.C + CH - 1) / CH, units = ((p.T + TP - 1) / TP) * cchunks;
  const int n_my = (int)blockIdx.x < units ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  xt_setup<L, kSlots, kBuf>(s, abort_p, warp, kCols, 4 * kColChunks);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // only now may the next kernel's blocks start: every block of this grid holds its tensor memory,
  // so none of them can be kept from it by a block that waits for this grid
  griddep_launch();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(gen + (s.tmem_slot - base));

  if (warp < kXtLoadWarps) {
    if (warp == 0 && lane == 0) {
      tma_prefetch_map(&mapX);
      mbar_expect_tx(s.bar_a, (uint32_t)kA);      // a constant of the library: no dependency
      bulk_load(s.a, a_image, (uint32_t)kA, s.bar_a);
      l2_hint_slice(l2_hint, l2_hint_bytes);
    }
    // this warp's units: i = warp, warp + 4, ...; (group, chunk) advances with carries
    const int d_u = kXtLoadWarps * (int)gridDim.x;
    const int u = blockIdx.x + warp * gridDim.x;
    int group = u / cchunks, chunk = u - group * cchunks;
    const int d_group = d_u / cchunks, d_chunk = d_u - d_group * cchunks;
    griddep_wait();
    for (int i = warp; i < n_my; i += kXtLoadWarps) {
      const int tau = group * TP + lane;
      const int rest = tau / p.TW, tw = tau - rest * p.TW, n = rest / p.TH, th = rest - n * p.TH;
      const int sl = i & (kSlots - 1), c0 = chunk * CH, n_tile = min(TP, p.T - group * TP);
      if (i >= kSlots && !__all_sync(0xffffffffu, mbar_wait<false>(s.bar_empty + 8u * sl,
                                                                   ((uint32_t)(i / kSlots) & 1u) ^ 1u, abort_p))) {
        *abort_p = 1u;
        break;
      }
      if (lane == 0) mbar_expect_tx(s.bar_full + 8u * sl, (uint32_t)(n_tile * R * CH));
      __syncwarp();
      if (lane < n_tile)
        tma_load_4d(s.slot + (uint32_t)(sl * kSlot + lane * G::KP * CH), &mapX, s.bar_full + 8u * sl, c0, tw * M - 1,
                    th * M - 1, n);
      group += d_group;
      chunk += d_chunk;
      if (chunk >= cchunks) { chunk -= cchunks; ++group; }
    }
  } else if (warp < kXiEpi0) {
    xt_mma_loop<L, kSlots, kBuf, kXiEpi0 - kXtMmaWarp, NA, 4, CH, 16384, kSlot>(s, n_my, warp - kXtMmaWarp, tmem_base, abort_p);
  } else {
    const int quad = warp & 3, sub = (warp - kXiEpi0) >> 2;
    const int r = quad * 32 + lane, xi = r / TP, j = r - xi * TP;
    const int col = (kColChunks == 4 ? sub : sub & 1) * 32;
    const int first = kColChunks == 4 ? 0 : sub >> 1, step = kColChunks == 4 ? 1 : 2;
    const F2 mult = f2_both(M == 6 ? p.mult_V * 0.0625f : p.mult_V), magic = M == 6 ? f2_both(kMagic) : u16x2_magic();
    const uint32_t lo = M == 6 ? s16x2_both((int)p.lo_V) : u16x2_both((int)p.lo_V);
    const uint32_t hi = M == 6 ? s16x2_both((int)p.hi_V) : u16x2_both((int)p.hi_V);
    const bool wide = (p.C & 31) == 0 && (reinterpret_cast<uintptr_t>(Vq) & 31u) == 0;
    // this warp's units advance by a constant stride: (group, chunk) with carries
    const int d_u = step * (int)gridDim.x, u0 = (int)blockIdx.x + first * (int)gridDim.x;
    const int d_group = d_u / cchunks, d_chunk = d_u - d_group * cchunks;
    int group = u0 / cchunks, chunk = u0 - group * cchunks;
    int8_t* const row0 = Vq + (long)xi * p.T * p.C;
    griddep_wait();
    for (int i = first; i < n_my; i += step) {
      const int c = chunk * CH + col, tau = group * TP + j;
      group += d_group;
      chunk += d_chunk;
      if (chunk >= cchunks) { chunk -= cchunks; ++group; }
      int corr = 0;
      if constexpr (Z) {
        const int rest = tau / p.TW, w0 = (tau - rest * p.TW) * M - 1, n = rest / p.TH, h0 = (rest - n * p.TH) * M - 1;
        const int ri = xi / G::T_, ci = xi - ri * G::T_;
        float rs = 0.0f, cs = 0.0f;
        if (xi < R)
          for (int k = 0; k < G::T_; ++k) {
            if ((unsigned)(h0 + k) < (unsigned)p.H) rs += p.BT[ri * G::T_ + k];
            if ((unsigned)(w0 + k) < (unsigned)p.W) cs += p.BT[ci * G::T_ + k];
          }
        corr = (int)(rs * cs * (M == 6 ? 16.0f : 1.0f)) * p.z_x;
      }
      const int b = i & (kBuf - 1);
      if (!__all_sync(0xffffffffu, mbar_wait(s.bar_acc_full + 8u * b, (uint32_t)(i / kBuf) & 1u, abort_p))) {
        *abort_p = 1u;
        break;
      }
      tc_fence_after();
      const uint32_t tacc = tmem_base + (uint32_t)(b * NA * CH + col) + ((uint32_t)(quad * 32) << 16);
      uint32_t v[32];
      tmem_ld32(tacc, v);
      if constexpr (NA == 2) {
        // the low part in two halves: 64 accumulator words at once spill at the 80 registers of a thread
        uint32_t l[16];
        tmem_ld16(tacc + CH, l);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = v[e] * 16u + l[e];
        tmem_ld16(tacc + CH + 16, l);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) v[16 + e] = v[16 + e] * 16u + l[e];
      } else {
        tmem_ld_wait();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s.bar_acc_empty + 8u * b);
      if (xi >= R || tau >= p.T || c >= p.C) continue;
      if constexpr (Z) {
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] -= (uint32_t)corr;
      }
      uint32_t w[8];
      quant32_fits16<M != 6, M != 6>(v, mult, magic, lo, hi, w);   // |V| <= 100 * 256
      store_row32(row0 + (long)tau * p.C + c, w, wide, p.C - c);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_p != 0u && threadIdx.x == 0) atomicExch(status, -6);  // WINO_ERR_TIMEOUT
  if (warp == kXtMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kCols);
  }
}

// ---------------------------------------------------------------------------
// Output transform.  m_q [t*t][T][K] -> y [N][H][W][K], int8 codes or floats.  Unit = (TP
// tiles, CH channels), the tile group varying fastest.  PK: the multiplier varies per output
// channel.  The bias in output-code units (and the multipliers) of all K channels are computed
// once per block into shared memory.
// ---------------------------------------------------------------------------
template <int M, int CH, bool PK>
__global__ void __launch_bounds__(kXoThreads, 1)
k_output_transform_tc(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap mapM,
                      const uint8_t* __restrict__ a_image, const float* __restrict__ bias, void* __restrict__ y,
                      float s_Y, int* __restrict__ status, const float* __restrict__ chan) {
  using G = OutGeom<M>;
  constexpr int TP = G::TP, kSlot = G::K * CH, kA = G::KB * 16384;
  constexpr int kSlots = (M == 2 ? 2 : 4) * (CH == 128 ? 1 : 2);
  constexpr int kBuf = 4, kColChunks = CH / 32;
  using L = XtSmem<kA, kSlot, kSlots>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const L s(base);
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  volatile uint32_t* abort_p = reinterpret_cast<volatile uint32_t*>(gen + (s.abort_slot - base));
  float* b_tab = reinterpret_cast<float*>(gen + (s.tail - base));     // [K]
  float* m_tab = b_tab + p.K;                                         // [K], PK only
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int groups = (p.T + TP - 1) / TP, units = groups * ((p.K + CH - 1) / CH);
  const int n_my = (int)blockIdx.x < units ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  xt_setup<L, kSlots, kBuf>(s, abort_p, warp, kBuf * CH, 4 * kColChunks);
  for (int k = threadIdx.x; k < p.K; k += kXoThreads) {
    float b = bias != nullptr ? __ldg(bias + k) : 0.0f;
    if (p.out_dtype == 0 && bias != nullptr)
      b = (float)((double)b / (double)(PK ? __ldg(chan + (long)kChSY * p.K + k) : s_Y));
    b_tab[k] = b;
    if constexpr (PK) m_tab[k] = __ldg(chan + (long)(p.out_dtype == 0 ? kChMultY : kChSAcc) * p.K + k);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_launch();   // as in the input transform
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(gen + (s.tmem_slot - base));

  if (warp < kXtLoadWarps) {
    if (warp == 0 && lane == 0) {
      tma_prefetch_map(&mapM);
      mbar_expect_tx(s.bar_a, (uint32_t)kA);
      for (int i = 0; i < G::KB; ++i) bulk_load(s.a + i * 16384, a_image + i * 16384, 16384u, s.bar_a);
      griddep_wait();
      int sl = 0;
      uint32_t ph = 0;
      for (int i = 0; i < n_my; ++i) {
        const int u = blockIdx.x + i * gridDim.x, chunk = u / groups, group = u - chunk * groups;
        if (i >= kSlots && !mbar_wait<false>(s.bar_empty + 8u * sl, ph ^ 1u, abort_p)) {
          *abort_p = 1u;
          break;
        }
        mbar_expect_tx(s.bar_full + 8u * sl, (uint32_t)kSlot);   // the full box counts, clipped rows included
        tma_load_3d(s.slot + (uint32_t)(sl * kSlot), &mapM, s.bar_full + 8u * sl, chunk * CH, group * TP, 0);
        if (++sl == kSlots) { sl = 0; ph ^= 1u; }
      }
    }
  } else if (warp < kXoEpi0) {
    xt_mma_loop<L, kSlots, kBuf, 1, 1, G::K / 32, CH, kA, kSlot>(s, n_my, 0, tmem_base, abort_p);
  } else {
    const int quad = warp & 3, sub = (warp - kXoEpi0) >> 2;
    const int r = quad * 32 + lane, j = r / G::PX, pix = r - j * G::PX, ip = pix / M, jp = pix - ip * M;
    const int col = (kColChunks == 4 ? sub : sub & 1) * 32;
    const int first = kColChunks == 4 ? 0 : sub >> 1, step = kColChunks == 4 ? 1 : 2;
    const F2 magic = f2_both(kMagic), mult = f2_both(p.out_dtype == 0 ? p.mult_Y : p.s_acc);
    const float lo = p.lo_Y, hi = p.hi_Y;
    const bool wide = (p.K & 31) == 0 && (reinterpret_cast<uintptr_t>(y) & 31u) == 0;
    // this row's tile: advanced by the units' stride with carries, divided out only at the
    // start and where a new channel chunk begins
    int group = -1, chunk = 0, tw = 0, th = 0, n = 0;
    const int d_group = step * (int)gridDim.x, d_tau = d_group * TP;
    const int d_rest = d_tau / p.TW, d_w = d_tau - d_rest * p.TW, d_n = d_rest / p.TH, d_h = d_rest - d_n * p.TH;
    griddep_wait();
    for (int i = first; i < n_my; i += step) {
      const int u = blockIdx.x + i * gridDim.x;
      if (group >= 0 && group + d_group < groups) {
        group += d_group;
        tw += d_w; if (tw >= p.TW) { tw -= p.TW; ++th; }
        th += d_h; if (th >= p.TH) { th -= p.TH; ++n; }
        n += d_n;
      } else {
        chunk = u / groups;
        group = u - chunk * groups;
        const int tau = group * TP + j, rest = tau / p.TW;
        tw = tau - rest * p.TW;
        n = rest / p.TH;
        th = rest - n * p.TH;
      }
      const int h = th * M + ip, w = tw * M + jp, k = chunk * CH + col;
      const bool valid = group * TP + j < p.T && h < p.H && w < p.W && k < p.K;
      const int b = i & (kBuf - 1);
      if (!__all_sync(0xffffffffu, mbar_wait(s.bar_acc_full + 8u * b, (uint32_t)(i / kBuf) & 1u, abort_p))) {
        *abort_p = 1u;
        break;
      }
      tc_fence_after();
      uint32_t v[32];
      tmem_ld32(tmem_base + (uint32_t)(b * CH + col) + ((uint32_t)(quad * 32) << 16), v);
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s.bar_acc_empty + 8u * b);
      if (!valid) continue;
      const long o = (((long)n * p.H + h) * p.W + w) * p.K + k;
      const float4* bt = reinterpret_cast<const float4*>(b_tab + k);
      const float4* mt = reinterpret_cast<const float4*>(m_tab + k);
      uint32_t out[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const bool in = k + 4 * q < p.K;
        const float4 bb = in ? bt[q] : make_float4(0.f, 0.f, 0.f, 0.f);
        F2 m0 = mult, m1 = mult;
        if constexpr (PK) {
          const float4 mm = in ? mt[q] : make_float4(0.f, 0.f, 0.f, 0.f);
          m0 = f2_make(mm.x, mm.y);
          m1 = f2_make(mm.z, mm.w);
        }
        const F2 y0 = v_fma(f2_make(__int2float_rn((int)v[4 * q]), __int2float_rn((int)v[4 * q + 1])), m0,
                            f2_make(bb.x, bb.y));
        const F2 y1 = v_fma(f2_make(__int2float_rn((int)v[4 * q + 2]), __int2float_rn((int)v[4 * q + 3])), m1,
                            f2_make(bb.z, bb.w));
        uint32_t a0, a1, a2, a3;
        f2_split(y0, a0, a1);
        f2_split(y1, a2, a3);
        if (p.out_dtype == 0) {
          auto clamp = [&](uint32_t a) { return fminf(fmaxf(__uint_as_float(a), lo), hi); };
          f2_split(v_add(f2_make(clamp(a0), clamp(a1)), magic), a0, a1);
          f2_split(v_add(f2_make(clamp(a2), clamp(a3)), magic), a2, a3);
          if (p.z_Y != 0) { a0 += p.z_Y; a1 += p.z_Y; a2 += p.z_Y; a3 += p.z_Y; }
          out[q] = __byte_perm(__byte_perm(a0, a1, 0x0040u), __byte_perm(a2, a3, 0x0040u), 0x5410u);
        } else if (in) {
          *reinterpret_cast<uint4*>(reinterpret_cast<float*>(y) + o + 4 * q) = make_uint4(a0, a1, a2, a3);
        }
      }
      if (p.out_dtype == 0) store_row32(reinterpret_cast<int8_t*>(y) + o, out, wide, p.K - k);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_p != 0u && threadIdx.x == 0) atomicExch(status, -6);  // WINO_ERR_TIMEOUT
  if (warp == kXtMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kBuf * CH);
  }
}

// ---------------------------------------------------------------------------
// The constant operands, in the layout of shared memory (K-major rows of 128 bytes, 128-byte
// swizzle, 16 KB per 128 K indices), one copy per device for all plans.
// ---------------------------------------------------------------------------
constexpr int kImgIn2 = 0, kImgIn4 = 16384, kImgIn6 = 2 * 16384, kImgOut2 = 4 * 16384, kImgOut4 = 8 * 16384;
constexpr int kImgBytes = 11 * 16384;
__device__ __align__(1024) uint8_t g_xt_images[kImgBytes];

void put(uint8_t* img, int row, int k, int value) {
  img[(k >> 7) * 16384 + row * 128 + ((((k & 127) >> 4) ^ (row & 7)) << 4) + (k & 15)] = (uint8_t)(int8_t)value;
}
template <int M> void fill_in(uint8_t* img) {
  using G = InGeom<M>;
  for (int j = 0; j < G::TP; ++j)
    for (int xi = 0; xi < G::R; ++xi)
      for (int ab = 0; ab < G::R; ++ab) {
        const float v = std_bt<M>(xi / G::T_, ab / G::T_) * std_bt<M>(xi % G::T_, ab % G::T_) * (M == 6 ? 16.0f : 1.0f);
        const int e = (int)v, hi = (e + (e >= 0 ? 8 : -8)) / 16;     // |e - 16 hi| <= 8
        if (G::NA == 1) {
          put(img, xi * G::TP + j, j * G::KP + ab, e);
        } else {
          put(img, xi * G::TP + j, j * G::KP + ab, hi);
          put(img + 16384, xi * G::TP + j, j * G::KP + ab, e - 16 * hi);
        }
      }
}
template <int M> void fill_out(uint8_t* img) {
  using G = OutGeom<M>;
  constexpr int T_ = M + 2;
  for (int j = 0; j < G::TP; ++j)
    for (int pix = 0; pix < G::PX; ++pix)
      for (int xi = 0; xi < G::T2; ++xi)
        put(img, j * G::PX + pix, xi * G::TP + j, (int)(std_at<M>(pix / M, xi / T_) * std_at<M>(pix % M, xi % T_)));
}

template <int M, int CH, bool Z>
int input_go(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const uint8_t* img, int8_t* Vq, int* status,
             cudaStream_t st) {
  using G = InGeom<M>;
  constexpr size_t smem = XtSmem<G::NA * 16384, 128 * CH, CH == 128 ? 4 : 8>::kBytes + 1024;
  static DeviceOnce once;
  if (int rc = set_max_smem(once, o.device, k_input_transform_tc<M, CH, Z>, smem)) return rc;
  const long units = (long)((p.T + G::TP - 1) / G::TP) * ((p.C + CH - 1) / CH);
  const int grid = units < o.num_sms ? (int)units : o.num_sms;
  return launch_kernel(k_input_transform_tc<M, CH, Z>, dim3((unsigned)grid), dim3(kXiThreads), smem, st, o.pdl, p, mapX,
                       img, Vq, status, static_cast<const uint8_t*>(o.l2_hint), (uint32_t)o.l2_hint_bytes);
}
template <int M>
int input_pick(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const uint8_t* img, int8_t* Vq, int* status,
             cudaStream_t st) {
  const bool z = p.z_x != 0;
  if (xt_chunk(p.C) == 128)
    return z ? input_go<M, 128, true>(p, o, mapX, img, Vq, status, st)
             : input_go<M, 128, false>(p, o, mapX, img, Vq, status, st);
  return z ? input_go<M, 64, true>(p, o, mapX, img, Vq, status, st)
           : input_go<M, 64, false>(p, o, mapX, img, Vq, status, st);
}
template <int M, int CH, bool PK>
int output_go(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const uint8_t* img, const float* bias,
              void* y, float s_Y, int* status, cudaStream_t st) {
  using G = OutGeom<M>;
  const size_t smem = XtSmem<G::KB * 16384, G::K * CH, (M == 2 ? 2 : 4) * (CH == 128 ? 1 : 2)>::kBytes + 1024 +
                      (size_t)p.K * (PK ? 8 : 4);
  static DeviceOnce once;
  if (int rc = set_max_smem(once, o.device, k_output_transform_tc<M, CH, PK>, 227 * 1024)) return rc;
  const long units = (long)((p.T + G::TP - 1) / G::TP) * ((p.K + CH - 1) / CH);
  const int grid = units < o.num_sms ? (int)units : o.num_sms;
  return launch_kernel(k_output_transform_tc<M, CH, PK>, dim3((unsigned)grid), dim3(kXoThreads), smem, st, o.pdl, p,
                       mapM, img, bias, y, s_Y, status, o.chan);
}
template <int M>
int output_pick(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const uint8_t* img, const float* bias,
                void* y, float s_Y, int* status, cudaStream_t st) {
  const bool pk = o.chan != nullptr;
  if (xt_chunk(p.K) == 128)
    return pk ? output_go<M, 128, true>(p, o, mapM, img, bias, y, s_Y, status, st)
              : output_go<M, 128, false>(p, o, mapM, img, bias, y, s_Y, status, st);
  return pk ? output_go<M, 64, true>(p, o, mapM, img, bias, y, s_Y, status, st)
            : output_go<M, 64, false>(p, o, mapM, img, bias, y, s_Y, status, st);
}

}  // namespace

int xt_images(int device, const uint8_t** out) {
  static DeviceOnce once;
  static uint8_t* addr[DeviceOnce::kMaxDevices];
  if (device < 0 || device >= DeviceOnce::kMaxDevices) return -5;
  const int rc = once.run(device, [&]() -> int {
    std::vector<uint8_t> img(kImgBytes, 0);
    fill_in<2>(img.data() + kImgIn2);
    fill_in<4>(img.data() + kImgIn4);
    fill_in<6>(img.data() + kImgIn6);
    fill_out<2>(img.data() + kImgOut2);
    fill_out<4>(img.data() + kImgOut4);
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_xt_images) != cudaSuccess ||
        cudaMemcpy(ptr, img.data(), kImgBytes, cudaMemcpyHostToDevice) != cudaSuccess) {
      cudaGetLastError();
      return -5;
    }
    addr[device] = static_cast<uint8_t*>(ptr);
    return 0;
  });
  *out = rc == 0 ? addr[device] : nullptr;
  return rc;
}

bool input_tc_supported(const Params& p, bool std_mats) { return std_mats && p.C % 16 == 0 && p.v_fits_16; }
bool output_tc_supported(const Params& p, bool std_mats) {
  return std_mats && p.m != 6 && p.K % 16 == 0 && p.K <= 2048 && p.qM_enabled;
}
void input_tc_box(const Params& p, uint32_t box[4]) {
  box[0] = (uint32_t)xt_chunk(p.C); box[1] = box[2] = (uint32_t)p.t; box[3] = 1;
}
void output_tc_box(const Params& p, uint32_t box[3]) {
  box[0] = (uint32_t)xt_chunk(p.K);
  box[1] = (uint32_t)(p.m == 2 ? OutGeom<2>::TP : OutGeom<4>::TP);
  box[2] = (uint32_t)(p.t * p.t);
}
int launch_input_transform_tc(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const uint8_t* images,
                              int8_t* Vq, int* status, cudaStream_t st) {
  return p.m == 2 ? input_pick<2>(p, o, mapX, images + kImgIn2, Vq, status, st)
       : p.m == 4 ? input_pick<4>(p, o, mapX, images + kImgIn4, Vq, status, st)
                  : input_pick<6>(p, o, mapX, images + kImgIn6, Vq, status, st);
}
int launch_output_transform_tc(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const uint8_t* images,
                               const float* bias, void* y, float s_Y, int* status, cudaStream_t st) {
  return p.m == 2 ? output_pick<2>(p, o, mapM, images + kImgOut2, bias, y, s_Y, status, st)
                  : output_pick<4>(p, o, mapM, images + kImgOut4, bias, y, s_Y, status, st);
}

}  // namespace wino
