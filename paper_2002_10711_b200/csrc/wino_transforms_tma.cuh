// TMA-staged variants of the input and output transform kernels (paper: Eq. 1,
// Fig. 2, stages 1 and 4).  A block owns G consecutive tiles x CC channels:
//   - the (m+2)x(m+2)xCC input patches (or the t*t x G x CC block of m_q) arrive
//     in shared memory by TMA; for the input, coordinates may start at -1 and
//     run past the image: the hardware fills those bytes with zero, which is
//     the padding (with an input zero point every thread then writes the code
//     of the real value zero over its own channels' bytes there);
//   - every thread transforms two channels of one tile in packed fp32 (or one channel,
//     which has twice the warps: see the launchers), reading and writing shared memory at
//     compile-time offsets;
//   - the result leaves by one TMA store (rows past the last tile, or pixels past
//     the image edge, are clipped by the hardware).
// What bounds them at ordinary sizes: the latency of load, arithmetic and store of the one or
// two waves a layer is, then issue slots.  One channel per thread spends a shared-memory
// wavefront on every 32 codes read or written and two clamp instructions on every code.
#pragma once
#include "wino_ptx.cuh"
#include "wino_spread.h"
#include "wino_trace.cuh"
#include "wino_transform_math.cuh"

namespace wino {

__device__ __forceinline__ uint32_t lds_u16(uint32_t addr) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
  return (uint32_t)v;
}
__device__ __forceinline__ void sts_u16(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ int lds_s8(uint32_t addr) {
  int v;
  asm volatile("ld.shared.s8 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u8(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Two signed bytes as floats: the low byte at weight 1 in a float of exponent 2^23, the high
// byte in one of exponent 2^15, both with the sign bit flipped: one lop3 each, one packed add.
// unbias: minus the two offsets, minus the zero point.
__device__ __forceinline__ F2 codes_unbias(int z) { return f2_make(-(8388736.0f + (float)z), -(32896.0f + (float)z)); }
__device__ __forceinline__ F2 codes_to_f2(uint32_t h, F2 unbias) {
  return v_add(f2_bits((h & 0xFFu) ^ 0x4B000080u, (h & 0xFF00u) ^ 0x47008000u), unbias);
}

#ifdef WINO_TRACE
static __device__ TraceTable g_in_trace, g_out_trace;
#endif
#if WINO_M == 4
WINO_ST_READER(wino_trace_input, g_in_trace)
WINO_ST_READER(wino_trace_output, g_out_trace)
#endif

// Dense F6 (kDensePair), while its threads all are resident at once: entries of the matrices read
// as pairs spare the two moves that make one of a float, at the price of the registers that hold
// them (255 and 168).  46 images of 22x22, 64 to 128 channels: 6.1 -> 5.2 us in, 6.2 -> 5.4 us out.
// From the second wave on more warps hide more than the moves cost (9.1 us with floats, 9.7 with
// pairs, on 128 such images), so the limits are the threads per SM of one wave.
constexpr int kPairInThreads = 256, kPairOutThreads = 384;
// Blocks of `threads` threads (whole warps) that make up so many.
constexpr int pair_blocks(int limit, int threads) { return limit / ((threads + 31) / 32 * 32); }

// Plans whose rounded products of Q_V fit 16 bits (the clamp is done on two codes at a time).
// MINB: blocks per SM asked of the compiler.  CPT: channels per thread (1: input zero point 0 only).
template <int M, int MODE, int CC, int G, int MINB, int CPT>
__global__ void __launch_bounds__((CC / CPT) * G, MINB)
k_input_transform_tma(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap mapX,
                      const __grid_constant__ CUtensorMap mapV, int* __restrict__ status,
                      const uint8_t* __restrict__ l2_hint, uint32_t l2_hint_bytes) {
  constexpr int T_ = M + 2, T2 = T_ * T_, TPT = CC / CPT;
  constexpr uint32_t kTileBytes = T2 * CC;
  constexpr uint32_t kTileStride = (kTileBytes + 127u) & ~127u;   // TMA destinations stay 128-byte aligned
  constexpr uint32_t kUnitBytes = G * kTileStride;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 127u) & ~127u;
  const uint32_t s_in = base;                 // [G][T2][CC]
  const uint32_t s_out = base + kUnitBytes;   // [T2][G][CC]
  const uint32_t bar = s_out + kUnitBytes;
  __shared__ uint32_t abort_flag;

  // unit = (tile group, channel chunk)
  const int cchunks = p.C / CC;
  const int group = (int)blockIdx.x / cchunks, c0 = ((int)blockIdx.x - group * cchunks) * CC;
  const int tau0 = group * G, ntile = min(G, p.T - tau0);
  const int g = threadIdx.x / TPT, c = (int)threadIdx.x % TPT * CPT;   // tile, first channel

  int trace_step = 0;
  (void)trace_step;
  if (threadIdx.x == 0) {
    WINO_ST_BEGIN(g_in_trace, trace_step);
    WINO_ST(g_in_trace, trace_step, 0);
  }
  griddep_launch();
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_flag = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_map(&mapX);
    tma_prefetch_map(&mapV);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    // the lanes of warp 0 load a tile each; patch coordinates first: nothing but the loads
    // themselves is left for after the wait
    const int lane = threadIdx.x, tau = tau0 + lane, rest = tau / p.TW;
    const int cw = (tau - rest * p.TW) * M - 1, cn = rest / p.TH, ch = (rest - cn * p.TH) * M - 1;
    // ask for the patches to be brought into L2 while the preceding kernel is still running
    // (a hint only: nothing is read into the SM before the wait below)
    if (lane < ntile) tma_prefetch_l2_4d(&mapX, c0, cw, ch, cn);
    if (lane == 0) l2_hint_slice(l2_hint, l2_hint_bytes);   // what the next kernel will want from HBM
    griddep_wait();   // only this warp reads or writes buffers that other kernels touch
    if (lane == 0) {
      WINO_ST(g_in_trace, trace_step, 1);
      mbar_expect_tx(bar, (uint32_t)ntile * kTileBytes);
    }
    __syncwarp();
    if (lane < ntile) tma_load_4d(s_in + (uint32_t)lane * kTileStride, &mapX, bar, c0, cw, ch, cn);
    // one thread polls (bounded); the others sleep in the barrier below
    if (lane == 0) {
      if (!mbar_wait(bar, 0u, &abort_flag)) {
        abort_flag = 1u;
        atomicExch(status, -6);  // WINO_ERR_TIMEOUT
      }
      WINO_ST(g_in_trace, trace_step, 2);
    }
  }
  __syncthreads();
  if (*(volatile uint32_t*)&abort_flag != 0u) return;
  (void)mbar_try_wait(bar, 0u);   // every thread observes the completed phase itself
  if (g < ntile) {
    const uint32_t rd = s_in + (uint32_t)g * kTileStride + (uint32_t)c;
    const uint32_t wr = s_out + (uint32_t)(g * CC + c);
    if constexpr (CPT == 1) {
      float V[T2];
      input_transform_2d<M, MODE>(p, [&](int l, float (&dcol)[T_]) {
#pragma unroll
        for (int a = 0; a < T_; ++a) dcol[a] = small_int_to_float(lds_s8(rd + (uint32_t)((a * T_ + l) * CC)));
      }, V);
#pragma unroll
      for (int xi = 0; xi < T2; ++xi)
        sts_u8(wr + (uint32_t)(xi * G * CC), __float_as_uint(quant_magic(V[xi], p.mult_V, p.lo_V, p.hi_V)));
    } else {
      if (p.z_x != 0) {
        const int tau = tau0 + g, rest = tau / p.TW, w0 = (tau - rest * p.TW) * M - 1, h0 = rest % p.TH * M - 1;
        const uint32_t pad = ((uint32_t)p.z_x & 0xFFu) * 0x0101u;
#pragma unroll 1
        for (int ab = 0; ab < T2; ++ab)
          if ((unsigned)(h0 + ab / T_) >= (unsigned)p.H || (unsigned)(w0 + ab % T_) >= (unsigned)p.W)
            sts_u16(rd + (uint32_t)(ab * CC), pad);
      }
      const F2 mult = f2_both(p.mult_V), mult_n = f2_both(-p.mult_V), magic = f2_both(kMagic);
      const uint32_t lo = s16x2_both((int)p.lo_V), hi = s16x2_both((int)p.hi_V);
      const F2 unbias = codes_unbias(p.z_x);
      F2 V[T2];
      input_transform_2d<M, MODE>(p, [&](int l, F2 (&dcol)[T_]) {
#pragma unroll
        for (int a = 0; a < T_; ++a) dcol[a] = codes_to_f2(lds_u16(rd + (uint32_t)((a * T_ + l) * CC)), unbias);
      }, V);
#pragma unroll
      for (int xi = 0; xi < T2; ++xi) {
        const bool neg = MODE == kExact && (pair_negated<T_>(xi / T_) != pair_negated<T_>(xi % T_));
        sts_u16(wr + (uint32_t)(xi * G * CC),
                __byte_perm(quant_s16x2(V[xi], neg ? mult_n : mult, magic, lo, hi), 0u, 0x0020u));
      }
    }
  }
  fence_async_smem();
  __syncthreads();
  if (threadIdx.x == 0) {
    WINO_ST(g_in_trace, trace_step, 3);
    tma_store_3d(&mapV, s_out, c0, tau0, 0);
    bulk_commit();
    bulk_wait_all();    // the bytes are in place before the block leaves
    WINO_ST(g_in_trace, trace_step, 4);
  }
}

// chan: null, or the scales vary per output channel (rows kChMultY and kChSY, or kChSAcc).  Float
// output goes to y directly, a pair of channels per store.
// MINB: blocks per SM asked of the compiler.  CPT: channels per thread (1: integer output only).
template <int M, int MODE, int KC, int G, int MINB, int CPT>
__global__ void __launch_bounds__((KC / CPT) * G, MINB)
k_output_transform_tma(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap mapM,
                       const __grid_constant__ CUtensorMap mapY, const float* __restrict__ bias,
                       float s_Y, int* __restrict__ status, const float* __restrict__ chan,
                       float* __restrict__ y_float) {
  constexpr int T_ = M + 2, T2 = T_ * T_, TPT = KC / CPT;
  constexpr uint32_t kInBytes = T2 * G * KC;          // [T2][G][KC]
  constexpr uint32_t kTileOutBytes = M * M * KC;      // [M][M][KC] per tile
  constexpr uint32_t kTileOut = (kTileOutBytes + 127u) & ~127u;   // stride: TMA sources 128-byte aligned
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 127u) & ~127u;
  const uint32_t s_in = base;
  const uint32_t s_out = base + ((kInBytes + 127u) & ~127u);   // [G][M][M][KC]
  const uint32_t bar = s_out + G * kTileOut;
  __shared__ uint32_t abort_flag;

  const int kchunks = p.K / KC;
  const int group = (int)blockIdx.x / kchunks, chunk = (int)blockIdx.x - group * kchunks;
  const int tau0 = group * G, k0 = chunk * KC;
  const int g = threadIdx.x / TPT, kc = (int)threadIdx.x % TPT * CPT;   // tile, first channel
  const int ntile = min(G, p.T - tau0);

  int trace_step = 0;
  (void)trace_step;
  if (threadIdx.x == 0) {
    WINO_ST_BEGIN(g_out_trace, trace_step);
    WINO_ST(g_out_trace, trace_step, 0);
  }
  griddep_launch();
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_flag = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    tma_prefetch_map(&mapM);
    griddep_wait();
    WINO_ST(g_out_trace, trace_step, 1);
    mbar_expect_tx(bar, kInBytes);   // the full box counts, clipped rows included
    tma_load_3d(s_in, &mapM, bar, k0, tau0, 0);
  }
  // F4, F6: every warp waits here, before the arithmetic below: done earlier, it takes issue slots
  // from the preceding kernel, beside which these blocks already sit (256 channels, 8x8, F4, batch
  // 256, us: alone 4.84, in the layer 15.95 like that, 4.72 and 15.84 like this; learnt matrices 6.00
  // and 19.88, 5.26 and 18.80).  F2, whose kernel is shorter, the other way round (128 channels,
  // 16x16, batch 64: 4.81 and 15.29 like this, 4.48 and 15.09 like that).
  if (M != 2) griddep_wait();
  // while the block's m_q is in flight: the pixel coordinates of the block's stores (lane of warp
  // 0 = tile) and this thread's bias in output-code units (a double-precision division, some
  // forty instructions), which would otherwise follow the load
  int sw = 0, sh = 0, sn = 0;
  if (threadIdx.x < 32) {
    const int tau = tau0 + (int)threadIdx.x, rest = tau / p.TW;
    sw = (tau - rest * p.TW) * M;
    sn = rest / p.TH;
    sh = (rest - sn * p.TH) * M;
  }
  F2 mult, b_pre;                              // CPT == 2
  float mult_1 = p.mult_Y, b_1 = 0.0f;         // CPT == 1
  const int k = k0 + kc;
  if constexpr (CPT == 1) {
    if (chan != nullptr) {
      mult_1 = __ldg(chan + (long)kChMultY * p.K + k);
      s_Y = __ldg(chan + (long)kChSY * p.K + k);
    }
    if (bias != nullptr) b_1 = (float)((double)__ldg(bias + k) / (double)s_Y);
  } else {
    mult = f2_both(y_float != nullptr ? p.s_acc : p.mult_Y);
    b_pre = f2_both(0.0f);
    float s0 = s_Y, s1 = s_Y;
    if (chan != nullptr) {
      const float* row = chan + (long)(y_float != nullptr ? kChSAcc : kChMultY) * p.K + k;
      mult = f2_make(__ldg(row), __ldg(row + 1));
      s0 = __ldg(chan + (long)kChSY * p.K + k);
      s1 = __ldg(chan + (long)kChSY * p.K + k + 1);
    }
    if (bias != nullptr) {
      b_pre = f2_make(__ldg(bias + k), __ldg(bias + k + 1));
      if (y_float == nullptr)
        b_pre = f2_make((float)((double)__ldg(bias + k) / (double)s0), (float)((double)__ldg(bias + k + 1) / (double)s1));
    }
  }
  if (M == 2) griddep_wait();
  if (threadIdx.x == 0) {
    if (!mbar_wait(bar, 0u, &abort_flag)) {
      abort_flag = 1u;
      atomicExch(status, -6);  // WINO_ERR_TIMEOUT
    }
    WINO_ST(g_out_trace, trace_step, 2);
  }
  __syncthreads();
  if (*(volatile uint32_t*)&abort_flag != 0u) return;
  (void)mbar_try_wait(bar, 0u);
  if (g < ntile) {
    const uint32_t rd = s_in + (uint32_t)(g * KC + kc);
    const uint32_t wr = s_out + (uint32_t)g * kTileOut + (uint32_t)kc;
    if constexpr (CPT == 1) {
      float Y[M * M];
      output_transform_2d<M, MODE>(p, [&](int i, float (&mrow)[T_]) {
#pragma unroll
        for (int j = 0; j < T_; ++j) mrow[j] = small_int_to_float(lds_s8(rd + (uint32_t)((i * T_ + j) * G * KC)));
      }, Y);
#pragma unroll
      for (int q = 0; q < M * M; ++q) {
        const float r = __fadd_rn(fminf(fmaxf(__fmaf_rn(Y[q], mult_1, b_1), p.lo_Y), p.hi_Y), kMagic);
        sts_u8(wr + (uint32_t)(q * KC), (uint32_t)(magic_to_int(r) + p.z_Y));
      }
    } else {
      const F2 unbias = codes_unbias(0);
      F2 Y[M * M];
      output_transform_2d<M, MODE>(p, [&](int i, F2 (&mrow)[T_]) {
#pragma unroll
        for (int j = 0; j < T_; ++j) mrow[j] = codes_to_f2(lds_u16(rd + (uint32_t)((i * T_ + j) * G * KC)), unbias);
      }, Y);
      if (y_float != nullptr) {
        const int tau = tau0 + g, rest = tau / p.TW, w0 = (tau - rest * p.TW) * M, n = rest / p.TH;
        const int h0 = (rest - n * p.TH) * M;
        float* yp = y_float + (((long)n * p.H + h0) * p.W + w0) * p.K + k;
#pragma unroll
        for (int q = 0; q < M * M; ++q) {
          const int ip = q / M, jp = q % M;
          uint32_t a, b;
          f2_split(v_fma(Y[q], mult, b_pre), a, b);
          if (h0 + ip < p.H && w0 + jp < p.W)
            *reinterpret_cast<uint2*>(yp + (long)(ip * p.W + jp) * p.K) = make_uint2(a, b);
        }
        return;
      }
      const F2 magic = f2_both(kMagic);
      const uint32_t z = s16x2_both(p.z_Y);
#pragma unroll
      for (int q = 0; q < M * M; ++q) {
        uint32_t a, b;
        f2_split(v_fma(Y[q], mult, b_pre), a, b);
        const F2 r = v_add(f2_make(fminf(fmaxf(__uint_as_float(a), p.lo_Y), p.hi_Y),
                                   fminf(fmaxf(__uint_as_float(b), p.lo_Y), p.hi_Y)), magic);
        uint32_t w = f2_low_halves(r);
        if (z != 0u) w = __vadd2(w, z);
        sts_u16(wr + (uint32_t)(q * KC), __byte_perm(w, 0u, 0x0020u));
      }
    }
  }
  if (y_float != nullptr) return;
  fence_async_smem();
  __syncthreads();
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0) WINO_ST(g_out_trace, trace_step, 3);
    if ((int)threadIdx.x < ntile) {
      tma_store_4d(&mapY, s_out + threadIdx.x * kTileOut, k0, sw, sh, sn);
      bulk_commit();
      bulk_wait_all();
    }
    if (threadIdx.x == 0) WINO_ST(g_out_trace, trace_step, 4);
  }
}

// ---------------------------------------------------------------------------
// Launchers.  CC (or KC) is the channel chunk, tma_chunk; narrower chunks take more tiles a block.
// ---------------------------------------------------------------------------
namespace {

// Blocks of a kernel that an SM holds, asked once per kernel and device.
class Resident {
 public:
  template <typename Kern>
  int blocks(int device, Kern kernel, int threads, size_t smem) {
    std::lock_guard<std::mutex> lock(mu_);
    int& n = n_[device >= 0 && device < DeviceOnce::kMaxDevices ? device : DeviceOnce::kMaxDevices];
    if (n == 0 || &n == n_ + DeviceOnce::kMaxDevices) {
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 1;
      }
    }
    return n;
  }
 private:
  std::mutex mu_;
  int n_[DeviceOnce::kMaxDevices + 1] = {};
};

// Launches the input transform; with one_wave only if its blocks are all resident at once, else it
// returns 1.
template <int M, int MODE, int CC, int MINB, int CPT>
int input_tma_go(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const CUtensorMap& mapV, int* status,
                 cudaStream_t st, bool one_wave = false) {
  constexpr int G = tma_in_group(M, CC);
  constexpr size_t smem = 2 * (size_t)G * ((((M + 2) * (M + 2) * CC) + 127) / 128 * 128) + 128 + 16;
  auto kernel = k_input_transform_tma<M, MODE, CC, G, MINB, CPT>;
  static DeviceOnce once;   // one per instantiation
  if (int rc = set_max_smem(once, o.device, kernel, spread_smem(smem, 2))) return rc;
  const long units = (long)((p.T + G - 1) / G) * (p.C / CC);
  const long sums = p.qM_enabled ? 0 : (long)p.t * p.t * p.T * p.K;
  const size_t ask = spread_smem(smem, in_blocks_per_sm(units, p.K, sums, o.num_sms));
  if (one_wave) {
    static Resident resident;
    if (units > (long)o.num_sms * resident.blocks(o.device, kernel, (CC / CPT) * G, smem)) return 1;
  }
  return launch_kernel(kernel, dim3((unsigned)units), dim3((CC / CPT) * G), ask, st, o.pdl, p, mapX, mapV, status,
                       static_cast<const uint8_t*>(o.l2_hint), (uint32_t)o.l2_hint_bytes);
}
// Which build.  A grid whose blocks are all resident at once is bound by the latency of one block,
// then by how many warps share its work; a second, mostly empty wave costs a quarter of the kernel.
// F4 and F6, Cook-Toom matrices, no zero point (whose padding only the other build patches):
//   - one channel per thread (twice the warps; 40 registers in F4, 72 in F6, 56 and 96 with several
//     tiles a block) while that grid is one wave, and for chunks of 112, 96, 80 and 48 channels,
//     which in pairs do not fill whole warps, always;
//   - else two channels per thread at 72 registers (F4, some spilling) where that makes one wave;
//   - else, F4 in 128-channel chunks, one channel per thread at 32 registers likewise;
//   - else two channels per thread at 80 registers (F2 48; F6 is slower within any limit).
// Measured on B200, us, two channels / this choice: F4  128 ch 16x16 batch 64 4.38 / 4.25, 256 ch
// 16x16 batch 72 6.62 / 5.90, 64 ch 32x32 batch 32 4.54 / 4.03, 192 ch 16x16 batch 64 6.04 / 4.48;
// F6  512 ch 4x4 batch 256 6.38 / 5.19, 160 ch 14x14 batch 64 6.66 / 5.36, 64 ch 12x12 batch 256
// 4.79 / 4.37, 192 ch 14x14 batch 64 6.66 / 5.23 (256 ch 16x16 batch 32 the other way, 4.54 / 4.89).
template <int M, int MODE, int CC>
int input_tma_launch(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const CUtensorMap& mapV,
                     int* status, cudaStream_t st) {
  constexpr int G = tma_in_group(M, CC);
  if constexpr (M != 2 && MODE == kExact) {
    constexpr bool kWholeWarps = CC * G % 64 == 0;
    if (p.z_x == 0) {
      const int rc = input_tma_go<M, MODE, CC, 1, 1>(p, o, mapX, mapV, status, st, kWholeWarps);
      if (rc <= 0) return rc;
    }
    if constexpr (M == 4 && kWholeWarps) {
      int rc = input_tma_go<M, MODE, CC, 14, 2>(p, o, mapX, mapV, status, st, true);
      if (rc <= 0) return rc;
      if constexpr (CC == 128) {
        if (p.z_x == 0) rc = input_tma_go<M, MODE, CC, 16, 1>(p, o, mapX, mapV, status, st, true);
        if (rc <= 0) return rc;
      }
    }
  }
  if constexpr (M == 6 && MODE == kDense) {
    constexpr int kPair = pair_blocks(kPairInThreads, (CC / 2) * G);
    if ((long)((p.T + G - 1) / G) * (p.C / CC) <= (long)kPair * o.num_sms)
      return input_tma_go<M, kDensePair, CC, kPair, 2>(p, o, mapX, mapV, status, st);
  }
  constexpr int kMin = MODE != kExact ? 1 : M == 2 ? 10 : M == 4 ? (CC * G <= 128 ? 12 : 6) : 1;
  return input_tma_go<M, MODE, CC, kMin, 2>(p, o, mapX, mapV, status, st);
}
template <int M, int MODE>
int input_tma_mode(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const CUtensorMap& mapV,
                   int* status, cudaStream_t st) {
  const int cc = tma_chunk(p.C);
  return cc == 128 ? input_tma_launch<M, MODE, 128>(p, o, mapX, mapV, status, st)
       : cc == 112 ? input_tma_launch<M, MODE, 112>(p, o, mapX, mapV, status, st)
       : cc == 96 ? input_tma_launch<M, MODE, 96>(p, o, mapX, mapV, status, st)
       : cc == 80 ? input_tma_launch<M, MODE, 80>(p, o, mapX, mapV, status, st)
       : cc == 48 ? input_tma_launch<M, MODE, 48>(p, o, mapX, mapV, status, st)
       : cc == 64 ? input_tma_launch<M, MODE, 64>(p, o, mapX, mapV, status, st)
       : cc == 32 ? input_tma_launch<M, MODE, 32>(p, o, mapX, mapV, status, st)
                  : input_tma_launch<M, MODE, 16>(p, o, mapX, mapV, status, st);
}

// As input_tma_go.
template <int M, int MODE, int KC, int MINB, int CPT>
int output_tma_go(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const CUtensorMap& mapY,
                  const float* bias, float s_Y, int* status, float* y_float, cudaStream_t st, bool one_wave = false) {
  constexpr int G = CPT == 1 ? 1 : tma_group(KC);
  constexpr size_t smem = (G * (M + 2) * (M + 2) * KC + 127) / 128 * 128 + (size_t)G * ((M * M * KC + 127) / 128 * 128) + 128 + 16;
  static DeviceOnce once;   // one per instantiation
  auto kernel = k_output_transform_tma<M, MODE, KC, G, MINB, CPT>;
  if (int rc = set_max_smem(once, o.device, kernel, spread_smem(smem, 2))) return rc;
  const long units = (long)((p.T + G - 1) / G) * (p.K / KC);
  const size_t ask = spread_smem(smem, out_blocks_per_sm(units, o.gemm_items, p.C, o.num_sms));
  if (one_wave) {
    static Resident resident;
    if (units > (long)o.num_sms * resident.blocks(o.device, kernel, (KC / CPT) * G, smem)) return 1;
  }
  return launch_kernel(kernel, dim3((unsigned)units), dim3((KC / CPT) * G), ask, st, o.pdl, p, mapM, mapY, bias, s_Y,
                       status, o.chan, y_float);
}
// Which build: one channel per thread by tma_out_group.  F4 in pairs at 64 registers (eight blocks per
// SM; seven at the compiler's own 72 cost 0.9 us on a layer of 1200 blocks).  F6 without a limit (161
// registers) while its blocks are all resident at once, from the second wave on at 128: 512 ch 4x4
// batch 100 3.4 us without a limit, 4.6 with; 128 ch 12x12 batch 250 5.9 and 5.4.
template <int M, int MODE, int KC>
int output_tma_launch(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const CUtensorMap& mapY,
                      const float* bias, float s_Y, int* status, float* y_float, cudaStream_t st) {
  if constexpr (MODE == kExact && ((M == 4 && KC == 128) || (M == 6 && KC % 64 == 0))) {
    if (tma_out_group(p, o.std_mats, o.chan != nullptr, o.num_sms) == 1)
      return output_tma_go<M, MODE, KC, M == 4 ? 16 : 1024 / KC, 1>(p, o, mapM, mapY, bias, s_Y, status, nullptr, st);
  }
  if constexpr (M == 6 && MODE == kDense) {
    constexpr int G = tma_group(KC), kPair = pair_blocks(kPairOutThreads, (KC / 2) * G);
    if ((long)((p.T + G - 1) / G) * (p.K / KC) <= (long)kPair * o.num_sms)
      return output_tma_go<M, kDensePair, KC, kPair, 2>(p, o, mapM, mapY, bias, s_Y, status, y_float, st);
  }
  if constexpr (M == 6 && MODE == kExact) {
    const int rc = output_tma_go<M, MODE, KC, 1, 2>(p, o, mapM, mapY, bias, s_Y, status, y_float, st, true);
    if (rc <= 0) return rc;
  }
  constexpr int kMin = M == 6 ? pair_blocks(512, (KC / 2) * tma_group(KC)) : M == 4 && MODE == kExact ? 8 : 1;
  return output_tma_go<M, MODE, KC, kMin, 2>(p, o, mapM, mapY, bias, s_Y, status, y_float, st);
}
template <int M, int MODE>
int output_tma_mode(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const CUtensorMap& mapY,
                    const float* bias, float s_Y, int* status, float* y_float, cudaStream_t st) {
  const int kc = tma_chunk(p.K);
  return kc == 128 ? output_tma_launch<M, MODE, 128>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 112 ? output_tma_launch<M, MODE, 112>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 96 ? output_tma_launch<M, MODE, 96>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 80 ? output_tma_launch<M, MODE, 80>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 64 ? output_tma_launch<M, MODE, 64>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 48 ? output_tma_launch<M, MODE, 48>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
       : kc == 32 ? output_tma_launch<M, MODE, 32>(p, o, mapM, mapY, bias, s_Y, status, y_float, st)
                  : output_tma_launch<M, MODE, 16>(p, o, mapM, mapY, bias, s_Y, status, y_float, st);
}

}  // namespace

int WINO_CAT(launch_input_transform_tma_m, WINO_M)(const Params& p, const LaunchOpt& o,
                                                    const CUtensorMap& mapX,
                                                    const CUtensorMap& mapV, int* status,
                                                    cudaStream_t st) {
  if (!o.std_mats) return input_tma_mode<WINO_M, kDense>(p, o, mapX, mapV, status, st);
  return input_tma_mode<WINO_M, kExact>(p, o, mapX, mapV, status, st);
}
int WINO_CAT(launch_output_transform_tma_m, WINO_M)(const Params& p, const LaunchOpt& o,
                                                     const CUtensorMap& mapM,
                                                     const CUtensorMap& mapY, const float* bias,
                                                     float s_Y, int* status, float* y_float, cudaStream_t st) {
  if (!o.std_mats) return output_tma_mode<WINO_M, kDense>(p, o, mapM, mapY, bias, s_Y, status, y_float, st);
  return output_tma_mode<WINO_M, kExact>(p, o, mapM, mapY, bias, s_Y, status, y_float, st);
}

}  // namespace wino
