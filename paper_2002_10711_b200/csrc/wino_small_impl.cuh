// The whole layer in one launch for layers of few tiles (paper: Eq. 1 with the quantizers of
// Fig. 2), any tile size, matrices and options: small batches, where the staged path's three
// launches and its two exchanges through global memory are most of the time.
//
// A block owns 8 consecutive tiles (one per warp) x 16*KB output channels and all t*t
// positions, so that V_q and the Hadamard sums never leave the SM.  Channels come in chunks of
// 64, every shared-memory row being the 64 bytes of one chunk:
//   1. the patches (one box per warp and chunk) and the block's slice of U_q arrive by TMA;
//   2. B^T d B and Q_V, two channels per thread in packed fp32, into shared memory as codes
//      (blocks of other output channels repeat this step, which limits the kernel to few tiles);
//   3. t*t products [16 k x channels] x [channels x 8 tiles] with int8 warp MMAs (m16n8k32: a
//      tile count of 8 fits the problem; a tcgen05 tile would be nearly all padding);
//   4. Q_M and the right factor of A^T m A, one (tile, k, row) per thread; then the left factor,
//      bias and Q_Y, one (tile, k, column) per thread.
// Wide layers split the chunks over the S blocks of a cluster; step 4 then adds the blocks'
// partial sums over distributed shared memory, each block finishing 8/S of the tiles.
//
// What bounds it: latency, i.e. the length of the instruction stream of each step times the few
// warps that share it.  Hence TMA for the operands (issuing 36 predicated loads per channel pair
// took 2700 cycles of a first version, the U_q slice by cp.async 2000) and step 4 in two short
// passes over all warps (one long pass per (tile, k) pair on half of them: 3600 cycles).
#pragma once
#include "wino_launch.h"
#include "wino_ptx.cuh"
#include "wino_transform_math.cuh"
#include "wino_warp_mma.cuh"

#define WINO_CAT_(a, b) a##b
#define WINO_CAT(a, b) WINO_CAT_(a, b)

namespace wino {
namespace {

// Eight warps, one per tile; two blocks per SM.  (Sixteen warps a block measured no faster: the
// input transform cannot use them below 128 channels, and it is the longest step.)
constexpr int kSmThreads = 256;
constexpr int kSmWarps = kSmThreads / 32;

__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ int lds_cluster(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// IMODE / OMODE: modes of the input and output transform (wino_transform_math.cuh).
// Operands by tensor copies (a.tma) or by small asynchronous copies.
template <int M, int IMODE, int OMODE, int KB>
__global__ void __launch_bounds__(kSmThreads, M == 6 ? 1 : 2)
k_layer_small(const __grid_constant__ Params p, const __grid_constant__ SmallGeom a,
              const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapU,
              const int8_t* __restrict__ x, const int8_t* __restrict__ Uq, const float* __restrict__ bias,
              void* __restrict__ y, float s_Y, const float* __restrict__ chan, int* __restrict__ status) {
  constexpr int T_ = M + 2, T2 = T_ * T_, KS = 16 * KB;
  constexpr int kTasks = (T2 * KB + kSmWarps - 1) / kSmWarps;   // (xi, 16 k) products per warp
  constexpr int kRowM = KS + 4;   // words between two tiles: the stores of a fragment hit 32 banks
  constexpr uint32_t kPatch = T2 * 64, kUChunk = T2 * KS * 64, kVChunk = T2 * 8 * 64;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 127u) & ~127u;
  const uint32_t s_u = base;                                   // [chunk][T2][KS][64]
  const uint32_t s_v = s_u + (uint32_t)a.chunks * kUChunk;     // [chunk][T2][8][64]
  const uint32_t s_x = s_v + (uint32_t)a.chunks * kVChunk;     // [chunk][8][T2][64]
  const uint32_t s_m = base;                                   // after the products: [T2][8][kRowM] sums,
  const uint32_t s_r = s_m + 4u * T2 * 8 * kRowM;              // [T_][M][8][kRowM] values of m A
  __shared__ __align__(8) unsigned long long bars[kSmWarps + 1];
  __shared__ uint32_t abort_flag;
  __shared__ long tile_at[8];      // output offset of the tile's first pixel (channel 0), -1: no such tile
  __shared__ int tile_left[8][2];  // image rows and columns from there on
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t bar_x = smem_u32(bars) + 8u * (uint32_t)warp, bar_u = smem_u32(bars) + 8u * kSmWarps;
  const uint32_t rank = a.S > 1 ? blockIdx.x % (unsigned)a.S : 0u;
  const int blk = a.S > 1 ? blockIdx.x / (unsigned)a.S : blockIdx.x;
  const int group = blk / a.n_kblk, k0 = (blk - group * a.n_kblk) * KS;
  const int c0 = (int)rank * a.chunks * 64;
  const int nq = min(a.chunks, (p.C - c0 + 63) / 64);          // chunks of this block (0 or less: none)
  const bool tma = a.tma != 0;

  // this warp's tile
  const int tau_w = group * 8 + warp;
  const int rest_w = tau_w / p.TW, tw_w = tau_w - rest_w * p.TW;
  const int n_w = rest_w / p.TH, th_w = rest_w - n_w * p.TH;
  const int w0 = tw_w * M - 1, h0 = th_w * M - 1;
  const bool on = tau_w < p.T && nq > 0;

  griddep_launch();
  if (tid == 0) abort_flag = 0u;
  if (lane == 0) {
    mbar_init(bar_x, 1);
    if (warp == 7) mbar_init(bar_u, 1);
    tile_at[warp] = tau_w < p.T ? (((long)n_w * p.H + th_w * M) * p.W + tw_w * M) * p.K : -1l;
    tile_left[warp][0] = p.H - th_w * M;
    tile_left[warp][1] = p.W - tw_w * M;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (tma) {
      tma_prefetch_map(&mapX);
      tma_prefetch_map(&mapU);
    }
  }
  __syncthreads();   // barriers and the abort flag are set up
  if (tma && warp == 7 && lane == 0)   // weights that are not in L2 come in while the preceding kernel runs
    for (int q = 0; q < nq; ++q) tma_prefetch_l2_3d(&mapU, c0 + 64 * q, k0, 0);
  griddep_wait();

  // 1. operands
  if (tma) {
    if (lane == 0) {
      if (on) {
        mbar_expect_tx(bar_x, (uint32_t)nq * kPatch);
        for (int q = 0; q < nq; ++q)
          tma_load_4d(s_x + (uint32_t)(q * 8 + warp) * kPatch, &mapX, bar_x, c0 + 64 * q, w0, h0, n_w);
      }
      if (warp == 7 && nq > 0) {
        mbar_expect_tx(bar_u, (uint32_t)nq * kUChunk);
        for (int q = 0; q < nq; ++q)
          tma_load_3d(s_u + (uint32_t)q * kUChunk, &mapU, bar_u, c0 + 64 * q, k0, 0);
      }
    }
    __syncwarp();
  } else {
    // the same rows by asynchronous copies of 16, 8 or 4 bytes, zeros where TMA would have filled
    // them in; a thread keeps its column and walks down the rows
    const int lg = (p.C & 15) == 0 ? 2 : (p.C & 7) == 0 ? 3 : 4, cols = 1 << lg, per = 64 >> lg;
    const int at = (tid & (cols - 1)) * per;
    for (int q = 0; q < nq; ++q) {
      const int c = c0 + q * 64 + at;
      for (int row = tid >> lg; row < T2 * KS; row += kSmThreads >> lg) {
        const int xi = row / KS, k = k0 + (row & (KS - 1));
        const bool in = c < p.C && k < p.K;
        cp_async_zfill(s_u + (uint32_t)q * kUChunk + (uint32_t)(row * 64 + at),
                       Uq + (in ? ((long)xi * p.K + k) * p.C + c : 0), per, in);
      }
      if (on)
        for (int pix = lane >> lg; pix < T2; pix += 32 >> lg) {
          const int h = h0 + pix / T_, wv = w0 + pix % T_;
          const bool in = c < p.C && (unsigned)h < (unsigned)p.H && (unsigned)wv < (unsigned)p.W;
          cp_async_zfill(s_x + (uint32_t)(q * 8 + warp) * kPatch + (uint32_t)(pix * 64 + at),
                         x + (in ? (((long)n_w * p.H + h) * p.W + wv) * p.C + c : 0), per, in);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }

  // what step 4 needs per output channel, while the operands are on their way: a thread keeps
  // the same channel throughout
  const int kk = tid & (KS - 1), k = k0 + kk;
  const bool k_on = k < p.K;
  const float b_real = bias != nullptr && k_on ? __ldg(bias + k) : 0.0f;
  const float mult_M = k_on ? chan_or(chan, p.K, kChMultM, k, p.mult_M) : 0.0f;
  const float mult_Y = k_on ? chan_or(chan, p.K, kChMultY, k, p.mult_Y) : 0.0f;
  const float s_acc = k_on ? chan_or(chan, p.K, kChSAcc, k, p.s_acc) : 0.0f;
  float b_scaled = 0.0f;
  if (p.out_dtype == 0 && bias != nullptr && k_on)
    b_scaled = (float)((double)b_real / (double)chan_or(chan, p.K, kChSY, k, s_Y));

  // 2. input transform, one chunk of one tile per warp and round (channel pair per lane).  With
  // fewer than eight tiles the other warps take further chunks
  const int n_tile = min(8, p.T - group * 8);
  if (nq > 0) {
    const F2 unbias = f2_make(-(8388736.0f + (float)p.z_x), -(32896.0f + (float)p.z_x));
    const F2 mult = f2_both(p.mult_V), mult_n = f2_both(-p.mult_V), magic = f2_both(kMagic);
    const uint32_t lo = s16x2_both((int)p.lo_V), hi = s16x2_both((int)p.hi_V);
#pragma unroll 1
    for (int task = warp; task < n_tile * nq; task += kSmWarps) {
      const int q = task / n_tile, tile = task - q * n_tile;
      if (tma && !mbar_wait<false>(smem_u32(bars) + 8u * (uint32_t)tile, 0u, &abort_flag)) {
        *(volatile uint32_t*)&abort_flag = 1u;
        if (lane == 0) atomicExch(status, -6);  // WINO_ERR_TIMEOUT
      }
      if (p.z_x != 0) {
        // padding is the real value zero, i.e. the code z_x
        const uint32_t pad = ((uint32_t)p.z_x & 0xFFu) * 0x01010101u;
        const int th0 = p.H - tile_left[tile][0] - 1, tw0 = p.W - tile_left[tile][1] - 1;
        for (int i = lane; i < T2 * 16; i += 32) {
          const int pix = i >> 4, h = th0 + pix / T_, wv = tw0 + pix % T_;
          if ((unsigned)h >= (unsigned)p.H || (unsigned)wv >= (unsigned)p.W)
            sts32(s_x + (uint32_t)(q * 8 + tile) * kPatch + (uint32_t)(pix * 64 + 4 * (i & 15)), pad);
        }
        __syncwarp();
      }
      const uint32_t src = s_x + (uint32_t)(q * 8 + tile) * kPatch + 2u * (uint32_t)lane;
      const uint32_t dst = s_v + (uint32_t)q * kVChunk + 64u * (uint32_t)tile + 2u * (uint32_t)lane;
      F2 V[T2];
      input_transform_2d<M, IMODE>(p, [&](int l, F2 (&dcol)[T_]) {
#pragma unroll
        for (int r = 0; r < T_; ++r) {
          uint16_t h;
          asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(src + 64u * (uint32_t)(r * T_ + l)));
          // low byte at weight 1 in a float of exponent 2^23, high byte in one of exponent 2^15,
          // both with the sign bit flipped: one lop3 each
          dcol[r] = v_add(f2_bits(((uint32_t)h & 0xFFu) ^ 0x4B000080u, ((uint32_t)h & 0xFF00u) ^ 0x47008000u), unbias);
        }
      }, V);
#pragma unroll
      for (int i = 0; i < T_; ++i)
#pragma unroll
        for (int j = 0; j < T_; ++j) {
          const bool neg = IMODE == kExact && (pair_negated<T_>(i) != pair_negated<T_>(j));
          const uint32_t c = quant_s16x2(V[i * T_ + j], neg ? mult_n : mult, magic, lo, hi);
          asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + 512u * (uint32_t)(i * T_ + j)),
                       "h"((uint16_t)__byte_perm(c, 0u, 0x0020u)) : "memory");
        }
    }
  }
  if (tma && nq > 0 && !mbar_wait<false>(bar_u, 0u, &abort_flag)) {
    *(volatile uint32_t*)&abort_flag = 1u;
    if (lane == 0) atomicExch(status, -6);
  }
  __syncthreads();

  // 3. products.  Fragments are read 16 bytes at a time: both operands' channels are permuted
  // alike inside a chunk, which leaves the sums as they are
  const int g = lane >> 2, t = lane & 3;
  int acc[kTasks][4];
#pragma unroll
  for (int j = 0; j < kTasks; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0;
#pragma unroll 1
  for (int q = 0; q < nq; ++q) {
    const uint32_t fu = s_u + (uint32_t)q * kUChunk + (uint32_t)((warp * 16 + g) * 64 + t * 16);
    const uint32_t fv = s_v + (uint32_t)q * kVChunk + (uint32_t)(g * 64 + t * 16);
#pragma unroll
    for (int j = 0; j < kTasks; ++j) {
      const int task = warp + kSmWarps * j;   // xi * KB + k block
      if (kSmWarps * (j + 1) <= T2 * KB || task < T2 * KB) {
        const uint32_t at = fu + (uint32_t)(j * kSmWarps * 1024);
        const uint4 a0 = lds128(at), a1 = lds128(at + 512u);
        const uint4 b = lds128(fv + (uint32_t)((task / KB) * 512));
        mma_s8(acc[j], a0.x, a1.x, a0.y, a1.y, b.x, b.y);
        mma_s8(acc[j], a0.z, a1.z, a0.w, a1.w, b.z, b.w);
      }
    }
  }
  __syncthreads();   // the sums take the operands' place
#pragma unroll
  for (int j = 0; j < kTasks; ++j) {
    const int task = warp + kSmWarps * j;
    if (kSmWarps * (j + 1) <= T2 * KB || task < T2 * KB) {
      const uint32_t d = s_m + 4u * (uint32_t)(((task / KB) * 8 + 2 * t) * kRowM + (task & (KB - 1)) * 16 + g);
      sts32(d, (uint32_t)acc[j][0]);
      sts32(d + 4u * kRowM, (uint32_t)acc[j][1]);
      sts32(d + 32u, (uint32_t)acc[j][2]);
      sts32(d + 4u * kRowM + 32u, (uint32_t)acc[j][3]);
    }
  }
  if (a.S > 1) cluster_sync();
  else __syncthreads();

  // 4. Q_M and m A, one row of one (tile, k) per thread and round; consecutive lanes take
  // consecutive channels
  const int tile0 = (int)rank * (8 / a.S);
  const int lg_pairs = 31 - __clz(8 * KS / a.S);     // S is a power of two
  const float lo_m = __fadd_rn(p.lo_M, kMagic), hi_m = __fadd_rn(p.hi_M, kMagic);
  const int qM = p.qM_enabled;
#pragma unroll 2
  for (int i = tid; i < (T_ << lg_pairs); i += kSmThreads) {
    const int row = i >> lg_pairs, tile = tile0 + (i - (row << lg_pairs)) / KS;
    const uint32_t src = s_m + 4u * (uint32_t)((row * T_ * 8 + tile) * kRowM + kk);
    int v[T_];
    if (a.S == 1) {
#pragma unroll
      for (int j = 0; j < T_; ++j) v[j] = (int)lds32(src + 4u * (uint32_t)(j * 8 * kRowM));
    } else {
#pragma unroll
      for (int j = 0; j < T_; ++j) v[j] = 0;
      for (int r = 0; r < a.S; ++r) {
        const uint32_t peer = cluster_addr(src, (uint32_t)r);
#pragma unroll
        for (int j = 0; j < T_; ++j) v[j] += lds_cluster(peer + 4u * (uint32_t)(j * 8 * kRowM));
      }
    }
    float m[T_], R[M];
#pragma unroll
    for (int j = 0; j < T_; ++j) {
      m[j] = __int2float_rn(v[j]);
      const float q = magic_to_float(fminf(fmaxf(__fmaf_rn(m[j], mult_M, kMagic), lo_m), hi_m));
      m[j] = qM ? q : m[j];
    }
    at_pass<M, OMODE, -1>(p, m, R);
#pragma unroll
    for (int jp = 0; jp < M; ++jp)
      sts32(s_r + 4u * (uint32_t)(((row * M + jp) * 8 + tile) * kRowM + kk), __float_as_uint(R[jp]));
  }
  __syncthreads();
#pragma unroll 2
  for (int i = tid; i < (M << lg_pairs); i += kSmThreads) {
    const int jp = i >> lg_pairs, tile = tile0 + (i - (jp << lg_pairs)) / KS;
    float c[T_], Y[M];
#pragma unroll
    for (int r = 0; r < T_; ++r)
      c[r] = __uint_as_float(lds32(s_r + 4u * (uint32_t)(((r * M + jp) * 8 + tile) * kRowM + kk)));
    at_pass<M, OMODE, M - 1>(p, c, Y);   // the last column's form of F6 holds for every column
    const long first = tile_at[tile];
    const int rows = tile_left[tile][0];
    if (first < 0 || !k_on || jp >= tile_left[tile][1]) continue;
    const long at = first + (long)(jp * p.K + k), step = (long)p.W * p.K;
    if (p.out_dtype == 0) {
      int8_t* yp = reinterpret_cast<int8_t*>(y) + at;
#pragma unroll
      for (int ip = 0; ip < M; ++ip) {
        const float yf = __fmaf_rn(Y[ip], mult_Y, b_scaled);
        const float r = __fadd_rn(fminf(fmaxf(yf, p.lo_Y), p.hi_Y), kMagic);
        if (ip < rows) yp[ip * step] = (int8_t)(magic_to_int(r) + p.z_Y);
      }
    } else {
      float* yp = reinterpret_cast<float*>(y) + at;
#pragma unroll
      for (int ip = 0; ip < M; ++ip)
        if (ip < rows) yp[ip * step] = __fmaf_rn(Y[ip], s_acc, b_real);
    }
  }
  if (a.S > 1) cluster_sync();   // the peers may still be reading this block's sums
}

template <int M, int IMODE, int OMODE, int KB>
int small_launch(const Params& p, const LaunchOpt& o, const SmallGeom& g, const SmallArgs& s, cudaStream_t st) {
  static DeviceOnce once;
  auto kernel = k_layer_small<M, IMODE, OMODE, KB>;
  if (int rc = set_max_smem(once, o.device, kernel, 226 * 1024)) return rc;
  return launch_kernel_cluster(kernel, dim3((unsigned)g.grid), dim3(kSmThreads), (unsigned)g.S, g.smem, st, o.pdl,
                               p, g, *s.mapX, *s.mapU, s.x, s.Uq, s.bias, s.y, s.s_Y, o.chan, s.status);
}
template <int M, int IMODE, int OMODE>
int small_kb(const Params& p, const LaunchOpt& o, const SmallGeom& g, const SmallArgs& s, cudaStream_t st) {
  if constexpr (M == 2)
    if (g.KB == 4) return small_launch<M, IMODE, OMODE, 4>(p, o, g, s, st);
  return g.KB == 2 ? small_launch<M, IMODE, OMODE, 2>(p, o, g, s, st) : small_launch<M, IMODE, OMODE, 1>(p, o, g, s, st);
}

}  // namespace

int WINO_CAT(launch_small_m, WINO_M)(const Params& p, const LaunchOpt& o, const SmallGeom& g, const SmallArgs& s,
                                     cudaStream_t st) {
  if (!o.std_mats) return small_kb<WINO_M, kDense, kDense>(p, o, g, s, st);
  // A^T is exact on codes, on un-quantized sums nowhere
  if (p.qM_enabled) return small_kb<WINO_M, kExact, kExact>(p, o, g, s, st);
  return small_kb<WINO_M, kExact, kSparse>(p, o, g, s, st);
}

}  // namespace wino
