// Direct int8 3x3 convolution (cross-correlation, zero padding 1, stride 1 or 2)
// with int32 accumulation: the lossless candidate the paper compares the
// Winograd-aware layers with (Sections 4 and 5.3), and the layer type of the
// network's strided convolutions, for which no Winograd form exists (Section 5.1).
// Channel counts the implicit GEMM does not take: integer dot products on the ALUs, thread =
// (output pixel, 4 or 8 output channels); at most 4 input channels: warp-level MMAs.
#include "wino_launch.h"
#include "wino_narrow_rows.cuh"
#include "wino_warp_mma.cuh"

namespace wino {

struct DirectParams {
  int N, C, H, W, K, stride, Ho, Wo;
  int z_x, z_w, z_Y;
  float mult, s_in, s_Y, lo_Y, hi_Y;
  int out_dtype;
  // per-output-channel scales (device arrays of K floats, nullable) and the per-layer scales
  const float* s_w_K;
  const float* s_Y_K;
  float s_x, s_w;
};

// Channel k's output arithmetic: the multiplier on the accumulator (s_x * s_w[k] / s_Y[k] for
// integer output, s_x * s_w[k] for float output; the product of the two scales is exact in
// double) and the output scale the bias is divided by.
__device__ __forceinline__ void channel_scales(const DirectParams& p, int k, float& mult, float& s_in,
                                               float& s_Y) {
  mult = p.mult; s_in = p.s_in; s_Y = p.s_Y;
  if (p.s_w_K != nullptr || p.s_Y_K != nullptr) {
    const double s_in_k = (double)p.s_x * (double)(p.s_w_K != nullptr ? __ldg(p.s_w_K + k) : p.s_w);
    if (p.s_Y_K != nullptr) s_Y = __ldg(p.s_Y_K + k);
    mult = (float)(s_in_k / (double)s_Y);
    s_in = (float)s_in_k;
  }
}

// KPT output channels per thread.  Consecutive lanes take consecutive output
// pixels, so a weight word is one broadcast load for the warp and every lane
// walks the contiguous channels of its own input pixel.
template <int KPT>
__global__ void __launch_bounds__(128)
k_direct_conv(const DirectParams p, const int8_t* __restrict__ x, const int8_t* __restrict__ w,
              const float* __restrict__ bias, void* __restrict__ y) {
  const int KG = p.K / KPT, C4 = p.C >> 2;
  const long npix = (long)p.N * p.Ho * p.Wo;
  const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  griddep_launch();
  griddep_wait();
  if (idx >= npix * KG) return;
  const int kg = (int)(idx / npix);          // slow index: a warp shares its output channels
  long pix = idx - (long)kg * npix;
  const int wo = (int)(pix % p.Wo); pix /= p.Wo;
  const int ho = (int)(pix % p.Ho);
  const int n = (int)(pix / p.Ho);
  const int* x32 = reinterpret_cast<const int*>(x);
  const int* w32 = reinterpret_cast<const int*>(w);
  int acc[KPT];
#pragma unroll
  for (int j = 0; j < KPT; ++j) acc[j] = 0;
  const bool plain = p.z_x == 0 && p.z_w == 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int h = ho * p.stride - 1 + a;
    if (h < 0 || h >= p.H) continue;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int wv = wo * p.stride - 1 + b;
      if (wv < 0 || wv >= p.W) continue;          // padding is the real value zero
      const int* xp = x32 + (((long)n * p.H + h) * p.W + wv) * C4;
      const int* wp = w32 + (((long)(kg * KPT) * 3 + a) * 3 + b) * C4;
      for (int c4 = 0; c4 < C4; ++c4) {
        const int xv = __ldg(xp + c4);
#pragma unroll
        for (int j = 0; j < KPT; ++j) {
          const int wv4 = __ldg(wp + (long)j * 9 * C4 + c4);
          if (plain) {
            acc[j] = __dp4a(xv, wv4, acc[j]);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              acc[j] += ((int)(int8_t)(xv >> (8 * q)) - p.z_x) * ((int)(int8_t)(wv4 >> (8 * q)) - p.z_w);
          }
        }
      }
    }
  }
  const long o = (((long)n * p.Ho + ho) * p.Wo + wo) * p.K + kg * KPT;
#pragma unroll
  for (int j4 = 0; j4 < KPT; j4 += 4) {
    if (p.out_dtype == 0) {
      uint32_t word = 0u;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = kg * KPT + j4 + j;
        float mult, s_in, s_Y;
        channel_scales(p, k, mult, s_in, s_Y);
        const float b = bias != nullptr ? (float)((double)__ldg(bias + k) / (double)s_Y) : 0.0f;
        const float yf = __fmaf_rn(__int2float_rn(acc[j4 + j]), mult, b);
        const float r = __fadd_rn(fminf(fmaxf(yf, p.lo_Y), p.hi_Y), kMagic);
        word |= ((uint32_t)(magic_to_int(r) + p.z_Y) & 0xFFu) << (8 * j);
      }
      *reinterpret_cast<uint32_t*>(reinterpret_cast<int8_t*>(y) + o + j4) = word;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float b = bias != nullptr ? __ldg(bias + kg * KPT + j4 + j) : 0.0f;
        float mult, s_in, s_Y;
        channel_scales(p, kg * KPT + j4 + j, mult, s_in, s_Y);
        reinterpret_cast<float*>(y)[o + j4 + j] = __fmaf_rn(__int2float_rn(acc[j4 + j]), s_in, b);
      }
    }
  }
}

// At most four input channels (a network's first layer, Section 5.1): the 9 * C codes under a
// pixel's window fit one or two K steps of an int8 warp MMA (m16n8k32), so the layer is an
// implicit GEMM whose A operand is gathered.  A warp takes 32 pixels: every lane gathers the
// window of one (aligned words, funnel shifts) and leaves it in shared memory, from where it
// comes back as A fragments; the 64 filters of the block are kept as B fragments in registers.
// The K order is free as long as windows and filters agree: a row's 3 * C bytes are padded to
// words (C = 3: the ninth bytes of the three rows share one).  Which filter is which column is free
// too: lane t of a quad takes channels 16 t .. 16 t + 15, so that it stores 16 bytes and a quad 64.
// With zero points, sum (x - z_x)(w - z_w) = sum x w - z_w sum x - z_x sum w + 9 C z_x z_w over the
// whole window, pixels outside the image holding the code z_x.
// Bound by the quantizer's issue slots and the launch.  64 images 32x32, 3 -> 64 channels: 114 us
// byte by byte, 10.0 with dot products and one pixel per thread, 5.1 like this.
constexpr int kNarrowK = 64, kNarrowThreads = 128;

// Three rows in K order: 8 words (one K step), or 16 (C = 4: two).
template <int C>
__device__ __forceinline__ void narrow_k(const uint32_t (&r)[3][3], uint32_t (&k)[C == 4 ? 16 : 8]) {
#pragma unroll
  for (int i = 0; i < (C == 4 ? 16 : 8); ++i) k[i] = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (C == 1) {
      k[a] = r[a][0];
    } else if (C == 4) {
      k[3 * a] = r[a][0]; k[3 * a + 1] = r[a][1]; k[3 * a + 2] = r[a][2];
    } else {
      k[2 * a] = r[a][0]; k[2 * a + 1] = r[a][1];
      if (C == 3) k[6] |= (r[a][2] & 0xFFu) << (8 * a);
    }
  }
}
// TAIL: x or w ends within a word.
template <int C, bool Z, bool TAIL>
__global__ void __launch_bounds__(kNarrowThreads)
k_direct_conv_narrow(const DirectParams p, const int8_t* __restrict__ x, const int8_t* __restrict__ w,
                     const float* __restrict__ bias, void* __restrict__ y, int wide) {
  constexpr int KW = C == 4 ? 16 : 8, STEPS = KW / 8;      // words of K, MMA K steps
  __shared__ __align__(16) uint32_t s_f[kNarrowK * KW];    // filters in K order
  __shared__ __align__(16) uint32_t s_a[kNarrowThreads * KW];
  __shared__ __align__(8) float s_mult[kNarrowK], s_b[kNarrowK];
  __shared__ int s_corr[kNarrowK];
  const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int k0 = blockIdx.y * kNarrowK;
  griddep_launch();
  if (tid < kNarrowK) {   // parameters of the layer: no dependency on the preceding kernel
    const int k = min(k0 + tid, p.K - 1);
    float mult, s_in, s_Y;
    channel_scales(p, k, mult, s_in, s_Y);
    const float b = bias != nullptr ? __ldg(bias + k) : 0.0f;
    s_mult[tid] = p.out_dtype == 0 ? mult : s_in;
    s_b[tid] = p.out_dtype == 0 && bias != nullptr ? (float)((double)b / (double)s_Y) : b;
  }
  griddep_wait();
  if (tid < kNarrowK) {
    uint32_t r[3][3], kw[KW];
    const int k = k0 + tid;
    narrow_filter<C, TAIL>(w, p.K, k, r);
    narrow_k<C>(r, kw);
    int sum = 0;
#pragma unroll
    for (int i = 0; i < KW; ++i) {
      s_f[tid * KW + i] = kw[i];
      sum = __dp4a((int)kw[i], 0x01010101, sum);
    }
    s_corr[tid] = -p.z_x * sum + 9 * C * p.z_x * p.z_w;
  }
  __syncthreads();
  // B fragments: column n = g of product j is channel 16 (g / 2) + 2 j + (g & 1)
  uint32_t bf[8][STEPS][2];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < STEPS; ++q) {
      const uint2 v = *reinterpret_cast<const uint2*>(s_f + (16 * (g >> 1) + 2 * j + (g & 1)) * KW + 8 * q + 2 * t);
      bf[j][q][0] = v.x;
      bf[j][q][1] = v.y;
    }
  const long npix = (long)p.N * p.Ho * p.Wo;
  const uint32_t fill = ((uint32_t)p.z_x & 0xFFu) * 0x01010101u;
  uint32_t* mine = s_a + (tid & ~31) * KW;
  for (long first = (blockIdx.x * (long)kNarrowThreads + (tid & ~31)); first < npix;
       first += (long)gridDim.x * kNarrowThreads) {
    const long idx = first + lane;
    uint32_t kw[KW];
    int xsum = 0;
    {
      uint32_t r[3][3] = {};
      if (idx < npix) {
        const long rest = idx / p.Wo;
        const int wo = (int)(idx - rest * p.Wo), n = (int)(rest / p.Ho), ho = (int)(rest - (long)n * p.Ho);
        narrow_window<C, TAIL>(x, p.N, p.H, p.W, n, ho * p.stride - 1, wo * p.stride - 1, fill, r);
      }
      narrow_k<C>(r, kw);
    }
    if constexpr (Z) {
#pragma unroll
      for (int i = 0; i < KW; ++i) xsum = __dp4a((int)kw[i], 0x01010101, xsum);
      xsum *= -p.z_w;
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < KW; i += 4)
      *reinterpret_cast<uint4*>(mine + lane * KW + i) = make_uint4(kw[i], kw[i + 1], kw[i + 2], kw[i + 3]);
    __syncwarp();
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      uint2 a0[STEPS], a1[STEPS];
#pragma unroll
      for (int q = 0; q < STEPS; ++q) {
        a0[q] = *reinterpret_cast<const uint2*>(mine + (16 * half + g) * KW + 8 * q + 2 * t);
        a1[q] = *reinterpret_cast<const uint2*>(mine + (16 * half + g + 8) * KW + 8 * q + 2 * t);
      }
      const int c0 = Z ? __shfl_sync(0xffffffffu, xsum, 16 * half + g) : 0;
      const int c1 = Z ? __shfl_sync(0xffffffffu, xsum, 16 * half + g + 8) : 0;
      uint32_t o0[4] = {0u, 0u, 0u, 0u}, o1[4] = {0u, 0u, 0u, 0u};   // 16 codes of rows g and g + 8
      const long p0 = first + 16 * half + g, p1 = p0 + 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        int d[4] = {0, 0, 0, 0};
#pragma unroll
        for (int q = 0; q < STEPS; ++q) mma_s8(d, a0[q].x, a1[q].x, a0[q].y, a1[q].y, bf[j][q][0], bf[j][q][1]);
        const int kc = 16 * t + 2 * j;
        if constexpr (Z) {
          const int s0 = s_corr[kc], s1 = s_corr[kc + 1];
          d[0] += c0 + s0; d[1] += c0 + s1; d[2] += c1 + s0; d[3] += c1 + s1;
        }
        const float2 m = *reinterpret_cast<const float2*>(s_mult + kc), b = *reinterpret_cast<const float2*>(s_b + kc);
        float f[4];
        f[0] = __fmaf_rn(__int2float_rn(d[0]), m.x, b.x);
        f[1] = __fmaf_rn(__int2float_rn(d[1]), m.y, b.y);
        f[2] = __fmaf_rn(__int2float_rn(d[2]), m.x, b.x);
        f[3] = __fmaf_rn(__int2float_rn(d[3]), m.y, b.y);
        if (p.out_dtype == 0) {
          uint32_t c[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            c[e] = (uint32_t)(magic_to_int(__fadd_rn(fminf(fmaxf(f[e], p.lo_Y), p.hi_Y), kMagic)) + p.z_Y);
          // two codes of each row into half j & 1 of word j / 2
          const uint32_t h0 = __byte_perm(c[0], c[1], 0x0040u), h1 = __byte_perm(c[2], c[3], 0x0040u);
          o0[j >> 1] = (j & 1) ? __byte_perm(o0[j >> 1], h0, 0x5410u) : (h0 & 0xFFFFu);
          o1[j >> 1] = (j & 1) ? __byte_perm(o1[j >> 1], h1, 0x5410u) : (h1 & 0xFFFFu);
        } else {
          float* yp = reinterpret_cast<float*>(y);
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (k0 + kc + e < p.K && p0 < npix) yp[p0 * p.K + k0 + kc + e] = f[e];
            if (k0 + kc + e < p.K && p1 < npix) yp[p1 * p.K + k0 + kc + e] = f[2 + e];
          }
        }
      }
      if (p.out_dtype == 0) {
        const int kc = k0 + 16 * t;
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          const long px = rr == 0 ? p0 : p1;
          if (px >= npix || kc >= p.K) continue;
          int8_t* yp = reinterpret_cast<int8_t*>(y) + px * p.K + kc;
          const uint32_t q0 = rr == 0 ? o0[0] : o1[0], q1 = rr == 0 ? o0[1] : o1[1], q2 = rr == 0 ? o0[2] : o1[2],
                         q3 = rr == 0 ? o0[3] : o1[3];
          if (wide) {
            *reinterpret_cast<uint4*>(yp) = make_uint4(q0, q1, q2, q3);
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (kc + e < p.K) yp[e] = (int8_t)((e < 4 ? q0 : e < 8 ? q1 : e < 12 ? q2 : q3) >> (8 * (e & 3)));
          }
        }
      }
    }
  }
}

// Any channel counts: thread = (output pixel, output channel), byte loads.  Odd channel counts
// above four only; nothing here is tuned.
__global__ void __launch_bounds__(128)
k_direct_conv_bytes(const DirectParams p, const int8_t* __restrict__ x, const int8_t* __restrict__ w,
                    const float* __restrict__ bias, void* __restrict__ y) {
  const long npix = (long)p.N * p.Ho * p.Wo;
  const long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  griddep_launch();
  griddep_wait();
  if (idx >= npix * p.K) return;
  const int k = (int)(idx % p.K);             // consecutive lanes: consecutive output channels
  long pix = idx / p.K;
  const int wo = (int)(pix % p.Wo); pix /= p.Wo;
  const int ho = (int)(pix % p.Ho);
  const int n = (int)(pix / p.Ho);
  int acc = 0;
  for (int a = 0; a < 3; ++a) {
    const int h = ho * p.stride - 1 + a;
    if (h < 0 || h >= p.H) continue;
    for (int b = 0; b < 3; ++b) {
      const int wv = wo * p.stride - 1 + b;
      if (wv < 0 || wv >= p.W) continue;      // padding is the real value zero
      const int8_t* xp = x + (((long)n * p.H + h) * p.W + wv) * p.C;
      const int8_t* wp = w + (((long)k * 3 + a) * 3 + b) * p.C;
      for (int c = 0; c < p.C; ++c) acc += ((int)__ldg(xp + c) - p.z_x) * ((int)__ldg(wp + c) - p.z_w);
    }
  }
  const long o = (((long)n * p.Ho + ho) * p.Wo + wo) * p.K + k;
  float mult, s_in, s_Y;
  channel_scales(p, k, mult, s_in, s_Y);
  if (p.out_dtype == 0) {
    const float b = bias != nullptr ? (float)((double)__ldg(bias + k) / (double)s_Y) : 0.0f;
    const float yf = __fmaf_rn(__int2float_rn(acc), mult, b);
    const float r = __fadd_rn(fminf(fmaxf(yf, p.lo_Y), p.hi_Y), kMagic);
    reinterpret_cast<int8_t*>(y)[o] = (int8_t)(magic_to_int(r) + p.z_Y);
  } else {
    const float b = bias != nullptr ? __ldg(bias + k) : 0.0f;
    reinterpret_cast<float*>(y)[o] = __fmaf_rn(__int2float_rn(acc), s_in, b);
  }
}

int launch_direct_conv(int num_sms, int N, int C, int H, int W, int K, int stride, int z_x, int z_w, int z_Y,
                       float mult, float s_in, float s_Y, float lo_Y, float hi_Y, int out_dtype,
                       const int8_t* x, const int8_t* w, const float* bias, void* y,
                       const float* s_w_K, const float* s_Y_K, float s_x, float s_w, cudaStream_t st) {
  DirectParams p;
  p.s_w_K = s_w_K; p.s_Y_K = s_Y_K; p.s_x = s_x; p.s_w = s_w;
  p.N = N; p.C = C; p.H = H; p.W = W; p.K = K; p.stride = stride;
  p.Ho = (H - 1) / stride + 1; p.Wo = (W - 1) / stride + 1;
  p.z_x = z_x; p.z_w = z_w; p.z_Y = z_Y;
  p.mult = mult; p.s_in = s_in; p.s_Y = s_Y; p.lo_Y = lo_Y; p.hi_Y = hi_Y;
  p.out_dtype = out_dtype;
  const long npix = (long)N * p.Ho * p.Wo;
  if (C <= 4 && (K + kNarrowK - 1) / kNarrowK <= 65535) {
    // up to four blocks an SM; a warp takes further groups of 32 pixels where there are more
    const int kb = (K + kNarrowK - 1) / kNarrowK;
    const long want = (npix + kNarrowThreads - 1) / kNarrowThreads, most = (4l * num_sms + kb - 1) / kb;
    const dim3 grid((unsigned)(want < most ? want : most), (unsigned)kb);
    const int wide = K % 16 == 0 ? 1 : 0;   // y is 16-byte aligned
    const bool z = z_x != 0 || z_w != 0;
    const bool tail = narrow_has_tail((long)N * H * W * C) || narrow_has_tail((long)K * 9 * C);
    auto go = [&](auto plain, auto with_z, auto plain_tail, auto with_z_tail) {
      return launch_kernel(tail ? (z ? with_z_tail : plain_tail) : z ? with_z : plain, grid, dim3(kNarrowThreads), 0, st,
                           true, p, x, w, bias, y, wide);
    };
    return C == 1 ? go(k_direct_conv_narrow<1, false, false>, k_direct_conv_narrow<1, true, false>,
                       k_direct_conv_narrow<1, false, true>, k_direct_conv_narrow<1, true, true>)
         : C == 2 ? go(k_direct_conv_narrow<2, false, false>, k_direct_conv_narrow<2, true, false>,
                       k_direct_conv_narrow<2, false, true>, k_direct_conv_narrow<2, true, true>)
         : C == 3 ? go(k_direct_conv_narrow<3, false, false>, k_direct_conv_narrow<3, true, false>,
                       k_direct_conv_narrow<3, false, true>, k_direct_conv_narrow<3, true, true>)
                  : go(k_direct_conv_narrow<4, false, false>, k_direct_conv_narrow<4, true, false>,
                       k_direct_conv_narrow<4, false, false>, k_direct_conv_narrow<4, true, false>);
  }
  if (C % 4 != 0 || K % 4 != 0) {
    const long blocks = (npix * K + 127) / 128;
    if (blocks > 0x7fffffffl) return -2;   // WINO_ERR_UNSUPPORTED: more blocks than a grid holds
    return launch_kernel(k_direct_conv_bytes, dim3((unsigned)blocks), dim3(128), 0, st, true, p, x, w,
                         bias, y);
  }
  if (K % 8 == 0)
    return launch_kernel(k_direct_conv<8>, dim3((unsigned)((npix * (K / 8) + 127) / 128)), dim3(128),
                         0, st, true, p, x, w, bias, y);
  return launch_kernel(k_direct_conv<4>, dim3((unsigned)((npix * (K / 4) + 127) / 128)), dim3(128), 0,
                       st, true, p, x, w, bias, y);
}

}  // namespace wino
