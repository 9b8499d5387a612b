// Direct int8 3x3 convolution (cross-correlation, zero padding 1, stride 1 or 2)
// with int32 accumulation: the lossless candidate the paper compares the
// Winograd-aware layers with (Sections 4 and 5.3), and the layer type of the
// network's strided convolutions, for which no Winograd form exists (Section 5.1).
// Integer dot products on the ALUs; thread = (output pixel, 4 or 8 output channels).
#include "wino_launch.h"

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

// At most four input channels (a network's first layer, Section 5.1).  The 9 * C codes under a
// pixel's window fit NW = ceil(9 * C / 4) registers, so a thread takes one output pixel, gathers
// its window once and walks 32 output channels whose filters, packed the same way, lie in shared
// memory (every lane reads the same words: broadcasts).  Window and filter pad with zeros.
// With zero points, sum (x - z_x)(w - z_w) = sum x w - z_w sum x - z_x sum w + 9 C z_x z_w over the
// whole window, pixels outside the image holding the code z_x.
// Bound by the ALU pipe: NW dot products and seven quantizer instructions per output.  64 images
// 32x32, 3 -> 64 channels: 10.0 us, where the byte-wise kernel below took 114.
constexpr int kNarrowK = 32, kNarrowThreads = 128;
template <int C>
__global__ void __launch_bounds__(kNarrowThreads)
k_direct_conv_narrow(const DirectParams p, const int8_t* __restrict__ x, const int8_t* __restrict__ w,
                     const float* __restrict__ bias, void* __restrict__ y, int store) {
  constexpr int NW = (9 * C + 3) / 4, taps = 9 * C, row_bytes = 3 * C;
  constexpr int WS = (NW + 3) / 4 * 4;     // words between two filters: whole 16-byte reads
  __shared__ __align__(16) uint32_t s_w[kNarrowK * WS];
  __shared__ int s_corr[kNarrowK];         // - z_x sum w + 9 C z_x z_w
  __shared__ float s_mult[kNarrowK], s_b[kNarrowK];
  const int k0 = blockIdx.y * kNarrowK;
  griddep_launch();
  for (int i = threadIdx.x; i < kNarrowK * WS; i += kNarrowThreads) s_w[i] = 0u;
  __syncthreads();
  griddep_wait();
  const int nk = min(kNarrowK, p.K - k0);
  for (int i = threadIdx.x; i < nk * taps; i += kNarrowThreads) {
    const int k = i / taps, j = i - k * taps;
    reinterpret_cast<int8_t*>(s_w + k * WS)[j] = w[(long)(k0 + k) * taps + j];
  }
  const long npix = (long)p.N * p.Ho * p.Wo;
  const long idx = blockIdx.x * (long)kNarrowThreads + threadIdx.x;
  uint32_t win[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) win[i] = 0u;
  if (idx < npix) {
    const int rest = (int)(idx / p.Wo), wo = (int)(idx - (long)rest * p.Wo);
    const int n = rest / p.Ho, ho = rest - n * p.Ho;
    const int h0 = ho * p.stride - 1, w0 = wo * p.stride - 1;
    const int8_t* xp = x + (((long)n * p.H + h0) * p.W + w0) * p.C;
    // byte 4 i + j of the window: row (4 i + j) / (3 C); within a row the bytes are contiguous
#pragma unroll
    for (int i = 0; i < NW; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int at = 4 * i + j;
        if (at < taps) {
          const int a = at / row_bytes, r = at - a * row_bytes, b = r / C;
          const bool in = (unsigned)(h0 + a) < (unsigned)p.H && (unsigned)(w0 + b) < (unsigned)p.W;
          const int v = in ? (int)__ldg(xp + (long)a * p.W * C + r) : p.z_x;
          win[i] |= ((uint32_t)v & 0xFFu) << (8 * j);
        }
      }
  }
  __syncthreads();
  if (threadIdx.x < nk) {
    const int k = threadIdx.x;
    int sum = 0;
    for (int j = 0; j < NW; ++j) sum = __dp4a((int)s_w[k * WS + j], 0x01010101, sum);
    s_corr[k] = -p.z_x * sum + taps * p.z_x * p.z_w;
    float mult, s_in, s_Y;
    channel_scales(p, k0 + k, mult, s_in, s_Y);
    const float b = bias != nullptr ? __ldg(bias + k0 + k) : 0.0f;
    s_mult[k] = p.out_dtype == 0 ? mult : s_in;
    s_b[k] = p.out_dtype == 0 && bias != nullptr ? (float)((double)b / (double)s_Y) : b;
  }
  __syncthreads();
  if (idx >= npix) return;
  int corr = 0;
  if (p.z_w != 0) {
#pragma unroll
    for (int i = 0; i < NW; ++i) corr = __dp4a((int)win[i], 0x01010101, corr);
    corr *= -p.z_w;
  }
  const long o = idx * p.K + k0;
#pragma unroll 1
  for (int q = 0; q < nk; q += 16) {
    uint32_t out[4];
#pragma unroll
    for (int e4 = 0; e4 < 4; ++e4) {
      uint32_t word = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = q + 4 * e4 + e;      // (channels past K: zero filters of the padded table)
        int acc = corr + s_corr[k];
        const uint4* f = reinterpret_cast<const uint4*>(s_w + k * WS);
#pragma unroll
        for (int i = 0; i < WS / 4; ++i) {
          const uint4 v = f[i];
          acc = __dp4a((int)win[4 * i], (int)v.x, acc);
          if (4 * i + 1 < NW) acc = __dp4a((int)win[4 * i + 1 < NW ? 4 * i + 1 : 0], (int)v.y, acc);
          if (4 * i + 2 < NW) acc = __dp4a((int)win[4 * i + 2 < NW ? 4 * i + 2 : 0], (int)v.z, acc);
          if (4 * i + 3 < NW) acc = __dp4a((int)win[4 * i + 3 < NW ? 4 * i + 3 : 0], (int)v.w, acc);
        }
        const float yf = __fmaf_rn(__int2float_rn(acc), s_mult[k], s_b[k]);
        if (p.out_dtype == 0) {
          const float r = __fadd_rn(fminf(fmaxf(yf, p.lo_Y), p.hi_Y), kMagic);
          word |= ((uint32_t)(magic_to_int(r) + p.z_Y) & 0xFFu) << (8 * e);
        } else if (k < nk) {
          reinterpret_cast<float*>(y)[o + k] = yf;
        }
      }
      out[e4] = word;
    }
    if (p.out_dtype == 0) {
      int8_t* yp = reinterpret_cast<int8_t*>(y) + o + q;
      if (store == 16) {
        *reinterpret_cast<uint4*>(yp) = make_uint4(out[0], out[1], out[2], out[3]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (q + j < nk) yp[j] = (int8_t)(out[j >> 2] >> (8 * (j & 3)));
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

int launch_direct_conv(int N, int C, int H, int W, int K, int stride, int z_x, int z_w, int z_Y,
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
  if (C <= 4 && (K + kNarrowK - 1) / kNarrowK <= 65535 && (npix + kNarrowThreads - 1) / kNarrowThreads <= 0x7fffffffl) {
    const dim3 grid((unsigned)((npix + kNarrowThreads - 1) / kNarrowThreads), (unsigned)((K + kNarrowK - 1) / kNarrowK));
    const int store = K % 16 == 0 ? 16 : 1;   // y is 16-byte aligned
    auto kernel = C == 1 ? k_direct_conv_narrow<1> : C == 2 ? k_direct_conv_narrow<2>
                : C == 3 ? k_direct_conv_narrow<3> : k_direct_conv_narrow<4>;
    return launch_kernel(kernel, grid, dim3(kNarrowThreads), 0, st, true, p, x, w, bias, y, store);
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
