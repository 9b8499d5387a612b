// Internal interface between the host planner (wino_host.cu) and the kernel
// translation units.  Every function enqueues work on `st` and returns 0 or a
// negative WINO_ERR_* code; none allocates or synchronizes.
#pragma once
#include <cstdio>
#include <mutex>
#include <utility>

#include <cuda.h>
#include <cuda_runtime.h>
#include "wino_common.cuh"

namespace wino {

// SMs of a B200: what is assumed where no device can be asked (plans made without one).
constexpr int kDefaultSms = 148;

// Launch options shared by all kernels.
struct LaunchOpt {
  bool std_mats = false;      // B^T and A^T are the built-in Cook-Toom matrices
  bool pdl = false;           // programmatic dependent launch on the stream
  int device = 0;             // the plan's device (current when the launcher runs)
  int num_sms = kDefaultSms;  // its SM count
  // A buffer a later kernel of the same call will read and that no kernel of the call
  // writes (the transformed weights): the input transform's blocks ask for it to be brought
  // into L2 while they run.  A hint only; null: none.
  const void* l2_hint = nullptr;
  size_t l2_hint_bytes = 0;   // a multiple of 16
  // Per-output-channel multipliers, device array [5][K] (rows kChMultU ... kChSY), or null
  // for the per-layer values of Params.  Read by the weight transform, the GEMM epilogues
  // and the output transforms.
  const float* chan = nullptr;
  bool chan_m_fits_16 = false;   // with these multipliers every rounded product of Q_M is below 2^15
  // Work items of the tensor-core GEMM in front of an output transform, 0 if it is another GEMM.
  long gemm_items = 0;
};

// "Done once per device" bookkeeping.  cudaFuncSetAttribute applies to the device
// that is current when it is called, so the opt-in to more than 48 KB of dynamic
// shared memory has to be repeated on every device a kernel is launched on.
// run(dev, fn) calls fn() the first time it sees `dev` (and again if fn failed)
// under a lock, so concurrent first launches from several host threads are safe.
// Device indices beyond the table always run fn.
class DeviceOnce {
 public:
  static constexpr int kMaxDevices = 64;
  template <typename Fn>
  int run(int dev, Fn fn) {
    if (dev < 0 || dev >= kMaxDevices) return fn();
    std::lock_guard<std::mutex> lock(mu_);
    if (done_[dev]) return 0;
    const int rc = fn();
    if (rc == 0) done_[dev] = true;
    return rc;
  }
 private:
  std::mutex mu_;
  bool done_[kMaxDevices] = {};
};

// Opt a kernel in to `smem` bytes of dynamic shared memory on device `dev`.
template <typename Kern>
int set_max_smem(DeviceOnce& once, int dev, Kern kernel, size_t smem) {
  return once.run(dev, [&]() -> int {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
#ifdef WINO_TRACE
    if (e != cudaSuccess)
      std::fprintf(stderr, "shared-memory attribute failed: %s (%zu bytes)\n", cudaGetErrorString(e), smem);
#endif
    return e == cudaSuccess ? 0 : -5;
  });
}

// absmax (nullable): one word, max |U| of the layer; absmax_K (nullable): K words, max |U| of
// each filter; both as float bits, caller-zeroed.
int launch_weight_transform(const Params& p, const LaunchOpt& o, const int8_t* w, int8_t* Uq,
                            unsigned* absmax, unsigned* absmax_K, cudaStream_t st);
int launch_input_transform(const Params& p, const LaunchOpt& o, const int8_t* x, int8_t* Vq,
                           unsigned* absmax, cudaStream_t st);
int launch_output_transform(const Params& p, const LaunchOpt& o, float s_Y, const void* mbuf,
                            const float* bias, void* y, unsigned* absmax2, cudaStream_t st);
int launch_gemm_warp(const Params& p, const LaunchOpt& o, const int8_t* Vq, const int8_t* Uq,
                     void* out, int out_mode, unsigned* absmaxM, cudaStream_t st);

// TMA-staged transform kernels (input needs C % 16 == 0; output needs Q_M on and K % 16 == 0).
// Channel chunk per block: the widest multiple of 16 up to 128 that divides the channels (narrow chunks
// are short rows, which the copy engine delivers no faster than long ones).
constexpr int tma_chunk(int channels) {
  for (int chunk = 128; chunk > 0; chunk -= 16)
    if (channels % chunk == 0) return chunk;
  return 0;
}
// Tiles per block: about 128 threads of two channels; half of that in the input transforms of F4
// and F6 (smaller blocks balance better over the SMs, 5.3 -> 5.1 us on a 256-channel 8x8 layer at
// batch 256, and a narrow layer has more of them; F2's shorter blocks do not gain).
constexpr int tma_group(int chunk) { return 256 / chunk; }
constexpr int tma_in_group(int m, int chunk) { return m == 2 ? tma_group(chunk) : chunk > 64 ? 1 : 128 / chunk; }
// Tiles per block of the output transform: one, with one channel per thread and 16 blocks per SM, for
// F4 in 128-channel chunks while all blocks are resident at once.  Measured on B200, us a layer, two
// channels per thread / one: 256 ch 8x8 batch 256 15.84 / 15.73, 128 ch 16x16 batch 64 12.68 / 12.43,
// batch 32 10.93 / 10.58, 384 ch 12x12 batch 32 15.76 / 15.48 (256 ch 8x8 batch 64 11.60 / 11.73);
// narrower chunks lose (96 ch: 11.80 / 12.45, 64 ch: 13.74 / 13.89).
// F6 likewise while a handful of blocks per SM is all there is: at 64 registers they start beside the
// GEMM, and a block is over sooner.  Layer, us, two channels per thread / one, blocks per SM in brackets: 128
// channels a block  128 ch 12x12 batch 64 (2) 9.9 / 9.2, batch 100 (3) 11.0 / 9.8, 512 ch 8x8 batch 32 (4) 12.7
// / 12.2, 128 ch 12x12 batch 150 (5) 12.6 / 13.1, 256 ch 12x12 batch 75 (5) 13.6 / 14.1;  64 channels  64 ch
// 12x12 batch 64 (2) 9.1 / 8.2, batch 150 (5) 10.4 / 9.7, batch 200 (6) 11.4 / 10.4, batch 275 (8) 12.4 / 13.1.
// With scales per output channel, of which a block reads three, up to two:  128 ch 12x12 batch 75 (3) 11.0 /
// 11.7, 512 ch 8x8 batch 37 (4) 16.3 / 16.9;  64 ch 12x12 batch 75 (3) 10.1 / 10.7, batch 150 (5) 10.9 / 12.1.
inline int tma_out_group(const Params& p, bool std_mats, bool per_channel, int num_sms) {
  const int chunk = tma_chunk(p.K);
  if (p.m == 6 && std_mats && p.out_dtype == 0 && (chunk == 128 || chunk == 64))
    return (long)p.T * (p.K / chunk) <= (per_channel ? 2l : chunk == 128 ? 4l : 6l) * num_sms ? 1 : tma_group(chunk);
  return p.m == 4 && std_mats && p.out_dtype == 0 && chunk == 128 && (long)p.T * (p.K / 128) <= 16l * num_sms
             ? 1 : tma_group(chunk);
}
int launch_input_transform_tma(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX,
                               const CUtensorMap& mapV, int* status, cudaStream_t st);
// y_float: the output when it is float (mapY is then not used), else null.
int launch_output_transform_tma(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM,
                                const CUtensorMap& mapY, const float* bias, float s_Y, int* status, float* y_float,
                                cudaStream_t st);

// Tensor-core transforms (wino_transforms_tc.cu): Cook-Toom matrices; the input side for m = 2, 4, 6,
// any input zero point, C a multiple of 16 and products of Q_V that fit 16 bits; the output side for
// m = 2, 4, Q_M on, K a multiple of 16 (at most 2048).  Channel chunk of a unit: 128 or 64.
// mapX: x as [N][H][W][C], box input_tc_box; mapM: m_q as [t*t][T][K], box output_tc_box; both with
// the swizzle of the chunk's width.  `images`: the constant operands (xt_images).
inline int xt_chunk(int channels) { return channels % 128 == 0 ? 128 : 64; }
int xt_images(int device, const uint8_t** out);
bool input_tc_supported(const Params& p, bool std_mats);
bool output_tc_supported(const Params& p, bool std_mats);
void input_tc_box(const Params& p, uint32_t box[4]);
void output_tc_box(const Params& p, uint32_t box[3]);
int launch_input_transform_tc(const Params& p, const LaunchOpt& o, const CUtensorMap& mapX, const uint8_t* images,
                              int8_t* Vq, int* status, cudaStream_t st);
int launch_output_transform_tc(const Params& p, const LaunchOpt& o, const CUtensorMap& mapM, const uint8_t* images,
                               const float* bias, void* y, float s_Y, int* status, cudaStream_t st);

// Kronecker matrices of the single-launch layer kernel, whose transforms are such products too.
// `kron`: device copy of the plan's tables (fill_kronecker_tables).
constexpr int kKronInRows = 48, kKronOutRows = 16;
constexpr int kKronBytes = (kKronInRows + kKronOutRows) * 64;
void fill_kronecker_tables(int m, int8_t* dst_host);

// The whole layer in one persistent launch (Cook-Toom F2 / F4, C and K multiples of
// 128, input zero point 0, Q_M on, int8 output).  `counters`: plan-owned device words,
// zero between launches (the kernel clears them when it finishes):
// [kFusedMaxMblk] cnt_in, [kFusedMaxMblk] cnt_m, then the exit ticket.
constexpr int kFusedMaxMblk = 1024;
constexpr int kFusedCounterWords = 2 * kFusedMaxMblk + 16;
struct FusedGeom { int BN, stages, n_mblk, n_nblk, n_items, grid; size_t smem; };
struct FusedMaps { const CUtensorMap *x, *v_store, *v_load, *u, *m_load, *y; };
bool layer_fused_supported(const Params& p, bool std_mats);
FusedGeom layer_fused_geometry(const Params& p, int num_sms);
int launch_layer_fused(const Params& p, const LaunchOpt& o, const FusedGeom& g, const FusedMaps& m,
                       const void* kron, unsigned* counters, int8_t* mq, const float* bias,
                       float s_Y, int* status, cudaStream_t st);

struct TcGeom { int BN, MB, cB, stages, tmem_cols, items, grid; size_t smem; };
TcGeom tc_geometry(const Params& p, int num_sms);
int launch_gemm_tc(const Params& p, const LaunchOpt& o, const TcGeom& g, const CUtensorMap& mapV,
                   const CUtensorMap& mapU, void* out, int out_mode, unsigned* absmaxM,
                   int* status, cudaStream_t st);
int launch_smallc(const Params& p, const LaunchOpt& o, const int8_t* x, const int8_t* Uq,
                  const float* bias, void* y, float s_Y, int* dbgM, cudaStream_t st);

// The whole layer in one launch for layers of few tiles (any m, matrices and options; C a
// multiple of 4): a block owns 8 tiles x 16*KB output channels, the S blocks of a cluster
// `chunks` chunks of 64 channels each.  `cost`: the launcher's estimate of the kernel's time, ns.
// The maps (C a multiple of 16): x as [N][H][W][C] with box {64, t, t, 1}, U_q as [t*t][K][C]
// with box {64, 16*KB, t*t}, no swizzle.
struct SmallGeom { int KB, chunks, S, n_kblk, grid, tma; size_t smem; long cost; };
struct SmallArgs {
  const CUtensorMap *mapX, *mapU;
  const int8_t *x, *Uq;
  const float* bias;
  void* y;
  float s_Y;
  int* status;
};
bool small_supported(const Params& p);
SmallGeom small_geometry(const Params& p, bool std_mats, int num_sms);
int launch_small(const Params& p, const LaunchOpt& o, const SmallGeom& g, const SmallArgs& s, cudaStream_t st);

// Fully fused F2 kernel for narrow layers (C in {32, 64}, K <= 64, Cook-Toom matrices).
bool fused_f2_supported(const Params& p, bool std_mats);
int launch_fused_f2(const Params& p, const LaunchOpt& o, const CUtensorMap& mapU, const int8_t* x,
                    const float* bias, void* y, float s_Y, int num_sms, int* status, int* dbgM,
                    cudaStream_t st);

// Direct int8 3x3 convolution (stride 1 or 2) on the ALUs.
// Tensor-core direct convolution (no zero points on x and w, C % 64 == 0, K % 32 == 0).
struct DirectTcArgs {
  int N, C, H, W, K;       // H, W: output height and width
  int stride;
  int element_strides;     // stride 2 by the element strides of the x map (odd input sizes)
  int BW, BH, BI;          // output tile: BW x BH pixels of BI images, BW * BH * BI = 128
  int nW, nH, nI;          // tiles along width, height, batch
  int BN, n_nblk;          // output-channel block and their number
  int cB, KB;              // channel bytes per stage (64 or 128) and stages per tap
  int stages, tmem_cols, acc_stride;
  int n_items;
  // Narrow layers whose whole weight tensor fits beside the input ring: the weights are
  // fetched once per block and stay in shared memory (w_resident), and a stage then holds the
  // input boxes of `taps_per_stage` = 3 taps, one row of the filter (1 otherwise).
  int w_resident, taps_per_stage;
  float mult, s_in, s_Y, lo_Y, hi_Y;
  int z_Y, out_dtype;
  // per-output-channel scales (device arrays of K floats, nullable) and the per-layer scales
  // they replace
  const float* s_w_K;
  const float* s_Y_K;
  float s_x, s_w;
};
bool direct_tc_supported(int C, int K, int stride, int z_x, int z_w);
DirectTcArgs direct_tc_geometry(int N, int C, int H, int W, int K, int stride, int num_sms);
int* direct_tc_status_word(int device);
int launch_direct_conv_tc(const DirectTcArgs& a, int device, int num_sms, const CUtensorMap& mapX,
                          const CUtensorMap& mapW, const float* bias, void* y, cudaStream_t st);
// s_w_K, s_Y_K (nullable device arrays of K floats): per-output-channel scales replacing s_w
// and s_Y; s_x, s_w: the per-layer scales behind mult and s_in.
int launch_direct_conv(int num_sms, int N, int C, int H, int W, int K, int stride, int z_x, int z_w, int z_Y,
                       float mult, float s_in, float s_Y, float lo_Y, float hi_Y, int out_dtype,
                       const int8_t* x, const int8_t* w, const float* bias, void* y,
                       const float* s_w_K, const float* s_Y_K, float s_x, float s_w, cudaStream_t st);

// Tensor-pipe probe: `iters` back-to-back 128x256x32 int8 MMAs on every SM.
int launch_mma_peak(int iters, int num_sms, int device, int* status, cudaStream_t st);

// Bounded-wait probe: one block waits, with the given cycle limit, on a barrier
// that nothing arrives at, records WINO_ERR_TIMEOUT in *status and exits normally.
int launch_wait_probe(long long limit_cycles, int* status, cudaStream_t st);

enum { kOutMq = 0, kOutI32 = 1 };
constexpr int kBM = 128;      // tiles per GEMM block (MMA M)
constexpr int kStageK = 128;  // channels (bytes) per shared-memory stage (TcGeom::cB: 64 in narrow layers)

// Generic launcher: cudaLaunchKernelEx with, where asked for, the programmatic stream
// serialization attribute (the kernel then calls griddep_wait()) and clusters of `cluster`
// blocks along x.
template <typename... KArgs, typename... Args>
int launch_kernel_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, unsigned cluster, size_t smem,
                          cudaStream_t st, bool pdl, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (pdl) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
#ifdef WINO_TRACE
  if (e != cudaSuccess)
    std::fprintf(stderr, "launch failed: %s (grid %u block %u smem %zu)\n", cudaGetErrorString(e), grid.x,
                 block.x, smem);
#endif
  return e == cudaSuccess ? 0 : -5;
}
template <typename... KArgs, typename... Args>
int launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                  bool pdl, Args&&... args) {
  return launch_kernel_cluster(kernel, grid, block, 1u, smem, st, pdl, std::forward<Args>(args)...);
}

}  // namespace wino
