// Host side of the small-layer kernel (wino_small_impl.cuh): which geometry, and dispatch over
// the tile size.
#include "wino_launch.h"

namespace wino {

#define WINO_DECL(m) \
  int launch_small_m##m(const Params&, const LaunchOpt&, const SmallGeom&, const SmallArgs&, cudaStream_t);
WINO_DECL(2)
WINO_DECL(4)
WINO_DECL(6)
#undef WINO_DECL

namespace {
// Bytes of shared memory of a block: U_q slice, codes, patches of its chunks.
size_t small_smem(int t2, int KB, int chunks) { return (size_t)chunks * t2 * (16 * KB + 16) * 64 + 256; }
}  // namespace

bool small_supported(const Params& p) {
  // 16-bit lanes of the input quantizer, 4-byte loads; a cluster of eight blocks with one chunk
  // each (F6) or up to three (F4, F2)
  return p.C % 4 == 0 && p.v_fits_16 && p.C <= (p.m == 6 ? 512 : 1024);
}

// Geometry by estimated time.  The grid runs in rounds of one or two blocks per SM; a round with one block
// per SM takes `one` (64-channel chunks; 16, 32 and 64 channels a block), `more` for every further chunk of a
// block, `exchange` in a cluster, `copies` a chunk without tensor copies, and as much of `load` as the round
// fills SMs: U_q and the patches then come through L2 to all of them at once.  Two blocks per SM (shared
// memory permitting, F2 and F4) take `two` times as long as one.  Clusters of four or eight do not fill every
// SM.  Learnt matrices and an input zero point, whose padding is patched, lengthen the input transform; at
// most four tiles leave half of a block's warps idle and take 0.92 of the time.
// Fitted on B200 to 8000 times of layers of 1 to 2048 blocks with every option and most geometries, per call,
// averaged over a loop of calls and a CUDA graph of them: 5.6 (F6) to 7.4 % (F2) standard deviation.  Where
// the geometry differs from that of an earlier fit without `load` (700 layers), 0.95 of the time.
SmallGeom small_geometry(const Params& p, bool std_mats, int num_sms) {
  static const double one[3][3] = {{3.1, 3.7, 5.2}, {4.6, 6.1, 0}, {6.7, 9.0, 0}};
  static const double more[3][3] = {{0.7, 0.8, 1.2}, {1.2, 1.0, 0}, {1.0, 1.0, 0}};
  static const double exchange[3] = {1.2, 1.0, 0.9}, copies[3] = {1.0, 2.4, 3.0};
  static const double load[3] = {0.9, 1.6, 0.9}, twice[3] = {1.1, 1.08, 1.0};
  static const double learnt[3] = {1.15, 1.17, 1.22}, zero[3] = {1.06, 1.10, 1.06};
  const int t2 = p.t * p.t, groups = (p.T + 7) / 8, all_chunks = (p.C + 63) / 64;
  const int mi = p.m / 2 - 1;
  SmallGeom best = {};
  best.cost = -1;
  for (int ki = 0; ki < (p.m == 2 ? 3 : 2); ++ki) {
    const int KB = 1 << ki;
    if (KB > 1 && 8 * KB >= p.K) break;          // half of the block's channels would not exist
    for (int S = 1; S <= 8; S *= 2) {
      if (S > 1 && S / 2 >= all_chunks) break;
      SmallGeom g = {};
      g.KB = KB; g.S = S;
      g.chunks = (all_chunks + S - 1) / S;
      g.n_kblk = (p.K + 16 * KB - 1) / (16 * KB);
      g.smem = small_smem(t2, KB, g.chunks);
      if (g.smem > 226 * 1024) continue;
      const long blocks = (long)groups * g.n_kblk * S;
      if (blocks > 0x7fffffffl) continue;
      g.grid = (int)blocks;
      const bool two = p.m != 6 && g.smem <= 113 * 1024;
      const long sms = S == 8 ? num_sms * 3l / 4 : S == 4 ? num_sms * 9l / 10 : num_sms;
      const long per_round = two ? 2 * sms : sms, rounds = (blocks + per_round - 1) / per_round;
      double t1 = one[mi][ki] + more[mi][ki] * (g.chunks - 1) + (S > 1 ? exchange[mi] : 0.0);
      // Tensor copies need whole 16-byte pieces; of rows narrower than a chunk they fill in the rest,
      // which the copy engine does slowly (16 channels, F2: 2.7 us with a block or two, 7.5 with 128,
      // where small copies take 3.3 and 5.1).
      g.tma = p.C % 16 == 0 && (p.C >= 64 || blocks <= 48);
      if (!g.tma) t1 += copies[mi] * (KB > 1 ? 1.5 : 1.0) * g.chunks * (p.C % 16 != 0 ? 1.15 : 1.0);
      const double full = (t1 + load[mi]) * (two ? twice[mi] : 1.0);
      const long last = blocks - (rounds - 1) * per_round;
      const double us = (rounds - 1) * full + (last > sms ? full : t1 + load[mi] * last / sms);
      g.cost = (long)(1000.0 * us * (std_mats ? 1.0 : learnt[mi]) * (p.z_x == 0 ? 1.0 : zero[mi]) * (p.T <= 4 ? 0.92 : 1.0));
      if (best.cost < 0 || g.cost < best.cost) best = g;
    }
  }
  return best;
}

int launch_small(const Params& p, const LaunchOpt& o, const SmallGeom& g, const SmallArgs& s, cudaStream_t st) {
  return p.m == 2 ? launch_small_m2(p, o, g, s, st)
       : p.m == 4 ? launch_small_m4(p, o, g, s, st)
                  : launch_small_m6(p, o, g, s, st);
}

}  // namespace wino
