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

// Geometry by estimated time.  The grid runs in rounds of one or two blocks per SM; a round with
// one block per SM takes `one` (measured on B200, us, one 64-channel chunk per block):
//     16*KB channels   16    32    64
//     F2               3.4   3.6   4.4
//     F4               4.3   5.3
//     F6               6.5   8.6
// plus `more` for every further chunk and 1.1 for the exchange in a cluster; two blocks per SM
// (shared memory permitting, F2 and F4) take 1.1 (F2) to 1.4 times as long as one.  Clusters of four or eight do not
// fill every SM.  Within 15 % of the measured time from 1 to 2048 blocks.
SmallGeom small_geometry(const Params& p, int num_sms) {
  static const double one[3][3] = {{3.4, 3.6, 4.4}, {4.3, 5.3, 0}, {6.5, 8.6, 0}};
  static const double more[3][3] = {{0.35, 0.6, 0.9}, {1.25, 1.4, 0}, {1.6, 1.6, 0}};
  static const double small_copies[3] = {1.0, 2.2, 3.2};
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
      double t1 = one[mi][ki] + more[mi][ki] * (g.chunks - 1) + (S > 1 ? 1.1 : 0.0);
      // Tensor copies need whole 16-byte pieces; of rows narrower than a chunk they fill in the rest,
      // which the copy engine does slowly (16 channels, F2: 2.7 us with a block or two, 7.5 with 128,
      // where small copies take 3.3 and 5.1).
      g.tma = p.C % 16 == 0 && (p.C >= 64 || blocks <= 48);
      if (!g.tma) t1 += small_copies[mi] * (KB > 1 ? 1.5 : 1.0) * g.chunks * (p.C % 16 != 0 ? 1.15 : 1.0);
      const double full = two ? t1 * (p.m == 2 ? 1.1 : 1.4) : t1;
      const bool last_full = blocks - (rounds - 1) * per_round > sms;
      g.cost = (long)(1000.0 * ((rounds - 1) * full + (last_full ? full : t1)));
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
