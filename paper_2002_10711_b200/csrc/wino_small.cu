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

// Geometry by estimated time.  The kernel's time is a latency (about a block's own time) while
// the grid fits the SMs once, and grows by a constant per block beyond that.  Measured on B200,
// back to back in a graph, one chunk per block, no cluster; latency in us, ns per further block:
//     16*KB channels      16            32            64
//     F2             3.4 / 10.7    3.6 / 12.9    4.4 / 17.3
//     F4             4.3 / 16.9    5.3 / 22.7
//     F6             6.5 / 43.6    8.5 / 58       (one block per SM)
// A further chunk adds a quarter to the cost per block, and doubles it where the shared memory
// then holds one block instead of two; a cluster costs 1 us and a third to a half per block, and
// clusters of four or eight blocks with an SM each leave SMs unused.  The estimate is within
// 20 % of the measured time from 1 to 2048 blocks.
SmallGeom small_geometry(const Params& p, int num_sms) {
  static const double latency[3][3] = {{3.4, 3.6, 4.4}, {4.3, 5.3, 0}, {6.5, 8.5, 0}};
  static const double per_block[3][3] = {{10.7, 12.9, 17.3}, {16.9, 22.7, 0}, {43.6, 58.0, 0}};
  static const double per_chunk[3] = {0.35, 1.25, 1.6};    // latency of a further chunk
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
      const bool one_per_sm = g.smem > 113 * 1024;
      double each = per_block[mi][ki] * (0.75 + 0.25 * g.chunks);
      if (one_per_sm && p.m != 6) each *= 1.75;
      if (S > 1) each *= p.m == 2 ? 1.5 : 1.3;
      if (S > 2 && one_per_sm) each *= 2.0;
      const double over = (double)blocks - (S > 2 && one_per_sm ? 0.75 : 1.0) * num_sms;
      double ns = 1000.0 * (latency[mi][ki] + per_chunk[mi] * (g.chunks - 1) + (S > 1 ? 1.0 : 0.0));
      if (over > 0) ns += over * each;
      if (p.C % 16 != 0) ns += 600.0 * p.m * g.chunks;   // operands by 4-byte loads
      g.cost = (long)ns;
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
