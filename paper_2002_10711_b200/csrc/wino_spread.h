// How many blocks of a transform kernel an SM may hold.  Host code, no CUDA.
//
// The transforms' blocks are launched while the preceding kernel runs and gather on whatever SMs it leaves
// free, up to sixteen on each of a few SMs; the kernel then takes as long as those.  Dynamic shared memory
// beyond what the blocks use keeps them apart.  Grids of more than eight blocks per SM even out by themselves.
#pragma once
#include <cstddef>

namespace wino {

// Dynamic shared memory of a block that uses `smem`, with which an SM holds at most `per` (0: as many as fit).
constexpr size_t kSpreadSmem = 220 * 1024;
inline size_t spread_smem(size_t smem, int per) {
  const size_t least = per == 0 ? 0 : kSpreadSmem / (size_t)per - 1024;
  return smem > least ? smem : least;
}

// A grid's blocks per SM, on average.  Measured on B200, us, without / with it:
//   input transform alone  128 ch 16x16 F4 batch 30 3.43 / 2.32, batch 40 3.72 / 2.57;  512 ch 4x4 F4 batch
//     100 3.11 / 2.06, F6 batch 140 4.81 / 3.54;  64 ch 16x16 F2 batch 30 2.50 / 2.16
//   output transform alone  256 ch 8x8 F4 batch 128 3.55 / 2.82;  96 ch 20x20 F4 batch 20 3.06 / 2.21;  128
//     ch 8x8 F2 batch 64 2.60 / 2.08
//   whole layers, with both  256 ch 8x8 F4 batch 128 12.67 / 10.29, batch 56 11.55 / 8.77, batch 32 8.04 /
//     8.09;  128 ch 28x28 F4 batch 8 9.06 / 7.23;  160 -> 192 ch 14x14 F4 batch 16 11.23 / 8.05;  512 ch 4x4
//     F4 batch 128 11.41 / 10.11;  128 ch 12x12 F6 batch 64 11.58 / 9.77
// The input transform's limit.  None in a layer of more than 64 output channels and many un-quantized sums
// (`sums` of them, 0 if they are quantized): what runs before it is as a rule another such layer's long
// pointer-based output transform, on whose last SMs the whole grid would then wait.  Layers, us, without /
// with the limit: 128 ch 8x8 F6 batch 150 (4.9 M sums) 25.0 / 26.6;  256 ch 8x8 F6 batch 75 (4.9 M) 27.6 /
// 30.0;  128 -> 256 ch 8x8 F4 batch 150 (5.5 M) 23.1 / 24.7;  256 ch 4x4 F2 batch 150 (2.5 M) 16.5 / 17.1;
// below  256 ch 8x8 F4 batch 50 (1.8 M) 18.2 / 16.6;  128 ch 4x4 F2 batch 150 (1.2 M) 13.4 / 11.4;  64 output
// channels  256 ch 8x8 F4 batch 100 (0.9 M) 14.0 / 13.3, 64 ch 8x8 F4 batch 400 (3.7 M) 18.3 / 17.4.
inline int in_blocks_per_sm(long units, int K, long sums, int num_sms) {
  const long per = (units + num_sms - 1) / num_sms;
  return per >= 2 && per <= 8 && (K <= 64 || sums <= 2200000) ? (int)per : 0;
}

// The output transform, behind a tensor-core GEMM of `items` work items and C input channels (items 0:
// another GEMM, whose SMs free themselves a block at a time).  The average, with these exceptions:
//   - none if some of the GEMM's blocks have an item more than others: the SMs that the others leave early
//     are then the place for the excess (128 ch 16x16 F4 batch 48, 216 items, 9.4 us without, 10.3 with;
//     batch 64, 288 items, 11.1 and 9.5);
//   - two, for less than one per SM, if the GEMM leaves free less than half as many SMs as there are blocks:
//     a whole grid of them gathers there.  Layer, us, without / one / two / three: 512 ch 8x8 F6 batch 4 (64
//     blocks, 20 SMs) 12.9 / 9.8 / 9.6 / 10.0, batch 8 (128) 13.7 / 11.4 / 9.9 / 10.1;  64 ch 8x8 F4 batch
//     100 (100 blocks, 4 SMs) 8.0 / 7.0 / 7.0 / 6.9.  With 84 SMs free it costs: 256 ch 12x12 F6 batch 18
//     (144 blocks) 8.6 / 10.6 / 10.4 / 10.5;
//   - three instead of two behind a GEMM of at most 128 channels: its blocks hold two stages and leave room
//     for another block, but two of a whole SM's share do not come to lie beside each other on enough SMs.
//     Us, two / three: 128 -> 256 ch 8x8 F4 batch 37 9.45 / 7.8, batch 32 9.3 / 7.6;  64 -> 256 9.0 / 7.6;
//     128 -> 256 ch 4x4 F2 batch 64 8.4 / 7.3;  128 ch 8x8 F4 batch 43 to 64 level.
inline int out_blocks_per_sm(long units, long items, int C, int num_sms) {
  if (items == 0 || !(items <= num_sms || (items <= 2l * num_sms && 10 * items >= 19l * num_sms))) return 0;
  const bool crowded = items <= num_sms && units > 2 * (num_sms - items);
  const long avg = (units + num_sms - 1) / num_sms, per = avg == 1 && crowded ? 2 : avg;
  if (per < 2 || per > 8) return 0;
  return per == 2 && C <= 128 ? 3 : (int)per;
}

}  // namespace wino
