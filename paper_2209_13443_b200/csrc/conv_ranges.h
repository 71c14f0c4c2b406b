// How many ranges the K loop of a tensor-core convolution is cut into when nobody sets the number (conv_tc.cuh).  Plain arithmetic,
// for the plan and for host tests.
#pragma once

namespace ee {

// A cluster of CTAs per tile runs with the deep operand ring, whose CTA owns its SM, while the grid leaves a quarter of the SMs
// free: a cluster needs all its CTAs inside one GPC, and the last clusters of a fuller grid wait for a second wave.
inline bool tc_cluster_deep(long ctas, int sms) { return ctas * 4 <= 3L * sms; }

// num_kb: K blocks of the layer.  tiles_max: its output tiles at max_batch.  The ranges fix how every sum is grouped, so they
// depend on the layer and max_batch and never on the batch that runs, and the cut is taken only where even max_batch runs as deep
// clusters, which is well within one wave.
// What it gives is accuracy.  Each of four accumulators takes a quarter of a layer's products, and about a quarter as many outputs miss
// the bf16 nearest to their sum in 64 bits.  In a chain of 3x3 layers on maps of 2x2 to 7x7, batch 1 to 64:
//   K blocks   misses per 10 000 outputs, whole / four ranges   us a layer, whole / what four ranges add
//        63       5.7-7.7 / 0.9-1.3                                 7.3-7.8 / +0.4 to +0.5
//        72       3.4-8.5 / 0.8-2.2                                8.0-10.5 / +0.5 to +0.6
//        90       7.2-8.3 / 2.2-2.6                                9.7-10.3 / +0.6 to +0.8
//       108       8.0-11  / 2.1-3.1                               11.8-12.1 / +0.5 to +0.7
//       144        11-14  / 3.4-3.7                                    15.7 / +0.3
//       216        16-21  / 5.0-9.3                               23.9-24.6 / -1.4
//       288        24-33  / 4.3-7.9                               32.8-37.7 / -2.0 to -7.1
// The line, about 60 blocks, lies where the two took the same time on tiles of 128 pixels (whole 2.0 + 0.122 us a block, a CTA of a
// cluster for each range 7.0 + 0.15 a block of a range).  Tiles of 64 pixels made whole layers the faster ones up to about 150 blocks; the
// line stays for the accuracy.  Past the deep clusters four ranges cost too much, 3x3 512->512 against one range, us a layer: 7x7 maps
// batch 16 +5.2, 64 +1.5; 6x6 batch 22 +5.1, 64 +5.3 (an accumulator per range in one CTA); 4x4 batch 64 +4.5.  Two ranges lost in every
// one of these (+0.7 to +9.9), three gave nothing where four gained.
inline int tc_auto_ranges(int num_kb, long tiles_max, int sms) {
  const int per = (num_kb + 3) / 4;
  return tc_cluster_deep(tiles_max * 4, sms) && 3 * per < num_kb && 7.0 + 0.15 * per < 2.0 + 0.122 * num_kb ? 4 : 1;
}

// How the ranges of a layer run whose tiles, of bn filters, fit in one wave: true = one after the other on the one-wave kernel, an
// accumulator for each, false = as a cluster of CTAs per tile.  The bits are the same.  Measured with four ranges, us a layer in a chain
// of launches, 3x3 layers on 2x2 to 7x7 maps of 1 to 64 samples, one wave against cluster:
//   72 K blocks 7.4 to 9.6 against 9.1 to 10.2, 108: 10.8 against 11.4, 144: 14.2 against 13.7 to 14.0, 216: 20.3 against 18.4,
//   288: 27.3 against 23.7, hence about 1.4 + 0.088 a block and 4.3 + 0.27 a block of a range.
// Half of tensor memory at most: the next kernel's CTA sets up beside this one.
inline bool tc_wave_ranges(int num_kb, int ranges, int bn) {
  return bn <= 64 && ranges * bn <= 256 && 1.4 + 0.088 * num_kb <= 4.3 + 0.27 * ((num_kb + ranges - 1) / ranges);
}

}  // namespace ee
