// How many ranges the K loop of a tensor-core convolution is cut into when nobody sets the number (conv_tc.cuh).  Plain arithmetic,
// for the plan and for host tests.
#pragma once

namespace ee {

// A cluster of CTAs per tile runs with the deep operand ring, whose CTA owns its SM, while the grid leaves a quarter of the SMs
// free: a cluster needs all its CTAs inside one GPC, and the last clusters of a fuller grid wait for a second wave.
inline bool tc_cluster_deep(long ctas, int sms) { return ctas * 4 <= 3L * sms; }

// num_kb: K blocks of the layer.  tiles_max: its output tiles at max_batch.  The ranges fix how every sum is grouped, so they
// depend on the layer and max_batch and never on the batch that runs: the cut has to pay at every batch, and is taken only
// where even max_batch runs as deep clusters.  There both routes are one wave, and a layer took, in a chain of launches, with the one-wave
// kernel of 128-pixel tiles that this cut was chosen for (us; 3x3 layers of the ResNet-50-shaped network's third and fourth stage, 36 and
// 72 K blocks; with the tiles that kernel has now, tc_wave_ranges says how such a layer's ranges run):
//   whole, on the one-wave kernel                  6.4, 10.8: 2.0 + 0.122 a block
//   four ranges, a CTA of a cluster for each       8.4,  9.7: 7.0 + 0.15 a block of a range
// so four pay from about 60 blocks on (3x3 layers on 7x7 maps of 1 to 16 samples, four against one: 54 blocks +0.4 us, 63 -0.7,
// 90 -2.9, 144 -7.2; with 64 filters 72 blocks -3.5).  Past the deep clusters they lose at every size: 3x3 512->512, four ranges against one,
// us a layer: 7x7 maps batch 8 -0.5, 16 +5.2, 64 +1.5; 6x6 batch 16 -0.5, 22 +5.1, 64 +5.3 (an accumulator per range in one CTA);
// 4x4 batch 48 -0.3, 64 +4.5; 3x3 and 2x2 -0.3 to -1.4 up to 64.  Two ranges lost in every one of these (+0.7 to +9.9), three
// gave nothing where four gain (-0.7 to +0.6).
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
