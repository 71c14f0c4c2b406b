// How the FC layer of an exit head is cut over CTAs (fc_cluster_kernel, head.cuh).  Plain arithmetic, for the launch and for host
// tests.
#pragma once
#include <stddef.h>

#include <algorithm>

namespace ee {

constexpr int kFcMaxSmem = 226 * 1024;   // dynamic; the scan's static arrays come on top
constexpr int kFcThreads = 256, kFcRing = 4, kFcBlocks = 16, kFcRows = 8, kFcSlot = kFcRows * 512;

struct FcShape {
  int S, CL;     // samples per tile, CTAs per tile
  int cluster;   // 1: the CTAs of a tile are a cluster; 0: they exchange through global memory (or CL is 1)
  int kb;        // classes per block
  int Cp;        // channels rounded up to whole ring slots
};
inline size_t fc_smem_bytes(const FcShape& f) {
  return (size_t)(kFcThreads / 32) * kFcRing * kFcSlot + (size_t)f.S * f.Cp * 4 + (size_t)f.S * (kFcBlocks / f.CL) * f.kb * 4 +
         (size_t)kFcBlocks * f.S * 16 + (kFcThreads / 32) * kFcRing * 8;
}
// 64 classes per CTA (clusters of 16 need the non-portable size), fewer CTAs for few classes.  Samples per tile: the fewest
// whose clusters run side by side (`room16` clusters of 16: not every GPC has 16 SMs), up to 8, as a second wave costs the
// whole kernel once more; past that the same tiles without clusters, 128 CTAs for 64 samples.  What bounds a CTA is then
// its FMAs and its shared memory, which every weight crosses twice per tile.  Many channels or classes: as many samples as
// the pooled tile and its logits leave shared memory for.  Nothing here changes a sum.  Pooling + FC of bf16 heads of 1000
// classes, batch 1 / 8 / 27 / 64, us: 4096 channels (tiles of four) 14.5 / 17 / 22 / 41 against 43 / 63 / 71 / 129 of fc_kernel, 8192
// (two) 22.5 / 27 / 50 / 95 against 79 / 119 / 133 / 244, 16384 (one) 39 / 42 / 116 / 262 against 148 / 234 / 242 / 476.
inline FcShape fc_shape(int B, int C, int K, int elem_bytes, int room16) {
  FcShape f;
  f.CL = 1;
  while (f.CL < 16 && f.CL * 64 < K) f.CL *= 2;
  f.kb = ((K + kFcBlocks - 1) / kFcBlocks + kFcRows - 1) / kFcRows * kFcRows;
  const int chunk = 512 / elem_bytes;
  f.Cp = (C + chunk - 1) / chunk * chunk;
  const int room = std::max(1, room16 * (16 / f.CL)), most = elem_bytes == 4 ? 4 : 8;   // eight fp64 sums per class do not fit the registers
  f.S = B <= room ? 1 : B <= 2 * room ? 2 : B <= 4 * room ? 4 : most;
  while (f.S > 1 && fc_smem_bytes(f) > (size_t)kFcMaxSmem) f.S /= 2;
  f.cluster = f.CL > 1 && ((B + f.S - 1) / f.S <= room || f.CL < 16);
  return f;
}
// A tile of one sample fits: the kernel takes the head at every batch.
inline bool fc_fits(int C, int K, int elem_bytes) { return fc_smem_bytes(fc_shape(1, C, K, elem_bytes, 1)) <= (size_t)kFcMaxSmem; }

}  // namespace ee
