// How the FC layer of an exit head is cut over CTAs (fc_cluster_kernel, head.cuh).  Plain arithmetic, for the launch and for host
// tests.
#pragma once
#include <stddef.h>

#include <algorithm>

namespace ee {

constexpr int kFcMaxSmem = 226 * 1024;   // dynamic; the scan's static arrays come on top
constexpr int kFcThreads = 256, kFcBlocks = 16, kFcRows = 8, kFcSlot = kFcRows * 512;
constexpr int kFcPoolSmem = kFcThreads * 32;   // partial sums of a kernel that pools as well: eight floats or four doubles a thread

struct FcShape {
  int S, CL;     // samples per tile, CTAs per tile
  int cluster;   // 1: the CTAs of a tile are a cluster; 0: they exchange through global memory (or CL is 1)
  int kb;        // classes per block
  int Cp;        // channels rounded up to whole ring slots
  int ws;          // warps that share a group of eight classes, each with every ws-th slot of its channels
  int ring;      // slots per warp, 2 to 6: what it walks and one, as far as they fit.  Slots that nobody uses would keep the kernel from
                 // its SM until the pooling kernel has left (37 samples of 28x28x512, two slots a warp: 15.7 us with six, 15.0 with four)
};
#ifdef __CUDACC__
__host__ __device__
#endif
inline size_t fc_smem_bytes(const FcShape& f) {
  return (size_t)(kFcThreads / 32) * f.ring * kFcSlot + (size_t)f.S * f.Cp * 4 + (size_t)f.S * (kFcBlocks / f.CL) * f.kb * 4 * (f.ws > 1 ? 1 + 2 * f.ws : 1) +
         (size_t)kFcBlocks * f.S * 16 + (kFcThreads / 32) * f.ring * 8 + 32;
}
// 64 classes per CTA (clusters of 16 need the non-portable size), fewer CTAs for few classes.  Samples per tile: the fewest
// whose clusters run side by side (`room16` clusters of 16: not every GPC has 16 SMs), up to 8, as a second wave costs the
// whole kernel once more; past that the same tiles without clusters, 128 CTAs for 64 samples.  What bounds a CTA is then
// its FMAs and its shared memory, which every weight crosses twice per tile.  Many channels or classes: as many samples as
// the pooled tile and its logits leave shared memory for.  None of these changes a sum.  Pooling + FC of bf16 heads of 1000
// classes, batch 1 / 8 / 27 / 64, us: 4096 channels (tiles of four) 14.5 / 17 / 22 / 41 against 43 / 63 / 71 / 129 of fc_kernel, 8192
// (two) 22.5 / 27 / 50 / 95 against 79 / 119 / 133 / 244, 16384 (one) 39 / 42 / 116 / 262 against 148 / 234 / 242 / 476.
// Few classes on many channels: a warp that walks all the channels of eight classes is a chain of slots, 0.6 us each, beside idle
// SMs and idle warps, so models of up to 32 samples give a tile at least eight CTAs, and warps without classes of their own share
// one's channels (a sum then has their shares added in ascending order: how depends on C, K and max_batch only).  fp32, 100
// classes, batch 4: 512 / 1024 / 2048 channels 8.6 / 11.0 / 15.7 -> 6.3 / 6.8 / 8.3 us; batch 30, 2048: 16.5 -> 11.3.  At batch 64 the
// clusters no longer run side by side and lose (17 -> 20).
inline FcShape fc_shape(int B, int C, int K, int elem_bytes, int room16, int max_batch = 1 << 30) {
  FcShape f;
  f.CL = 1;
  const int chunk = 512 / elem_bytes, nchunk = (C + chunk - 1) / chunk;
  while (f.CL < 16 && f.CL * 64 < K) f.CL *= 2;
  if (nchunk >= 4 && max_batch <= 32) f.CL = std::max(f.CL, 8);
  f.kb = ((K + kFcBlocks - 1) / kFcBlocks + kFcRows - 1) / kFcRows * kFcRows;
  f.Cp = nchunk * chunk;
  f.ws = 1;
  while (f.ws < kFcThreads / 32 && f.ws * 2 <= nchunk && f.ws * 2 * (kFcBlocks / f.CL) * f.kb <= kFcThreads / 32 * kFcRows) f.ws *= 2;
  f.ring = 4, f.S = 1;
  while (f.ws > 1 && fc_smem_bytes(f) > (size_t)kFcMaxSmem) f.ws /= 2;
  const int room = std::max(1, room16 * (16 / f.CL)), most = elem_bytes == 4 ? 4 : 8;   // eight fp64 sums per class do not fit the registers
  f.S = B <= room ? 1 : B <= 2 * room ? 2 : B <= 4 * room ? 4 : most;
  while (f.S > 1 && fc_smem_bytes(f) > (size_t)kFcMaxSmem) f.S /= 2;
  const int side = kFcThreads / 32 / f.ws, groups = kFcBlocks / f.CL * f.kb / kFcRows, slots = (groups + side - 1) / side * ((nchunk + f.ws - 1) / f.ws);
  for (f.ring = std::min(6, slots + 1); f.ring > 4 && fc_smem_bytes(f) > (size_t)kFcMaxSmem;) --f.ring;
  f.cluster = f.CL > 1 && ((B + f.S - 1) / f.S <= room || f.CL < 16);
  return f;
}
// The FC kernel pools as well: tiles of one CTA and one sample whose channel vectors fit side by side in its threads (`lanes` of
// them).  One pass over a small map costs less than a launch and a trip through global memory; a second pass costs more.  Head of
// fp32 maps, 10 classes, batch 8, with a pooling kernel / without, us: 16x16x16 7.8 / 6.4, 16x16x64 (one pass) 7.3 / 6.4, 32x32x16 8.2 / 6.8,
// 16x16x256 (four passes, batch 1) 7.3 / 10.9, 32x32x64 7.9 / 13.4; bf16 28x28x64, batch 64: 7.7 / 7.3.
inline bool fc_pools(const FcShape& f, int vectors, int lanes) {
  return f.CL == 1 && f.S == 1 && vectors <= lanes && fc_smem_bytes(f) + kFcPoolSmem <= (size_t)kFcMaxSmem;
}
// A tile of one sample fits: the kernel takes the head at every batch.
inline bool fc_fits(int C, int K, int elem_bytes) { return fc_smem_bytes(fc_shape(1, C, K, elem_bytes, 1)) <= (size_t)kFcMaxSmem; }

}  // namespace ee
