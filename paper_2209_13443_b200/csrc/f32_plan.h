// Tile and K cut of the fp32 model's convolutions (conv_f32.cuh).  Plain arithmetic, for the plan and for host tests.
#pragma once

namespace ee {

inline long f32_div(long a, long b) { return (a + b - 1) / b; }

struct F32Plan {
  int tile = 0;    // 0: 64 x 32, one K group; 1: 64 x 64, two; 2: 32 x 32, eight; 3: 16 x 32, eight
  int z = 1;       // CTAs of a cluster that share a tile's K
};

// K range of a CTA of the cluster: equal numbers of 16-wide steps, the unit the K groups take in turn, the last one shorter.  A ring
// stage at a range's end may be short.  (In whole stages of 128 the cut of K = 1152 over four CTAs, or of 2304 over eight, was
// three stages each and none for the last CTA, or the last two.)
inline int f32_k_per(int k, int z) { return (int)f32_div(f32_div(k, 16), z) * 16; }

// Tile and cluster size of a layer, from its geometry and max_batch.  Short K: one K group, larger tiles.  So too K up to 256 whose
// channels are copied one by one (!vec: stems on 3 channels), where addresses and copies of a row are the cost and a 64 x 32 tile has the
// fewest: 7x7 on 64 x 64 x 3, batch 6 24.3 us as 32 x 32 tiles, 11.9 so; a pass of that model 436 -> 422.  Grids of two waves of 64 x 64 tiles: that tile reads its operands least.
// Everything else has idle SMs: small tiles (16 rows where the layer never has more than 32), eight K groups, and as many CTAs per tile (up to 8) as keep the grid within
// two CTAs per SM while every CTA still has 64 of K, a 16-wide step for half its groups, and the last one any.  That line at 256 / 128 / 64 / 32, us a pass,
// nobody leaving: tiny model at 32 px, batch 1 60.5 / 57.1 / 53.6 / 53.7, batch 8 64.1 / 61.6 / 58.0 / 58.1, at 40 px, batch 8 67.7 / 65.4 / 67.7 / 67.7; ResNet-50-shaped
// model of batch 1 at 33 px 278 / 265 / 271 / 283, of 4 at 48 px 426 / 396 / 406 / 415, of 2 at 64 px 337 / 337 / 346 / 353, of 6 at 64 px 484 / 467 / 467 / 467.
inline F32Plan f32_plan(long m_max, int n, int k, int sms, bool vec = true) {
  F32Plan p;
  if (k < (vec ? 128 : 256)) return p;
  if (f32_div(m_max, 64) * f32_div(n, 64) >= 2L * sms) {
    p.tile = 1;
    return p;
  }
  p.tile = m_max <= 32 ? 3 : 2;   // 17 to 32 rows are two 16-row tiles: the same products, and half of them once samples have left
  const long tiles = f32_div(m_max, p.tile == 3 ? 16 : 32) * f32_div(n, 32);
  while (p.z < 8 && tiles * p.z * 2 <= 2L * sms && k >= p.z * 2 * 64 && f32_k_per(k, p.z * 2) * (p.z * 2L - 1) < k) p.z *= 2;
  return p;
}

}  // namespace ee
