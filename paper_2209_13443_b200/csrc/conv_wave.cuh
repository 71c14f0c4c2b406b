// Convolution tiles of grids with at most one tile per SM (small batches, the 14x14 and 7x7 maps): BM pixels x BN filters per
// CTA, the first of 64 x 32, 64 x 64, 128 x 32, 128 x 64 and 128 x 128 whose tiles fit in one wave.
//
// Such a layer is a chain of latencies: first operands (600 ns), the K loop of one tile, its epilogue, and about 1 us until the
// next launch may go on.  What this kernel does about them (clocks measured on one SM):
//  - The tensor core reads both operands at 128 bytes a clock, so a K block's four MMAs take BM + BN clocks and a few more (64 x 32:
//    110, 64 x 64: 133, 128 x 32: 162, 128 x 64: 194, 128 x 128: 257); TMA writes a 128-byte row a clock beside them.  Hence
//    small tiles first.  At 128 x 32 alone the 3x3 512 -> 512 layer on one 7x7 map took 10.6 us, at 64 x 32 10.4: another bound.
//  - That bound was the thread behind the MMAs: every wait on a barrier costs it about 100 clocks, whether the data is there or not, so a
//    K block with a wait of its own took 212 clocks at 64 x 32, with one MMA in place of four as well.  kG K blocks share a full
//    barrier (their slots are still given back one by one): 212 -> 140 clocks at two, 128 at four; 128 x 64 and 128 x 128 tiles, which
//    are bound by the MMAs and by the few slots that fit, lose from it (3x3 256 -> 256, batch 30: 9.3, 9.7 at two, 13.8 at four).
//  - A K block goes round the ring in about 1900 clocks (its loads 1100, its MMAs and their commit, the feeding thread), so the
//    K loop's pace is also that over the number of slots: all of shared memory is ring when the loop is long, and a small tile has
//    more slots (16 of 12 KB at 64 x 32, 6 of 32 KB at 128 x 128).
//  - Weights and activations have two feeding warps each, three at 64 x 32: a thread takes 140 to 280 clocks from one request to its
//    next, and that tile's MMAs a K block every 128 (3x3 512 -> 512, batch 1: 8.7 us with two, 7.2 with three; four gain nothing).
//  - The MMA thread asks for the next group's barrier before it issues this one's MMAs: the answer is there when it gets to it.
//  - Tensor memory is given back as soon as the accumulators are in registers, and every warp leaves when it is done: nobody waits for
//    the stores (0.1 us a launch).
//  - 32 or 64 columns per epilogue warp (four warps with 128 columns each took 2800 clocks, these take 700 or 1400).  The
//    residual's rows come to registers while the K loop runs.
// Bits are those of the other kernels: the same K order, one accumulator per output, one rounding.
// In a chain of launches, 128-pixel tiles and a wait per K block -> now, us: 3x3 512 -> 512 on 7x7, batch 1 10.6 -> 7.2; 3x3 256 -> 256
// on 14x14, batch 1 6.3 -> 4.6, batch 7 6.8 -> 5.7; 1x1 2048 -> 512, batch 1 5.8 -> 4.3; 1x1 512 -> 128 on 28x28 2.9 -> 2.4.
//
// PROJ: the residual operand is a 1x1 projection computed into a second accumulator (see the persistent kernel of conv_tc.cuh).
// RANGES: the layer's sums are cut into p.ranges ranges of K (conv_ranges.h); each has an accumulator, added in ascending order at the end.
#pragma once
#include "conv_tc.cuh"

namespace ee {

template <int BM, int BN>
struct WaveSmem {
  static constexpr int kEpiWarps = BN == 32 ? 4 : 8;
  static constexpr int kFeed = BM == 64 && BN == 32 ? 3 : 2;   // feeding warps of each operand
  static constexpr int kMma = 2 * kFeed, kEpi = kMma + 1;   // warps: weights, activations, MMA, then the epilogue
  static constexpr int kThreads = 32 * (kEpi + kEpiWarps);
  static constexpr int kG = BM == 64 ? (BN == 32 ? 4 : 2) : BN == 32 ? 2 : 1;   // K blocks per full barrier
  static constexpr int kABytes = BM * kTcBK * 2, kBBytes = BN * kTcBK * 2, kSlot = kABytes + kBBytes;
  static constexpr int kMaxSlots = (BM == 64 ? (BN == 32 ? 18 : 13) : BN == 32 ? 11 : BN == 64 ? 9 : 6) / kG * kG;
  static constexpr int kWarpRows = BM / 4;                  // pixels per epilogue warp: at 64 pixels a TMEM lane quarter holds 16 of them
  static_assert(kEpiWarps * kWarpRows * 64 <= kSlot, "output staging: 64 bytes per pixel of an epilogue warp in the drained first slot");
  static constexpr int kBars = 2 * kMaxSlots + 1, kTapsOff = (kBars * 8 + 4 + 15) / 16 * 16;   // barriers, the TMEM address, taps
  static constexpr int bytes(int slots) { return slots * kSlot + 4 * BN * 4 + kTapsOff + 256 + 1024; }   // + scale/bias, barriers, taps, alignment slack
  static_assert(bytes(kMaxSlots) <= 227 * 1024, "exceeds the shared memory of an SM");
};

template <int BM, int BN, bool PROJ, bool RANGES>
__global__ void __launch_bounds__(WaveSmem<BM, BN>::kThreads, 1)
conv_wave_tcgen05_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
                         const __grid_constant__ CUtensorMap tmA2, const __grid_constant__ CUtensorMap tmW2, TcParams p) {
  using S = WaveSmem<BM, BN>;
  constexpr int R = S::kMaxSlots;
  extern __shared__ uint8_t smem_raw[];
  const int ring = p.ring;   // slots, <= R
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  float* s_sb = reinterpret_cast<float*>(gen + ring * S::kSlot);      // scale | bias | scale2 | bias2
  uint64_t* bars = reinterpret_cast<uint64_t*>(gen + ring * S::kSlot + 4 * BN * 4);
  const uint32_t bar0 = base + (uint32_t)(ring * S::kSlot + 4 * BN * 4);
  auto full_bar = [&](int s) { return bar0 + 8u * (s / S::kG); };   // of the group that slot s belongs to
  auto empty_bar = [&](int s) { return bar0 + 8u * (R + s); };
  const uint32_t accum_bar = bar0 + 8u * (2 * R);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * R + 1);
  uint32_t* taps = reinterpret_cast<uint32_t*>(gen + ring * S::kSlot + 4 * BN * 4 + S::kTapsOff);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = (p.rev ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x) * BM, n0 = blockIdx.y * BN;
  const int num_kb1 = p.taps * p.cblocks, num_kb = num_kb1 + (PROJ ? p.cblocks2 : 0);
  uint32_t cols = PROJ ? 2 * BN : BN;   // accumulators, fp32 columns
  if (RANGES)
    while ((int)cols < p.ranges * BN) cols *= 2;

  if (threadIdx.x < 2 * R + 1) {
    mbar_init(bar0 + 8u * threadIdx.x, threadIdx.x < R ? 2 * S::kG : 1);   // full: an expect_tx each of weights and activations per K block
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == S::kEpi && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
    if (PROJ) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA2) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW2) : "memory");
    }
  }
  tap_table_fill(taps, p.kh, p.kw, p.stride);
  if (warp == S::kMma) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp < S::kMma) {
    // K blocks h, h + kFeed, ...: walked by counters (slot and phase, channel block x 64, position in the tap table)
    constexpr int F = S::kFeed;
    const int h = warp % F, dc = p.taps == 1 ? F * kTcBK : 0, dt = p.taps == 1 ? 0 : F;
    int i = h, s = h, c = p.taps == 1 ? h * kTcBK : 0, t = p.taps == 1 ? 0 : h;
    uint32_t ph = 1;
    while (t >= p.taps) t -= p.taps, c += kTcBK;
    auto step = [&] {
      i += F, c += dc, t += dt;
      while (t >= p.taps) t -= p.taps, c += kTcBK;
      if ((s += F) >= ring) s -= ring, ph ^= 1u;
    };
    // the last group may be short: whoever feeds its last block arrives for the missing ones
    auto fill = [&] {
      if (S::kG > 1 && h == (num_kb - 1) % F && num_kb % S::kG) {
        const uint32_t bar = full_bar((num_kb - 1) % ring);
        for (int k = num_kb % S::kG; k < S::kG; ++k) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
      }
    };
    if (warp < F) {
      if (elect_one()) {
        // no kernel writes weights: nothing to wait for but a free slot
        for (; i < num_kb; step()) {
          if (i >= ring && !mbar_wait(empty_bar(s), ph, p.err_flag)) break;
          mbar_expect_tx(full_bar(s), S::kBBytes);
          const uint32_t dst = base + (uint32_t)(s * S::kSlot + S::kABytes);
          if (PROJ && i >= num_kb1)
            tma_load_3d(dst, &tmW2, full_bar(s), (i - num_kb1) * kTcBK, 0, n0);
          else
            tma_load_3d(dst, &tmW, full_bar(s), c, (int)(taps[t] >> 16), n0);
        }
        if (i >= num_kb) fill();
      }
      __syncwarp();
      asm volatile("griddepcontrol.wait;" ::: "memory");
    } else {
      int cw = 0, ch = 0, cn = 0, cw2 = 0, ch2 = 0;
      if (p.im2col || (PROJ && p.im2col2)) {
        const int hw = p.Ho * p.Wo;
        cn = m0 / hw;
        const int rem = m0 - cn * hw, ho = rem / p.Wo, wo = rem - ho * p.Wo;
        cw = wo * p.stride - p.pad_w, ch = ho * p.stride - p.pad;
        if (PROJ) cw2 = wo * p.stride2, ch2 = ho * p.stride2;
      }
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (elect_one()) {
        bool ok = true;
        if (p.im2col) {
          for (; i < num_kb1; step()) {
            const uint32_t tap = taps[t];
            ok = i < ring || mbar_wait(empty_bar(s), ph, p.err_flag);
            if (!ok) break;
            mbar_expect_tx(full_bar(s), S::kABytes);
            tma_load_im2col_4d(base + (uint32_t)(s * S::kSlot), &tmA, full_bar(s), c, cw, ch, cn, (uint16_t)(tap & 255u), (uint16_t)(tap >> 8 & 255u));
          }
        } else {
          for (; i < num_kb1; step()) {
            ok = i < ring || mbar_wait(empty_bar(s), ph, p.err_flag);
            if (!ok) break;
            mbar_expect_tx(full_bar(s), S::kABytes);
            tma_load_2d(base + (uint32_t)(s * S::kSlot), &tmA, full_bar(s), c, m0);
          }
        }
        if (PROJ) {
          for (; ok && i < num_kb; step()) {
            if (i >= ring && !mbar_wait(empty_bar(s), ph, p.err_flag)) break;
            mbar_expect_tx(full_bar(s), S::kABytes);
            if (p.im2col2)
              tma_load_im2col_4d(base + (uint32_t)(s * S::kSlot), &tmA2, full_bar(s), (i - num_kb1) * kTcBK, cw2, ch2, cn, (uint16_t)0, (uint16_t)0);
            else
              tma_load_2d(base + (uint32_t)(s * S::kSlot), &tmA2, full_bar(s), (i - num_kb1) * kTcBK, m0);
          }
        }
        if (i >= num_kb) fill();
      }
      __syncwarp();
    }
  } else if (warp == S::kMma) {
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc(BN, BM);
      constexpr int G = S::kG;
      const uint64_t da0 = umma_desc(base), db0 = umma_desc(base + S::kABytes);
      bool ok = true;
      int s = 0, i = 0;
      uint32_t ph = 0;
      uint32_t range_acc = tmem_base;   // RANGES: accumulator of the open range
      int in_range = 0;                 // its blocks so far
      auto block = [&](int i, int s) {
        const uint64_t off = (uint64_t)(s * (S::kSlot >> 4));
        if (RANGES) {
          if (in_range == p.kb_per) in_range = 0, range_acc += (uint32_t)BN;
          umma_block(range_acc, da0 + off, db0 + off, idesc, in_range != 0);
          ++in_range;
        } else {
          umma_block(tmem_base + (PROJ && i >= num_kb1 ? (uint32_t)BN : 0u), da0 + off, db0 + off, idesc, i != 0 && !(PROJ && i == num_kb1));
        }
      };
      bool here = mbar_test_wait(full_bar(0), 0);
      for (; i + G <= num_kb; i += G) {
        if (!here) ok = mbar_wait(full_bar(s), ph, p.err_flag);
        if (!ok) break;
        const int cur = s;
        if ((s += G) == ring) s = 0, ph ^= 1u;
        here = mbar_test_wait(full_bar(s), ph);   // behind the last group: a phase that nobody waits for
#pragma unroll
        for (int k = 0; k < G; ++k) {
          block(i + k, cur + k);
          umma_commit(empty_bar(cur + k));
        }
      }
      if (ok && i < num_kb) {   // a short group: its slots are not used again
        if (!here) ok = mbar_wait(full_bar(s), ph, p.err_flag);
        for (; ok && i < num_kb; ++i, ++s) block(i, s);
      }
      if (ok) umma_commit(accum_bar);   // everything before it has read its operands as well
    }
    __syncwarp();
    asm volatile("bar.sync 2, %0;" ::"n"(32 * (S::kEpiWarps + 1)) : "memory");   // every epilogue warp has read its part
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cols) : "memory");
  } else {
    const int et = threadIdx.x - 32 * S::kEpi;
    for (int i = et; i < BN; i += 32 * S::kEpiWarps) {
      const bool in = n0 + i < p.N;
      s_sb[i] = (p.scale && in) ? p.scale[n0 + i] : 1.f;
      s_sb[BN + i] = (p.bias && in) ? p.bias[n0 + i] : 0.f;
      if (PROJ) {
        s_sb[2 * BN + i] = (p.scale2 && in) ? p.scale2[n0 + i] : 1.f;
        s_sb[3 * BN + i] = (p.bias2 && in) ? p.bias2[n0 + i] : 0.f;
      }
    }
    asm volatile("bar.sync 1, %0;" ::"n"(32 * S::kEpiWarps) : "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    constexpr int kCover = BN == 128 ? 64 : 32, kSteps = kCover / 32;   // columns of a warp, in steps of 32
    const int q = warp & 3, half = et >> 7, m = lane < S::kWarpRows ? m0 + q * S::kWarpRows + lane : p.M;
    uint4 r[4 * kSteps];
#pragma unroll
    for (int g = 0; g < 4 * kSteps; ++g) {
      const int n = n0 + half * kCover + g * 8;
      r[g] = make_uint4(0u, 0u, 0u, 0u);
      if (!PROJ && p.residual && m < p.M && n < p.N) r[g] = *reinterpret_cast<const uint4*>(p.residual + (size_t)m * p.N + n);
    }
    const bool ok = __all_sync(0xffffffffu, mbar_wait(accum_bar, 0, p.err_flag));
    bool read = false;   // this warp's part of the accumulator is in registers: the MMA warp may free it, nobody waits for the stores
    auto free_tmem = [&] {
      if (!read) {
        tc_fence_before();
        asm volatile("bar.arrive 2, %0;" ::"n"(32 * (S::kEpiWarps + 1)) : "memory");
        read = true;
      }
    };
    if (ok) {
      tc_fence_after();
      uint8_t* stage = gen + (warp - S::kEpi) * (S::kWarpRows * 64);   // rows of 64 bytes, their 16-byte chunks XORed with the row
#pragma unroll
      for (int st = 0; st < kSteps; ++st) {
        const int c0 = half * kCover + st * 32;
        if (n0 + c0 >= p.N) break;
        const uint32_t acc = tmem_base + (uint32_t)c0 + ((uint32_t)(q * 32) << 16);
        float v[32];
        uint4 o[4];
        if (PROJ) {   // rounded to bf16 as the projection's own layer would store it
          float w[32];
          tmem_ld32_issue(acc, v);
          tmem_ld32_issue(acc + (uint32_t)BN, w);
          tmem_ld_wait(v, w);
          epilogue32<false>(p.act2, w, s_sb + 2 * BN + c0, s_sb + 3 * BN + c0, nullptr, r + 4 * st);
        } else {
          tmem_ld32(acc, v);
          if (RANGES)
            for (int g = 1; g < p.ranges; ++g) {   // the order of the cluster's reduction
              float w[32];
              tmem_ld32(acc + (uint32_t)(g * BN), w);
#pragma unroll
              for (int e = 0; e < 32; ++e) v[e] += w[e];
            }
        }
        if (st + 1 == kSteps) free_tmem();
        if (PROJ || p.residual)
          epilogue32<true>(p.act, v, s_sb + c0, s_sb + BN + c0, r + 4 * st, o);
        else
          epilogue32<false>(p.act, v, s_sb + c0, s_sb + BN + c0, nullptr, o);
        if (st) __syncwarp();
#pragma unroll
        for (int g = 0; g < 4; ++g)
          if (lane < S::kWarpRows) *reinterpret_cast<uint4*>(stage + lane * 64 + ((g ^ (lane >> 1 & 3)) << 4)) = o[g];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < S::kWarpRows / 8; ++k) {   // eight rows per store, four lanes with 64 bytes of each
          const int row = k * 8 + (lane >> 2), g = lane & 3, mm = m0 + q * S::kWarpRows + row, n = n0 + c0 + g * 8;
          const uint4 x = *reinterpret_cast<const uint4*>(stage + row * 64 + ((g ^ (row >> 1 & 3)) << 4));
          if (mm < p.M && n < p.N) *reinterpret_cast<uint4*>(p.out + (size_t)mm * p.N + n) = x;
        }
      }
    }
    free_tmem();
  }
}

inline ee_status_t wave_context_init() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kernel, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  auto tile = [&](auto s, auto... kernels) {
    typedef decltype(s) S;
    (set(kernels, S::bytes(S::kMaxSlots)), ...);
  };
  tile(WaveSmem<64, 32>{}, conv_wave_tcgen05_kernel<64, 32, false, false>, conv_wave_tcgen05_kernel<64, 32, true, false>, conv_wave_tcgen05_kernel<64, 32, false, true>);
  tile(WaveSmem<64, 64>{}, conv_wave_tcgen05_kernel<64, 64, false, false>, conv_wave_tcgen05_kernel<64, 64, true, false>, conv_wave_tcgen05_kernel<64, 64, false, true>);
  tile(WaveSmem<128, 32>{}, conv_wave_tcgen05_kernel<128, 32, false, false>, conv_wave_tcgen05_kernel<128, 32, true, false>, conv_wave_tcgen05_kernel<128, 32, false, true>);
  tile(WaveSmem<128, 64>{}, conv_wave_tcgen05_kernel<128, 64, false, false>, conv_wave_tcgen05_kernel<128, 64, true, false>, conv_wave_tcgen05_kernel<128, 64, false, true>);
  tile(WaveSmem<128, 128>{}, conv_wave_tcgen05_kernel<128, 128, false, false>, conv_wave_tcgen05_kernel<128, 128, true, false>);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

// Slots: as many as the K loop has blocks for; a short loop leaves room on its SM for the next layer's CTA to set up.
template <int BM, int BN, bool PROJ, bool RANGES = false>
inline cudaError_t wave_launch_t(cudaStream_t st, const CUtensorMap& a, const CUtensorMap& w, const CUtensorMap& a2, const CUtensorMap& w2, TcParams p) {
  using S = WaveSmem<BM, BN>;
  p.ring = std::min(S::kMaxSlots, cdiv(std::max(S::kFeed, p.taps * p.cblocks + (PROJ ? p.cblocks2 : 0)), S::kG) * S::kG);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cdiv(p.M, BM), cdiv(p.N, BN));
  cfg.blockDim = dim3(S::kThreads);
  cfg.dynamicSmemBytes = S::bytes(p.ring);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, conv_wave_tcgen05_kernel<BM, BN, PROJ, RANGES>, a, w, a2, w2, p);
}

// a, a2: maps whose boxes have t.bm rows, w, w2: boxes of t.bn filters.
template <bool PROJ>
inline cudaError_t wave_launch(WaveTile t, cudaStream_t st, const CUtensorMap& a, const CUtensorMap& w, const CUtensorMap& a2, const CUtensorMap& w2, const TcParams& p) {
  if constexpr (!PROJ)
    if (p.ranges > 1) {
      if (t.bm == 64) return t.bn == 32 ? wave_launch_t<64, 32, false, true>(st, a, w, a2, w2, p) : wave_launch_t<64, 64, false, true>(st, a, w, a2, w2, p);
      return t.bn == 32 ? wave_launch_t<128, 32, false, true>(st, a, w, a2, w2, p) : wave_launch_t<128, 64, false, true>(st, a, w, a2, w2, p);
    }
  if (t.bm == 64) return t.bn == 32 ? wave_launch_t<64, 32, PROJ>(st, a, w, a2, w2, p) : wave_launch_t<64, 64, PROJ>(st, a, w, a2, w2, p);
  return t.bn == 32   ? wave_launch_t<128, 32, PROJ>(st, a, w, a2, w2, p)
         : t.bn == 64 ? wave_launch_t<128, 64, PROJ>(st, a, w, a2, w2, p)
                      : wave_launch_t<128, 128, PROJ>(st, a, w, a2, w2, p);
}

}  // namespace ee
