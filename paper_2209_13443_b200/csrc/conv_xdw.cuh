// Expand and depthwise layer of an inverted-residual block in one launch (bf16): a 1x1 convolution to the block's hidden channels on
// tcgen05.mma, whose output only the 3x3 pad-1 depthwise layer behind it reads, stays in shared memory.
//
// The hidden map is the block's largest tensor, six times its input.  Apart, the first layer writes it and the second reads it back
// (77 MB each way for 32 images of 112 x 112 x 96); on the small maps, where neither layer has work for more than a microsecond, it costs a launch.
// A CTA owns a block of up to 64 hidden channels (the 1x1 weights stay in shared memory, the depthwise ones in registers) and walks bands
// of output rows over all columns.  Per band the TMA unit brings the framed input rows (coordinates from -1, zero fill) as one
// [rows][W + 2] run of positions, 128 bytes a K block, which is the A operand as it lies; tiles of 128 positions are multiplied into
// as many accumulators; eight warps finish them (scale, bias, activation, one rounding to bf16; zeros outside the image, where the
// depthwise layer's padding is) into shared memory, meet at a barrier and run the depthwise layer on it as conv_dw.cuh does.  While they
// do, the next band's input is loaded and multiplied.  The frame is computed again by the neighbouring band: two rows of each.
// What bounds it: the eight workers, two a scheduler, which finish a band and then filter it, one after the other: about 2000
// clocks each on a 16 x 16 frame of 64 channels, the MMAs 400.  (Fetching narrow pixels by threads in place of TMA: 40.7 -> 42.6 us on
// 56 x 56 x 144, batch 32.)
// Each output sums the same products in the same K steps as the two layers apart, with the same roundings: the same bits.  (Beside this
// launch a 1x1 layer groups its pixels, conv_tc.cuh, only where a pixel's channels are part of one K step or whole ones.)
#pragma once
#include "conv_dw.cuh"

namespace ee {

struct XdwParams {
  int H, W, Ho, Wo, C;       // maps before and behind the depthwise layer, hidden channels
  int RB, bands, tiles;      // output rows of a band, bands of an image, bands of the batch
  int cb;                    // hidden channels of a block (dw_block_channels)
  int cin, kblocks;
  int positions, mtiles;     // (rows of a band's frame) * (W + 2), in tiles of 128
  int slots;                 // bands of input in flight
  int magic;                 // ceil(2^20 / (W + 2)): position * magic >> 20 is its row of the frame
  int act1, act2;
  int rev;
  const float* scale1;
  const float* bias1;
  const bf16* w;             // depthwise weights [C][3][3]
  const float* scale2;
  const float* bias2;
  bf16* y;
  int* err_flag;
};

constexpr int kXdwThreads = 320, kXdwMaxTiles = 8, kXdwMaxKb = 3;   // producer, MMA, eight workers

struct XdwSmem {   // byte offsets behind the aligned base
  int x_off, slot, h_off, pitch, sb_off, bar_off, bytes;
};
inline XdwSmem xdw_smem(int cb, int kblocks, int positions, int slots) {
  XdwSmem s;
  const int mtiles = (positions + 127) / 128;
  s.x_off = kblocks * 64 * 128;
  s.slot = kblocks * mtiles * 128 * 128;
  s.h_off = s.x_off + slots * s.slot;
  s.pitch = cb * 2 + 16;   // eight positions of a store or load phase in different banks
  s.sb_off = s.h_off + ((positions + kDwOver) * s.pitch + 127) / 128 * 128;   // strips read past the last row of the frame
  s.bar_off = s.sb_off + 4 * 64 * 4;
  s.bytes = s.bar_off + 128 + 1024;
  return s;
}

template <int STRIDE>
__global__ void __launch_bounds__(kXdwThreads, 1)
conv_expand_dw_tcgen05_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, XdwParams p, XdwSmem S) {
  constexpr int P = kDwStrip;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  float* s_sb = reinterpret_cast<float*>(gen + S.sb_off);
  const uint32_t bar0 = base + S.bar_off, w_bar = bar0, acc_full = bar0 + 8, acc_empty = bar0 + 16;
  auto x_full = [&](int s) { return bar0 + 24u + 8u * s; };
  auto x_empty = [&](int s) { return bar0 + 40u + 8u * s; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + S.bar_off + 64);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int my_tiles = (int)blockIdx.x < p.tiles ? (p.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int c0 = (int)blockIdx.y * p.cb, Wc = p.W + 2;
  uint32_t cols = 64;
  while ((int)cols < p.mtiles * 64) cols *= 2;
  if (threadIdx.x == 0) {
    mbar_init(w_bar, 1);
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 8);   // lane 0 of each worker
    for (int s = 0; s < 2; ++s) mbar_init(x_full(s), 1), mbar_init(x_empty(s), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  auto band_of = [&](int j, int& b, int& band) {
    const int tf = (int)blockIdx.x + j * (int)gridDim.x, t = p.rev ? p.tiles - 1 - tf : tf;
    b = t / p.bands, band = t - b * p.bands;
  };

  if (warp == 0) {
    if (elect_one()) {
      mbar_expect_tx(w_bar, (uint32_t)(p.kblocks * 64 * 128));   // no kernel writes weights
      for (int k = 0; k < p.kblocks; ++k) tma_load_3d(base + (uint32_t)(k * 64 * 128), &tmW, w_bar, k * kTcBK, 0, c0);
      asm volatile("griddepcontrol.wait;" ::: "memory");
      int s = 0;
      uint32_t ph = 1;
      for (int j = 0; j < my_tiles; ++j) {
        int b, band;
        band_of(j, b, band);
        if (!mbar_wait(x_empty(s), ph, p.err_flag)) break;
        mbar_expect_tx(x_full(s), (uint32_t)(p.kblocks * p.positions * 128));
        for (int k = 0; k < p.kblocks; ++k)
          tma_load_4d(base + (uint32_t)(S.x_off + s * S.slot + k * p.mtiles * 16384), &tmX, x_full(s), k * kTcBK, -1, band * p.RB * STRIDE - 1, b);
        if (++s == p.slots) s = 0, ph ^= 1u;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = umma_idesc((p.cb + 15) / 16 * 16);
      const uint64_t da0 = umma_desc(base + S.x_off), db0 = umma_desc(base);
      bool ok = my_tiles > 0 ? mbar_wait(w_bar, 0, p.err_flag) : true;
      int s = 0;
      uint32_t ph = 0;
      for (int j = 0; j < my_tiles && ok; ++j) {
        ok = mbar_wait(x_full(s), ph, p.err_flag) && (j == 0 || mbar_wait(acc_empty, (uint32_t)(j - 1) & 1u, p.err_flag));
        if (!ok) break;
        tc_fence_after();
        for (int m = 0; m < p.mtiles; ++m)
          for (int k = 0; k < p.kblocks; ++k) {
            const uint64_t da = da0 + (uint64_t)((s * S.slot + (k * p.mtiles + m) * 16384) >> 4), db = db0 + (uint64_t)(k * 512);
            const int steps = min(4, (p.cin - k * kTcBK + 15) / 16);   // channels past Cin are zeros
            for (int i = 0; i < steps; ++i) umma_bf16(tmem_base + (uint32_t)(m * 64), da + 2 * i, db + 2 * i, idesc, (uint32_t)(k != 0 || i != 0));
          }
        umma_commit(acc_full);
        umma_commit(x_empty(s));
        if (++s == p.slots) s = 0, ph ^= 1u;
      }
    }
    __syncwarp();
  } else {
    const int tid = (int)threadIdx.x - 64, q = warp & 3, half = tid >> 7;
    for (int i = tid; i < 64; i += 256) {
      const bool in = i < p.cb && c0 + i < p.C;
      s_sb[i] = (p.scale1 && in) ? p.scale1[c0 + i] : 1.f;
      s_sb[64 + i] = (p.bias1 && in) ? p.bias1[c0 + i] : 0.f;
      s_sb[128 + i] = (p.scale2 && in) ? p.scale2[c0 + i] : 1.f;
      s_sb[192 + i] = (p.bias2 && in) ? p.bias2[c0 + i] : 0.f;
    }
    const int nv = p.cb >> 3;                 // channel vectors per block
    const int cvec = tid % nv, item0 = tid / nv, item_step = kDwConsumers / nv;
    const bool live = item0 < item_step;      // nv need not divide 256: the threads of the ragged tail idle
    const int c = c0 + cvec * 8;
    const bool c_in = c < p.C;
    f32x2 wf[9][4];
    dw_weights(p.w + (size_t)c * 9, c_in, wf);
    asm volatile("bar.sync 1, 256;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint8_t* hid = gen + S.h_off;
    const int strips = (p.Wo + P - 1) / P, items = p.RB * strips;
    for (int j = 0; j < my_tiles; ++j) {
      int b, band;
      band_of(j, b, band);
      // a warp whose wait ran out keeps the barriers' count; what it stores then is garbage, and the model's error word says so
      const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_full, (uint32_t)j & 1u, p.err_flag));
      tc_fence_after();
      const int h0 = band * p.RB * STRIDE - 1;
      for (int m = half; m < p.mtiles && ok; m += 2) {
        const int pos = m * 128 + q * 32 + lane, fr = pos * p.magic >> 20, fc = pos - fr * Wc;
        const bool inside = fc > 0 && fc <= p.W && (unsigned)(h0 + fr) < (unsigned)p.H;
        uint8_t* line = hid + pos * S.pitch;
        for (int n0 = 0; n0 < p.cb; n0 += 32) {
          float v[32];
          uint4 o[4];
          const uint32_t at = tmem_base + (uint32_t)(m * 64 + n0) + ((uint32_t)(q * 32) << 16);
          if (p.cb - n0 > 16) {
            tmem_ld32(at, v);
            epilogue32<false>(p.act1, v, s_sb + n0, s_sb + 64 + n0, nullptr, o);
          } else {
            tmem_ld16(at, v);
            o[0] = epilogue8_act<false>(p.act1, v, s_sb + n0, s_sb + 64 + n0, o[0]);
            o[1] = epilogue8_act<false>(p.act1, v + 8, s_sb + n0 + 8, s_sb + 72 + n0, o[1]);
          }
#pragma unroll
          for (int g = 0; g < 4; ++g)
            if (pos < p.positions && n0 + g * 8 < p.cb) *reinterpret_cast<uint4*>(line + n0 * 2 + g * 16) = inside ? o[g] : make_uint4(0u, 0u, 0u, 0u);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty) : "memory");   // the next band's MMAs may start
      asm volatile("bar.sync 1, 256;" ::: "memory");   // the hidden band is complete
      if (live) {
        for (int it = item0; it < items; it += item_step) {
          const int ro = it / strips, st = it - ro * strips, wo0 = st * P, ho = band * p.RB + ro;
          f32x2 acc[P][4];
          dw_strip<STRIDE>(hid + (ro * STRIDE * Wc + wo0 * STRIDE) * S.pitch + cvec * 16, S.pitch, Wc * S.pitch, wf, acc);
          if (c_in && ho < p.Ho) dw_store(p.y + (((size_t)b * p.Ho + ho) * p.Wo + wo0) * p.C + c, p.C, p.Wo - wo0, acc, s_sb + 128 + cvec * 8, p.act2);
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");   // read by everybody: the next band may be written over it
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(cols) : "memory");
  }
}

// Band height and slots of input for a batch; RB = 0: a band of one output row does not fit.  The busiest CTA's time, in clocks:
// accumulators two at a time (a worker warp has every other one), passes of the workers over a band's strips, and a band's hand-over.
struct XdwPlan {
  int RB = 0, slots = 1;
};
inline XdwPlan xdw_plan(int sm_count, int B, int W, int Ho, int Wo, int stride, int cin, int hidden) {
  const int cb = dw_block_channels(hidden), chunks = cdiv(hidden, cb), ctas = std::max(1, sm_count / chunks);
  const int strips = cdiv(Wo, kDwStrip), per_pass = kDwConsumers / (cb / 8), kblocks = cdiv(cin, kTcBK);
  XdwPlan best;
  long least = -1;
  for (int rb = 1; rb <= Ho; ++rb) {
    const int positions = ((rb - 1) * stride + 3) * (W + 2), mtiles = cdiv(positions, 128);
    if (mtiles > kXdwMaxTiles || (rb - 1) * stride + 3 > 256) break;
    int slots = 2;
    if (xdw_smem(cb, kblocks, positions, 2).bytes > 226 * 1024) slots = 1;
    if (xdw_smem(cb, kblocks, positions, slots).bytes > 226 * 1024) break;
    const long tiles = (long)B * cdiv(Ho, rb);
    const long cost = (long)cdiv(tiles, std::min<long>(tiles, ctas)) * (cdiv(mtiles, 2) * 500 + (long)cdiv((long)rb * strips, per_pass) * (stride == 1 ? 1100 : 1500) + (slots == 2 ? 500 : 1500));
    if (least < 0 || cost < least) least = cost, best.RB = rb, best.slots = slots;
  }
  return best;
}

// A 1x1 layer L and the depthwise layer D behind it, which alone reads its output.  A map's size decides, not the batch (see
// xdw_active).  Stages of the MobileNetV2-shaped network, apart -> together, us.  Maps of 28 x 28 to 7 x 7 (stages 2 to 4): batch 1
// 131 -> 121, 13 176 -> 164, 32 233 -> 233.  First stage (112 x 112 and 56 x 56): batch 1 45.7 -> 43.2, but 13 100 -> 107 and 32 187 -> 197,
// where the workers' chain, not memory, bounds the kernel; of 130 px images (65 x 65 and 33 x 33) batch 32 117 -> 105, 111 of it with the 33 x 33
// maps alone.  So up to 34 x 34.
constexpr int kXdwMaxMap = 1156;
inline bool xdw_supported(const ee_layer_desc_t& l, const ee_layer_desc_t& d, int in_h, int in_w, int sm_count) {
  if (!(l.op == EE_OP_CONV && l.kh == 1 && l.kw == 1 && l.stride == 1 && l.pad == 0 && l.pad_w == 0 && l.residual_from == EE_NO_RESIDUAL)) return false;
  if (!(d.op == EE_OP_DWCONV && d.kh == 3 && d.kw == 3 && d.pad == 1 && d.pad_w == 1 && (d.stride == 1 || d.stride == 2) && d.residual_from == EE_NO_RESIDUAL)) return false;
  if (l.cin % 8 || l.cout % 8 || l.cout != d.cin || l.cin > kXdwMaxKb * kTcBK || in_w + 2 > 256 || (long)in_h * in_w > kXdwMaxMap) return false;
  return xdw_plan(sm_count, 1, in_w, (in_h - 1) / d.stride + 1, (in_w - 1) / d.stride + 1, d.stride, l.cin, l.cout).RB > 0;
}

inline ee_status_t xdw_context_init() {
  cudaError_t e = cudaFuncSetAttribute(conv_expand_dw_tcgen05_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_expand_dw_tcgen05_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

inline ee_status_t xdw_weight_map(const TcContext& c, const void* w, int cin, int cout, CUtensorMap* out) {
  const cuuint64_t dims[3] = {(cuuint64_t)cin, 1, (cuuint64_t)cout};
  const cuuint64_t strides[2] = {(cuuint64_t)cin * 2, (cuuint64_t)cin * 2};
  const cuuint32_t box[3] = {kTcBK, 1, 64}, es[3] = {1, 1, 1};
  return c.encode_tiled(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(w), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? EE_OK
             : EE_ERR_CUDA;
}

// maps: where the input's tensor maps are cached; tmW: the 1x1 weights [hidden][1][Cin] in boxes of 64 filters; g: the depthwise layer.
inline ee_status_t xdw_launch(TcContext& c, const TcLayer& maps, const CUtensorMap& tmW, int cin, int act1, const float* scale1, const float* bias1,
                              const ConvGeom& g, bool rev, const void* x, const void* w, const float* scale2, const float* bias2, void* y, int* err_flag,
                              cudaStream_t st) {
  if (((uintptr_t)x | (uintptr_t)w | (uintptr_t)y) & 15) return EE_ERR_INVALID_ARG;
  const XdwPlan plan = xdw_plan(c.sm_count, g.B, g.W, g.Ho, g.Wo, g.stride, cin, g.Cin);
  if (plan.RB < 1) return EE_ERR_INTERNAL;
  XdwParams p = {};
  const int rows = (plan.RB - 1) * g.stride + 3;
  p.H = g.H, p.W = g.W, p.Ho = g.Ho, p.Wo = g.Wo, p.C = g.Cin;
  p.RB = plan.RB, p.bands = cdiv(g.Ho, plan.RB), p.tiles = g.B * p.bands;
  p.cb = dw_block_channels(g.Cin);
  p.cin = cin, p.kblocks = cdiv(cin, kTcBK);
  p.magic = (1 << 20) / (g.W + 2) + 1;
  p.positions = rows * (g.W + 2), p.mtiles = cdiv(p.positions, 128), p.slots = plan.slots;
  p.act1 = act1, p.act2 = g.act, p.rev = rev ? 1 : 0;
  p.scale1 = scale1, p.bias1 = bias1, p.w = (const bf16*)w, p.scale2 = scale2, p.bias2 = bias2, p.y = (bf16*)y, p.err_flag = err_flag;
  const CUtensorMap* t = nullptr;
  const ee_status_t s = dw_input_map(c, maps, x, g.B, cin, g.H, g.W, kTcBK, rows, &t, true);
  if (s != EE_OK) return s;
  const CUtensorMap tmX = *t;
  const XdwSmem sm = xdw_smem(p.cb, p.kblocks, p.positions, p.slots);
  const int chunks = cdiv(g.Cin, p.cb);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::min(p.tiles, std::max(1, c.sm_count / chunks)), chunks);
  cfg.blockDim = dim3(kXdwThreads);
  cfg.dynamicSmemBytes = sm.bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = g.stride == 1 ? cudaLaunchKernelEx(&cfg, conv_expand_dw_tcgen05_kernel<1>, tmX, tmW, p, sm)
                                      : cudaLaunchKernelEx(&cfg, conv_expand_dw_tcgen05_kernel<2>, tmX, tmW, p, sm);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

}  // namespace ee
