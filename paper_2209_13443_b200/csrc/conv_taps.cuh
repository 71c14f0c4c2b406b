// Convolutions with several filter taps (3x3, 1x7, 7x1, ...; stride 1 or 2) whose A operand is read from shared memory
// once per tap but fetched once per filter COLUMN.
//
// The generic kernel of conv_tc.cuh gathers a 128-pixel x 64-channel A tile per tap (im2col map): 16 KB per K block, at
// 0.36 us per K block and SM against 0.26 us for plain tiles, and its 128 x 128 tiles leave most SMs idle when the map is
// small.  Here an output tile is R rows x NI images x Wp columns (Wp = the row length rounded up to 8, R * NI * Wp <= 128),
// ordered [row][image][column].  For filter column s and one 64-channel block, one tiled TMA load brings the input rows
// all taps (., s) of the tile touch, shifted by s: [R + kh - 1][NI][Wp] pixels of 128 bytes (zero fill outside the image is
// the padding).  Tap (r, s) is that block viewed from pixel r * NI * Wp on, a multiple of 8 rows = 1024 bytes, so the view
// is an aligned operand of the 128-byte swizzle and the tensor core reads it at full rate (views shifted by single
// columns cost it twice the time).  A 3x3 layer on 14x14 maps moves 60 KB per channel block instead of 144 KB.  With
// stride 2 the rows of one parity form a block (tiled map with element strides), two blocks per filter column.
//
// The tile width BN (128 ... 16 filters) is picked per launch so that the grid fills the SMs (tap_pick_bn).  It changes no
// sum: every output adds its K blocks in the order of tap_at, as in all kernels of this library.
//
// Warp roles: warp 0 weights (TMA), warp 1 TMEM and MMA, warps 2-5 epilogue (a thread owns one output pixel and stores its
// BN channels straight to global memory), warp 6 activations (TMA).  Every wait on an mbarrier is bounded.
#pragma once
#include "conv_tc.cuh"

namespace ee {

constexpr int kTapThreads = 224;

struct TapParams {
  int N, Ho, Wo, B;
  int R, NI, Wp, y_tiles;     // tile geometry; M tile t = (image group t / y_tiles, rows (t % y_tiles) * R ...)
  int kh, kw, stride, pad, pad_w, cblocks;
  int act, rev;
  int sa, sw, a_slot, a_bytes;   // ring depths, bytes of an A slot and of one load
  const float* scale;
  const float* bias;
  bf16* out;
  int* err_flag;
};

template <int BN>
__global__ void __launch_bounds__(kTapThreads, 2)
conv_taps_tcgen05_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, TapParams p) {
  constexpr int kWBytes = BN * kTcBK * 2, kCols = BN < 32 ? 32 : BN;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  const uint32_t w_base = base + (uint32_t)(p.sa * p.a_slot);
  const int after = p.sa * p.a_slot + p.sw * kWBytes;
  float* s_scale = reinterpret_cast<float*>(gen + after);
  float* s_bias = s_scale + BN;
  const uint32_t bar0 = base + (uint32_t)after + 2 * BN * 4;
  auto a_full = [&](int s) { return bar0 + 8u * s; };
  auto a_empty = [&](int s) { return bar0 + 8u * (p.sa + s); };
  auto w_full = [&](int s) { return bar0 + 8u * (2 * p.sa + s); };
  auto w_empty = [&](int s) { return bar0 + 8u * (2 * p.sa + p.sw + s); };
  const uint32_t accum_bar = bar0 + 8u * (2 * p.sa + 2 * p.sw);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + after + 2 * BN * 4 + 8 * (2 * p.sa + 2 * p.sw + 1));

  __shared__ uint32_t tab[kMaxTaps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = p.rev ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
  const int n0 = (int)blockIdx.y * BN;
  const int img0 = tile / p.y_tiles * p.NI, y0 = tile % p.y_tiles * p.R;
  const int taps = p.kh * p.kw, num_kb = taps * p.cblocks;
  const int parts = p.stride == 1 ? 1 : min(2, p.kh);   // A blocks per filter column

  tap_table_fill(tab, p.kh, p.kw, p.stride);
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2 * (p.sa + p.sw) + 1; ++s) mbar_init(bar0 + 8u * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {   // weights: written by no kernel, so the first ring slots need not wait for the previous one
    if (elect_one()) {
      int s = 0;
      uint32_t ph = 1;
      int c = 0, t = 0;
      for (int i = 0; i < num_kb; ++i) {
        const int tap = (int)(tab[t] >> 16);
        if (i >= p.sw && !mbar_wait(w_empty(s), ph, p.err_flag)) break;
        mbar_expect_tx(w_full(s), kWBytes);
        tma_load_3d(w_base + (uint32_t)(s * kWBytes), &tmW, w_full(s), c, tap, n0);
        if (++t == taps) t = 0, c += kTcBK;
        if (++s == p.sw) s = 0, ph ^= 1u;
        if (i == min(p.sw, num_kb) - 1) {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
      }
    } else {
      asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    __syncwarp();
  } else if (warp == 6) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (elect_one()) {
      int s = 0, col = 0, q = 0, cb = 0;
      uint32_t ph = 1;
      for (int c = 0; c < p.cblocks * p.kw * parts; ++c) {
        if (!mbar_wait(a_empty(s), ph, p.err_flag)) break;
        mbar_expect_tx(a_full(s), (uint32_t)p.a_bytes);
        tma_load_4d(base + (uint32_t)(s * p.a_slot), &tmX, a_full(s), cb * kTcBK, col - p.pad_w, img0, y0 * p.stride - p.pad + q);
        if (++q == parts) {
          q = 0;
          if (++col == p.kw) col = 0, ++cb;
        }
        if (++s == p.sa) s = 0, ph ^= 1u;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc(BN);
      const uint64_t da0 = umma_desc(base), db0 = umma_desc(w_base);
      const uint32_t row_shift = (uint32_t)(p.NI * p.Wp * 128) >> 4;
      int sa = 0, sw = 0, q = 0;
      uint32_t pa = 0, pw = 0;
      bool ok = true, acc = false;
      for (int c = 0; c < p.cblocks * p.kw * parts && ok; ++c) {
        const int n_taps = parts == 1 ? p.kh : (p.kh + 1 - q) / 2;   // filter rows of this block
        uint64_t da = da0 + (uint64_t)(uint32_t)(sa * p.a_slot >> 4);
        ok = mbar_wait(a_full(sa), pa, p.err_flag);
        for (int j = 0; j < n_taps && ok; ++j) {
          ok = mbar_wait(w_full(sw), pw, p.err_flag);
          if (!ok) break;
          tc_fence_after();
          umma_block(tmem_base, da, db0 + (uint64_t)(sw * (kWBytes >> 4)), idesc, acc);
          umma_commit(w_empty(sw));
          da += row_shift;
          acc = true;
          if (++sw == p.sw) sw = 0, pw ^= 1u;
        }
        if (ok) umma_commit(a_empty(sa));
        if (++sa == p.sa) sa = 0, pa ^= 1u;
        if (++q == parts) q = 0;
      }
      if (ok) umma_commit(accum_bar);
    }
    __syncwarp();
  } else {
    const int et = threadIdx.x - 64;
    for (int i = et; i < BN; i += 128) {
      const bool in = n0 + i < p.N;
      s_scale[i] = (p.scale && in) ? p.scale[n0 + i] : 1.f;
      s_bias[i] = (p.bias && in) ? p.bias[n0 + i] : 0.f;
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int q = warp & 3, row = q * 32 + lane;
    const int y = row / (p.NI * p.Wp), nx = row - y * p.NI * p.Wp, im = nx / p.Wp, x = nx - im * p.Wp;
    const bool inside = y < p.R && y0 + y < p.Ho && img0 + im < p.B && x < p.Wo;
    bf16* dst = p.out + (((size_t)(img0 + im) * p.Ho + y0 + y) * p.Wo + x) * p.N + n0;
    if (__all_sync(0xffffffffu, mbar_wait(accum_bar, 0, p.err_flag))) {
      tc_fence_after();
      const uint32_t acc = tmem_base + ((uint32_t)(q * 32) << 16);
#pragma unroll
      for (int c0 = 0; c0 < BN; c0 += 32) {
        if (n0 + c0 >= p.N) break;
        float v[32];
        tmem_ld32(acc + (uint32_t)c0, v);   // BN = 16: the upper half is not used
        if (inside) {
#pragma unroll
          for (int g = 0; g < (BN < 32 ? 2 : 4); ++g) {
            if (n0 + c0 + g * 8 >= p.N) break;
            *reinterpret_cast<uint4*>(dst + c0 + g * 8) =
                epilogue8_act<false>(p.act, v + g * 8, s_scale + c0 + g * 8, s_bias + c0 + g * 8, make_uint4(0u, 0u, 0u, 0u));
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kCols) : "memory");
  }
}

// ----------------------------------------------------------------------------- host side

// Tile geometry of a layer: the images per tile that need the fewest tiles at max_batch.
inline bool tap_plan(const ee_layer_desc_t& d, int out_h, int out_w, int max_batch, TapPlan* t) {
  t->on = false;
  if (d.op != EE_OP_CONV || d.kh * d.kw == 1 || d.cin % 8 != 0 || d.cout % 8 != 0 || d.kh > 7 || d.kw > 7 || d.stride > 2 ||
      d.residual_from != EE_NO_RESIDUAL || out_w > 128)
    return false;
  const int wp = (out_w + 7) / 8 * 8;
  long best = -1;
  for (int ni = 1; ni * wp <= kTcBM && ni <= max_batch; ++ni) {
    const int r = std::min(kTcBM / (ni * wp), out_h);
    const long tiles = (long)cdiv(max_batch, ni) * cdiv(out_h, r);
    if (best < 0 || tiles < best) best = tiles, t->ni = ni, t->r = r;
  }
  t->wp = wp;
  t->rows = d.stride == 1 ? t->r + d.kh - 1 : t->r + (d.kh + 1) / 2 - 1;
  t->a_bytes = t->rows * t->ni * wp * 128;
  t->on = t->rows <= 128 && t->a_bytes <= 40 * 1024;
  return t->on;
}

inline int tap_m_tiles(const TcLayer& L, int B) { return cdiv(B, L.tap.ni) * cdiv(L.out_h, L.tap.r); }

// Filters per tile.  A K block costs an SM the larger of what its L2 port takes (64 bytes per clock: the weights and the
// tap's share of the activations) and what the MMAs read (128 bytes per clock); tiles beyond one per SM add up.  About 1.5 us
// of epilogue go with 128 columns.
inline int tap_pick_bn(const TcContext& c, const TcLayer& L, int B) {
  const int parts = L.stride == 1 ? 1 : std::min(2, L.kh), num_kb = L.kh * L.kw * cdiv(L.cin, kTcBK);
  const double a_share = (double)L.tap.a_bytes * parts / L.kh;
  const long mt = tap_m_tiles(L, B);
  int pick = 128;
  double best = 0;
  for (int bn = 128; bn >= 16; bn /= 2) {
    if (bn > 16 && bn / 2 >= L.cout) continue;
    const double clk = std::max((a_share + bn * 128.0) / 64.0, (16384.0 + bn * 128.0) / 128.0);
    const double cost = (double)cdiv(mt * cdiv(L.cout, bn), c.sm_count) * (num_kb * clk + bn * 22.0);
    if (best == 0 || cost < best * 0.97) best = cost, pick = bn;
  }
  return pick;
}

template <int BN>
inline cudaError_t tap_launch_t(dim3 grid, cudaStream_t st, const CUtensorMap& x, const CUtensorMap& w, TapParams p, int sms) {
  // two CTAs per SM when the grid has more tiles than SMs, else a deeper weight ring
  const int fixed = 2 * BN * 4 + 512 + 1024 + 256, room = ((long)grid.x * grid.y > sms ? 113 : 200) * 1024;
  p.sa = std::min(4, std::max(2, (room - fixed - 4 * BN * 128) / p.a_slot));
  p.sw = std::min(12, std::max(3, (room - fixed - p.sa * p.a_slot) / (BN * 128)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kTapThreads);
  cfg.dynamicSmemBytes = p.sa * p.a_slot + std::max(p.sw * BN * 128, kTcBM * 128) + fixed;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, conv_taps_tcgen05_kernel<BN>, x, w, p);
}

inline ee_status_t tap_context_init() {
  cudaError_t e = cudaFuncSetAttribute(conv_taps_tcgen05_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_taps_tcgen05_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_taps_tcgen05_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(conv_taps_tcgen05_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

inline ee_status_t tap_launch(TcContext& c, const TcLayer& L, const void* src, void* dst, int B, const float* scale, const float* bias,
                              int* err_flag, cudaStream_t st) {
  if (((uintptr_t)src & 15) || ((uintptr_t)dst & 15)) return EE_ERR_INVALID_ARG;
  const CUtensorMap* t = nullptr;
  ee_status_t s = tc_buffer_map(c, L, src, B, 6, &t);
  if (s != EE_OK) return s;
  const CUtensorMap tmX = *t;
  TapParams p = {};
  p.N = L.cout, p.Ho = L.out_h, p.Wo = L.out_w, p.B = B;
  p.R = L.tap.r, p.NI = L.tap.ni, p.Wp = L.tap.wp, p.y_tiles = cdiv(L.out_h, L.tap.r);
  p.kh = L.kh, p.kw = L.kw, p.stride = L.stride, p.pad = L.pad, p.pad_w = L.pad_w, p.cblocks = cdiv(L.cin, kTcBK);
  p.act = L.act, p.rev = L.rev ? 1 : 0;
  // a view of 128 rows from the last filter row on may reach past its block: into the next slot or up to 16 KB behind the last
  p.a_bytes = L.tap.a_bytes, p.a_slot = (int)align_up((size_t)L.tap.a_bytes, 1024);
  p.scale = scale, p.bias = bias, p.out = (bf16*)dst, p.err_flag = err_flag;
  const int bn = tap_pick_bn(c, L, B);
  const dim3 grid(tap_m_tiles(L, B), cdiv(L.cout, bn));
  cudaError_t e;
  switch (bn) {
    case 128: e = tap_launch_t<128>(grid, st, tmX, L.tm_w_bn[3], p, c.sm_count); break;
    case 64: e = tap_launch_t<64>(grid, st, tmX, L.tm_w_bn[2], p, c.sm_count); break;
    case 32: e = tap_launch_t<32>(grid, st, tmX, L.tm_w_bn[1], p, c.sm_count); break;
    default: e = tap_launch_t<16>(grid, st, tmX, L.tm_w_bn[0], p, c.sm_count); break;
  }
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

}  // namespace ee
