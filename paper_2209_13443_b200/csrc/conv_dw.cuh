// Depthwise 3x3 pad-1 convolution on bf16 (stride 1 or 2) with the input staged in shared memory by TMA: the
// layers of the inverted-residual blocks that do 9 MACs per element.
//
// A kernel that loads through registers holds one item's inputs per thread and stalls on every item.  Here
// one producer warp per persistent CTA asks the TMA unit for whole input tiles, a band of output rows x all columns x
// one block of up to 64 channels, including the one-pixel frame of the padding (coordinates start at -1; the unit
// zero-fills outside the image), into a ring of three slots: two or three tiles (up to 72 KB each) are in flight per
// SM whatever the consumers do.  Eight consumer warps compute from shared memory: a thread owns one vector of eight
// channels (its 72 weights stay in registers as floats) and walks strips of four consecutive output pixels of the
// tile, reading each of the 3 x 6 (stride 2: 3 x 9) input vectors of a strip once.  A quarter warp reads the eight
// channel vectors of one pixel, 128 contiguous bytes, so the reads are conflict-free without swizzling.  Every output
// sums its nine taps in ascending (r, s) with fp32 FMAs, scale / bias / activation in fp32, one rounding to bf16.
#pragma once
#include <type_traits>

#include "conv_tc.cuh"

namespace ee {

struct DwParams {
  int H, W, C, Ho, Wo;
  int RB;          // output rows per tile
  int bands;       // ceil(Ho / RB)
  int tiles;       // B * bands, per channel block
  int cb;          // channels per block (dw_block_channels)
  int tile_bytes;  // ((RB - 1) * stride + 3) * (W + 2) * cb * 2
  int slot_bytes;  // tile_bytes rounded up to 128
  int act;
  int rev;         // 1: walk the tiles from the last one down
  const bf16* w;   // [C][3][3]
  const float* scale;
  const float* bias;
  bf16* y;         // [B][Ho][Wo][C]
  int* err_flag;
};

constexpr int kDwStages = 3;
constexpr int kDwConsumers = 256;
constexpr int kDwThreads = 32 + kDwConsumers;
constexpr int kDwMaxTileBytes = 72 * 1024;

// What a thread does with its vector of eight channels, here and in conv_xdw.cuh, whose bits have to agree.  What bounds it is instructions:
// nine FMAs an output are 4.5 packed ones (an SM does about 93 FMAs a clock, packed or not), so everything else has to be few.  Pairs of
// channels stay packed from the unpacking to the rounding, columns are offsets from one address, and the activation is chosen once a strip.  (17
// instructions an output, about 30 before.)  us, batch 32 / 13 / 1: 112 x 112 x 32 18.2 / 8.6 / 2.7 -> 16.7 / 8.1 / 2.6, 112 x 112 x 96 at stride 2
// 22.9 / 9.2 / 3.1 -> 20.0 / 8.3 / 2.9.  A thread that walks down its columns, sums of three rows open in registers, reads every vector once
// (13.7 and 17.5 at batch 32) but fills the register file, so that no neighbouring kernel sets up beside it: 9.3 and 9.4 at 13, 4.2 and 4.3 at 1.
typedef unsigned long long f32x2;   // two floats
__device__ __forceinline__ f32x2 f32x2_pack(uint32_t lo, uint32_t hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ f32x2 f32x2_fma(f32x2 a, f32x2 b, f32x2 c) {   // two independent round-to-nearest FMAs
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ void f32x2_unpack_bf16(uint4 x, f32x2 (&f)[4]) {
  const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) f[i] = f32x2_pack(w[i] << 16, w[i] & 0xffff0000u);
}
// Its 72 weights [8][3][3] as floats, [tap][channel pair]: unpacked from bf16 once, not at every product (two of three instructions of a strip
// were such shifts and masks).  Zeros where !take.
__device__ __forceinline__ void dw_weights(const bf16* w, bool take, f32x2 (&wf)[9][4]) {
  uint32_t wr[36];   // as stored: element e = channel e / 9, tap e % 9
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const uint4 v = take ? __ldg(reinterpret_cast<const uint4*>(w) + i) : make_uint4(0u, 0u, 0u, 0u);
    wr[4 * i] = v.x, wr[4 * i + 1] = v.y, wr[4 * i + 2] = v.z, wr[4 * i + 3] = v.w;
  }
  auto elem = [&](int e) { return (e & 1) ? wr[e >> 1] & 0xffff0000u : wr[e >> 1] << 16; };
#pragma unroll
  for (int t = 0; t < 9; ++t)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      wf[t][i] = f32x2_pack(elem(18 * i + t), elem(18 * i + 9 + t));
      asm volatile("" : "+l"(wf[t][i]));   // floats from here on: not to be unpacked again in the loop
    }
}
// The sums of a strip of kDwStrip output pixels, every output's taps in ascending (r, s).  at: the strip's first frame vector, columns `pitch` and
// rows `line` bytes apart.  Columns past the frame only feed outputs that are not stored: up to kDwOver vectors behind the last row are read.
constexpr int kDwOver = 8;
template <int STRIDE>
__device__ __forceinline__ void dw_strip(const uint8_t* at, int pitch, int line, const f32x2 (&w)[9][4], f32x2 (&acc)[kDwStrip][4]) {
  constexpr int COLS = (kDwStrip - 1) * STRIDE + 3;
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    uint4 v[COLS];
#pragma unroll
    for (int q = 0; q < COLS; ++q) v[q] = *reinterpret_cast<const uint4*>(at + r * line + q * pitch);
#pragma unroll
    for (int q = 0; q < COLS; ++q) {
      f32x2 f[4];
      f32x2_unpack_bf16(v[q], f);
#pragma unroll
      for (int p = 0; p < kDwStrip; ++p) {
        const int s = q - p * STRIDE;   // compile-time after unrolling
        if (s < 0 || s > 2) continue;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[p][i] = f32x2_fma(f[i], w[r * 3 + s][i], r == 0 && s == 0 ? 0ull : acc[p][i]);
      }
    }
  }
}
// y[0 .. cols) = act(scale * sum + bias), rounded to bf16; pixels at and past `cols` are not stored.  sb: eight scales and, 64 floats behind, biases.
__device__ __forceinline__ void dw_store(bf16* y, int C, int cols, const f32x2 (&acc)[kDwStrip][4], const float* sb, int act) {
  f32x2 sc[4], bi[4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const ulonglong2 s = reinterpret_cast<const ulonglong2*>(sb)[i], b = reinterpret_cast<const ulonglong2*>(sb + 64)[i];
    sc[2 * i] = s.x, sc[2 * i + 1] = s.y, bi[2 * i] = b.x, bi[2 * i + 1] = b.y;
  }
  auto put = [&](auto kind) {
#pragma unroll
    for (int p = 0; p < kDwStrip; ++p)
      if (p < cols) {
        uint32_t o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const f32x2 t = f32x2_fma(sc[i], acc[p][i], bi[i]);
          o[i] = pack_bf16x2(apply_act(__uint_as_float((uint32_t)t), decltype(kind)::value), apply_act(__uint_as_float((uint32_t)(t >> 32)), decltype(kind)::value));
        }
        *reinterpret_cast<uint4*>(y + (size_t)p * C) = make_uint4(o[0], o[1], o[2], o[3]);
      }
  };
  if (act == EE_ACT_RELU6) put(std::integral_constant<int, EE_ACT_RELU6>{});
  else if (act == EE_ACT_RELU) put(std::integral_constant<int, EE_ACT_RELU>{});
  else put(std::integral_constant<int, EE_ACT_NONE>{});
}

// POOL: the same staging for a 3x3 pad-1 window maximum (the max-pool behind a ResNet-style stem): taps outside the
// image are skipped (the frame's zeros must not win against negative inputs), no weights, no epilogue arithmetic.
template <int STRIDE, bool POOL>
__global__ void __launch_bounds__(kDwThreads, 1)
dwconv3x3_tma_kernel(const __grid_constant__ CUtensorMap tmX, DwParams p) {
  constexpr int P = kDwStrip;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_s = smem_u32(smem_raw);
  const uint32_t base = (raw_s + 127u) & ~127u;
  uint8_t* gen = smem_raw + (base - raw_s);
  const int bar_off = kDwStages * p.slot_bytes + kDwOver * 128;   // behind the last slot: what strips read past its frame
  const uint32_t bar0 = base + bar_off;
  __shared__ __align__(16) float s_sb[128];   // scale | bias of the channel block
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kDwStages + s); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int my_tiles = (int)blockIdx.x < p.tiles ? (p.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  const int c0 = (int)blockIdx.y * p.cb;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kDwStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), kDwConsumers / 32);   // lane 0 of each consumer warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmX) : "memory");
  }
  if (!POOL && threadIdx.x < 64) {   // no kernel writes weights, scale or bias: fetched while the layer in front still runs
    const int i = (int)threadIdx.x;
    const bool in = i < p.cb && c0 + i < p.C;
    s_sb[i] = p.scale && in ? p.scale[c0 + i] : 1.f;
    s_sb[64 + i] = p.bias && in ? p.bias[c0 + i] : 0.f;
  }
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (lane == 0) {
      for (int j = 0; j < my_tiles; ++j) {
        const int tf = (int)blockIdx.x + j * (int)gridDim.x, t = p.rev ? p.tiles - 1 - tf : tf;
        const int b = t / p.bands, band = t - b * p.bands;
        const int s = j % kDwStages;
        if (!mbar_wait(empty(s), ((uint32_t)(j / kDwStages) & 1u) ^ 1u, p.err_flag)) break;
        mbar_expect_tx(full(s), (uint32_t)p.tile_bytes);
        tma_load_4d(base + (uint32_t)(s * p.slot_bytes), &tmX, full(s), c0, -1, band * p.RB * STRIDE - 1, b);
      }
    }
    return;
  }

  const int tid = (int)threadIdx.x - 32;
  const int nv = p.cb >> 3;                 // channel vectors per block
  const int cvec = tid % nv, item0 = tid / nv, item_step = kDwConsumers / nv;
  const bool live = item0 < item_step;      // nv need not divide 256: the threads of the ragged tail idle
  const int c = c0 + cvec * 8;
  const bool c_in = c < p.C;
  f32x2 wf[9][4];
  if constexpr (!POOL) dw_weights(p.w + (size_t)c * 9, c_in, wf);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int strips = (p.Wo + P - 1) / P;
  const int Wc = p.W + 2, pitch = p.cb * 2;
  const int items = p.RB * strips;
  for (int j = 0; j < my_tiles; ++j) {
    const int tf = (int)blockIdx.x + j * (int)gridDim.x, t = p.rev ? p.tiles - 1 - tf : tf;
    const int b = t / p.bands, band = t - b * p.bands;
    const int s = j % kDwStages;
    if (!__all_sync(0xffffffffu, mbar_wait(full(s), (uint32_t)(j / kDwStages) & 1u, p.err_flag))) break;
    const uint8_t* tile = gen + (size_t)s * p.slot_bytes;
    if (live) {
      for (int it = item0; it < items; it += item_step) {
        const int ro = it / strips, st = it - ro * strips;
        const int wo0 = st * P;
        const int ho = band * p.RB + ro;
        const uint8_t* at = tile + (ro * STRIDE * Wc + wo0 * STRIDE) * pitch + cvec * 16;
        bf16* y = p.y + (((size_t)b * p.Ho + ho) * p.Wo + wo0) * p.C + c;
        if constexpr (POOL) {
          float acc[P][8];
#pragma unroll
          for (int pp = 0; pp < P; ++pp)
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[pp][e] = -INFINITY;
#pragma unroll
          for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int q = 0; q < (P - 1) * STRIDE + 3; ++q) {
              const int hi = ho * STRIDE - 1 + r, wi = wo0 * STRIDE - 1 + q;
              if (hi < 0 || hi >= p.H || wi < 0 || wi >= p.W) continue;
              Vec16<bf16> f;
              f.unpack(*reinterpret_cast<const uint4*>(at + (r * Wc + q) * pitch));
#pragma unroll
              for (int pp = 0; pp < P; ++pp)
                if (q - pp * STRIDE >= 0 && q - pp * STRIDE < 3) {
#pragma unroll
                  for (int e = 0; e < 8; ++e) acc[pp][e] = fmaxf(acc[pp][e], f.v[e]);
                }
            }
          if (c_in && ho < p.Ho)
#pragma unroll
            for (int pp = 0; pp < P; ++pp)
              if (pp < p.Wo - wo0) {
                Vec16<bf16> o;
#pragma unroll
                for (int e = 0; e < 8; ++e) o.v[e] = acc[pp][e];
                o.store(y + (size_t)pp * p.C);
              }
        } else {
          f32x2 acc[P][4];
          dw_strip<STRIDE>(at, pitch, Wc * pitch, wf, acc);
          if (c_in && ho < p.Ho) dw_store(y, p.C, p.Wo - wo0, acc, s_sb + cvec * 8, p.act);
        }
      }
    }
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty(s)) : "memory");
  }
}

// Layers this kernel takes: depthwise 3x3 (or a 3x3 max-pool, w == nullptr), pad 1, stride 1 or 2, channels a multiple
// of 8, at most 254 columns, and a tile of one output row that fits a ring slot.
// Channels per block: the channels are cut into ceil(C / 64) blocks of equal size (a multiple of 8), so that no block
// is mostly empty (144 channels: 3 x 48, not 64 + 64 + 16).
inline int dw_block_channels(int C) {
  const int blocks = (C + 63) / 64;
  return ((C + blocks - 1) / blocks + 7) / 8 * 8;
}

inline bool dw_tma_supported(const ConvGeom& g, const void* x, const void* w, const void* y) {
  if (!(g.kh == 3 && g.kw == 3 && g.pad == 1 && (g.stride == 1 || g.stride == 2) && g.Cin % 8 == 0 && g.Cin == g.Cout)) return false;
  if ((((uintptr_t)x | (uintptr_t)w | (uintptr_t)y) & 15) != 0 || g.W + 2 > 256) return false;
  const int cb = dw_block_channels(g.Cin);
  return 3 * (g.W + 2) * cb * 2 <= kDwMaxTileBytes;
}

inline ee_status_t dw_context_init() {
  const int bytes = kDwStages * kDwMaxTileBytes + kDwOver * 128 + 256 + 128;
  cudaError_t e = cudaFuncSetAttribute(dwconv3x3_tma_kernel<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(dwconv3x3_tma_kernel<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(dwconv3x3_tma_kernel<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(dwconv3x3_tma_kernel<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

// Tensor map of a depthwise layer's input, NHWC as (C, W, H, B), box = (cb, W + 2, rows, 1), no swizzle; cached in the
// layer like the other maps of caller buffers.
// operand: 128-byte swizzle, boxes that are the rows of a K-major operand (conv_xdw.cuh).
inline ee_status_t dw_input_map(const TcContext& c, const TcLayer& L, const void* ptr, int batch, int C, int H, int W, int cb, int rows,
                                const CUtensorMap** out, bool operand = false) {
  const int kind = operand ? 10 : 5;
  for (auto& e : L.a_maps)
    if (e.ptr == ptr && e.batch == batch && e.kind == kind) {
      *out = &e.tm;
      return EE_OK;
    }
  TcLayer::Cached e;
  e.ptr = ptr, e.batch = batch, e.kind = kind;
  const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)batch};
  const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)C * 2 * W, (cuuint64_t)C * 2 * W * H};
  const cuuint32_t box[4] = {(cuuint32_t)cb, (cuuint32_t)(W + 2), (cuuint32_t)rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  if (c.encode_tiled(&e.tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     operand ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return EE_ERR_CUDA;
  if (L.a_maps.size() < 48) {
    L.a_maps.push_back(e);
    *out = &L.a_maps.back().tm;
  } else {
    L.a_maps[L.next_evict] = e;
    *out = &L.a_maps[L.next_evict].tm;
    L.next_evict = (L.next_evict + 1) % L.a_maps.size();
  }
  return EE_OK;
}

// L: only its map cache is used (a depthwise layer has no tensor-core plan).
inline ee_status_t dw_tma_launch(TcContext& c, const TcLayer& L, const ConvGeom& g, const void* x, const void* w, const float* scale,
                                 const float* bias, void* y, int* err_flag, cudaStream_t st) {
  DwParams p;
  p.H = g.H, p.W = g.W, p.C = g.Cin, p.Ho = g.Ho, p.Wo = g.Wo;
  p.cb = dw_block_channels(g.Cin);
  const int row_bytes = (g.W + 2) * p.cb * 2;
  int in_rows = kDwMaxTileBytes / row_bytes;                      // input rows a slot holds
  if (in_rows > 256) in_rows = 256;
  int rb_max = (in_rows - 3) / g.stride + 1;
  if (rb_max > g.Ho) rb_max = g.Ho;
  // Band height: a CTA's eight consumer warps take 256 / (cb / 8) strips per pass over a tile, a tile costs about one
  // more pass (waiting for the slot, hand-over), and the busiest CTA walks ceil(tiles / CTAs) tiles.  Take the height
  // that minimises that CTA's passes (bytes moved rise with shorter bands: each band re-reads two frame rows).
  const int chunks = cdiv(g.Cin, p.cb);
  const int ctas_x = std::max(1, c.sm_count / chunks);
  const int strips = (g.Wo + kDwStrip - 1) / kDwStrip;
  const int per_pass = kDwConsumers / std::max(1, p.cb / 8);
  long best = -1;
  p.RB = 1;
  for (int rb = 1; rb <= rb_max; ++rb) {
    const long tiles = (long)g.B * cdiv(g.Ho, rb);
    const long cost = cdiv(tiles, std::min<long>(tiles, ctas_x)) * (cdiv((long)rb * strips, per_pass) + 1);
    if (best < 0 || cost <= best) best = cost, p.RB = rb;   // ties: the taller band (fewer frame rows re-read)
  }
  const int rows = (p.RB - 1) * g.stride + 3;
  p.bands = cdiv(g.Ho, p.RB);
  p.tiles = g.B * p.bands;
  p.tile_bytes = rows * row_bytes;
  p.slot_bytes = (int)align_up((size_t)p.tile_bytes, 128);
  p.act = g.act;
  p.rev = L.rev ? 1 : 0;
  p.w = (const bf16*)w, p.scale = scale, p.bias = bias, p.y = (bf16*)y;
  p.err_flag = err_flag;
  const CUtensorMap* t = nullptr;
  ee_status_t s = dw_input_map(c, L, x, g.B, g.Cin, g.H, g.W, p.cb, rows, &t);
  if (s != EE_OK) return s;
  const CUtensorMap tmX = *t;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::min(p.tiles, std::max(1, c.sm_count / chunks)), chunks);
  cfg.blockDim = dim3(kDwThreads);
  cfg.dynamicSmemBytes = kDwStages * p.slot_bytes + kDwOver * 128 + 256 + 128;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (w)
    e = g.stride == 1 ? cudaLaunchKernelEx(&cfg, dwconv3x3_tma_kernel<1, false>, tmX, p) : cudaLaunchKernelEx(&cfg, dwconv3x3_tma_kernel<2, false>, tmX, p);
  else
    e = g.stride == 1 ? cudaLaunchKernelEx(&cfg, dwconv3x3_tma_kernel<1, true>, tmX, p) : cudaLaunchKernelEx(&cfg, dwconv3x3_tma_kernel<2, true>, tmX, p);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

}  // namespace ee
