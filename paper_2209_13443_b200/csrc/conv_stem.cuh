// Stride-2 stem convolutions on 3-channel bf16 images (7x7 of the ResNet-style backbones, 3x3 of the MobileNet-style ones), as
// an implicit GEMM on tcgen05.mma.
//
// A 3-channel pixel is 6 bytes, so no TMA load can fetch operand rows, and the operand is built by threads: the row of filter
// row rf and output pixel ox is the kw * 3 contiguous elements of image row 2 oy - pad + rf from 6 ox - 3 pad on.  These do
// not depend on oy but through the image row, and consecutive output rows share all but two of theirs.  So the unit is a PAIR of
// image rows (2 P - pad, 2 P - pad + 1): 128 pixels x 64 columns, built once into a ring slot and read by the up to
// (kh + 1) / 2 output rows P, P - 1, ...; an output row costs one new pair and its MMAs.  (Built per output row, seven
// filter rows went through shared memory for each of them and a row took 2950 clocks of an SM.)
//
// One persistent CTA per SM walks a contiguous range of output rows.  Four gather warps (one thread per output pixel) read the
// image straight from global memory, a pair ahead of the one they store; one thread issues the MMAs into four accumulators in
// turn; eight epilogue warps, 32 channels of 32 pixels each, finish the rows.  (A second set of gather warps left each thread 96
// registers, and with nearly all of L1 given to shared memory what spilled came back from L2.)
//
// Columns of a pair: a filter row is a dummy column, the kw * 3 taps and zeros (24 columns at 7x7, 16 at 3x3), its second row
// follows.  The dummy makes every run start at an even element (6 ox - 10 or 6 ox - 4).  The last filter row of an output row is the
// first row of its last pair, whose other row must not enter the sum, not even times zero: at 7x7 its columns 16..23 are there
// once more as columns 48..55, so that K steps 0 and 3 hold it alone.
// What bounds it: the gather, about 1600 clocks a pair (its loads come from L2, and 26 words in two sets are what the registers
// hold), against 530 of MMAs and 1500 of epilogue a row.  224 x 224 x 64 images with the pool 78.4 -> 66.9 us, 59 with the pool's
// integer keys (bf16x2_max); 161 x 161 images ran on the generic gather, whose tiles read every image row seven times.
#pragma once
#include <type_traits>

#include "conv_tc.cuh"
#include "stem_words.h"

namespace ee {

struct StemParams {
  int tiles;            // B * Ho output rows
  int H, W, Ho, Wo, N;  // image and output (Wo <= 128) sizes, Cout (<= 64)
  int act;
  int rev;              // 1: walk the output rows from the last range down
  int Hp, Wp, rows;     // fused pooling only: pooled height and width, rows = B * Hp pooled rows
  long total;           // elements of the image batch
  const float* scale;
  const float* bias;
  const bf16* x;
  bf16* out;
  int* err_flag;
};

constexpr int kStemThreads = 416;      // MMA warp, 4 gather warps, 8 epilogue warps
constexpr int kStemRing = 8, kStemAccs = 4, kStemCin = 3;

template <int KH>
struct StemGeom {
  static constexpr int kPad = KH / 2, kPairs = (KH + 1) / 2;
  static constexpr int kCols = KH == 7 ? 24 : 16;            // columns of a filter row
  static constexpr int kRead = (1 + KH * kStemCin + 1) / 2;  // words that hold taps
  static constexpr int kSteps = 2 * kCols / 16;              // K steps of a pair
  static constexpr int kPacked = kPairs * kTcBK;             // columns of the packed weights, a K block per pair
  static constexpr int kABytes = kTcBM * kTcBK * 2, kWBytes = 64 * kTcBK * 2;
  static constexpr int kWOff = kStemRing * kABytes;
  static constexpr int kOOff = kWOff + kPairs * kWBytes;
  static constexpr int kScaleOff = kOOff + 4 * kTcBM * 64;   // staging: two tiles of 128 pixels x 32 channels per channel half
  static constexpr int kBarOff = kScaleOff + 2 * 64 * 4;
  static constexpr int kBytes = kBarOff + 256 + 1024;
  static_assert(kBytes <= 227 * 1024, "exceeds the shared memory of an SM");
};

// The output rows of a CTA, in order: body(j, n, oy, fresh_pairs, free_pairs, fresh, emit, t) for its j-th row, row oy of image n.
// fresh_pairs: pairs that no row before it had (all of them where the walk starts or jumps), free_pairs: pairs that no row
// behind it needs.  Without pooling t is the row's index over the batch.  With the 3x3 stride-2 pad-1 max-pool fused behind the
// convolution a CTA owns a range of POOLED rows (t = the pooled row's index over the batch) and walks the convolution rows
// they cover in ascending order: rows 2py-1 .. 2py+1 for the first pooled row of the range or of an image (`fresh` marks the row
// that starts a new running maximum), rows 2py and 2py+1 for the others (row 2py-1 was the row before); `emit` marks the
// last row of a pooled row.  body returns false to stop the walk.
template <bool POOL, int PAIRS, typename F>
__device__ __forceinline__ void stem_walk(const StemParams& p, F&& body) {
  const long g = p.rev ? (long)gridDim.x - 1 - blockIdx.x : (long)blockIdx.x;
  const int all = POOL ? p.rows : p.tiles, per = POOL ? p.Hp : p.Ho;
  const int r0 = (int)(g * all / gridDim.x), r1 = (int)((g + 1) * all / gridDim.x);
  int n = r0 / per, y = r0 - n * per, j = 0;
  for (int r = r0; r < r1; ++r) {
    const bool first = r == r0 || y == 0, last = r + 1 == r1 || y + 1 == per;
    if constexpr (POOL) {
      const int lo = first ? max(2 * y - 1, 0) : 2 * y, hi = min(2 * y + 1, p.Ho - 1);
      for (int c = lo; c <= hi; ++c, ++j)
        if (!body(j, n, c, first && c == lo ? PAIRS : 1, last && c == hi ? PAIRS : 1, first && c == lo, c == hi, r)) return;
    } else {
      if (!body(j++, n, y, first ? PAIRS : 1, last ? PAIRS : 1, false, false, r)) return;
    }
    if (++y == per) y = 0, ++n;
  }
}

// Maximum of bf16 pairs.  NONNEG: behind a ReLU the order of the values is that of their bits, and the 16-bit integer maximum is
// an instruction of full rate; the bf16 one took 60 clocks each here.  A pooling layer of its own drops NaN (fmaxf), so here it must
// lose too: the keys of NONNEG are the bits plus one, by which the conversion's one NaN, 0x7FFF, becomes the least integer.
template <bool NONNEG>
__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  if (NONNEG) {
    uint32_t m;
    asm("max.s16x2 %0, %1, %2;" : "=r"(m) : "r"(a), "r"(b));
    return m;
  }
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
constexpr uint32_t kPoolKey = 0x00010001u;   // both halves: they hold 0 .. 0x7FFF (or 0x8000, -0), so nothing is carried or borrowed
// A window's maximum as it is stored: no number in the window (every tap NaN) is -inf, what a maximum over none starts from.
template <bool NONNEG>
__device__ __forceinline__ uint32_t bf16x2_pooled(uint32_t m) {
  const uint32_t nan = __vcmpeq2(m, NONNEG ? 0x80008000u : 0x7FFF7FFFu);
  return (NONNEG ? m - kPoolKey : m) & ~nan | (0xFF80FF80u & nan);
}

// The words (elements e0 + 2 j, e0 + 2 j + 1; e0 even) of a filter row's run in one image row, in two steps: `load` only requests
// aligned words (stem_words.h says which), `finish` makes the run's words of them.  Words outside the row are loads that do not
// happen, so nothing looks at a word before it is stored: a mask behind each load made every pair wait for memory (5200 clocks
// a pair).  Rows of an odd number of elements start at an odd element every other time; their words are put together from two
// aligned ones.
template <int NW>
struct StemRun {
  uint32_t a[NW + 1];
  int kind;   // of StemAsk, the same for the whole warp
  __device__ __forceinline__ void load(const StemParams& p, int n, int y, int e0, StemTaps in) {
    const int row_elems = p.W * kStemCin;
    if (y < 0 || y >= p.H) in.first = in.second = 0;
    const long rb = ((long)n * p.H + y) * row_elems;
    const StemAsk ask = stem_ask(rb, row_elems, p.total, in);
    kind = ask.kind;
    const bf16* row = p.x + (rb + e0);
    auto at = [&](int e, uint32_t ok) {
      uint32_t w;
      asm volatile("{\n .reg .pred q;\n setp.ne.u32 q, %2, 0;\n mov.u32 %0, 0;\n @q ld.global.nc.u32 %0, [%1];\n}" : "=r"(w) : "l"(row + e), "r"(ok));
      return w;
    };
    if (kind != 2) {
#pragma unroll
      for (int j = 0; j < NW; ++j) a[j] = at(2 * j, ask.mask & 1u << j);
      if (kind == 3) a[NW] = in.first ? (uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p.x) + (p.total - 1)) : 0u;
    } else {
#pragma unroll
      for (int j = 0; j <= NW; ++j) a[j] = at(2 * j - 1, ask.mask & 1u << j);
    }
  }
  __device__ __forceinline__ void finish(int e0, int row_elems, uint32_t in, uint32_t* w) const {
#pragma unroll
    for (int j = 0; j < NW; ++j) w[j] = a[j];
    if (!(row_elems & 1)) return;
#pragma unroll
    for (int j = 0; j < NW; ++j) {
      const bool end = e0 + 2 * j == row_elems - 1;   // the row's last element, alone in its word
      if (kind == 2) w[j] = in >> j & 1u ? __byte_perm(a[j], a[j + 1], 0x5432) : 0u;
      if (end) w[j] = kind == 3 ? a[NW] : w[j] & 0xffffu;
    }
  }
};

// tmW: packed weights (columns, 1, Cout) with a 64 x 1 x 64 box, 128-byte swizzle.
//
// POOL: the epilogue threads keep the running maximum over the convolution rows of a pooled row in registers (a
// thread owns one pixel column, 32 channels), and on the last of them put it in a staging tile, take the maximum
// over the three columns of every pooled pixel there and store the pooled row; the convolution's own output never
// reaches global memory.  max() of bf16 values is exact and NaN loses on both routes, so the result equals pooling the stored
// convolution output bit for bit.
template <int KH, bool POOL>
__global__ void __launch_bounds__(kStemThreads, 1)
conv_stem_tcgen05_kernel(const __grid_constant__ CUtensorMap tmW, StemParams p) {
  extern __shared__ uint8_t smem_raw[];
  using S = StemGeom<KH>;
  constexpr int PAIRS = S::kPairs;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  float* s_scale = reinterpret_cast<float*>(gen + S::kScaleOff);
  float* s_bias = s_scale + 64;
  const uint32_t bar0 = base + S::kBarOff;
  const uint32_t w_bar = bar0;
  auto pair_full = [&](int s) { return bar0 + 8u * (1 + s); };
  auto pair_empty = [&](int s) { return bar0 + 8u * (1 + kStemRing + s); };
  auto acc_full = [&](int b) { return bar0 + 8u * (1 + 2 * kStemRing + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (1 + 2 * kStemRing + kStemAccs + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gen + S::kBarOff + 8 * 30);
  volatile int* s_abort = reinterpret_cast<volatile int*>(gen + S::kBarOff + 8 * 31);   // POOL: an epilogue warp gave up

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x < 1 + 2 * kStemRing + 2 * kStemAccs) {
    const int i = threadIdx.x;
    // pair_full: lane 0 of each gather warp, after every lane's proxy fence; acc_empty: lane 0 of each epilogue warp
    mbar_init(bar0 + 8u * i, i >= 1 && i <= kStemRing ? 4 : i > 2 * kStemRing + kStemAccs ? 8 : 1);
    if (i == 0) *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kStemAccs * 64) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (threadIdx.x == 0) {   // the whole weight matrix stays resident; no kernel writes it, so it need not wait
    mbar_expect_tx(w_bar, PAIRS * S::kWBytes);
    for (int i = 0; i < PAIRS; ++i) tma_load_3d(base + S::kWOff + i * S::kWBytes, &tmW, w_bar, i * kTcBK, 0, 0);
  }
  __syncwarp();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc(64);
      const uint64_t da0 = umma_desc(base), db0 = umma_desc(base + S::kWOff);
      int q = 0;   // pairs the rows so far have met
      if (mbar_wait(w_bar, 0, p.err_flag))
        stem_walk<POOL, PAIRS>(p, [&](int j, int, int, int fresh_pairs, int free_pairs, bool, bool, int) {
          const int b = j & (kStemAccs - 1);
          // the epilogue must have drained this accumulator
          if (j >= kStemAccs && !mbar_wait(acc_empty(b), (uint32_t)(j / kStemAccs - 1) & 1u, p.err_flag)) return false;
          tc_fence_after();
          q += fresh_pairs;
          const uint32_t acc = tmem_base + (uint32_t)(b * 64);
#pragma unroll
          for (int k = 0; k < PAIRS; ++k) {
            const int pq = q - PAIRS + k, s = pq & (kStemRing - 1);
            if (k >= PAIRS - fresh_pairs && !mbar_wait(pair_full(s), (uint32_t)(pq / kStemRing) & 1u, p.err_flag)) return false;
            const uint64_t da = da0 + (uint64_t)(s * (S::kABytes >> 4)), db = db0 + (uint64_t)(k * (S::kWBytes >> 4));
            if (k + 1 < PAIRS) {
#pragma unroll
              for (int i = 0; i < S::kSteps; ++i) umma_bf16(acc, da + 2 * i, db + 2 * i, idesc, (uint32_t)(k != 0 || i != 0));
            } else {   // the last filter row alone
              umma_bf16(acc, da, db, idesc, 1u);
              if (KH == 7) umma_bf16(acc, da + 6, db + 6, idesc, 1u);
            }
          }
          umma_commit(acc_full(b));
          for (int k = 0; k < free_pairs; ++k) umma_commit(pair_empty((q - PAIRS + k) & (kStemRing - 1)));
          return true;
        });
    }
    __syncwarp();
  } else if (warp < 5) {
    // gather warps: thread r builds row r (output pixel ox = r) of every pair
    const int r = (int)threadIdx.x - 32;
    const int ox = min(r, p.Wo - 1);   // rows past Wo repeat the last pixel; nobody reads them
    const int e0 = 2 * kStemCin * ox - S::kPad * kStemCin - 1;   // image-row element of column 0 (even)
    const StemTaps in = stem_taps(e0, p.W * kStemCin, S::kRead);
    uint8_t* aline = gen + r * 128;
    constexpr int NW = S::kRead, CH = S::kCols / 8;   // words, 16-byte chunks of a filter row
    StemRun<NW> wa[2], wb[2];
    auto load = [&](int n, int P, StemRun<NW>* r) {
      r[0].load(p, n, 2 * P - S::kPad, e0, in);
      r[1].load(p, n, 2 * P - S::kPad + 1, e0, in);
    };
    auto store = [&](int q, const StemRun<NW>* run) {
      const int s = q & (kStemRing - 1);
      if (q >= kStemRing && !mbar_wait(pair_empty(s), (uint32_t)(q / kStemRing - 1) & 1u, p.err_flag)) return false;
      uint8_t* line = aline + s * S::kABytes;
      uint32_t w[NW];
      auto put = [&](int c, int c_src) {   // chunk c_src of the filter row (words 4 c_src .. + 3) as chunk c
        uint32_t v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = 4 * c_src + e < NW ? w[4 * c_src + e] : 0u;
        if (c_src == 0) v[0] &= 0xFFFF0000u;   // dummy column | first tap
        *reinterpret_cast<uint4*>(line + ((c ^ (r & 7)) << 4)) = make_uint4(v[0], v[1], v[2], v[3]);
      };
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        run[half].finish(e0, p.W * kStemCin, in.first, w);
#pragma unroll
        for (int c = 0; c < CH; ++c) put(half * CH + c, c);
        if (KH == 7 && half == 0) {
          put(6, 2);
          put(7, 3);   // past the row: zeros
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the tensor core
      __syncwarp();   // one arrival per warp: 128 of them on one barrier took 1000 clocks
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(pair_full(s)) : "memory");
      return true;
    };
    int q = 0;
    bool ok = true;
    stem_walk<POOL, PAIRS>(p, [&](int, int n, int oy, int fresh_pairs, int, bool, bool, int) {
      for (int k = PAIRS - fresh_pairs; k < PAIRS && ok; ++k, ++q) {
        // two sets of registers in turn: a pair's words are on their way while those of the one before are stored
        if (q & 1) {
          load(n, oy + k, wb);
          ok = store(q - 1, wa);
        } else {
          load(n, oy + k, wa);
          if (q) ok = store(q - 1, wb);
        }
      }
      return ok;
    });
    if (ok && q) (q & 1) ? store(q - 1, wa) : store(q - 1, wb);
  } else {
    // epilogue warps 5..12: TMEM lane quarter = warp % 4, 32 channels each
    const int quarter = warp & 3, half = (warp - 5) >> 2, et = (int)threadIdx.x - 160 - 128 * half;
    const int row = quarter * 32 + lane;
    if (threadIdx.x < 160 + 64) {
      const int c = threadIdx.x - 160;
      const bool in = c < p.N;
      s_scale[c] = (p.scale && in) ? p.scale[c] : 1.f;
      s_bias[c] = (p.bias && in) ? p.bias[c] : 0.f;
    }
    asm volatile("bar.sync 3, 256;" ::: "memory");   // once, before the row loop
    const bool idle = half * 32 >= p.N;               // no channels for this half: it only keeps the accumulators' count
    const float* sc = s_scale + half * 32;
    const float* bi = s_bias + half * 32;
    uint8_t* stage = gen + S::kOOff + half * (2 * kTcBM * 64);
    uint32_t vm[16];   // POOL: running maximum over the rows of the open pooled row: this thread's pixel column, 32 channels
#pragma unroll
    for (int i = 0; i < 16; ++i) vm[i] = 0u;
    bool live = true;
    const bool nonneg = p.act != EE_ACT_NONE;
    int emitted = 0;
    // Where a pooled row goes out, the four warps of a half meet at a barrier, so a warp whose wait ran out must not
    // leave: it raises s_abort and from then on only keeps the barrier's count; the others see the flag at their
    // next row and do the same.
    stem_walk<POOL, PAIRS>(p, [&](int j, int, int, int, int, bool fresh, bool emit, int t) {
      const int b = j & (kStemAccs - 1);
      if (POOL) live = live && !__any_sync(0xffffffffu, *s_abort != 0);
      if (live && !__all_sync(0xffffffffu, mbar_wait(acc_full(b), (uint32_t)(j / kStemAccs) & 1u, p.err_flag))) {
        live = false;
        *s_abort = 1;
      }
      if (!POOL && !live) return false;
      if (live) {
        tc_fence_after();
        float v[32];
        if (!idle) tmem_ld32(tmem_base + (uint32_t)(b * 64 + half * 32) + ((uint32_t)(quarter * 32) << 16), v);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty(b)) : "memory");   // the MMA warp may refill it
        if (idle) return true;
        uint32_t cur[16];   // this row's values
        uint4 o[4];
        epilogue32<false>(p.act, v, sc, bi, nullptr, o);
#pragma unroll
        for (int g = 0; g < 4; ++g) cur[4 * g] = o[g].x, cur[4 * g + 1] = o[g].y, cur[4 * g + 2] = o[g].z, cur[4 * g + 3] = o[g].w;
        if constexpr (!POOL) {
          uint8_t* mine = stage + quarter * 2048;   // 32 pixels of 64 bytes, their 16-byte chunks XORed with the pixel
#pragma unroll
          for (int g = 0; g < 4; ++g) *reinterpret_cast<uint4*>(mine + lane * 64 + ((g ^ (lane >> 1 & 3)) << 4)) = make_uint4(cur[4 * g], cur[4 * g + 1], cur[4 * g + 2], cur[4 * g + 3]);
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 4; ++k) {   // eight pixels per store, four lanes with 64 bytes of each
            const int px = k * 8 + (lane >> 2), g = lane & 3, ox = quarter * 32 + px, ch = half * 32 + g * 8;
            const uint4 x = *reinterpret_cast<const uint4*>(mine + px * 64 + ((g ^ (px >> 1 & 3)) << 4));
            if (ox < p.Wo && ch < p.N) *reinterpret_cast<uint4*>(p.out + ((size_t)t * p.Wo + ox) * p.N + ch) = x;
          }
          __syncwarp();
        } else {
          uint8_t* tile = stage + (emitted & 1) * (kTcBM * 64);
          if (nonneg) {
#pragma unroll
            for (int e = 0; e < 16; ++e) cur[e] += kPoolKey;
          }
          if (fresh) {
#pragma unroll
            for (int e = 0; e < 16; ++e) vm[e] = cur[e];
          } else if (nonneg) {
#pragma unroll
            for (int e = 0; e < 16; ++e) vm[e] = bf16x2_max<true>(vm[e], cur[e]);
          } else {
#pragma unroll
            for (int e = 0; e < 16; ++e) vm[e] = bf16x2_max<false>(vm[e], cur[e]);
          }
          if (emit) {
#pragma unroll
            for (int g = 0; g < 4; ++g)
              *reinterpret_cast<uint4*>(tile + row * 64 + ((g ^ (row >> 1 & 3)) << 4)) = make_uint4(vm[4 * g], vm[4 * g + 1], vm[4 * g + 2], vm[4 * g + 3]);
#pragma unroll
            for (int e = 0; e < 16; ++e) vm[e] = cur[e];   // the last row of a pooled row is the first row of the next one
          }
        }
      }
      if (!POOL || !emit || idle) return true;
      // the row of running maxima is staged; the tile is written again two pooled rows on, past the barrier of the next one
      asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
      const uint8_t* tile = stage + (emitted++ & 1) * (kTcBM * 64);
      if (!live) return true;
      auto columns = [&](auto sign) {
        constexpr bool NONNEG = decltype(sign)::value;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int idx = et + k * 128, px = idx >> 2, g = idx & 3, ch = half * 32 + g * 8;   // pooled pixel, 16-byte channel group
          if (px < p.Wp && ch < p.N) {
            auto at = [&](int c) { return *reinterpret_cast<const uint4*>(tile + c * 64 + ((g ^ (c >> 1 & 3)) << 4)); };
            auto most = [](uint4 m, uint4 a) {
              return make_uint4(bf16x2_max<NONNEG>(m.x, a.x), bf16x2_max<NONNEG>(m.y, a.y), bf16x2_max<NONNEG>(m.z, a.z), bf16x2_max<NONNEG>(m.w, a.w));
            };
            const int c1 = 2 * px;   // columns 2px-1 .. 2px+1, a column past the row's ends replaced by the middle one
            const uint4 x = at(c1), l = at(max(c1 - 1, 0)), r = at(min(c1 + 1, p.Wo - 1));
            const uint4 m = most(most(x, l), r);
            *reinterpret_cast<uint4*>(p.out + ((size_t)t * p.Wp + px) * p.N + ch) =
                make_uint4(bf16x2_pooled<NONNEG>(m.x), bf16x2_pooled<NONNEG>(m.y), bf16x2_pooled<NONNEG>(m.z), bf16x2_pooled<NONNEG>(m.w));
          }
        }
      };
      if (nonneg) columns(std::true_type{}); else columns(std::false_type{});
      return true;
    });
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kStemAccs * 64) : "memory");
  }
}

// Weight rows [Cout][KH][KH * 3] into the K layout above.
template <int KH>
__global__ void pack_stem_weights_kernel(const bf16* __restrict__ w, bf16* __restrict__ out, int rows) {
  using S = StemGeom<KH>;
  constexpr int run = KH * kStemCin;
  const long total = (long)rows * S::kPacked;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int k = (int)(idx % S::kPacked), pair = k / kTcBK, c = k % kTcBK;
    const long co = idx / S::kPacked;
    int r = -1, j = 0;   // filter row and column of its run
    if (pair + 1 < S::kPairs) {
      if (c < 2 * S::kCols) r = 2 * pair + c / S::kCols, j = c % S::kCols;
    } else if (c < 16) {
      r = KH - 1, j = c;
    } else if (KH == 7 && c >= 48 && c < 56) {
      r = KH - 1, j = c - 32;
    }
    out[idx] = r >= 0 && j >= 1 && j <= run ? w[(co * KH + r) * run + j - 1] : __float2bfloat16_rn(0.f);
  }
}

// ----------------------------------------------------------------------------- host side

inline bool stem_supported(const ee_layer_desc_t& d, int out_w) {
  return d.op == EE_OP_CONV && d.cin == kStemCin && (d.kh == 7 || d.kh == 3) && d.kw == d.kh && d.stride == 2 && d.pad == d.kh / 2 && d.pad_w == d.kh / 2 &&
         d.cout % 8 == 0 && d.cout <= 64 && out_w <= kTcBM;
}
inline int stem_packed_cols(int kh) { return kh == 7 ? StemGeom<7>::kPacked : StemGeom<3>::kPacked; }
inline void stem_pack(int kh, const bf16* w, bf16* out, int rows, cudaStream_t st) {
  const int blocks = cdiv((long)rows * stem_packed_cols(kh), 256);
  if (kh == 7)
    pack_stem_weights_kernel<7><<<blocks, 256, 0, st>>>(w, out, rows);
  else
    pack_stem_weights_kernel<3><<<blocks, 256, 0, st>>>(w, out, rows);
}

inline ee_status_t stem_context_init() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kernel, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set(conv_stem_tcgen05_kernel<7, false>, StemGeom<7>::kBytes);
  set(conv_stem_tcgen05_kernel<7, true>, StemGeom<7>::kBytes);
  set(conv_stem_tcgen05_kernel<3, false>, StemGeom<3>::kBytes);
  set(conv_stem_tcgen05_kernel<3, true>, StemGeom<3>::kBytes);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

// The pooling layer the stem kernel can take into its epilogue: 3x3 windows, stride 2, one pixel of padding.
inline bool stem_pool_supported(const ee_layer_desc_t& pool) {
  return pool.op == EE_OP_MAXPOOL && pool.kh == 3 && pool.kw == 3 && pool.stride == 2 && pool.pad == 1 && pool.pad_w == 1;
}

// L: the layer's GEMM view planned by tc_plan_layer over the packed weights (tm_w), with the g_* fields holding the
// geometry of the real convolution.  pool: dst is the output of the 3x3 stride-2 pad-1 max-pool behind the convolution,
// [B][(Ho-1)/2+1][(Wo-1)/2+1][Cout].
inline ee_status_t stem_launch(TcContext& c, const TcLayer& L, const void* src, void* dst, int B, const float* scale, const float* bias,
                               int* err_flag, cudaStream_t st, bool pool = false) {
  if (((uintptr_t)src & 15) || ((uintptr_t)dst & 15)) return EE_ERR_INVALID_ARG;
  StemParams p;
  p.tiles = B * L.out_h;
  p.H = L.g_h, p.W = L.g_w, p.Ho = L.out_h, p.Wo = L.out_w, p.N = L.cout;
  p.act = L.act;
  p.rev = L.rev ? 1 : 0;
  p.Hp = (L.out_h - 1) / 2 + 1, p.Wp = (L.out_w - 1) / 2 + 1, p.rows = B * p.Hp;
  p.total = (long)B * L.g_h * L.g_w * kStemCin;
  p.scale = scale, p.bias = bias;
  p.x = (const bf16*)src, p.out = (bf16*)dst;
  p.err_flag = err_flag;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(std::min(pool ? p.rows : p.tiles, c.sm_count));
  cfg.blockDim = dim3(kStemThreads);
  cfg.dynamicSmemBytes = L.g_kh == 7 ? StemGeom<7>::kBytes : StemGeom<3>::kBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (L.g_kh == 7)
    e = pool ? cudaLaunchKernelEx(&cfg, conv_stem_tcgen05_kernel<7, true>, L.tm_w, p) : cudaLaunchKernelEx(&cfg, conv_stem_tcgen05_kernel<7, false>, L.tm_w, p);
  else
    e = pool ? cudaLaunchKernelEx(&cfg, conv_stem_tcgen05_kernel<3, true>, L.tm_w, p) : cudaLaunchKernelEx(&cfg, conv_stem_tcgen05_kernel<3, false>, L.tm_w, p);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

}  // namespace ee
