// Stride-2 stem convolutions on 3-channel bf16 images (7x7 of the ResNet-style backbones, 3x3 of the MobileNet-style ones), as
// an implicit GEMM on tcgen05.mma.
//
// A 3-channel pixel is 6 bytes, so no TMA load can fetch operand rows.  But in an image row whose pixels are padded to four channels, 8
// bytes, the operand row of output pixel ox is the run of pixels from 2 ox - pad on, 16 bytes further for every ox: read without
// swizzle, as groups of eight rows of 16 bytes with 128 bytes from group to group, the image row IS the operand, whose rows overlap, and
// a filter row is one (3x3) or two (7x7) K steps at fixed offsets into it.  Nothing is built per output pixel; a row that several
// output rows read is in shared memory once.
//
// A run starts at an odd pixel, and the pixel in front of it must not enter the sum, not even times zero.  So an image row is two
// arrays of pixel pairs: "odd", with zeros in place of the even pixel, and "both".  A K step is two pairs, the second at any distance
// from the first (the descriptor's leading offset): taps 0 | 1 2 from "odd" and "both", taps 3 4 | 5 6 from "both".
//
// One persistent CTA per SM walks a contiguous range of output rows; the unit is a PAIR of image rows (2 P - pad, 2 P - pad + 1) in a ring,
// read by the up to (kh + 1) / 2 output rows P, P - 1, ...  Four gather warps, a thread per pixel pair, fetch three words of a row
// with cp.async, eight pairs of rows ahead, and put them into the arrays; one thread issues the MMAs into four accumulators in turn;
// eight epilogue warps, 32 channels of 32 pixels each, finish the rows.
// What bounds it: none of its parts alone.  7x7 and pool on 64 images of 224 x 224 take 50 us, without the pooled rows' exchange 38, without any
// epilogue 30: gather (650 clocks a row; 1430 to 1600 when every output pixel gathered its own runs), MMAs (780) and epilogue with the pool behind
// it (1500; sixteen warps of 16 channels take as long, and at 80 registers spill) overlap only in part.  A stage of the
// stem, the pool and an 8-channel 1x1 layer, gather per output pixel -> this, us: 7x7, batch 64 of 224 x 224 images 77.9 -> 74.9, batch 7
// 30.8 -> 27.6, batch 21 of 161 x 161 41.1 -> 37.2; 3x3 without a pool, batch 32 of 224 x 224 74.3 -> 63.6.
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

constexpr int kStemEpi = 8, kStemThreads = 32 * (5 + kStemEpi);      // MMA warp, 4 gather warps, epilogue warps
constexpr int kStemRing = 8, kStemAccs = 4, kStemCin = 3, kStemAhead = 8;

template <int KH>
struct StemGeom {
  static constexpr int kPad = KH / 2, kPairs = (KH + 1) / 2;
  static constexpr int kCols = KH == 7 ? 32 : 16;            // columns of a filter row
  static constexpr int kPacked = kPairs * kTcBK;             // columns of the packed weights, a K block per pair
  static constexpr int kLine = 136 * 16;                     // bytes of one array of an image row: two pixel pairs of padding, 128, and six
  static constexpr int kRow = 2 * kLine;                     // "odd" and "both"
  static constexpr int kABytes = 2 * kRow, kWBytes = 64 * kTcBK * 2;
  static constexpr int kWOff = (kStemRing * kABytes + 1023) / 1024 * 1024;
  static constexpr int kOOff = kWOff + kPairs * kWBytes;
  static constexpr int kScaleOff = kOOff + 4 * kTcBM * 64;   // staging: two tiles of 128 pixels x 32 channels per channel half
  static constexpr int kRawOff = kScaleOff + 2 * 64 * 4;     // words on their way: [pair][image row][word][thread]
  static constexpr int kBarOff = kRawOff + kStemAhead * 2 * 4 * 128 * 4;
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

// The pairs that the rows of stem_walk meet, in order: image n, rows 2 P - pad and 2 P - pad + 1 of it.
template <bool POOL, int PAIRS>
struct StemPairs {
  const StemParams& p;
  int r, r1, per, n, y;   // y: pooled row (POOL) or output row
  int P, last;            // pairs of the open row still to come: P .. last
  __device__ __forceinline__ explicit StemPairs(const StemParams& q) : p(q) {
    const long g = p.rev ? (long)gridDim.x - 1 - blockIdx.x : (long)blockIdx.x;
    const int all = POOL ? p.rows : p.tiles;
    per = POOL ? p.Hp : p.Ho;
    r = (int)(g * all / gridDim.x), r1 = (int)((g + 1) * all / gridDim.x);
    n = r / per, y = r - n * per;
    open(true);
  }
  __device__ __forceinline__ void open(bool first) {
    const int lo = POOL ? (first ? max(2 * y - 1, 0) : 2 * y) : y, hi = POOL ? min(2 * y + 1, p.Ho - 1) : y;
    P = first ? lo : lo + PAIRS - 1, last = hi + PAIRS - 1;
  }
  __device__ __forceinline__ bool more() const { return r < r1; }
  __device__ __forceinline__ void next() {
    if (++P <= last) return;
    ++r;
    if (++y == per) y = 0, ++n;
    open(y == 0);
  }
};

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

// A pixel pair (elements e0 .. e0 + 5 of an image row, e0 even) in two steps: `load` only requests aligned words (stem_words.h says
// which) into the thread's own column of a staging buffer, `finish` makes the pair's three words of them.  Copies, not registers,
// hold what is on its way: kStemAhead pairs of rows.  Words outside the row arrive as zeros.  Rows of an odd number of elements start at
// an odd element every other time; their words are put together from two aligned ones.
struct StemRun {
  static constexpr int NW = 3;
  __device__ __forceinline__ static void load(const StemParams& p, uint32_t dst, int n, int y, int e0, StemTaps in) {
    const int row_elems = p.W * kStemCin;
    if (y < 0 || y >= p.H) in.first = in.second = 0;
    const long rb = ((long)n * p.H + y) * row_elems;
    const StemAsk ask = stem_ask(rb, row_elems, p.total, in);
    const bf16* src = p.x + (rb + e0 + ask.off);
#pragma unroll
    for (int j = 0; j <= NW; ++j) {
      const int bytes = stem_word_bytes(ask, in, j);
      if (j < NW || ask.kind == 2) asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + j * 512), "l"(bytes ? src + 2 * j : p.x), "r"(bytes) : "memory");
    }
  }
  __device__ __forceinline__ static void finish(const StemParams& p, const uint32_t* col, int n, int y, int e0, uint32_t in, uint32_t* w) {
    const int row_elems = p.W * kStemCin;
#pragma unroll
    for (int j = 0; j < NW; ++j) w[j] = col[j * 128];
    if (!(row_elems & 1)) return;
    const bool odd = (((long)n * p.H + y) * row_elems & 1) != 0;
    uint32_t next = odd ? col[NW * 128] : 0u;
#pragma unroll
    for (int j = NW - 1; j >= 0; --j) {
      const uint32_t a = w[j];
      if (odd) w[j] = in >> j & 1u ? __byte_perm(a, next, 0x5432) : 0u;
      if (e0 + 2 * j == row_elems - 1) w[j] &= 0xffffu;   // the row's last element, alone in its word
      next = a;
    }
  }
};

// Descriptor of an operand without swizzle: groups of eight rows of 16 bytes, 128 bytes from one to the next; a K step's second half lies `lead` bytes further.
__device__ __forceinline__ uint64_t stem_desc(uint32_t addr, int lead) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | (uint64_t)(lead >> 4) << 16 | (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46;
}

// The epilogue of a thread's pixel column with the pool behind it: the running maximum over the rows of a pooled row in registers,
// then the maximum over three columns through shared memory.  Where a pooled row goes out, the four warps of a half meet at a
// barrier, so a warp whose wait ran out must not leave: it raises s_abort and from then on only keeps the barrier's count; the
// others see the flag at their next pooled row and do the same.
template <bool NONNEG, typename W, typename V>
__device__ __forceinline__ void stem_pool_rows(const StemParams& p, uint8_t* stage, volatile int* s_abort, int r0, int r1, int half, int row, int et,
                                               bool idle, W&& arrived, V&& values) {
  uint4 vm[4];   // the open pooled row
  auto most = [](uint4 m, uint4 a) {
    return make_uint4(bf16x2_max<NONNEG>(m.x, a.x), bf16x2_max<NONNEG>(m.y, a.y), bf16x2_max<NONNEG>(m.z, a.z), bf16x2_max<NONNEG>(m.w, a.w));
  };
  // the two pooled pixels whose 16-byte channel group this thread finishes: columns 2 px - 1 .. 2 px + 1, a column past the row's
  // ends replaced by the middle one
  const int g = et & 3, ch = half * 32 + g * 8, px0 = et >> 2;
  uint32_t at[2][3];
  bool mine[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int px = px0 + 32 * k;
    mine[k] = px < p.Wp && ch < p.N;
    const int c[3] = {2 * px, max(2 * px - 1, 0), min(2 * px + 1, p.Wo - 1)};
#pragma unroll
    for (int i = 0; i < 3; ++i) at[k][i] = (uint32_t)(c[i] * 64 + ((g ^ (c[i] >> 1 & 3)) << 4));
  }
  bf16* out = p.out + ((size_t)r0 * p.Wp + px0) * p.N + ch;
  bool live = true;
  int y = r0 % p.Hp, j = 0;
  for (int t = r0; t < r1; ++t, out += (size_t)p.Wp * p.N) {
    live = live && !__any_sync(0xffffffffu, *s_abort != 0);
    bool fresh = t == r0 || y == 0;          // else vm holds the row above, the last one of the pooled row before
    const int last = min(2 * y + 1, p.Ho - 1);
    for (int c = fresh ? max(2 * y - 1, 0) : 2 * y; c <= last; ++c, ++j) {
      if (!live) continue;
      if (!arrived(j)) {
        live = false;
        *s_abort = 1;
        continue;
      }
      uint4 cur[4];
      values(j, cur);
      if (idle) continue;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (NONNEG) cur[i].x += kPoolKey, cur[i].y += kPoolKey, cur[i].z += kPoolKey, cur[i].w += kPoolKey;
        vm[i] = fresh ? cur[i] : most(vm[i], cur[i]);
      }
      fresh = false;
      if (c == last) {
        uint8_t* line = stage + (t & 1) * (kTcBM * 64) + row * 64;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          *reinterpret_cast<uint4*>(line + ((i ^ (row >> 1 & 3)) << 4)) = vm[i];
          vm[i] = cur[i];                    // the last row of a pooled row is the first row of the next one
        }
      }
    }
    if (++y == p.Hp) y = 0;
    if (idle) continue;
    // the row of running maxima is staged; the tile is written again two pooled rows on, past the barrier of the next one
    asm volatile("bar.sync %0, 128;" ::"r"(1 + half) : "memory");
    if (!live) continue;
    const uint8_t* tile = stage + (t & 1) * (kTcBM * 64);
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (mine[k]) {
        auto col = [&](int i) { return *reinterpret_cast<const uint4*>(tile + at[k][i]); };
        uint4 m = most(most(col(0), col(1)), col(2));
        if (NONNEG && ((m.x | m.y | m.z | m.w) & 0x80008000u) == 0)   // no NaN (and no -0) among them
          m = make_uint4(m.x - kPoolKey, m.y - kPoolKey, m.z - kPoolKey, m.w - kPoolKey);
        else
          m = make_uint4(bf16x2_pooled<NONNEG>(m.x), bf16x2_pooled<NONNEG>(m.y), bf16x2_pooled<NONNEG>(m.z), bf16x2_pooled<NONNEG>(m.w));
        *reinterpret_cast<uint4*>(out + (size_t)(32 * k) * p.N) = m;
      }
  }
}

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
    mbar_init(bar0 + 8u * i, i >= 1 && i <= kStemRing ? 4 : i > 2 * kStemRing + kStemAccs ? kStemEpi : 1);
    if (i == 0) *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the padding that no gather thread writes: pixel pairs -2, -1, 128 and 129 of every array
  for (int i = threadIdx.x; i < kStemRing * 4 * 4; i += kStemThreads) {
    const int e = i & 3;
    *reinterpret_cast<uint4*>(gen + (i >> 2) * S::kLine + (e < 2 ? e : 128 + e) * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 0) {
    if (lane == 0) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(kStemAccs * 64) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) {   // the whole weight matrix stays resident; no kernel writes it, so it need not wait
    mbar_expect_tx(w_bar, PAIRS * S::kWBytes);
    for (int i = 0; i < PAIRS; ++i) tma_load_3d(base + S::kWOff + i * S::kWBytes, &tmW, w_bar, i * kTcBK, 0, 0);
  }
  __syncwarp();
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == 0) {
    if (elect_one()) {
      constexpr uint32_t idesc = umma_idesc(64);
      // K step 0 of a filter row: taps 0, 1 and 2 (the odd pixel of a pair, the next pair whole), step 1: taps 3 to 6
      const uint64_t d0 = stem_desc(base + (KH == 7 ? 0 : 16), S::kLine + 16), d1 = stem_desc(base + S::kLine + 32, 16), db0 = umma_desc(base + S::kWOff);
      int q = 0;   // pairs the rows so far have met
      bool acc_here = false, pair_here = false;   // asked for while the row before was being computed: a wait costs its thread 200 clocks
      if (mbar_wait(w_bar, 0, p.err_flag))
        stem_walk<POOL, PAIRS>(p, [&](int j, int, int, int fresh_pairs, int free_pairs, bool, bool, int) {
          const int b = j & (kStemAccs - 1);
          // the epilogue must have drained this accumulator
          if (j >= kStemAccs && !acc_here && !mbar_wait(acc_empty(b), (uint32_t)(j / kStemAccs - 1) & 1u, p.err_flag)) return false;
          tc_fence_after();
          q += fresh_pairs;
          const uint32_t acc = tmem_base + (uint32_t)(b * 64);
#pragma unroll
          for (int k = 0; k < PAIRS; ++k) {
            const int pq = q - PAIRS + k, s = pq & (kStemRing - 1);
            if (k >= PAIRS - fresh_pairs && !(pair_here && k == PAIRS - fresh_pairs) && !mbar_wait(pair_full(s), (uint32_t)(pq / kStemRing) & 1u, p.err_flag)) return false;
            const uint64_t off = (uint64_t)(s * (S::kABytes >> 4)), db = db0 + (uint64_t)(k * (S::kWBytes >> 4));
#pragma unroll
            for (int half = 0; half < 2; ++half) {
              if (half == 1 && k + 1 == PAIRS) break;   // the last filter row alone
              const uint64_t row = off + (uint64_t)(half * (S::kRow >> 4));
              umma_bf16(acc, d0 + row, db + half * (S::kCols / 8), idesc, (uint32_t)(k != 0 || half != 0));
              if (KH == 7) umma_bf16(acc, d1 + row, db + half * (S::kCols / 8) + 2, idesc, 1u);
            }
          }
          pair_here = mbar_test_wait(pair_full(q & (kStemRing - 1)), (uint32_t)(q / kStemRing) & 1u);
          acc_here = j + 1 >= kStemAccs && mbar_test_wait(acc_empty((j + 1) & (kStemAccs - 1)), (uint32_t)((j + 1) / kStemAccs - 1) & 1u);
          umma_commit(acc_full(b));
          for (int k = 0; k < free_pairs; ++k) umma_commit(pair_empty((q - PAIRS + k) & (kStemRing - 1)));
          return true;
        });
    }
    __syncwarp();
  } else if (warp < 5) {
    // gather warps: thread r puts pixels 2 r and 2 r + 1 of every image row into its arrays
    const int r = (int)threadIdx.x - 32, e0 = 2 * kStemCin * r;   // image-row element of pixel 2 r
    const StemTaps in = r < p.Wo ? stem_taps(e0, p.W * kStemCin, 3) : StemTaps{0u, 0u};   // behind the row: zeros
    uint8_t* at = gen + (r + 2) * 16;
    const uint32_t raw0 = base + S::kRawOff + r * 4;
    const uint32_t* col0 = reinterpret_cast<const uint32_t*>(gen + S::kRawOff) + r;
    // Rows of an even number of elements: every word is whole and aligned, and a pair of rows costs a thread two addresses.
    const bool even = (p.W & 1) == 0;
    const uint32_t size = r < p.Wo ? 4u : 0u;
    const char* src0 = reinterpret_cast<const char*>(p.x) + (r < p.Wo ? 2 * e0 : 0);
    const uint32_t row_bytes = (uint32_t)p.W * (2 * kStemCin);
    auto load = [&](int q, int n, int P) {
      const uint32_t dst = raw0 + (uint32_t)(q & (kStemAhead - 1)) * 4096u;
      const int y = 2 * P - S::kPad;
      if (even) {
        const char* src = src0 + (long)(n * p.H + y) * row_bytes;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const bool in = (unsigned)(y + half) < (unsigned)p.H;
          const char* at = in ? src + half * row_bytes : src0;
#pragma unroll
          for (int j = 0; j < 3; ++j)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + half * 2048 + j * 512), "l"(at + 4 * j), "r"(in ? size : 0u) : "memory");
        }
      } else {
        StemRun::load(p, dst, n, y, e0, in);
        StemRun::load(p, dst + 2048u, n, y + 1, e0, in);
      }
    };
    auto store = [&](int q, int n, int P) {
      const int s = q & (kStemRing - 1);
      if (q >= kStemRing && !mbar_wait(pair_empty(s), (uint32_t)(q / kStemRing - 1) & 1u, p.err_flag)) return false;
      const uint32_t* col = col0 + (q & (kStemAhead - 1)) * 1024;
      uint8_t* row = at + s * S::kABytes;
#pragma unroll
      for (int half = 0; half < 2; ++half, row += S::kRow) {
        uint32_t w[3];
        if (even) {
#pragma unroll
          for (int j = 0; j < 3; ++j) w[j] = col[half * 512 + j * 128];
        } else {
          StemRun::finish(p, col + half * 512, n, 2 * P - S::kPad + half, e0, in.first, w);
        }
        const uint32_t lo = __byte_perm(w[1], w[2], 0x5432), hi = w[2] >> 16;   // the odd pixel
        *reinterpret_cast<uint4*>(row) = make_uint4(0u, 0u, lo, hi);
        *reinterpret_cast<uint4*>(row + S::kLine) = make_uint4(w[0], w[1] & 0xffffu, lo, hi);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the tensor core
      __syncwarp();   // one arrival per warp: 128 of them on one barrier took 1000 clocks
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(pair_full(s)) : "memory");
      return true;
    };
    // two walks over the same pairs, the first kStemAhead - 1 pairs in front of the second
    StemPairs<POOL, PAIRS> ahead(p), here(p);
    bool ok = true;
    for (int q = 0; q < kStemAhead - 1; ++q) {
      if (ahead.more()) load(q, ahead.n, ahead.P), ahead.next();
      cp_async_commit();
    }
    for (int q = 0; ok && here.more(); ++q) {
      if (ahead.more()) load(q + kStemAhead - 1, ahead.n, ahead.P), ahead.next();
      cp_async_commit();
      cp_async_wait<kStemAhead - 1>();
      ok = store(q, here.n, here.P);
      here.next();
    }
    cp_async_wait<0>();
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
    const uint32_t acc0 = tmem_base + (uint32_t)(half * 32) + ((uint32_t)(quarter * 32) << 16);
    auto arrived = [&](int j) { return __all_sync(0xffffffffu, mbar_wait(acc_full(j & (kStemAccs - 1)), (uint32_t)(j / kStemAccs) & 1u, p.err_flag)); };
    auto values = [&](int j, uint4* o) {   // of row j: this thread's pixel column, 32 channels
      tc_fence_after();
      float v[32];
      if (!idle) tmem_ld32(acc0 + (uint32_t)((j & (kStemAccs - 1)) * 64), v);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty(j & (kStemAccs - 1))) : "memory");   // the MMA warp may refill it
      if (!idle) epilogue32<false>(p.act, v, sc, bi, nullptr, o);
    };
    const long g0 = p.rev ? (long)gridDim.x - 1 - blockIdx.x : (long)blockIdx.x;
    const int all = POOL ? p.rows : p.tiles, r0 = (int)(g0 * all / gridDim.x), r1 = (int)((g0 + 1) * all / gridDim.x);
    uint4 cur[4];
    if constexpr (!POOL) {
      uint8_t* mine = stage + quarter * 2048;   // 32 pixels of 64 bytes, their 16-byte chunks XORed with the pixel
      for (int t = r0; t < r1; ++t) {
        if (!arrived(t - r0)) break;
        values(t - r0, cur);
        if (idle) continue;
#pragma unroll
        for (int g = 0; g < 4; ++g) *reinterpret_cast<uint4*>(mine + lane * 64 + ((g ^ (lane >> 1 & 3)) << 4)) = cur[g];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) {   // eight pixels per store, four lanes with 64 bytes of each
          const int px = k * 8 + (lane >> 2), g = lane & 3, ox = quarter * 32 + px, ch = half * 32 + g * 8;
          const uint4 x = *reinterpret_cast<const uint4*>(mine + px * 64 + ((g ^ (px >> 1 & 3)) << 4));
          if (ox < p.Wo && ch < p.N) *reinterpret_cast<uint4*>(p.out + ((size_t)t * p.Wo + ox) * p.N + ch) = x;
        }
        __syncwarp();
      }
    } else if (p.act != EE_ACT_NONE) {
      stem_pool_rows<true>(p, stage, s_abort, r0, r1, half, row, et, idle, arrived, values);
    } else {
      stem_pool_rows<false>(p, stage, s_abort, r0, r1, half, row, et, idle, arrived, values);
    }
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
  const long total = (long)rows * S::kPacked;
  for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    const int k = (int)(idx % S::kPacked), pair = k / kTcBK, c = k % kTcBK;
    const long co = idx / S::kPacked;
    const int r = 2 * pair + c / S::kCols, tap = c % S::kCols / 4 - 1, ch = c % 4;   // four columns a pixel, the first pixel of a row a dummy
    const bool in = c < 2 * S::kCols && r < KH && tap >= 0 && tap < KH && ch < kStemCin;
    out[idx] = in ? w[((co * KH + r) * KH + tap) * kStemCin + ch] : __float2bfloat16_rn(0.f);
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
