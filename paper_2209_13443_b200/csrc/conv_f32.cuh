// Convolutions of the fp32 model: implicit GEMM on the double-precision matrix instruction.
//
// The fp32 model multiplies floats exactly and sums in fp64 (see Accum in common.cuh), so its bound is the fp64 rate
// (one DFMA per lane and two clocks) for large maps and, for the small maps this model is used on, latency: a layer
// has few output tiles and a long K, e.g. 24 x 512 outputs over K = 4608.  Both are answered by mma.m16n8k16.f64 (2048
// FMAs per instruction; operands converted from float once per fragment instead of once per product) and by cutting
// K: the 8 warps of a CTA are KG groups that take every KG-th 16-wide K step of a tile, and a cluster of Z CTAs cuts
// the K range of the tile once more.  Partial tiles (fp64) are added in ascending group order in each CTA, sent to the CTA
// that finishes their share of the tile (distributed shared memory) and added there in ascending CTA order.
// Z, KG and the tile depend on the layer and max_batch only, so a sample's sums are grouped the same way in any batch.
//
// A K group has a ring of its own, 16 of K a step, which its threads fill, and waits for nobody else: where a group is one warp, the
// fragments of one warp are fetched and converted while the other warp of its scheduler multiplies.  (With stages of 128 that all eight warps
// shared, a block-wide barrier each, loads, conversions and products took turns: of 9.7 us of a 3x3 512 -> 512 layer 1.7 and 3.5 were the
// last two.)  us a layer of the 64 x 64 model: 3x3 64 -> 64, batch 6 11.0 -> 9.9, 3x3 512 -> 512, 2 9.7 -> 8.3, 1x1 512 -> 2048, 2 5.2 -> 4.3;
// a pass at batch 6 479 -> 448, tiny model at 8 69 -> 64.
//
// What a small layer's time is (clocks of one CTA, 32 x 32 tile): 2050 of MMAs per 128 of K, which is the fp64 rate, and around
// them first operands, reduction and epilogue.  So weights are requested before the wait for the layer in front, scale, bias
// and residual come to registers during the K loop (fetched at the end they took 5000), tap positions are counted, not divided,
// and partial sums travel as asynchronous stores that the barrier of their receiver counts.  ResNet-50-shaped fp32 model at 64 x 64, batch 6:
// 630 -> 567 us a pass with these; K cut in equal numbers of 16-wide steps instead of whole ring stages (f32_plan.h) 526 -> 513.
#pragma once
#include "common.cuh"
#include "conv_simt.cuh"
#include "conv_tc.cuh"
#include "f32_plan.h"

namespace ee {

constexpr int kF32Threads = 256;

template <int WM, int WN, int KG, int MF, int NF>
struct F32Tile {   // WM x WN warps per K group, each MF x NF fragments of 16 x 8
  static constexpr int kBM = WM * MF * 16, kBN = WN * NF * 8, kKS = 16 * KG;   // output tile; K that the groups take together per step
  static constexpr int kGroup = 32 * WM * WN;              // threads of a K group
  static constexpr int kStages = KG == 8 && MF == 2 ? 3 : 4;   // steps in a group's ring
  static constexpr int kStageFloats = (kBM + kBN) * 16;    // rows of 16 floats, their four 16-byte chunks XORed with half the row: a fragment's 8 rows then lie in all banks
  static constexpr int kPRow = kBN + 2;                    // doubles per row of a partial tile
  static constexpr int kRing = KG * kStages * kStageFloats * 4, kPart = KG * kBM * kPRow * 8;
  static constexpr int kOuts = kBM * kBN / kF32Threads;    // outputs per thread
  static constexpr int kMain = kRing > kPart ? kRing : kPart;
  // a cluster's CTAs receive their share of the partial tiles behind the ring; the 64 x 64 tile is not cut further
  static constexpr int kRecv = KG == 8 ? kBM * kBN * 8 : 0;
  static constexpr int kBytes = kMain + kRecv + 16;        // and a barrier that counts it
  static_assert(WM * WN * KG == 8, "8 warps");
  static_assert(KG != 8 || 2 * (kBytes + kBM * 16 + 1024) <= 228 * 1024, "the plan counts two CTAs of these tiles an SM");
  static_assert(kBytes <= 227 * 1024, "exceeds the shared memory of an SM");
};

__device__ __forceinline__ void mma_f64(double* c, const double* a, const double* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7, %8, %9, %10, %11}, {%12, %13, %14, %15}, {%0, %1, %2, %3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(a[4]), "d"(a[5]), "d"(a[6]), "d"(a[7]), "d"(b[0]), "d"(b[1]), "d"(b[2]), "d"(b[3]));
}
__device__ __forceinline__ double lds_f64(uint32_t at) {   // a float of shared memory
  float x;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(at) : "memory");
  return x;
}
template <int BYTES>   // 16 or 4; `in` false fills zeros
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void* src, bool in) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
// Two doubles into the shared memory of CTA `rank` of the cluster; its barrier `bar` counts them.  addr, bar: as in this CTA.
__device__ __forceinline__ void st_async_f64x2(uint32_t addr, uint32_t bar, uint32_t rank, double v0, double v1) {
  asm volatile(
      "{\n .reg .b32 a, b;\n mapa.shared::cluster.u32 a, %0, %2;\n mapa.shared::cluster.u32 b, %1, %2;\n"
      " st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [a], {%3, %4}, [b];\n}"
      ::"r"(addr), "r"(bar), "r"(rank), "l"(__double_as_longlong(v0)), "l"(__double_as_longlong(v1))
      : "memory");
}

// V: floats per copy (4 when Cin is a multiple of 4 and the pointers are 16-byte aligned, else 1).  k_per: K range of a CTA.
template <int WM, int WN, int KG, int MF, int NF, int V>
__global__ void __launch_bounds__(kF32Threads, KG == 1 || KG == 8 ? 2 : 1)   // two CTAs an SM, which the plan counts on: 128 registers
conv_igemm_f64mma_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ scale,
                         const float* __restrict__ bias, const float* __restrict__ residual, float* __restrict__ y, ConvGeom g, int k_per,
                         int* err_flag, long long wait_cycles) {
  using S = F32Tile<WM, WN, KG, MF, NF>;
  constexpr int BM = S::kBM, BN = S::kBN, KS = S::kKS, STAGES = S::kStages;
  constexpr int UNITS = 16 / V;                       // copies per row and step
  constexpr int STEP = S::kGroup / UNITS;             // rows covered by one pass of a group
  constexpr int RA = (BM + STEP - 1) / STEP, RB = (BN + STEP - 1) / STEP;
  extern __shared__ __align__(16) uint8_t f32_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, kg = __shfl_sync(0xffffffffu, tid / S::kGroup, 0);   // the compiler is to know that a warp has one
  const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(f32_smem);
  const uint32_t ring_s = smem_s + (uint32_t)(kg * (STAGES * S::kStageFloats)) * 4u;   // of this thread's K group
  const int M = g.B * g.Ho * g.Wo, N = g.Cout, K = g.kh * g.kw * g.Cin;
  const int m0 = (int)blockIdx.x * BM, n0 = (int)blockIdx.y * BN;
  const int z = (int)blockIdx.z, Z = (int)gridDim.z;
  const int k_begin = z * k_per, k_end = min(K, k_begin + k_per);
  const int k_mine = k_begin + kg * 16, steps = max(0, (k_end - k_mine + KS - 1) / KS);   // this group's steps: k_mine, k_mine + KS, ...

  const int ku = tid % UNITS, r0 = tid % S::kGroup / UNITS;   // this thread copies column ku of rows r0, r0 + STEP, ...
  // An output row's first tap: sample x image rows, row and column.  Each thread keeps those of its rows, but for the 32-row tile copied in 4 bytes: there
  // they are 16, which with 16 addresses of weights took 254 registers and an SM to itself, half of what the plan counts on.  Read from shared
  // memory, and weights eight at a time, 126.  us a layer, one CTA an SM / spilled / so: 3x3 on 8 x 8 x 126, batch 4 23.2 / 14.3 / 12.0, on 14 x 14 x 30, 6
  // 12.5 / 9.0 / 7.5, 1x1 on 7 x 7 x 512 from an unaligned pointer, 6 24.8 / 24.7 / 19.4; where the grid never fills the chip, 3x3 on 7 x 7 x 62, 2, 6.8 / 8.4 / 7.3.
  constexpr bool TABLE = KG == 8 && MF == 2 && V == 1;
  auto row_at = [&](int r) {
    const int m = m0 + r;
    const bool in = r < BM && m < M;
    const int mm = in ? m : 0;
    const int wo = mm % g.Wo, q = mm / g.Wo, ho = q % g.Ho, b = q / g.Ho;
    return make_int4(b * g.H, in ? ho * g.stride - g.pad : -(1 << 20), wo * g.stride - g.pad_w, 0);   // far outside the image: zeros
  };
  __shared__ int4 s_rows[TABLE ? BM : 1];
  int4 my_rows[TABLE ? 1 : RA];
  if constexpr (TABLE) {
    if (tid < BM) s_rows[tid] = row_at(tid);
    __syncthreads();
  } else {
#pragma unroll
    for (int i = 0; i < RA; ++i) my_rows[i] = row_at(r0 + i * STEP);
  }
  auto place = [&](int row) { return ((ku * V / 4 ^ (row >> 1 & 3)) << 4) + ku * V % 4 * 4; };   // byte of this thread's column in a row
  // position of this thread's column in a step: K index, channel, filter row and column, walked by counters
  int k = k_mine + ku * V, ci = k % g.Cin, fs = k / g.Cin % g.kw, fr_ = k / g.Cin / g.kw;
  const int dci = KS % g.Cin, dtap = KS / g.Cin;
  auto load_b = [&](int step) {   // weights
    const uint32_t st = ring_s + (uint32_t)((step % STAGES) * S::kStageFloats) * 4u;
    const int kb = k_mine + step * KS + ku * V;
#pragma unroll (TABLE ? RB / 2 : RB)
    for (int i = 0; i < RB; ++i) {
      const int row = r0 + i * STEP, n = n0 + row;
      if (BN % STEP == 0 || row < BN) {
        const bool in = kb < k_end && n < N;
        cp_async_zfill<V * 4>(st + (uint32_t)((BM + row) * 64 + place(row)), in ? w + (size_t)n * K + kb : w, in);
      }
    }
  };
  auto load_a = [&](int step) {
    const uint32_t st = ring_s + (uint32_t)((step % STAGES) * S::kStageFloats) * 4u;
#pragma unroll
    for (int i = 0; i < RA; ++i) {
      const int row = r0 + i * STEP;
      if (BM % STEP == 0 || row < BM) {
        int4 at;
        if constexpr (TABLE) at = s_rows[row];
        else at = my_rows[i];
        const int hi = at.y + fr_, wi = at.z + fs;
        const bool in = k < k_end && hi >= 0 && hi < g.H && wi >= 0 && wi < g.W;
        cp_async_zfill<V * 4>(st + (uint32_t)(row * 64 + place(row)), in ? x + ((size_t)(at.x + hi) * g.W + wi) * g.Cin + ci : x, in);
      }
    }
    k += KS, ci += dci, fs += dtap;
    if (ci >= g.Cin) ci -= g.Cin, ++fs;
    while (fs >= g.kw) fs -= g.kw, ++fr_;
  };

  // no kernel writes weights, scale or bias: requested before the layer in front has finished
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s)
    if (s < steps) load_b(s);
  const uint32_t arrived = smem_s + (uint32_t)(S::kMain + S::kRecv);   // counts the partial sums that this CTA finishes
  if (Z > 1) {
    if (tid == 0) {
      mbar_init(arrived, 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      mbar_expect_tx(arrived, (uint32_t)(BM * BN * 8));
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  }
  // outputs z * share + 2 tid and its neighbour, + 512, ...: two channels per thread (512 is a multiple of every BN, Z is 1, 2, 4 or 8)
  const int share = BM * BN / Z, out_first = z * share + 2 * tid;
  const int nc = n0 + out_first % BN;
  float sc[2], bi[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) sc[h] = scale && nc + h < N ? scale[nc + h] : 1.f, bi[h] = bias && nc + h < N ? bias[nc + h] : 0.f;
  // The next layer's CTAs may set up and fetch their weights while this layer still waits: they wait for its end themselves.  A layer's own
  // prologue is long here (copies of 4 to 16 bytes), and behind the wait it was not over when its turn came: 497 -> 485 us a pass (64 x 64, batch 6).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < steps) load_a(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float res[S::kOuts];
#pragma unroll
  for (int i = 0; i < S::kOuts; i += 2) {
    const int m = m0 + (out_first + i * kF32Threads) / BN;
#pragma unroll
    for (int h = 0; h < 2; ++h) res[i + h] = residual && 2 * tid + i * kF32Threads < share && m < M && nc + h < N ? residual[(size_t)m * N + nc + h] : 0.f;
  }
  const int wmn = warp % (WM * WN), wm = wmn / WN, wn = wmn % WN;
  const int fr = lane >> 2, fk = lane & 3;            // fragment row (column of B) and K position of this lane
  double acc[MF][NF][4];
#pragma unroll
  for (int i = 0; i < MF; ++i)
#pragma unroll
    for (int j = 0; j < NF; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0;
  uint32_t chunk[4];   // of K 4 e .. 4 e + 3, in this lane's rows
#pragma unroll
  for (int e = 0; e < 4; ++e) chunk[e] = ring_s + (uint32_t)(fr * 64 + ((e ^ (fr >> 1 & 3)) << 4) + fk * 4);
  int at = 0;   // step % STAGES
  for (int step = 0; step < steps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    // this step has landed for the whole group; the one refilled below was read a step ago
    if constexpr (S::kGroup == 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1 + kg), "n"(S::kGroup) : "memory");
    if (step + STAGES - 1 < steps) {
      load_a(step + STAGES - 1);
      load_b(step + STAGES - 1);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t stage = (uint32_t)(at * S::kStageFloats * 4), a_at = stage + (uint32_t)(wm * MF * 16 * 64), b_at = stage + (uint32_t)((BM + wn * NF * 8) * 64);
    if (++at == STAGES) at = 0;
    double b[NF][4];
#pragma unroll
    for (int j = 0; j < NF; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) b[j][e] = lds_f64(chunk[e] + b_at + j * 8 * 64);
#pragma unroll
    for (int i = 0; i < MF; ++i) {
      double a[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) a[e] = lds_f64(chunk[e >> 1] + a_at + (i * 16 + 8 * (e & 1)) * 64);
#pragma unroll
      for (int j = 0; j < NF; ++j) mma_f64(acc[i][j], a, b[j]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // partial tiles: [KG][BM][kPRow] doubles over the drained ring
  double* part = reinterpret_cast<double*>(f32_smem);
  {
    double* p = part + ((size_t)kg * BM + wm * MF * 16 + fr) * S::kPRow + wn * NF * 8 + 2 * fk;
#pragma unroll
    for (int i = 0; i < MF; ++i)
#pragma unroll
      for (int j = 0; j < NF; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          *reinterpret_cast<double2*>(p + (i * 16 + 8 * h) * S::kPRow + j * 8) = make_double2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
  }
  __syncthreads();
  auto group_sum = [&](int o) {   // of two outputs side by side
    double2 v = *reinterpret_cast<const double2*>(part + o);
#pragma unroll
    for (int q = 1; q < KG; ++q) {
      const double2 t = *reinterpret_cast<const double2*>(part + q * BM * S::kPRow + o);
      v.x += t.x, v.y += t.y;
    }
    return v;
  };
  double* recv = reinterpret_cast<double*>(f32_smem + S::kMain);   // [Z][share]
  if (Z > 1) {
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");   // every CTA of the cluster runs
    const uint32_t recv_s = smem_s + (uint32_t)S::kMain;
#pragma unroll
    for (int i = 0; i < S::kOuts; i += 2) {
      const int idx = 2 * tid + i * kF32Threads, q = idx / share;
      const double2 v = group_sum(idx / BN * S::kPRow + idx % BN);
      st_async_f64x2(recv_s + (uint32_t)(z * share + idx - q * share) * 8u, arrived, (uint32_t)q, v.x, v.y);
    }
    // Nothing but the data is waited for; a barrier of the cluster behind plain stores cost a pass of the ResNet-50-shaped model at 64 px 6 us of
    // 427 at batch 6, 18 of 365 at batch 2.  Whoever waits here has been sent everything, so a CTA may leave while its own stores are on their way; one whose
    // wait ran out stays until it has been.
    if (!mbar_wait_cluster(arrived, 0, err_flag, wait_cycles) && !cluster_drain(arrived, 0, err_flag)) return;
  }
#pragma unroll
  for (int i = 0; i < S::kOuts; i += 2) {
    const int rel = 2 * tid + i * kF32Threads, idx = z * share + rel, m = m0 + idx / BN;
    if (rel >= share || m >= M) continue;
    double v[2] = {0.0, 0.0};
    if (Z > 1) {
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q < Z) {
          const double2 t = *reinterpret_cast<const double2*>(recv + q * share + rel);
          v[0] += t.x, v[1] += t.y;
        }
    } else {
      const double2 t = group_sum(idx / BN * S::kPRow + idx % BN);
      v[0] = t.x, v[1] = t.y;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (nc + h >= N) continue;
      double t = (double)sc[h] * v[h] + (double)bi[h];
      if (residual) t += (double)res[i + h];
      y[(size_t)m * N + nc + h] = (float)apply_act(t, g.act);
    }
  }
}

// ----------------------------------------------------------------------------- host side

template <int WM, int WN, int KG, int MF, int NF, int V>
inline cudaError_t f32_launch_t(const F32Plan& p, const float* x, const float* w, const float* scale, const float* bias, const float* residual,
                                float* y, const ConvGeom& g, int* err_flag, long long wait_cycles, cudaStream_t st) {
  using S = F32Tile<WM, WN, KG, MF, NF>;
  if (p.z > 1 && S::kRecv == 0) return cudaErrorInvalidValue;   // no room for what a cluster's CTAs send
  const int K = g.kh * g.kw * g.Cin;
  const int k_per = f32_k_per(K, p.z);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cdiv((long)g.B * g.Ho * g.Wo, S::kBM), cdiv(g.Cout, S::kBN), p.z);
  cfg.blockDim = dim3(kF32Threads);
  cfg.dynamicSmemBytes = S::kBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = p.z;
  cfg.attrs = attr;
  cfg.numAttrs = p.z > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, conv_igemm_f64mma_kernel<WM, WN, KG, MF, NF, V>, x, w, scale, bias, residual, y, g, k_per, err_flag, wait_cycles);
}

template <int V>
inline cudaError_t f32_launch_v(const F32Plan& p, const float* x, const float* w, const float* scale, const float* bias, const float* residual,
                                float* y, const ConvGeom& g, int* err_flag, long long wait_cycles, cudaStream_t st) {
  switch (p.tile) {
    case 1: return f32_launch_t<2, 2, 2, 2, 4, V>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st);
    case 2: return f32_launch_t<1, 1, 8, 2, 4, V>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st);
    case 3: return f32_launch_t<1, 1, 8, 1, 4, V>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st);
    default: return f32_launch_t<4, 2, 1, 1, 2, V>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st);
  }
}

inline cudaError_t f32_launch(const F32Plan& p, const float* x, const float* w, const float* scale, const float* bias, const float* residual,
                              float* y, const ConvGeom& g, int* err_flag, long long wait_cycles, cudaStream_t st) {
  const bool vec = g.Cin % 4 == 0 && (((uintptr_t)x | (uintptr_t)w) & 15) == 0;
  return vec ? f32_launch_v<4>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st) : f32_launch_v<1>(p, x, w, scale, bias, residual, y, g, err_flag, wait_cycles, st);
}

inline ee_status_t f32_context_init() {
  cudaError_t e = cudaSuccess;
  auto set = [&](auto kernel, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  set(conv_igemm_f64mma_kernel<4, 2, 1, 1, 2, 4>, F32Tile<4, 2, 1, 1, 2>::kBytes);
  set(conv_igemm_f64mma_kernel<4, 2, 1, 1, 2, 1>, F32Tile<4, 2, 1, 1, 2>::kBytes);
  set(conv_igemm_f64mma_kernel<2, 2, 2, 2, 4, 4>, F32Tile<2, 2, 2, 2, 4>::kBytes);
  set(conv_igemm_f64mma_kernel<2, 2, 2, 2, 4, 1>, F32Tile<2, 2, 2, 2, 4>::kBytes);
  set(conv_igemm_f64mma_kernel<1, 1, 8, 2, 4, 4>, F32Tile<1, 1, 8, 2, 4>::kBytes);
  set(conv_igemm_f64mma_kernel<1, 1, 8, 2, 4, 1>, F32Tile<1, 1, 8, 2, 4>::kBytes);
  set(conv_igemm_f64mma_kernel<1, 1, 8, 1, 4, 4>, F32Tile<1, 1, 8, 1, 4>::kBytes);
  set(conv_igemm_f64mma_kernel<1, 1, 8, 1, 4, 1>, F32Tile<1, 1, 8, 1, 4>::kBytes);
  return e == cudaSuccess ? EE_OK : EE_ERR_CUDA;
}

}  // namespace ee
