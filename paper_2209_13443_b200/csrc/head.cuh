// Exit head and batch bookkeeping kernels: global average pool, FC, softmax top-1 + threshold,
// stable compaction scan, survivor gather, refill copy.
//
// The exit head is the intermediate classifier whose softmax top-1 probability is the
// confidence that is compared with the exit's threshold (paper Section II-B; Section IV,
// Benchmarks).  The scan produces B_rem = B_act - B_exit and the order-preserving list of the
// remaining samples, the gather is their write-back to the next subnet's input buffer
// (Section III-B, Preemption Mechanism), the refill copy appends B_incr new samples
// (Algorithm 1: B_merged = B_rem + B_incr).
//
// All reductions run in a fixed order that depends on the layer shape only, never on the
// batch size or on scheduling, so a sample's logits are bit-identical in any batch.
#pragma once
#include "conv_tc.cuh"
#include "fc_shape.h"

namespace ee {

constexpr int kGapThreads = 256;

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Adds the rows grp, grp + groups, ... of a [HW][C] map to acc, one vector of VEC channels at p, in ascending order, eight loads in flight: what
// a row group of gap_kernel does, and of an FC kernel that pools by itself.
template <typename T, int VEC, typename A>
__device__ __forceinline__ void pool_rows(const T* p, int HW, int C, int grp, int groups, A* acc) {
  int r = grp;
  if constexpr (VEC > 1) {
    for (; r + 7 * groups < HW; r += 8 * groups) {
      Vec16<T> t[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) t[u].load(p + (size_t)(r + u * groups) * C);
#pragma unroll
      for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int e = 0; e < VEC; ++e) acc[e] += t[u].v[e];
    }
  }
  for (; r < HW; r += groups) {
    if constexpr (VEC > 1) {
      Vec16<T> t;
      t.load(p + (size_t)r * C);
#pragma unroll
      for (int e = 0; e < VEC; ++e) acc[e] += t.v[e];
    } else {
      acc[0] += Elem<T>::ld(p + (size_t)r * C);
    }
  }
}

// gap[b][c] = mean over the HW rows of sample b's [HW][C] map, in one pass.  A CTA owns one sample and a slab of
// `lanes` channel vectors: its 256 threads form 256 / lanes row groups, group g adds rows g, g + groups, ... in
// ascending order (eight loads in flight), then the first lanes * VEC threads add the group sums in ascending group
// order.  `lanes` depends on the layer shape only (few rows: wide slabs; many rows: many row groups), so the
// grouping of a sample's sum is the same in every batch.  Block (0, 0) also zeroes the n_zero counters that the
// FC kernel behind it in the stream relies on.  Launched with programmatic stream serialization.
template <typename T, int VEC>
__global__ void __launch_bounds__(kGapThreads)
gap_kernel(const T* __restrict__ x, int HW, int C, int lanes, float* __restrict__ gap, unsigned* __restrict__ zero_me, int n_zero,
           int rev) {
  typedef typename Accum<T>::type A;   // fp64 sums for the fp32 model
  __shared__ A red[kGapThreads * VEC];
  const int tid = threadIdx.x, b = rev ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;   // rev: last sample first
  const int cv = C / VEC;
  const int groups = kGapThreads / lanes;
  const int grp = tid / lanes, lv = tid - grp * lanes;
  const int v = blockIdx.x * lanes + lv;
  pdl_launch_dependents();
  pdl_wait();
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = tid; i < n_zero; i += kGapThreads) zero_me[i] = 0u;
  A acc[VEC];
#pragma unroll
  for (int e = 0; e < VEC; ++e) acc[e] = (A)0;
  if (v < cv) pool_rows<T, VEC>(x + (size_t)b * HW * C + (size_t)v * VEC, HW, C, grp, groups, acc);
#pragma unroll
  for (int e = 0; e < VEC; ++e) red[(grp * lanes + lv) * VEC + e] = acc[e];
  __syncthreads();
  if (tid < lanes * VEC) {
    const int c = blockIdx.x * lanes * VEC + tid;   // red[q][lv][e] with lv * VEC + e == tid
    if (c < cv * VEC) {
      A sum = (A)0;
      for (int q = 0; q < groups; ++q) sum += red[q * lanes * VEC + tid];
      gap[(size_t)b * C + c] = (float)(sum / (A)HW);
    }
  }
}

// Channel vectors per CTA of gap_kernel for a [HW][C] map: about 16 rows per thread, between 8 and 64 row groups.
inline int gap_lanes(int hw) {
  int groups = 8;
  while (groups < 64 && groups * 16 < hw) groups *= 2;
  return kGapThreads / groups;
}

// ----------------------------------------------------------------------------- pooling in row blocks (bf16 models)
//
// gap[b][c] = (sum over the HW rows of sample b) / HW with the sum grouped in a way that a convolution's epilogue can
// start: the rows are cut into nb = HW / G blocks of G consecutive rows, G the largest power of two up to 32 that
// divides HW, so that a block never straddles two samples and, for G = 32 or 16, is exactly the rows one epilogue warp
// (or half of it) holds.  Block sum: the pairwise tree T(g, o, s) = T(g/2, o, 2s) + T(g/2, o + s, 2s), T(1, o, .) =
// row o - what a shuffle butterfly over the lanes with distances G/2, ..., 2, 1 computes.  Sample sum: row group q of
// 256 / lanes adds the blocks q, q + groups, ... in ascending order, then the group sums are added in ascending
// order.  A tensor-core kernel that writes the block sums of its output tile (conv_tc.cuh, gap partials) followed by
// this kernel with G = 1 over those sums gives the same bits as this kernel over the stored feature map.
inline int gap_block_rows(int hw) {
  int g = 1;
  while (g < 32 && hw % (2 * g) == 0) g *= 2;
  return g;
}
// Channel vectors side by side in a CTA for nb blocks per sample: as many row groups as there are blocks, between 8 and 64.
inline int gap_block_lanes(int nb) {
  int groups = 8;
  while (groups < 64 && groups * 2 <= nb) groups *= 2;
  return kGapThreads / groups;
}

template <int g, int VEC, typename LD>
__device__ __forceinline__ void gap_tree(LD&& load, int o, int s, float* out) {
  if constexpr (g == 1) {
    load(o, out);
  } else {
    float a[VEC], b[VEC];
    gap_tree<g / 2, VEC>(load, o, 2 * s, a);
    gap_tree<g / 2, VEC>(load, o + s, 2 * s, b);
#pragma unroll
    for (int e = 0; e < VEC; ++e) out[e] = a[e] + b[e];
  }
}

// Adds the sums of the blocks grp, grp + groups, ... of G rows, one vector of VP channels at p, to acc: a row group of gap_blocks_kernel, and of an FC
// kernel that pools by itself.
// MANY: a row group has more than two blocks of one or two rows (gap_many), which are few loads each: eight rows are in flight
// together, added in the same order, kept as the words they came in.
template <int VP, int G, bool MANY = false, typename T>
__device__ __forceinline__ void pool_blocks(const T* p, int nb, int C, int grp, int groups, float* acc) {
  auto sum = [&](auto&& row_at) {   // of a block's G rows
    float t[VP];
    gap_tree<G, VP>([&](int row, float* out) {
      const Vec16<T> r = row_at(row);
#pragma unroll
      for (int e = 0; e < VP; ++e) out[e] = r.v[e];
    }, 0, 1, t);
#pragma unroll
    for (int e = 0; e < VP; ++e) acc[e] += t[e];
  };
  constexpr int U = MANY ? 8 / G : 1;
  for (int j = grp; j < nb; j += U * groups) {
    if constexpr (MANY) {
      uint4 raw[8];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j + u * groups < nb)
#pragma unroll
          for (int row = 0; row < G; ++row) raw[u * G + row] = *reinterpret_cast<const uint4*>(p + ((size_t)(j + u * groups) * G + row) * C);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j + u * groups < nb)
          sum([&](int row) {
            Vec16<T> r;
            r.unpack(raw[u * G + row]);
            return r;
          });
    } else {
      const T* pb = p + (size_t)j * G * C;
      sum([&](int row) {
        Vec16<T> r;
        r.load(pb + (size_t)row * C);
        return r;
      });
    }
  }
}
// Pooling + FC, us, 41 x 41 x 256 (odd: blocks of one row) at batch 37 / 64 without and with: 17.8 / 24.3 -> 15.7 / 21.8, 27 rows a group; in a
// pass, where the map comes from HBM, 21 of them took 23 and take 13.  Up to two blocks a group it costs registers (32 -> 60) and with them
// CTAs side by side: 11 x 11 x 1024 at 64 19.8 -> 21.7.  Blocks of four rows and more have their loads in flight as it is.
inline bool gap_many(int G, int nb, int lanes) { return G <= 2 && nb > 2 * (kGapThreads / lanes); }

// The same for a thread that has half of every block's tree (gap_tree), rows h, h + 2, ...: the lane beside it has the other half, and both get the
// sums.  Every lane of the warp calls it; take = false: without rows.
template <int VP, int G, typename T>
__device__ __forceinline__ void pool_blocks_halved(const T* p, int nb, int C, int grp, int groups, int h, bool take, float* acc) {
  const int rounds = (nb + groups - 1) / groups;   // the same for every lane
  for (int i = 0; i < rounds; ++i) {
    const int j = grp + i * groups;
    const bool in = take && j < nb;
    float t[VP];
#pragma unroll
    for (int e = 0; e < VP; ++e) t[e] = 0.f;
    if (in)
      gap_tree<G / 2, VP>([&](int row, float* out) {
        Vec16<T> x;
        x.load(p + ((size_t)j * G + row) * C);
#pragma unroll
        for (int e = 0; e < VP; ++e) out[e] = x.v[e];
      }, h, 2, t);
#pragma unroll
    for (int e = 0; e < VP; ++e) {
      const float other = __shfl_xor_sync(0xffffffffu, t[e], 1);
      if (in) acc[e] += t[e] + other;
    }
  }
}
// Few samples leave most SMs without a CTA: blocks of 16 and 32 rows are then halved, and a CTA has half as many channel vectors.  Pooling + FC, us, 56 x 56 x 256
// at batch 1 / 4 / 7 whole 7.64 / 8.60 / 9.41, halved 7.19 / 8.46 / 9.52, 28 x 28 x 512 6.37 / 7.34 / 7.54 and 6.13 / 7.27 / 7.67: the line is
// between 32 CTAs and 56.  A pass of the ResNet-50-shaped model at batch 1: 229.4 -> 227.2.
inline bool gap_halved(int G, int lanes, int ctas, int sms) { return G >= 16 && lanes >= 2 && 4 * ctas <= sms; }

// T = bf16 (VEC 8, the feature map) or float (VEC 4, block sums written by a convolution's epilogue; G = 1).  HALVED: `lanes` is half of what the
// shape asks for, row groups are as many.
template <typename T, int VEC, int G, bool MANY = false, bool HALVED = false>
__global__ void __launch_bounds__(kGapThreads)
gap_blocks_kernel(const T* __restrict__ x, int nb, int HW, int C, int lanes, float* __restrict__ gap, unsigned* __restrict__ zero_me,
                  int n_zero, int rev) {
  __shared__ float red[kGapThreads * VEC];
  const int tid = threadIdx.x, b = rev ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
  const int cv = C / VEC;
  const int at = HALVED ? tid / 2 : tid, groups = kGapThreads / (HALVED ? 2 : 1) / lanes;
  const int grp = at / lanes, lv = at - grp * lanes;
  const int v = blockIdx.x * lanes + lv;
  pdl_launch_dependents();
  pdl_wait();
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = tid; i < n_zero; i += kGapThreads) zero_me[i] = 0u;
  float acc[VEC];
#pragma unroll
  for (int e = 0; e < VEC; ++e) acc[e] = 0.f;
  const T* p = x + (size_t)b * nb * G * C + (size_t)v * VEC;
  if constexpr (HALVED)
    pool_blocks_halved<VEC, G>(p, nb, C, grp, groups, tid % 2, v < cv, acc);
  else if (v < cv)
    pool_blocks<VEC, G, MANY>(p, nb, C, grp, groups, acc);
  if (!HALVED || tid % 2 == 0)
#pragma unroll
    for (int e = 0; e < VEC; ++e) red[(grp * lanes + lv) * VEC + e] = acc[e];
  __syncthreads();
  if (tid < lanes * VEC) {
    const int c = blockIdx.x * lanes * VEC + tid;
    if (c < cv * VEC) {
      float sum = 0.f;
      for (int q = 0; q < groups; ++q) sum += red[q * lanes * VEC + tid];
      gap[(size_t)b * C + c] = sum / (float)HW;
    }
  }
}

constexpr int kFcPackedBatch = 56;   // survivors of that many samples and the number of tiles done, 56 at most, fit a 64-bit word

struct DecideArgs {  // everything the exit decision needs besides the logits
  const float* shift;
  const int32_t* shift_cls;
  float thr;
  int always_exit;
  float* conf;
  int32_t* pred;
  uint8_t* mask;
  const int32_t* ids;
  int32_t* surv_idx;
  int32_t* ids_out;
  int32_t* n_surv;
  unsigned* tile_done;  // per sample tile: CTAs of the FC kernel that have written its logits; zero between launches
  unsigned* done;       // sample tiles whose exit decisions are written; zero between launches
  unsigned long long* packed;      // cluster FC kernel, up to kFcPackedBatch samples: tiles done and survivors in one word; zero between launches
  volatile int32_t* n_surv_host;   // optional: device address of a pinned host word that receives the count (exit_scan)
  bool host_out;                   // conf or pred is host memory: they reach it before the count does
};

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc, int src_bytes) {  // bytes past src_bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gsrc), "r"(src_bytes)
               : "memory");
}

// Exit decision of samples [b_lo, b_hi), one warp per sample (warp w of nwarps takes b_lo + w, b_lo + w + nwarps, ...):
// optional logit shift, max / lowest argmax, conf = 1 / sum exp(z - max), exit = always || conf >= thr (NaN never
// exits).  The logits may have been written by other CTAs and are read through L2.
__device__ __forceinline__ void exit_decide_samples(float* z, int b_lo, int b_hi, int K, int warp, int nwarps, const DecideArgs& d) {
  const int lane = threadIdx.x & 31;
  constexpr int kRegs = 32;  // logits per lane held in registers: one pass over memory for K <= 1024
  for (int b = b_lo + warp; b < b_hi; b += nwarps) {
    float* zb = z + (size_t)b * K;
    const int cls = (d.shift && d.shift_cls) ? d.shift_cls[b] : -1;
    const float sh = cls >= 0 && cls < K ? d.shift[b] : 0.f;
    float m = -INFINITY;
    int arg = 0x7fffffff;
    float zr[kRegs];
#pragma unroll
    for (int i = 0; i < kRegs; ++i) {
      const int k = lane + 32 * i;
      zr[i] = k < K ? __ldcg(zb + k) : -INFINITY;
    }
#pragma unroll
    for (int i = 0; i < kRegs; ++i) {
      const int k = lane + 32 * i;
      if (k == cls) {
        zr[i] += sh;
        zb[k] = zr[i];
      }
      if (zr[i] > m) {
        m = zr[i];
        arg = k;
      }
    }
    for (int k = lane + 32 * kRegs; k < K; k += 32) {  // classes past the register window
      float v = __ldcg(zb + k);
      if (k == cls) {
        v += sh;
        zb[k] = v;
      }
      if (v > m) {
        m = v;
        arg = k;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, m, o);
      const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
      if (om > m || (om == m && oa < arg)) {
        m = om;
        arg = oa;
      }
    }
    __syncwarp();
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < kRegs; ++i)
      if (lane + 32 * i < K) s += expf(zr[i] - m);
    for (int k = lane + 32 * kRegs; k < K; k += 32) s += expf(__ldcg(zb + k) - m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const float cf = 1.0f / s;
      if (d.conf) d.conf[b] = cf;
      if (d.pred) d.pred[b] = arg == 0x7fffffff ? 0 : arg;
      d.mask[b] = (uint8_t)((d.always_exit || cf >= d.thr) ? 1 : 0);
    }
  }
}

// One CTA of THREADS threads: ballot + prefix-sum scan over the not-exit flags of samples [0, B) gives the ascending
// survivor list, the survivors' ids and their count (B_rem).  The flags may have been written by other CTAs.
template <int THREADS>
__device__ __forceinline__ void exit_scan(int B, const DecideArgs& d) {
  __shared__ int warp_tot[32];
  __shared__ int pass_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int base = 0;  // identical in every thread
  for (int p0 = 0; p0 < B; p0 += THREADS) {
    const int b = p0 + tid;
    const bool keep = b < B && __ldcg(d.mask + b) == 0;
    const int id = b < B && d.ids && d.ids_out ? d.ids[b] : 0;   // asked for together with the flag
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    const int pre = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    if (warp == 0) {
      const int t = lane < THREADS / 32 ? warp_tot[lane] : 0;
      int inc = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += n;
      }
      warp_tot[lane] = inc - t;  // exclusive offset of each warp
      if (lane == 31) pass_total = inc;
    }
    __syncthreads();
    if (keep) {
      const int pos = base + warp_tot[warp] + pre;
      d.surv_idx[pos] = b;
      if (d.ids && d.ids_out) d.ids_out[pos] = id;
    }
    base += pass_total;
    __syncthreads();
  }
  if (tid == 0) {
    d.n_surv[0] = base;
    if (d.n_surv_host) {
      if (d.host_out) __threadfence_system();   // the other CTAs' decisions are ordered before this one's counter by device-wide fences
      *d.n_surv_host = base;   // B_exit goes to the scheduler: the host polls this word
    }
  }
}

// The FC layer, softmax top-1, threshold and survivor scan of a batch of pooled vectors: CL CTAs per tile of S samples,
// z[b][k] = bfc[k] + sum_c wfc[k][c] * gap[b][c].
//
// The layer is a few MFLOP over at most a few MB of weights, so nothing but latency bounds it.  Every wait on another
// SM through global memory costs about a microsecond, so a tile's CTAs form a cluster and send what the decision
// needs into its leader's shared memory, and the weights, which no kernel writes, are on their way into
// shared memory before the kernel waits for the pooled vectors.
//   1. The classes are cut into 16 blocks of kb (a multiple of 8), CTA r owns 16 / CL of them.  A warp takes groups of eight
//      classes: its weights stream through a ring of its own, [8 classes][512 bytes of channels] per slot, one TMA box
//      each (as eight row copies a slot took 1200 clocks), requested ring - 1 slots ahead; no barrier across warps.  A lane adds its 16 bytes of channels
//      of every slot in ascending order, then a halving butterfly (distances 16, 8, ..., 1) forms all 8 S sums at once:
//      the tree of a sum does not depend on S, so a logit is the same bits in any batch.
//   2. Per (sample, block): maximum, lowest argmax and sum of exp(z - max) go into the leader CTA's shared memory as asynchronous stores
//      that count on a barrier there: only the leader waits, and only for the data.  Maximum and argmax are one warp reduction
//      each, and the caller's shifts are fetched beside the pooled vectors: from the last sum to the decision 1.6 -> 0.7 us, every head
//      on this route 0.9 to 1.1 us (cluster barrier, shuffles and two dependent loads before; 1 sample of 28 x 28 x 512 7.8 -> 6.8).  More tiles
//      than clusters fit side by side: no clusters, the triples go through global memory and the CTA that finishes a tile
//      last is its leader.
//   3. The leader adds the 16 triples in a fixed order: conf = 1 / sum_r s_r exp(m_r - m), exit = always || conf >= thr (NaN
//      never exits).  With several tiles the leader that finishes last has the survivors of all of them in the word that counts
//      the tiles (up to kFcPackedBatch samples; else it runs the stable scan over the flags in memory).
// Waits on copies are bounded.  Launched with programmatic stream serialization.  Pooling kernel + this kernel on B200, 37 samples
// of 28 x 28 x 512 and 1000 classes: 17.4 us with 16 classes a CTA behind block-wide barriers, 14.9 with this split.  Survivors in
// one atomic and six slots, a chain of heads, us: 1 sample of 14 x 14 x 1024 7.6 -> 7.2, 7 samples 9.8 -> 8.6, 13 of 17 x 17 x 192
// 7.9 -> 7.0, fp32 8 of 16 x 16 x 16 with 10 classes 7.8 -> 5.5 (6.4 of that by pooling here).

__device__ __forceinline__ uint32_t hc_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t hc_map(const void* smem_ptr, uint32_t rank) {   // the same variable in CTA `rank` of the cluster
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(smem_ptr)), "r"(rank));
  return r;
}
__device__ __forceinline__ void hc_st_f32(uint32_t cluster_addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr), "f"(v) : "memory");
}
// 16 bytes into another CTA's shared memory; its barrier `bar` counts them.
__device__ __forceinline__ void st_async16(uint32_t cluster_addr, uint32_t cluster_bar, float a, float b, float c, float d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];"
               ::"r"(cluster_addr), "r"(cluster_bar), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}
// Largest m of a warp (no lane holds NaN) and the smallest arg of the lanes that hold it, in every lane.
__device__ __forceinline__ void warp_argmax(float& m, int& arg) {
  float top;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(top) : "f"(m));
  arg = (int)__reduce_min_sync(0xffffffffu, m == top ? (unsigned)arg : 0x7fffffffu);
  m = top;
}
__device__ __forceinline__ void hc_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void hc_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// C in whole 16-byte vectors (a row of the weights is then a multiple of 16 bytes), shared memory for a tile of one sample.
inline bool fc_cluster_supported(int C, int K, int elem_bytes, const void* wfc) {
  return C % (16 / elem_bytes) == 0 && ((uintptr_t)wfc & 15) == 0 && fc_fits(C, K, elem_bytes);
}

__device__ __forceinline__ void fc_fma2(float (&a)[2], float w0, float w1, float g0, float g1) {   // two independent FMAs, one instruction
  asm("{\n .reg .b64 w, g, a;\n mov.b64 w, {%2, %3};\n mov.b64 g, {%4, %5};\n mov.b64 a, {%0, %1};\n fma.rn.f32x2 a, w, g, a;\n"
      " mov.b64 {%0, %1}, a;\n}"
      : "+f"(a[0]), "+f"(a[1])
      : "f"(w0), "f"(w1), "f"(g0), "f"(g1));
}
__device__ __forceinline__ void fc_fma2(double (&a)[2], float w0, float w1, float g0, float g1) {
  a[0] = acc_fma(w0, g0, a[0]);
  a[1] = acc_fma(w1, g1, a[1]);
}

// POOL (tiles of one CTA): the CTA pools its samples' feature maps itself, in place of a pooling kernel in front of it, summed as
// gap_kernel and gap_blocks_kernel do (same bits).
struct PoolArgs {
  const void* x;   // [B][HW][C] feature maps, or their block sums [B][nb][C] (fp32) when `sums`
  int HW, nb, G;   // bf16: blocks of G rows
  int lanes;       // gap_block_lanes / gap_lanes of the map
  int sums;
};
// Pools the tile's samples, `lanes` channel vectors of VP channels at a time.  put(s, c, value).
template <int VP, typename A, typename SUM, typename PUT>
__device__ __forceinline__ void pool_tile(int samples, int C, int lanes, A* red, SUM&& sum, PUT&& put) {
  static_assert(kFcThreads == kGapThreads, "row groups as in the pooling kernels");
  const int tid = threadIdx.x, groups = kFcThreads / lanes, grp = tid / lanes, lv = tid - grp * lanes;
  const int cv = C / VP, items = samples * cv;
  for (int i0 = 0; i0 < items; i0 += lanes) {
    const int it = i0 + lv;
    A acc[VP];
#pragma unroll
    for (int e = 0; e < VP; ++e) acc[e] = (A)0;
    if (it < items) sum(it / cv, it % cv, grp, groups, acc);
#pragma unroll
    for (int e = 0; e < VP; ++e) red[(grp * lanes + lv) * VP + e] = acc[e];
    __syncthreads();
    if (tid < lanes * VP && i0 + tid / VP < items) {
      const int i = i0 + tid / VP;
      A t = (A)0;
      for (int q = 0; q < groups; ++q) t += red[q * lanes * VP + tid];
      put(i / cv, i % cv * VP + tid % VP, t);
    }
    __syncthreads();
  }
}

template <typename T, int S, bool POOL>
__global__ void __launch_bounds__(kFcThreads)
fc_cluster_kernel(const __grid_constant__ CUtensorMap tmW, const float* __restrict__ gap, const float* __restrict__ bfc, int B, int C, int K,
                  float* z, float4* exchange, DecideArgs d, FcShape f, PoolArgs pa, int* err_flag, long long wait_cycles) {
  typedef typename Accum<T>::type A;                        // fp64 sums for the fp32 model
  constexpr int VEC = 16 / (int)sizeof(T), CHUNK = 32 * VEC, NV = kFcRows * S, WARPS = kFcThreads / 32;
  extern __shared__ __align__(128) uint8_t fc_smem[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint8_t* ring = fc_smem + (size_t)warp * f.ring * kFcSlot;                             // this warp's slots
  float* gs = reinterpret_cast<float*>(fc_smem + (size_t)WARPS * f.ring * kFcSlot);      // [S][Cp] pooled vectors, see below
  const int my_blocks = kFcBlocks / f.CL, kc = my_blocks * f.kb;
  float* zs = gs + (size_t)S * f.Cp;                                                      // [S][kc] this CTA's logits
  float* part = zs + (size_t)S * kc;                                                      // [16][S][4] (leader): max, argmax, sum
  uint64_t* s_done = reinterpret_cast<uint64_t*>(part + kFcBlocks * S * 4);               // [3]: survivors, is this the last tile; a barrier
  const uint32_t triples = smem_u32(s_done + 2);                                          // (leader) counts the tile's triples as they arrive
  const uint32_t bars = smem_u32(s_done + 3) + (uint32_t)(warp * f.ring * 8);             // this warp's slot barriers
  A* cross = reinterpret_cast<A*>(s_done + 3 + WARPS * f.ring + 1);                           // [ws][S][kc] sums of the warps that share classes
  const uint32_t rank = blockIdx.x % (unsigned)f.CL;   // also the CTA's rank in its cluster
  const int tile = (int)blockIdx.x / f.CL, tiles = (int)gridDim.x / f.CL, b0 = tile * S;
  const int k0 = (int)rank * kc;
  const int nchunk = f.Cp / CHUNK, ngroups = max(0, min(kc, K - k0) + kFcRows - 1) / kFcRows;
  // warp -> group wg, wg + side, ... of classes, slots wc, wc + ws, ... of their channels
  const int ws = f.ws, side = WARPS / ws, wg = warp / ws, wc = warp - wg * ws, my_chunks = (nchunk - 1 - wc) / ws + 1;
  const int my_groups = wg < ngroups ? (ngroups - 1 - wg) / side + 1 : 0, slots = my_groups * my_chunks;

  if (tid == 0) {
    mbar_init(triples, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(triples, kFcBlocks * S * 16);
  }
  __syncwarp();
  if (f.cluster) hc_cluster_arrive();   // every CTA of the cluster runs and its barrier is set up (waited for before the first remote store)
  if (lane == 0) {
    for (int i = 0; i < f.ring; ++i) mbar_init(bars + 8u * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  // slot lt of this warp: classes of group lg, channels of chunk lc; classes past K and channels past C arrive as zeros
  int lt = 0, lg = wg, lc = wc, ls = 0;
  auto load = [&]() {
    if (lt < slots) {
      if (lane == 0) {
        const uint32_t bar = bars + 8u * ls;
        mbar_expect_tx(bar, kFcSlot);
        tma_load_2d(smem_u32(ring + ls * kFcSlot), &tmW, bar, lc * CHUNK, k0 + lg * kFcRows);
      }
      if (++ls == f.ring) ls = 0;
      if ((lc += ws) >= nchunk) lc = wc, lg += side;
    }
    ++lt;
  };
  for (int t = 0; t < f.ring - 1; ++t) load();
  // bias of the classes this lane finishes in a group (see the butterfly below): the first group's ahead of the wait
  constexpr int LEFT = NV > 32 ? NV / 32 : 1, REP = NV < 32 ? 32 / NV : 1;   // values per lane, lanes per value
  float bias[LEFT];
  auto load_bias = [&](int g) {
#pragma unroll
    for (int j = 0; j < LEFT; ++j) {
      const int k = k0 + g * kFcRows + ((lane / REP) * LEFT + j) % kFcRows;
      bias[j] = bfc && k < K && g < ngroups ? bfc[k] : 0.f;
    }
  };
  load_bias(wg);
  pdl_launch_dependents();
  pdl_wait();
  const bool packed = d.packed && B <= kFcPackedBatch;
  // a warp's triples are all of one sample: S is 1, 2, 4 or 8, the step between them the eight warps
  const int my_s = warp % S, my_b = b0 + my_s;
  const int my_cls = my_b < B && d.shift && d.shift_cls ? d.shift_cls[my_b] : -1;
  const float my_shift = my_b < B && d.shift ? d.shift[my_b] : 0.f;
  const int my_id = packed && tid < B && d.ids && d.ids_out ? d.ids[tid] : 0;   // of the scan, should this CTA run it
  // pooled vectors: within a chunk the float4 `e` of lane l's VEC channels sits at [e][l], so that a warp's reads are 512
  // consecutive bytes
  auto place = [&](int s, int c) { return s * f.Cp + c / CHUNK * CHUNK + (c % VEC / 4 * 32 + c % CHUNK / VEC) * 4; };   // of float4 c / 4
  if constexpr (!POOL) {
    for (int i = tid; i < S * (f.Cp / 4); i += kFcThreads) {
      const int s = i / (f.Cp / 4), c = (i - s * (f.Cp / 4)) * 4;
      const bool in = b0 + s < B && c < C;
      cp_async16(gs + place(s, c), in ? gap + (size_t)(b0 + s) * C + c : gap, in ? 16 : 0);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
  } else {
    const int here = min(S, B - b0), pad4 = (f.Cp - C) / 4;
    for (int i = tid; i < S * pad4; i += kFcThreads) *reinterpret_cast<float4*>(gs + place(i / pad4, C + i % pad4 * 4)) = make_float4(0.f, 0.f, 0.f, 0.f);
    void* red = fc_smem + fc_smem_bytes(f);
    auto put = [&](int s, int c, A total) { gs[place(s, c) + c % 4] = (float)(total / (A)pa.HW); };
    if constexpr (sizeof(T) == 4) {
      pool_tile<VEC>(here, C, pa.lanes, (A*)red, [&](int s, int v, int grp, int groups, A* acc) {
        pool_rows<T, VEC>((const T*)pa.x + (size_t)(b0 + s) * pa.HW * C + (size_t)v * VEC, pa.HW, C, grp, groups, acc);
      }, put);
    } else if (pa.sums) {
      pool_tile<4>(here, C, pa.lanes, (A*)red, [&](int s, int v, int grp, int groups, A* acc) {
        pool_blocks<4, 1>((const float*)pa.x + (size_t)(b0 + s) * pa.nb * C + (size_t)v * 4, pa.nb, C, grp, groups, acc);
      }, put);
    } else {
      pool_tile<VEC>(here, C, pa.lanes, (A*)red, [&](int s, int v, int grp, int groups, A* acc) {
        const T* p0 = (const T*)pa.x + (size_t)(b0 + s) * pa.HW * C + (size_t)v * VEC;
        switch (pa.G) {
          case 32: pool_blocks<VEC, 32>(p0, pa.nb, C, grp, groups, acc); break;
          case 16: pool_blocks<VEC, 16>(p0, pa.nb, C, grp, groups, acc); break;
          case 8: pool_blocks<VEC, 8>(p0, pa.nb, C, grp, groups, acc); break;
          case 4: pool_blocks<VEC, 4>(p0, pa.nb, C, grp, groups, acc); break;
          case 2: pool_blocks<VEC, 2>(p0, pa.nb, C, grp, groups, acc); break;
          default: pool_blocks<VEC, 1>(p0, pa.nb, C, grp, groups, acc); break;
        }
      }, put);
    }
  }

  A acc[kFcRows][S][2];   // even and odd channels
#pragma unroll
  for (int q = 0; q < kFcRows; ++q)
#pragma unroll
    for (int s = 0; s < S; ++s) acc[q][s][0] = acc[q][s][1] = (A)0;
  int ch = wc, grp = wg, cs = 0;
  uint32_t cp = 0;
  bool ok = true;
  for (int t = 0; t < slots; ++t) {
    __syncwarp();           // every lane is done with the slot refilled next
    if (ok) load();
    ok = ok && mbar_wait(bars + 8u * cs, cp, err_flag);
    const uint8_t* slot = ring + cs * kFcSlot + lane * 16;
    if (++cs == f.ring) cs = 0, cp ^= 1u;
    if (ok) {
      float gv[S][VEC];
#pragma unroll
      for (int s = 0; s < S; ++s)
#pragma unroll
        for (int e = 0; e < VEC / 4; ++e) {
          const float4 v = *reinterpret_cast<const float4*>(gs + (size_t)s * f.Cp + ch * CHUNK + (e * 32 + lane) * 4);
          gv[s][4 * e] = v.x, gv[s][4 * e + 1] = v.y, gv[s][4 * e + 2] = v.z, gv[s][4 * e + 3] = v.w;
        }
#pragma unroll
      for (int q = 0; q < kFcRows; ++q) {
        Vec16<T> w;
        w.load(reinterpret_cast<const T*>(slot + q * 512));
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
          for (int e = 0; e < VEC; e += 2) fc_fma2(acc[q][s], w.v[e], w.v[e + 1], gv[s][e], gv[s][e + 1]);
      }
    }
    __syncwarp();
    if ((ch += ws) >= nchunk) {   // the group's sums are complete: all 8 S of them in one halving butterfly
      A v[NV];
#pragma unroll
      for (int q = 0; q < kFcRows; ++q)
#pragma unroll
        for (int s = 0; s < S; ++s) {
          v[s * kFcRows + q] = acc[q][s][0] + acc[q][s][1];
          acc[q][s][0] = acc[q][s][1] = (A)0;
        }
      int n = NV;             // values a lane still holds (a compile-time constant after unrolling)
#pragma unroll
      for (int dd = 16; dd >= 1; dd >>= 1) {
        if (n > 1) {
          const bool up = (lane & dd) != 0;
#pragma unroll
          for (int i = 0; i < NV / 2; ++i)
            if (i < n / 2) {
              const A send = up ? v[i] : v[i + n / 2], keep = up ? v[i + n / 2] : v[i];
              v[i] = keep + __shfl_xor_sync(0xffffffffu, send, dd);
            }
          n /= 2;
        } else {
          v[0] += __shfl_xor_sync(0xffffffffu, v[0], dd);
        }
      }
#pragma unroll
      for (int j = 0; j < LEFT; ++j) {
        const int idx = (lane / REP) * LEFT + j, s = idx / kFcRows, kl = grp * kFcRows + idx % kFcRows;
        if (lane % REP == 0) {
          if (ws == 1) zs[s * kc + kl] = (float)(v[j] + (A)bias[j]);
          else cross[((size_t)wc * S + s) * kc + kl] = v[j];
        }
      }
      grp += side, ch = wc;
      load_bias(grp);
    }
  }
  __syncthreads();
  if (ws > 1) {   // the shares of the warps that shared classes, in ascending order
    for (int i = tid; i < S * kc; i += kFcThreads) {
      const int s = i / kc, k = i - s * kc;
      A sum = (A)0;
      for (int w = 0; w < ws; ++w) sum += cross[((size_t)w * S + s) * kc + k];
      zs[s * kc + k] = (float)(sum + (A)(bfc && k0 + k < K ? bfc[k0 + k] : 0.f));
    }
    __syncthreads();
  }

  // ---- 2. one warp per (block, sample)
  if (f.cluster) hc_cluster_wait();
  for (int it = warp; it < my_blocks * S; it += WARPS) {
    const int s = my_s, bl = it / S, b = my_b, kf = k0 + bl * f.kb;
    const int nk = max(0, min(f.kb, K - kf));
    float m = -INFINITY, sum = 0.f;
    int arg = 0x7fffffff;
    if (b < B) {
      float* zb = zs + s * kc + bl * f.kb;
      if (lane == 0 && my_cls >= kf && my_cls < kf + nk) zb[my_cls - kf] += my_shift;
      __syncwarp();
      for (int j = lane; j < nk; j += 32) {
        const float v = zb[j];
        if (z) z[(size_t)b * K + kf + j] = v;
        if (v > m) m = v, arg = kf + j;
      }
      warp_argmax(m, arg);
      for (int j = lane; j < nk; j += 32) sum += expf(zb[j] - m);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    if (lane == 0) {
      const int at = ((int)rank * my_blocks + bl) * S + s;
      float* mine = part + (size_t)at * 4;
      if (f.cluster)
        st_async16(hc_map(mine, 0), hc_map(s_done + 2, 0), m, __int_as_float(arg), sum, 0.f);
      else if (f.CL == 1)
        *reinterpret_cast<float4*>(mine) = make_float4(m, __int_as_float(arg), sum, 0.f);
      else
        __stcg(exchange + (size_t)tile * kFcBlocks * S + at, make_float4(m, __int_as_float(arg), sum, 0.f));
    }
  }
  bool late = false;
  if (f.cluster) {
    if (rank != 0) return;
    if (warp < S && b0 + warp < B) late = !__all_sync(0xffffffffu, mbar_wait_cluster(triples, 0, err_flag, wait_cycles));   // else every block's triple is here
  } else {
    if (f.CL > 1) __threadfence();
    __syncthreads();
    if (f.CL > 1) {
      int* last = reinterpret_cast<int*>(zs);
      if (tid == 0) *last = atomicAdd(d.tile_done + tile, 1u) == (unsigned)(f.CL - 1) ? 1 : 0;
      __syncthreads();
      if (!*last) return;
      __threadfence();
      if (tid == 0) d.tile_done[tile] = 0;
      for (int i = tid; i < kFcBlocks * S; i += kFcThreads) reinterpret_cast<float4*>(part)[i] = __ldcg(exchange + (size_t)tile * kFcBlocks * S + i);
      __syncthreads();
    }
  }
  // ---- 3. decision: one warp per sample, lane r holds block r.  A sample whose triples are late has confidence 0 and class 0, and the leader then stays,
  // behind the barrier that follows, until what is sent to it has landed.
  int* leave = reinterpret_cast<int*>(gs);   // [S] bit 0: leaves, bit 1: late.  Not where triples may still arrive; the pooled vectors have been read
  if (warp < S && b0 + warp < B) {
    const int s = warp, b = b0 + s;
    float mr = -INFINITY, sr = 0.f;
    int arg = 0x7fffffff;
    if (lane < kFcBlocks && !late) {
      const float* t3 = part + ((size_t)lane * S + s) * 4;
      mr = t3[0], arg = __float_as_int(t3[1]), sr = t3[2];
    }
    float m = mr;
    warp_argmax(m, arg);
    float tot = sr * (lane < kFcBlocks ? expf(mr - m) : 0.f);
#pragma unroll
    for (int o = kFcBlocks; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) {
      const float cf = late ? 0.f : 1.0f / tot;
      if (d.conf) d.conf[b] = cf;
      if (d.pred) d.pred[b] = arg == 0x7fffffff ? 0 : arg;
      const int leaves = d.always_exit || cf >= d.thr ? 1 : 0;
      d.mask[b] = (uint8_t)leaves;
      leave[s] = leaves | (late ? 2 : 0);
    }
  }
  if (packed) {
    // The survivors and the number of tiles done travel in one atomic: who finishes last has every decision in hand, and nothing is
    // written, fenced and read again (2 us of a head that takes 8 to 10).
    __syncthreads();
    if (tid == 0) {
      unsigned long long keep = 0;
      int any = 0;
      for (int s = 0; s < S && b0 + s < B; ++s) keep |= (unsigned long long)(~leave[s] & 1) << (b0 + s), any |= leave[s];
      unsigned long long last = 1;
      if (tiles > 1) {
        if (d.host_out) __threadfence();
        const unsigned long long before = atomicAdd(d.packed, (1ull << kFcPackedBatch) + keep);
        last = (int)(before >> kFcPackedBatch) == tiles - 1;
        keep = (before + keep) & ((1ull << kFcPackedBatch) - 1);
        if (last) *d.packed = 0;
      }
      s_done[0] = keep, s_done[1] = last | (any & 2);
    }
    __syncthreads();
    const unsigned long long keep = s_done[0], state = s_done[1];
    if (state & 2) cluster_drain(triples, 0, err_flag);
    if (!(state & 1)) return;
    if (tid < B && (keep >> tid & 1)) {
      const int pos = __popcll(keep & ((1ull << tid) - 1));
      d.surv_idx[pos] = tid;
      if (d.ids && d.ids_out) d.ids_out[pos] = my_id;
    }
    if (tid == 0) {
      d.n_surv[0] = __popcll(keep);
      if (d.n_surv_host) {
        if (d.host_out) __threadfence_system();   // conf and pred reach the host before the count does
        *d.n_surv_host = __popcll(keep);          // B_exit goes to the scheduler: the host polls this word
      }
    }
    return;
  }
  __threadfence();
  __syncthreads();
  if (f.cluster) {
    int any = 0;
    for (int s = 0; s < S && b0 + s < B; ++s) any |= leave[s];
    if (any & 2) cluster_drain(triples, 0, err_flag);
  }
  if (tiles > 1) {         // the leader that finishes last scans
    int* flag = reinterpret_cast<int*>(part);
    if (tid == 0) *flag = atomicAdd(d.done, 1u) == (unsigned)(tiles - 1) ? 1 : 0;
    __syncthreads();
    if (!*flag) return;
    __threadfence();
    if (tid == 0) *d.done = 0;
  }
  exit_scan<kFcThreads>(B, d);
}

// pool: null = `gap` holds the pooled vectors.
template <typename T, int S>
inline cudaError_t fc_cluster_launch_t(const float* gap, const PoolArgs* pool, const CUtensorMap& wfc, const float* bfc, int B, int C, int K, float* z,
                                       float4* exchange, const DecideArgs& d, const FcShape& f, int* err_flag, long long wait_cycles, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((B + S - 1) / S * f.CL));
  cfg.blockDim = dim3(kFcThreads);
  cfg.dynamicSmemBytes = fc_smem_bytes(f) + (pool ? kFcPoolSmem : 0);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = f.CL;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = f.cluster ? 2 : 1;
  if constexpr (S == 1)   // fc_pools: tiles of one sample
    if (pool) return cudaLaunchKernelEx(&cfg, fc_cluster_kernel<T, 1, true>, wfc, gap, bfc, B, C, K, z, exchange, d, f, *pool, err_flag, wait_cycles);
  if (pool) return cudaErrorInvalidValue;
  return cudaLaunchKernelEx(&cfg, fc_cluster_kernel<T, S, false>, wfc, gap, bfc, B, C, K, z, exchange, d, f, PoolArgs{}, err_flag, wait_cycles);
}
// d.done and d.tile_done must be zero when the kernel starts and are zero again when it ends.  exchange: 16 float4 per sample
// of every tile, less than the batch's logits take wherever it is used (more than 512 classes).
template <typename T>
inline cudaError_t fc_cluster_launch(const FcShape& f, const float* gap, const PoolArgs* pool, const CUtensorMap& wfc, const float* bfc, int B, int C, int K, float* z,
                                     float4* exchange, const DecideArgs& d, int* err_flag, long long wait_cycles, cudaStream_t st) {
  switch (f.S) {
    case 1: return fc_cluster_launch_t<T, 1>(gap, pool, wfc, bfc, B, C, K, z, exchange, d, f, err_flag, wait_cycles, st);
    case 2: return fc_cluster_launch_t<T, 2>(gap, pool, wfc, bfc, B, C, K, z, exchange, d, f, err_flag, wait_cycles, st);
    case 4: return fc_cluster_launch_t<T, 4>(gap, pool, wfc, bfc, B, C, K, z, exchange, d, f, err_flag, wait_cycles, st);
  }
  if constexpr (sizeof(T) == 2) return fc_cluster_launch_t<T, 8>(gap, pool, wfc, bfc, B, C, K, z, exchange, d, f, err_flag, wait_cycles, st);
  return cudaErrorInvalidValue;
}
template <typename T, int S>
inline cudaError_t fc_cluster_attr() {
  cudaError_t e = cudaSuccess;
  for (auto kernel : {fc_cluster_kernel<T, S, false>, fc_cluster_kernel<T, S, S == 1>}) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFcMaxSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  return e;
}
inline cudaError_t fc_context_init() {
  cudaError_t e = cudaSuccess;
  for (cudaError_t r : {fc_cluster_attr<bf16, 1>(), fc_cluster_attr<bf16, 2>(), fc_cluster_attr<bf16, 4>(), fc_cluster_attr<bf16, 8>(), fc_cluster_attr<float, 1>(),
                        fc_cluster_attr<float, 2>(), fc_cluster_attr<float, 4>()})
    if (e == cudaSuccess) e = r;
  return e;
}

// Clusters of 16 of this kernel that run side by side on the current device (a GPC with fewer than 16 SMs holds none).
inline int fc_room() {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(16 * 16);
  cfg.blockDim = dim3(kFcThreads);
  cfg.dynamicSmemBytes = kFcMaxSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 16, attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, fc_cluster_kernel<bf16, 8, false>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 4;
  }
  return std::max(1, n);
}
// FC weights [K][C] as boxes of eight classes x 512 bytes of channels.
template <typename T>
inline ee_status_t fc_weight_map(const TcContext& c, const void* w, int C, int K, CUtensorMap* out) {
  const cuuint64_t dims[2] = {(cuuint64_t)C, (cuuint64_t)K};
  const cuuint64_t strides[1] = {(cuuint64_t)C * sizeof(T)};
  const cuuint32_t box[2] = {512 / sizeof(T), kFcRows};
  const cuuint32_t es[2] = {1, 1};
  return c.encode_tiled(out, sizeof(T) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(w), dims,
                        strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS
             ? EE_OK
             : EE_ERR_CUDA;
}

// The same layer for any C, K and alignment (channels that are not whole 16-byte vectors, or too many of them or of classes for
// the shared memory of fc_cluster_kernel): CTA (x, y)
// owns 16 classes (two per warp) of eight samples and walks the channels 128 at a time with plain loads.  The CTA that
// completes a sample tile's logits (a counter per tile) takes that tile's exit decisions; the CTA that completes the last
// tile's decisions runs the scan and leaves all counters at zero.
constexpr int kFcWarps = 8, kFcClassesPerWarp = 2, kFcChunk = 128, kFcSamples = 8;
constexpr int kFcClasses = kFcWarps * kFcClassesPerWarp;

template <typename T>
__global__ void __launch_bounds__(kFcThreads)
fc_kernel(const float* __restrict__ gap, const T* __restrict__ wfc, const float* __restrict__ bfc, int B, int C, int K, float* z,
          DecideArgs d) {
  constexpr int PER = kFcChunk / 32, S = kFcSamples;  // channels per lane per chunk (4)
  __shared__ __align__(16) float gs[S][kFcChunk];
  __shared__ __align__(16) T wsm[kFcClasses][kFcChunk];
  __shared__ bool last_flag;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int k0 = blockIdx.x * kFcClasses, b0 = blockIdx.y * S;
  const int nchunk = (C + kFcChunk - 1) / kFcChunk;
  pdl_launch_dependents();
  pdl_wait();
  typedef typename Accum<T>::type A;   // fp64 sums for the fp32 model
  A acc[kFcClassesPerWarp][S];
#pragma unroll
  for (int q = 0; q < kFcClassesPerWarp; ++q)
#pragma unroll
    for (int s2 = 0; s2 < S; ++s2) acc[q][s2] = (A)0;
  for (int chunk = 0; chunk < nchunk; ++chunk) {
    const int c0 = chunk * kFcChunk;
    __syncthreads();
    for (int i = tid; i < S * kFcChunk; i += kFcThreads) {
      const int sidx = i / kFcChunk, c = i % kFcChunk;
      gs[sidx][c] = (b0 + sidx < B && c0 + c < C) ? gap[(size_t)(b0 + sidx) * C + c0 + c] : 0.f;
    }
    for (int i = tid; i < kFcClasses * kFcChunk; i += kFcThreads) {
      const int cls = i / kFcChunk, c = i % kFcChunk;
      Elem<T>::st(&wsm[cls][c], (k0 + cls < K && c0 + c < C) ? Elem<T>::ld(wfc + (size_t)(k0 + cls) * C + c0 + c) : 0.f);
    }
    __syncthreads();
    float wv[kFcClassesPerWarp][PER];
#pragma unroll
    for (int q = 0; q < kFcClassesPerWarp; ++q)
#pragma unroll
      for (int e = 0; e < PER; ++e) wv[q][e] = Elem<T>::ld(&wsm[warp * kFcClassesPerWarp + q][lane * PER + e]);
#pragma unroll
    for (int s2 = 0; s2 < S; ++s2) {
      const float4 g = *reinterpret_cast<const float4*>(&gs[s2][lane * PER]);
      const float gv[PER] = {g.x, g.y, g.z, g.w};
#pragma unroll
      for (int q = 0; q < kFcClassesPerWarp; ++q)
#pragma unroll
        for (int e = 0; e < PER; ++e) acc[q][s2] = acc_fma(wv[q][e], gv[e], acc[q][s2]);
    }
  }
#pragma unroll
  for (int q = 0; q < kFcClassesPerWarp; ++q) {
    const int k = k0 + warp * kFcClassesPerWarp + q;
    const float bk = (bfc && k < K) ? bfc[k] : 0.f;
#pragma unroll
    for (int s2 = 0; s2 < S; ++s2) {
      A v = acc[q][s2];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && k < K && b0 + s2 < B) z[(size_t)(b0 + s2) * K + k] = (float)(v + (A)bk);
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last_flag = atomicAdd(d.tile_done + blockIdx.y, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last_flag) return;
  __threadfence();
  exit_decide_samples(z, b0, min(B, b0 + S), K, warp, kFcWarps, d);
  __threadfence();
  __syncthreads();
  if (tid == 0) {
    d.tile_done[blockIdx.y] = 0;
    last_flag = atomicAdd(d.done, 1u) == gridDim.y - 1;
  }
  __syncthreads();
  if (!last_flag) return;
  __threadfence();
  if (tid == 0) *d.done = 0;
  exit_scan<kFcThreads>(B, d);
}

// ----------------------------------------------------------------------------- the whole exit head in one launch
//
// bf16 models: global average pool, FC, softmax top-1, threshold and the survivor scan as ONE kernel of 8-CTA
// clusters, one cluster per tile of S samples (S = 1, 2 or 4 by the batch; no sum depends on S).
//   1. Pool.  CTA r of a cluster pools the channels [r, r+1) * C/8 of the tile's samples (row groups in ascending order
//      as in gap_kernel, the grouping a function of C only) and writes its slab of the pooled vectors into the shared
//      memory of all eight CTAs (distributed shared memory); a cluster barrier publishes them.
//   2. FC.  CTA r owns the classes [r, r+1) * ceil(K/8).  Their weights stream through a 4-deep cp.async ring of
//      [64 classes][256 channels] blocks whose first three blocks are requested before the kernel waits for its
//      predecessor in the stream (the weights are constants).  Warp w takes classes 8w..8w+7 of a block, a lane the
//      channels 8 lane..8 lane+7: per (sample, class) a lane adds its channels in ascending order over the blocks, then
//      a shuffle tree, so a logit is the same bits in every batch and at every position.
//   3. Decision.  Every CTA reduces its classes to (max, lowest argmax, sum of exp(z - max)) per sample and writes the
//      triple into the leader CTA's shared memory; after a second cluster barrier the leader combines the eight triples in
//      rank order: conf = 1 / sum_r s_r exp(m_r - m), exit = always || conf >= thr.
//   4. Scan.  The leader of the cluster that finishes last (one counter per launch, left at zero) runs the stable scan.
// No wait in this kernel spins: cluster barriers and cp.async groups only.  Launched with programmatic stream
// serialization.
constexpr int kHcCluster = 8, kHcThreads = 256, kHcRing = 4, kHcBlockClasses = 64, kHcBlockCh = 256, kHcMaxKc = 128;

struct HcShape {   // functions of the head's shape (C, K) only
  int Cp;          // C rounded up to whole 256-channel blocks
  int cvp;         // 16-byte channel vectors a CTA pools: ceil(C / 8 / 8)
  int L;           // power of two >= cvp: vectors side by side in the pooling loop (256 / L row groups)
  int kc;          // classes per CTA: ceil(K / 8)
  int nchunk;      // channel blocks: Cp / 256
  int ngroup;      // class blocks of a CTA: ceil(kc / 64)
};
inline HcShape hc_shape(int C, int K) {
  HcShape h;
  h.Cp = (C + kHcBlockCh - 1) / kHcBlockCh * kHcBlockCh;
  h.cvp = (C / 8 + kHcCluster - 1) / kHcCluster;
  h.L = 1;
  while (h.L < h.cvp) h.L *= 2;
  h.kc = (K + kHcCluster - 1) / kHcCluster;
  h.nchunk = h.Cp / kHcBlockCh;
  h.ngroup = (h.kc + kHcBlockClasses - 1) / kHcBlockClasses;
  return h;
}
inline size_t hc_smem_bytes(int S, const HcShape& h) {
  return (size_t)S * h.Cp * 4 + (size_t)kHcRing * kHcBlockClasses * kHcBlockCh * 2 + (size_t)S * kHcThreads * 8 * 4 +
         (size_t)S * kHcMaxKc * 4 + (size_t)kHcCluster * S * 4 * 4 + 16;
}
inline int hc_tile_samples(int B) { return B <= 18 ? 1 : B <= 37 ? 2 : 4; }   // up to 18 clusters of 8 fill the 148 SMs
inline bool hc_supported(int C, int K, const void* x, const void* wfc) {
  if (C < 8 || C % 8 != 0 || C > 2048 || K < 1 || K > kHcCluster * kHcMaxKc) return false;
  if (((uintptr_t)x & 15) || ((uintptr_t)wfc & 15)) return false;
  return hc_shape(C, K).L <= kHcThreads;
}

template <int S>
__global__ void __cluster_dims__(kHcCluster, 1, 1) __launch_bounds__(kHcThreads)
head_cluster_kernel(const bf16* __restrict__ x, int HW, int C, const bf16* __restrict__ wfc, const float* __restrict__ bfc, int B, int K,
                    float* z, DecideArgs d, HcShape h) {
  extern __shared__ __align__(16) uint8_t hc_smem[];
  float* gsm = reinterpret_cast<float*>(hc_smem);                                   // [S][Cp] pooled vectors of the tile
  bf16* ring = reinterpret_cast<bf16*>(gsm + (size_t)S * h.Cp);                     // [4][64][256]
  float* red = reinterpret_cast<float*>(ring + (size_t)kHcRing * kHcBlockClasses * kHcBlockCh);   // [S][256][8]
  float* zs = red + (size_t)S * kHcThreads * 8;                                     // [S][128] this CTA's logits
  float* part = zs + (size_t)S * kHcMaxKc;                                          // [8][S][4] (leader): max, argmax, sum
  int* flag = reinterpret_cast<int*>(part + kHcCluster * S * 4);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = hc_cluster_rank();
  const int tile = (int)blockIdx.x / kHcCluster, b0 = tile * S;
  const int k0 = (int)rank * h.kc, k1 = min(K, k0 + h.kc), nk = max(k1 - k0, 0);
  const int T = h.ngroup * h.nchunk;   // ring blocks of this CTA, class block major

  hc_cluster_arrive();   // #1: every CTA of the cluster runs (waited for before the first remote store)
  auto block_load = [&](int t, int buf) {
    const int g = t / h.nchunk, ch = t - g * h.nchunk;
    bf16* dst = ring + (size_t)buf * kHcBlockClasses * kHcBlockCh;
#pragma unroll
    for (int i = 0; i < kHcBlockClasses * (kHcBlockCh / 8) / kHcThreads; ++i) {
      const int idx = tid + i * kHcThreads, row = idx >> 5, c = ch * kHcBlockCh + (idx & 31) * 8;
      const int k = k0 + g * kHcBlockClasses + row;
      const bool in = k < k1 && c < C;
      cp_async16(dst + row * kHcBlockCh + (idx & 31) * 8, in ? wfc + (size_t)k * C + c : wfc, in ? 16 : 0);
    }
  };
#pragma unroll
  for (int t = 0; t < kHcRing - 1; ++t) {
    if (t < T) block_load(t, t);
    cp_async_commit();
  }
  for (int i = tid; i < S * (h.Cp - C); i += kHcThreads) gsm[(i / (h.Cp - C)) * h.Cp + C + i % (h.Cp - C)] = 0.f;   // channel padding
  pdl_launch_dependents();
  pdl_wait();

  // ---- 1. pool
  {
    const int groups = kHcThreads / h.L, grp = tid / h.L, lv = tid - grp * h.L;
    const int v = (int)rank * h.cvp + lv;
    const bool mine = lv < h.cvp && v < C / 8;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      float acc[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = 0.f;
      if (mine && b0 + s < B) {
        const bf16* p0 = x + (size_t)(b0 + s) * HW * C + (size_t)v * 8;
        int r = grp;
        for (; r + 15 * groups < HW; r += 16 * groups) {   // sixteen 16-byte loads in flight per thread; added in row order
          uint4 t[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) t[u] = __ldg(reinterpret_cast<const uint4*>(p0 + (size_t)(r + u * groups) * C));
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const uint32_t w4[4] = {t[u].x, t[u].y, t[u].z, t[u].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              acc[2 * i] += __uint_as_float(w4[i] << 16);
              acc[2 * i + 1] += __uint_as_float(w4[i] & 0xffff0000u);
            }
          }
        }
        for (; r < HW; r += groups) {
          Vec16<bf16> t;
          t.load(p0 + (size_t)r * C);
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[e] += t.v[e];
        }
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) red[((size_t)s * kHcThreads + grp * h.L + lv) * 8 + e] = acc[e];
    }
    __syncthreads();
    hc_cluster_wait();   // #1
    if (tid < h.L * 8) {
      const int lv2 = tid >> 3, c = ((int)rank * h.cvp + lv2) * 8 + (tid & 7);
      if (lv2 < h.cvp && c < C) {
#pragma unroll
        for (int s = 0; s < S; ++s) {
          float sum = 0.f;
          for (int q = 0; q < groups; ++q) sum += red[((size_t)s * kHcThreads + q * h.L) * 8 + tid];
          const float mean = sum / (float)HW;
#pragma unroll
          for (uint32_t peer = 0; peer < (uint32_t)kHcCluster; ++peer) hc_st_f32(hc_map(gsm + (size_t)s * h.Cp + c, peer), mean);
        }
      }
    }
    hc_cluster_arrive();   // #2: the pooled vectors are complete in every CTA
    hc_cluster_wait();
  }

  // ---- 2. FC
  float acc[8][S];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int s = 0; s < S; ++s) acc[q][s] = 0.f;
  for (int t = 0; t < T; ++t) {
    const int buf = t % kHcRing;
    cp_async_wait<kHcRing - 2>();
    __syncthreads();   // block t landed for every thread; the buffer refilled below was read one iteration ago
    if (t + kHcRing - 1 < T) block_load(t + kHcRing - 1, (t + kHcRing - 1) % kHcRing);
    cp_async_commit();
    const int g = t / h.nchunk, ch = t - g * h.nchunk;
    float gv[S][8];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const float4 a = *reinterpret_cast<const float4*>(gsm + (size_t)s * h.Cp + ch * kHcBlockCh + lane * 8);
      const float4 b = *reinterpret_cast<const float4*>(gsm + (size_t)s * h.Cp + ch * kHcBlockCh + lane * 8 + 4);
      gv[s][0] = a.x, gv[s][1] = a.y, gv[s][2] = a.z, gv[s][3] = a.w, gv[s][4] = b.x, gv[s][5] = b.y, gv[s][6] = b.z, gv[s][7] = b.w;
    }
    const bf16* wb = ring + (size_t)buf * kHcBlockClasses * kHcBlockCh + (warp * 8) * kHcBlockCh + lane * 8;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      Vec16<bf16> w;
      w.load(wb + q * kHcBlockCh);
#pragma unroll
      for (int s = 0; s < S; ++s)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[q][s] = fmaf(w.v[e], gv[s][e], acc[q][s]);
    }
    if (ch == h.nchunk - 1) {   // the classes of this block are complete
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int kl = g * kHcBlockClasses + warp * 8 + q;
        const float bk = (bfc && kl < nk) ? bfc[k0 + kl] : 0.f;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          float v = acc[q][s];
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane == 0 && kl < nk) zs[s * kHcMaxKc + kl] = v + bk;
          acc[q][s] = 0.f;
        }
      }
    }
  }
  cp_async_wait<0>();
  __syncthreads();

  // ---- 3. decision
  if (warp < S && b0 + warp < B) {
    const int s = warp, b = b0 + s;
    const int cls = (d.shift && d.shift_cls) ? d.shift_cls[b] : -1;
    const float sh = cls >= 0 && cls < K ? d.shift[b] : 0.f;
    float zr[kHcMaxKc / 32];
    float m = -INFINITY;
    int arg = 0x7fffffff;
#pragma unroll
    for (int i = 0; i < kHcMaxKc / 32; ++i) {
      const int j = lane + 32 * i;
      zr[i] = j < nk ? zs[s * kHcMaxKc + j] : -INFINITY;
      if (j < nk) {
        if (k0 + j == cls) zr[i] += sh;
        if (z) z[(size_t)b * K + k0 + j] = zr[i];
        if (zr[i] > m) m = zr[i], arg = k0 + j;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, m, o);
      const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
      if (om > m || (om == m && oa < arg)) m = om, arg = oa;
    }
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < kHcMaxKc / 32; ++i)
      if (lane + 32 * i < nk) sum += expf(zr[i] - m);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) {
      float* mine = part + ((size_t)rank * S + s) * 4;
      hc_st_f32(hc_map(mine, 0), m);
      hc_st_f32(hc_map(mine + 1, 0), __int_as_float(arg));
      hc_st_f32(hc_map(mine + 2, 0), sum);
    }
  }
  hc_cluster_arrive();   // #3: the leader holds every CTA's triple
  hc_cluster_wait();
  if (rank != 0) return;
  if (tid < S && b0 + tid < B) {
    const int s = tid, b = b0 + s;
    float m = -INFINITY;
    int arg = 0x7fffffff;
    for (int r = 0; r < kHcCluster; ++r) {   // ranks hold ascending classes: strict > keeps the lowest argmax
      const float mr = part[(r * S + s) * 4];
      if (mr > m) m = mr, arg = __float_as_int(part[(r * S + s) * 4 + 1]);
    }
    float tot = 0.f;
    for (int r = 0; r < kHcCluster; ++r) {
      const float mr = part[(r * S + s) * 4];
      if (mr != -INFINITY) tot += part[(r * S + s) * 4 + 2] * expf(mr - m);   // a rank without classes holds -inf
    }
    const float cf = 1.0f / tot;
    if (d.conf) d.conf[b] = cf;
    if (d.pred) d.pred[b] = arg == 0x7fffffff ? 0 : arg;
    d.mask[b] = (uint8_t)((d.always_exit || cf >= d.thr) ? 1 : 0);
  }
  // ---- 4. scan, by the last tile
  __threadfence();
  __syncthreads();
  if (tid == 0) *flag = atomicAdd(d.done, 1u) == gridDim.x / kHcCluster - 1 ? 1 : 0;
  __syncthreads();
  if (!*flag) return;
  __threadfence();
  if (tid == 0) *d.done = 0;
  exit_scan<kHcThreads>(B, d);
}

template <int S>
inline cudaError_t hc_launch_t(const bf16* x, int HW, int C, const bf16* wfc, const float* bfc, int B, int K, float* z, const DecideArgs& d,
                               cudaStream_t st) {
  const HcShape h = hc_shape(C, K);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((B + S - 1) / S * kHcCluster));
  cfg.blockDim = dim3(kHcThreads);
  cfg.dynamicSmemBytes = hc_smem_bytes(S, h);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, head_cluster_kernel<S>, x, HW, C, wfc, bfc, B, K, z, d, h);
}
// d.done must be zero when the kernel starts and is zero again when it ends; d.tile_done is not used.
inline cudaError_t hc_launch(const bf16* x, int HW, int C, const bf16* wfc, const float* bfc, int B, int K, float* z, const DecideArgs& d,
                             cudaStream_t st) {
  switch (hc_tile_samples(B)) {
    case 1: return hc_launch_t<1>(x, HW, C, wfc, bfc, B, K, z, d, st);
    case 2: return hc_launch_t<2>(x, HW, C, wfc, bfc, B, K, z, d, st);
    default: return hc_launch_t<4>(x, HW, C, wfc, bfc, B, K, z, d, st);
  }
}
inline cudaError_t hc_context_init() {
  const size_t most = hc_smem_bytes(4, hc_shape(2048, kHcCluster * kHcMaxKc));
  cudaError_t e = cudaFuncSetAttribute(head_cluster_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(head_cluster_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(head_cluster_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  return e;
}

constexpr int kCopyThreads = 256, kCopyUnroll = 8;

// feat_out[j] = feat[surv_idx[j]] for j < *n_surv, in vectors of type V (16 bytes whenever the row size
// allows), grid (chunks, max_rows).
template <typename V>
__global__ void __launch_bounds__(kCopyThreads)
gather_rows_kernel(const V* __restrict__ src, size_t vecs_per_row, const int32_t* __restrict__ surv_idx,
                   const int32_t* __restrict__ n_surv, V* __restrict__ dst, int rev) {
  pdl_launch_dependents();
  pdl_wait();
  const int j = rev ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;   // rev: last row first, each row from its end
  const unsigned bx = rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
  if (j >= *n_surv) return;
  const V* s = src + (size_t)surv_idx[j] * vecs_per_row;
  V* d = dst + (size_t)j * vecs_per_row;
  const size_t v0 = (size_t)bx * (kCopyThreads * kCopyUnroll) + threadIdx.x;
  V r[kCopyUnroll];
#pragma unroll
  for (int u = 0; u < kCopyUnroll; ++u) {
    const size_t v = v0 + (size_t)u * kCopyThreads;
    if (v < vecs_per_row) r[u] = __ldcs(s + v);
  }
#pragma unroll
  for (int u = 0; u < kCopyUnroll; ++u) {
    const size_t v = v0 + (size_t)u * kCopyThreads;
    if (v < vecs_per_row) d[v] = r[u];
  }
}

// The same inside one buffer of B rows: rows surv_idx[j] > j of `feat` move down to row j, j ascending.  A thread owns a column of
// vectors and moves its own down all rows, kMoveRows loads ahead of the stores: a store to row j hits what an earlier load has fetched
// or nobody needs (surv_idx ascends, and j <= surv_idx[j] < surv_idx[j'] for every later j'), and threads do not share columns.  Rows
// in front of the first sample that left stay where they are, and a batch that nobody leaves is not copied at all.
// Bound by HBM once rows move.  First stage of the ResNet-50-shaped model at batch 64, gathered from the workspace -> closed up in
// place, us: 0, 1, 19 of 64 leave 317 / 317 / 306 -> 280 / 291 / 304; third stage, batch 7 107 -> 98.  256 threads or eight rows at a time: 19
// leave 306 to 308; a search for the first row that moves, through shared memory: 312, and 2 us on small maps.
constexpr int kMoveThreads = 128, kMoveRows = 16;
template <typename V>
__global__ void __launch_bounds__(kMoveThreads)
move_rows_kernel(V* feat, size_t vecs_per_row, const int32_t* __restrict__ surv_idx, const int32_t* __restrict__ n_surv, int B) {
  const size_t v = (size_t)blockIdx.x * kMoveThreads + threadIdx.x;
  V* at = feat + v;
  pdl_launch_dependents();
  pdl_wait();
  const int n = *n_surv;   // and, asked for together with it, the first rows' sources
  if (v >= vecs_per_row) return;
  for (int j0 = 0; j0 < B; j0 += kMoveRows) {
    int from[kMoveRows];
    V r[kMoveRows];
#pragma unroll
    for (int u = 0; u < kMoveRows; ++u) from[u] = j0 + u < B ? surv_idx[j0 + u] : 0;
    if (j0 >= n || n == B) return;
#pragma unroll
    for (int u = 0; u < kMoveRows; ++u)
      if (j0 + u < n && from[u] != j0 + u) r[u] = __ldcs(at + (size_t)from[u] * vecs_per_row);
#pragma unroll
    for (int u = 0; u < kMoveRows; ++u)
      if (j0 + u < n && from[u] != j0 + u) at[(size_t)(j0 + u) * vecs_per_row] = r[u];
  }
}

// Flat copy of n vectors plus n_ids int32 (the appended arrivals of a refill).
template <typename V>
__global__ void __launch_bounds__(kCopyThreads)
append_rows_kernel(const V* __restrict__ src, V* __restrict__ dst, size_t n, const int32_t* __restrict__ ids_src,
                   int32_t* __restrict__ ids_dst, int n_ids) {
  pdl_launch_dependents();
  pdl_wait();
  const size_t stride = (size_t)gridDim.x * kCopyThreads;
  for (size_t v = (size_t)blockIdx.x * kCopyThreads + threadIdx.x; v < n; v += stride) dst[v] = __ldcs(src + v);
  if (ids_src && ids_dst && blockIdx.x == 0)
    for (int i = threadIdx.x; i < n_ids; i += kCopyThreads) ids_dst[i] = ids_src[i];
}

}  // namespace ee
