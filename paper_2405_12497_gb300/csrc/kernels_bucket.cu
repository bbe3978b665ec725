// kernels_bucket.cu -- the bucket-major scan of large batches (§3.3.2, §4).
//
// When many queries of a batch probe the same buckets, the products <x_b,
// q_u> of one bucket's codes with the quantized queries of all its probes
// are one matrix product. It runs on the tensor cores (tcgen05 kind::f8f6f4:
// a code bit is the E4M3 value 2, a quantized query value 0..15 is itself,
// and the FP32 accumulator holds the exact integer 2 <x_b, q_u>), and the
// estimator, its bound and the candidates come from the accumulator:
//
//   1. bucket_tau0_kernel   per query, the k-th smallest upper bound of its
//                           first codes (nearest probes): tau0 >= tau_ub. Of a
//                           short query these are all its codes: its
//                           candidates, and steps 2 to 4 are without it
//   2. bucket_count / bucket_plan / bucket_quant: (query, probe) pairs
//                           grouped by bucket, quantized (§3.3.1) into
//                           operand rows; work items {bucket, pairs, codes};
//                           the room a query's candidate list may take
//   3. bucket_scan<1>       every code: upper bounds <= tau0, per query;
//      bucket_tau_kernel    tau_ub, the k-th smallest of them (exact)
//   4. bucket_scan<2>       every code again: the candidates LB <= tau_ub
//   5. bucket_tail_kernel   pilot, re-rank and top-k per query (the rule of
//                           finish_query; most rows through their 8-bit copy)
//
// The results are those of the per-query scan bit for bit: the products are
// exact, the estimator is evaluated in the same FP32 order, and the re-rank
// rule depends on the candidate set only, not on the order it was found in.
// A query whose candidate list outgrows its capacity goes to the redo list,
// which the per-query kernel runs, a CTA for each: some milliseconds for a
// query of 256 large buckets, however few they are. So the lists share one
// pool, and where most queries probe few codes (learned counts) the others get
// room for several times the even share (13 of 10k queries of a learned batch,
// 10M x 256, had up to 54k candidates against a share of 32k: 6.29 ms with
// them redone, 4.66 all per query, 3.68 so).
//
// Measured (GB300, order to re-rank of one batch, per-query kernel -> this):
//   10k queries x 62 probes, 1M x 128, K 4096, k 100        4.83 -> 2.30 ms
//   10k queries x 128 probes, 2M x 256, K 4096, k 100      17.5  -> 6.44 ms
//   4000 queries x 16 probes, 1M x 128, K 4096, k 10        0.57 -> 0.37 ms
//   1000 queries x 32 probes, 200k x 960, K 1024, k 100     1.27 -> 0.95 ms
// Of the first: quantization 0.22, tau0 0.13, passes 0.43 and 0.71, tail 0.86.
// The quantization keeps 74% of the issue slots busy. The passes keep half of
// them busy and the tensor pipe 5 and 3%, DRAM below 10%: they wait for the
// hits' list slots and the items' constants (most stalls are on global loads and
// atomics), and their time hardly follows their work (8000 learned queries:
// 0.17 ms for pass 2 with all pairs or a quarter less). The tail is bound by the
// latency of its short steps (loads, then barriers; DRAM 36%).
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "internal.h"
#include "query_common.cuh"
#include "tc_util.cuh"

namespace rbq {
namespace {

constexpr int kGM = 128;                 // codes per tile (TMEM lanes)
constexpr int kGN = 128;                 // most pairs per item (TMEM columns)
constexpr int kGChunk = 128;             // code bits per operand stage (1 byte each)
constexpr int kGStages = 2;
constexpr int kGStageBytes = kGM * kGChunk;
constexpr int kGQueue = 28;              // queued hits per lane
constexpr int kGQueueFlush = 12;         // flushed above (16 columns may add 16 more)
constexpr int kGEpiWarps = 8, kGProdWarps = 4;
constexpr int kGMmaWarp = kGEpiWarps + kGProdWarps, kGItemWarp = kGMmaWarp + 1;
constexpr int kGThreads = (kGItemWarp + 1) * 32;
constexpr int kGTilesPerItem = 4;        // code tiles per work item
constexpr int kGPad = 16;                // a bucket's pair slots start at a multiple of this
constexpr int kQJ = 4;                   // probes per quantization run
constexpr int kGTau0Probes = 16;         // probes the first threshold may look at
constexpr float kGSlack = 0x1.0p-18f;    // prefilter slack (bucket_scan_kernel)
constexpr int kGLevels = 6;              // list capacities: the even share << level

struct BucketParams {
  const uint64_t* codes;
  const float4* factors;
  const int32_t* bucket_off;
  int W, dpad, nt;           // nt: pairs per item
  const int32_t* boff;       // K + 1 padded pair offsets
  const int32_t* bcnt;       // K pair counts
  const int4* items;         // {bucket, first pair, first tile, tiles}
  const int* nitems;
  int* work;                 // work counter
  const uint8_t* qop;        // pair slots: operand rows, 8 slots x (16-byte chunk, slot) order
  const float4* smeta;       // pair slots: A, B, E, add
  const float* spsum;        // pair slots: sum(q_u)
  const int32_t* sq;         // pair slots: query
  const float* tau;          // queries: the pass's threshold
  uint32_t* ulist;           // pass 1: queries x capu upper-bound keys
  int4* list;                // pass 2: the lists {position, LB, estimate, UB}
  const int2* lrow;          // pass 2: queries: a list's first entry and capacity
  int* cnt;                  // queries: hits of this pass
  int cap;                   // pass 1
  int* err;
};

// ------------------------------------------------------------ packed FP32
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t pack2u(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Append e to the lane's queue at qp (32 lanes interleaved) unless w > t (a
// NaN is kept). Predicated and without a memory clobber, so that the columns
// of a chunk may overlap.
__device__ __forceinline__ void queue_unless_above(uint32_t& qp, float w, float t, uint32_t e) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.gt.f32 p, %1, %2;\n@!p st.shared.u32 [%0], %3;\n"
      "@!p add.u32 %0, %0, 128;\n}"
      : "+r"(qp)
      : "f"(w), "f"(t), "r"(e));
}

// Instruction descriptor of kind::f8f6f4 with E4M3 operands (format 0) and an
// FP32 accumulator, both operands K-major.
__device__ __forceinline__ uint32_t make_idesc_f8(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// ------------------------------------------------------------- pair grouping
// Probes of query q that are searched.
__device__ __forceinline__ int probes_of(const FusedParams& P, int64_t q) {
  return P.nprobe_q ? min(max(P.nprobe_q[q], 1), P.nprobe) : P.nprobe;
}

// Whether the first threshold looks at all codes of a query (np probes).
__device__ __forceinline__ bool short_query(int codes, int np, int want_max) {
  return codes <= want_max && np <= kGTau0Probes;
}

// One warp per query (learned counts are mostly far below nprobe); short ones
// are marked and not counted. Of the others also, where counts differ, the runs
// of kQJ probes for the quantization, and of all the entries that all candidate lists would take at each level of capacity
// (share << level, and never more than the query's codes): lsum.
__global__ void __launch_bounds__(256) bucket_count_kernel(FusedParams P, int share, int want_max,
                                                           int32_t* __restrict__ bcnt,
                                                           unsigned long long* __restrict__ lsum,
                                                           int* __restrict__ is_short,
                                                           int* __restrict__ nruns,
                                                           int2* __restrict__ runs) {
  __shared__ int s_codes[8], s_runs[8], s_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  int codes = 0, nr = 0;
  if (q < P.nq) {
    const int np = probes_of(P, q);
    int first = -1;  // the lane's only probe of a query that may be short
    for (int j = lane; j < np; j += 32) {
      const int c = P.probe_ids[q * P.nprobe + j];
      if (c >= 0) {
        if (np > kGTau0Probes) atomicAdd(bcnt + c, 1); else first = c;
        codes += __ldg(P.bucket_off + c + 1) - __ldg(P.bucket_off + c);
      }
    }
    __syncwarp();
    codes = __reduce_add_sync(kFull, codes);
    const bool brief = short_query(codes, np, want_max);
    if (first >= 0 && !brief) atomicAdd(bcnt + first, 1);
    if (lane == 0) is_short[q] = brief;
    if (P.nprobe_q && !brief) nr = (np + kQJ - 1) / kQJ;
  }
  if (lane == 0) {
    s_codes[wid] = codes;
    s_runs[wid] = nr;
  }
  __syncthreads();
  if (P.nprobe_q && threadIdx.x == 32) {
    int sum = 0;
    for (int w = 0; w < 8; ++w) sum += s_runs[w];
    s_base = atomicAdd(nruns, sum);
  }
  if (threadIdx.x < kGLevels) {
    unsigned long long sum = 0;
    for (int w = 0; w < 8; ++w) sum += min((int64_t)s_codes[w], (int64_t)share << threadIdx.x);
    atomicAdd(lsum + threadIdx.x, sum);
  }
  if (!P.nprobe_q) return;
  __syncthreads();
  int at = s_base;
  for (int w = 0; w < wid; ++w) at += s_runs[w];
  for (int i = lane; i < nr; i += 32) runs[at + i] = make_int2((int)q, i * kQJ);
}

// Exclusive block scan of one int per thread (1024 threads); returns the
// value before this thread, *total the sum.
__device__ int scan1024(int v, int* total) {
  __shared__ int wt[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wt[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int t = wt[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, t, o);
      if (lane >= o) t += y;
    }
    wt[lane] = t;
  }
  __syncthreads();
  const int before = wid ? wt[wid - 1] : 0;
  *total = wt[31];
  __syncthreads();
  return before + x - v;
}

// Padded slot offsets of the buckets and the work items: every bucket's
// pairs in blocks of nt, every block's codes in runs of kGTilesPerItem
// tiles. The large items (at least half of the largest possible) come first:
// each CTA claims an item or two ahead, and a large one claimed last would
// keep the others waiting. One block.
__global__ void __launch_bounds__(1024) bucket_plan_kernel(const int32_t* __restrict__ bcnt,
                                                           const int32_t* __restrict__ bucket_off,
                                                           int K, int nt, int32_t* __restrict__ boff,
                                                           int4* __restrict__ items,
                                                           int* __restrict__ nitems) {
  const int per = (K + 1023) / 1024;
  const int c0 = min(K, (int)threadIdx.x * per), c1 = min(K, c0 + per);
  const int half = nt * kGTilesPerItem / 2;
  // every item of bucket c: f(item, is it large)
  auto each = [&](int c, auto f) {
    const int n = bcnt[c], tiles = (bucket_off[c + 1] - bucket_off[c] + kGM - 1) / kGM;
    for (int n0 = 0; n0 < n; n0 += nt)
      for (int t0 = 0; t0 < tiles; t0 += kGTilesPerItem) {
        const int t = min(kGTilesPerItem, tiles - t0);
        f(make_int4(c, n0, t0, t), min(nt, n - n0) * t >= half);
      }
  };
  int slots = 0, big = 0, rest = 0;
  for (int c = c0; c < c1; ++c) {
    slots += (bcnt[c] + kGPad - 1) / kGPad * kGPad;
    each(c, [&](int4, bool large) { (large ? big : rest) += 1; });
  }
  int tot_s, tot_b, tot_r;
  int so = scan1024(slots, &tot_s), bo = scan1024(big, &tot_b), ro = scan1024(rest, &tot_r);
  ro += tot_b;
  for (int c = c0; c < c1; ++c) {
    boff[c] = so;
    so += (bcnt[c] + kGPad - 1) / kGPad * kGPad;
    each(c, [&](int4 e, bool large) { items[large ? bo++ : ro++] = e; });
  }
  if (threadIdx.x == 0) {
    boff[K] = tot_s;
    *nitems = tot_b + tot_r;
  }
}

// Randomized quantization (§3.3.1, the arithmetic of quant_core) of a query
// against a run of kQJ probes, one warp per run: the rotated query stays in
// registers, each value goes to its pair's operand row as an E4M3 byte, and
// the per-pair constants are formed by one lane per pair at the end.
//
// The byte order inside each 32 coordinates is that of the code expansion
// (expand_code): coordinate 8 j + t is byte 4 t + j.
//
// The quotient (qd - v_l) / Delta is only needed inside floor(x + u): it is
// taken from a multiplication by 1 / Delta unless the sum falls within 3e-5
// of an integer (the multiplied form is within 5e-6 of the correctly rounded
// one for x < 16), where the division decides.
// With one count for all queries a warp takes every quant_runs-th run of its
// query. LISTED: the warps take the runs in turn, from a list
// (bucket_count_kernel): per-query counts are mostly far below nprobe, and a
// warp per possible run was mostly warps without work (nprobe_max 256, 7.6
// probes on average: 92 us per 8000 queries), while with four warps to each
// query most idled as those of 100 probes and more held up the rest (52 us; so
// 29; with one count the list is 1 to 2% of a search slower).
__host__ __device__ inline int quant_runs(int nprobe) {
  const int r = (nprobe + kQJ - 1) / kQJ;
  return r < 4 ? r : 4;
}
template <bool LISTED>
__global__ void __launch_bounds__(256) bucket_quant_kernel(FusedParams P,
                                                           const int* __restrict__ is_short,
                                                           const int* __restrict__ nruns,
                                                           const int2* __restrict__ list,
                                                           const int32_t* __restrict__ boff,
                                                           int32_t* __restrict__ bfill,
                                                           uint8_t* __restrict__ qop,
                                                           float4* __restrict__ smeta,
                                                           float* __restrict__ spsum,
                                                           int32_t* __restrict__ sq) {
  const int lane = threadIdx.x & 31;
  const int w = (blockIdx.x * 256 + threadIdx.x) >> 5;
  const int runs = quant_runs(P.nprobe);
  int64_t q = w / runs;
  if (!LISTED && (q >= P.nq || is_short[q])) return;
  // items: runs of the list, or first probes of the query's runs
  const int end = LISTED ? *nruns : probes_of(P, q);
  const int step = LISTED ? (int)gridDim.x * 8 : runs * kQJ;
  const int dpad = P.dpad;
  const int qmax = (1 << P.bq) - 1;
  const uint32_t sub = (uint32_t)(lane >> 1) & 3u;  // byte of the operand word
  for (int i = LISTED ? w : (int)(w - q * runs) * kQJ; i < end; i += step) {
  int j0 = i;
  if (LISTED) {
    const int2 run = __ldg(list + i);
    q = run.x;
    j0 = run.y;
  }
  const int nj = min(kQJ, (LISTED ? probes_of(P, q) : end) - j0);
  const float* rq = P.rq + q * dpad;
  // lane j < nj: pair j's cluster, slot and constants
  int c_l = -1, slot_l = 0, sum_l = 0;
  float vl_l = 0.0f, delta_l = 0.0f, add_l = 0.0f, nq2_l = 0.0f;
  if (lane < nj) {
    const int64_t pj = q * P.nprobe + j0 + lane;
    c_l = P.probe_ids[pj];
    add_l = P.probe_dist[pj];
    nq2_l = P.probe_nq2 ? P.probe_nq2[pj] : add_l;
    if (c_l >= 0) slot_l = boff[c_l] + atomicAdd(bfill + c_l, 1);
  }
  for (int j = 0; j < nj; ++j) {
    const int c = __shfl_sync(kFull, c_l, j);
    const int slot = __shfl_sync(kFull, slot_l, j);
    if (c < 0) continue;
    const float* pc = P.ptc + (int64_t)c * dpad;
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    for (int k0 = 4 * lane; k0 < dpad; k0 += 128) {
      const float4 a = *reinterpret_cast<const float4*>(rq + k0);
      const float4 b = __ldg(reinterpret_cast<const float4*>(pc + k0));
      const uint32_t x0 = float_key(__fsub_rn(a.x, b.x)), x1 = float_key(__fsub_rn(a.y, b.y));
      const uint32_t x2 = float_key(__fsub_rn(a.z, b.z)), x3 = float_key(__fsub_rn(a.w, b.w));
      kmin = min(kmin, min(min(x0, x1), min(x2, x3)));
      kmax = max(kmax, max(max(x0, x1), max(x2, x3)));
    }
    const float vl = key_float(__reduce_min_sync(kFull, kmin));
    const float vr = key_float(__reduce_max_sync(kFull, kmax));
    const float delta = __fdiv_rn(__fsub_rn(vr, vl), (float)qmax);
    const float inv = __frcp_rn(delta);
    int sum = 0;
    uint8_t* row = qop + (int64_t)(slot >> 3) * 8 * dpad + (slot & 7) * 16;
    for (int b0 = 0; b0 < dpad; b0 += 128) {
      const int k0 = b0 + 4 * lane;
      float qf[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      if (delta > 0.0f && k0 < dpad) {
        const float4 a = *reinterpret_cast<const float4*>(rq + k0);
        const float4 b = __ldg(reinterpret_cast<const float4*>(pc + k0));
        const float qd[4] = {__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z),
                             __fsub_rn(a.w, b.w)};
        const U4 r = philox4x32_10(P.seed, (uint32_t)(k0 >> 2), (uint32_t)(P.q_offset + q),
                                   (uint32_t)c, kTagQuant);
        const uint32_t ws[4] = {r.x, r.y, r.z, r.w};
        bool near = false;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float u = __fmul_rn(__uint2float_rn(ws[e] >> 8), 0x1.0p-24f);
          const float y = __fmaf_rn(__fsub_rn(qd[e], vl), inv, u);
          const float f = floorf(y), fr = y - f;
          near = near || !(fr >= 3e-5f && fr <= 1.0f - 3e-5f);
          qf[e] = fminf(f, (float)qmax);
        }
        if (near) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float u = __fmul_rn(__uint2float_rn(ws[e] >> 8), 0x1.0p-24f);
            const float x = __fdiv_rn(__fsub_rn(qd[e], vl), delta);
            const int v = __float2int_rd(__fadd_rn(x, u));
            qf[e] = (float)(v > qmax ? qmax : v);
          }
        }
      }
      sum += (int)qf[0] + (int)qf[1] + (int)qf[2] + (int)qf[3];
      // the four values as E4M3 bytes, then a 4 x 4 byte transpose over the
      // lanes l, l ^ 2, l ^ 4, l ^ 6: word r of a chunk holds value r of the
      // four lanes with this lane's parity
      uint16_t lo, hi;
      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(qf[1]), "f"(qf[0]));
      asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(qf[3]), "f"(qf[2]));
      uint32_t x = (uint32_t)lo | ((uint32_t)hi << 16);
      uint32_t y = __shfl_xor_sync(kFull, x, 2);
      x = (sub & 1u) ? __byte_perm(x, y, 0x3715) : __byte_perm(x, y, 0x6240);
      y = __shfl_xor_sync(kFull, x, 4);
      x = (sub & 2u) ? __byte_perm(x, y, 0x3276) : __byte_perm(x, y, 0x5410);
      if (k0 < dpad) {
        const int chunk = (b0 >> 4) + (lane >> 3) * 2 + (lane & 1);
        *reinterpret_cast<uint32_t*>(row + chunk * 128 + 4 * sub) = x;
      }
    }
    sum = warp_sum_i(sum);
    if (lane == j) {
      vl_l = vl;
      delta_l = delta;
      sum_l = sum;
    }
  }
  if (lane < nj && c_l >= 0) {
    smeta[slot_l] = quant_meta(delta_l, vl_l, nq2_l, add_l, P.eps0, dpad);
    spsum[slot_l] = (float)sum_l;
    sq[slot_l] = (int32_t)q;
  }
  }
}

// ---------------------------------------------------------- first threshold
struct ListPool {
  const unsigned long long* sum;  // kGLevels (bucket_count_kernel)
  unsigned* used;
  unsigned size;                  // entries (below 2^31)
  int share;
};

// tau0 of a query: the k-th smallest upper bound of its first `want` codes
// (in probe order, at most kGTau0Probes probes), +inf when there are fewer
// than k. The k-th smallest of any subset bounds tau_ub from above. Of a
// short query (at most want_max codes in kGTau0Probes probes) all are looked
// at: that is tau_ub itself, the candidates are written here, and tau0 = -inf
// keeps the tau kernel from the query: its pairs are not grouped, quantized or
// scanned. Also clears the query's hit
// counters and takes its candidate list from the pool, at the highest level at
// which all lists fit (level 0 does: the pool has a share for each). One CTA
// per query.
// (The CTA is short steps that wait on each other: the CTAs resident set the
// rate, so registers are held to what six -- four for longer codes -- allow.)
template <int WT, int BQT>
__global__ void __launch_bounds__(kThreads, WT == 2 ? 6 : 4) bucket_tau0_kernel(
    FusedParams P, int want_max, ListPool lp, float* __restrict__ tau0, float* __restrict__ taub,
    int* __restrict__ ucnt, int* __restrict__ lcnt, int2* __restrict__ lrow,
    int4* __restrict__ list) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ SelState s_sel;
  __shared__ float4 s_meta[kGTau0Probes];
  __shared__ int s_psum[kGTau0Probes], s_pbeg[kGTau0Probes], s_pref[kGTau0Probes + 1];
  __shared__ int s_np;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int64_t q = blockIdx.x;
  const int W = P.W, bq = P.bq;
  FusedSmem S;
  S.planes = reinterpret_cast<uint64_t*>(smem);
  S.pmeta = s_meta;
  S.psum = s_psum;
  S.pbeg = s_pbeg;
  S.pref = s_pref;
  uint32_t* ub = reinterpret_cast<uint32_t*>(smem + sizeof(uint64_t) * kGTau0Probes * bq * W);
  int* hist = reinterpret_cast<int*>(ub + want_max);
  uint32_t* coll = reinterpret_cast<uint32_t*>(hist + kHistBins);
  float2* both = reinterpret_cast<float2*>(coll + 256);  // a short query's LB, estimate
  const int np_all = probes_of(P, q), np = min(np_all, kGTau0Probes);
  // the codes to look at: a third of the query's codes where that is fewer
  // than want_max (at least 4 k): a code costs here over twice what it costs
  // in pass 1, which a looser tau0 only gives some more hits
  int codes = 0;
  for (int i = tid; i < np_all; i += kThreads) {
    const int c = P.probe_ids[q * P.nprobe + i];
    if (c >= 0) codes += P.bucket_off[c + 1] - P.bucket_off[c];
  }
  codes = __reduce_add_sync(kFull, codes);
  if (lane == 0) s_sel.warp_cnt[wid] = codes;
  __syncthreads();
  codes = 0;
  for (int w = 0; w < kThreads / 32; ++w) codes += s_sel.warp_cnt[w];
  const bool all = short_query(codes, np_all, want_max);  // tau0 is tau_ub then
  const int want = all ? codes : min(want_max, max(codes / 3, 4 * P.k));
  if (wid == 0) {  // the probes that hold the first `want` codes
    int len = 0;
    if (lane < np) {
      const int c = P.probe_ids[q * P.nprobe + lane];
      if (c >= 0) len = P.bucket_off[c + 1] - P.bucket_off[c];
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const unsigned full = __ballot_sync(kFull, incl >= want || lane >= np - 1);
    if (lane == 0) s_np = __ffs(full);
  }
  if (tid == 0) {
    ucnt[q] = 0;
    lcnt[q] = 0;
  }
  __syncthreads();
  const int m = s_np;
  if (wid == kThreads / 32 - 1) {  // (a warp that seldom has a probe to quantize)
    const bool fits = lane < kGLevels && lp.sum[lane] <= lp.size;
    const int l = 31 - __clz((int)(__ballot_sync(kFull, fits) | 1u));
    const int cap = (int)min((int64_t)codes, (int64_t)lp.share << l);
    if (lane == 0) lrow[q] = make_int2((int)atomicAdd(lp.used, (unsigned)cap), cap);
  }
  for (int j = wid; j < m; j += kThreads / 32) {
    const int64_t pj = q * P.nprobe + j;
    const float add = P.probe_dist[pj];
    quantize_probe(P, S, q, j, j, P.probe_ids[pj], P.probe_nq2 ? P.probe_nq2[pj] : add, add);
  }
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    s_pref[0] = 0;
    for (int j = 0; j < m; ++j) {
      run += s_pref[j + 1];
      s_pref[j + 1] = run;
    }
  }
  __syncthreads();
  const int n = min(want, s_pref[m]);
  int j = 0;
  for (int t = tid; t < n; t += kThreads) {
    while (s_pref[j + 1] <= t) ++j;
    const int64_t pos = s_pbeg[j] + (t - s_pref[j]);
    CodeRegs<WT> cr;
    const uint64_t* code = P.codes + pos * W;
    load_code<WT>(cr, code);
    const float4 f = __ldg(P.factors + pos);
    const int ip = code_ip<WT, BQT>(cr, code, S.planes + (size_t)j * bq * W, W, bq);
    const float4 mt = s_meta[j];
    const float t1 = (float)(2 * ip - s_psum[j]);
    const float xq = __fadd_rn(__fmul_rn(mt.x, t1), __fmul_rn(mt.y, f.w));
    const float dist = __fsub_rn(__fadd_rn(f.x, mt.w), __fmul_rn(f.y, xq));
    const float er = __fmul_rn(f.z, mt.z);
    ub[t] = float_key(__fadd_rn(dist, er));
    if (all) both[t] = make_float2(__fsub_rn(dist, er), dist);
  }
  __syncthreads();
  float tau = __int_as_float(0x7f800000);
  if (n >= P.k) {
    int rem, eq;
    tau = key_float(hist_select(n, P.k, s_sel, hist, coll, 256, rem, eq,
                                [ub](int i) { return ub[i]; }));
  }
  if (tid == 0) {
    tau0[q] = all ? __int_as_float(0xff800000) : tau;
    if (all) taub[q] = tau;
  }
  if (!all) return;
  int4* L = list + lrow[q].x;  // (n entries at most: the query's codes)
  if (tid == 0) s_np = 0;
  __syncthreads();
  j = 0;
  for (int t0 = 0; t0 < n; t0 += kThreads) {
    const int t = t0 + tid;
    float2 e = make_float2(0.0f, 0.0f);
    if (t < n) e = both[t];
    const bool in = t < n && e.x <= tau;
    const int slot = warp_reserve(in, &s_np);
    if (in) {
      while (s_pref[j + 1] <= t) ++j;
      L[slot] = make_int4(s_pbeg[j] + (t - s_pref[j]), __float_as_int(e.x), __float_as_int(e.y),
                          __float_as_int(key_float(ub[t])));
    }
  }
  __syncthreads();
  if (tid == 0) lcnt[q] = s_np;
}

// tau_ub of a query: the k-th smallest upper bound of its pass-1 list (which
// holds every code with UB <= tau0, so at least k when tau0 is finite). Of a
// list that outgrew its capacity the kept part gives a bound of tau_ub (the
// tail then finds tau_ub itself).
__global__ void __launch_bounds__(kThreads) bucket_tau_kernel(const uint32_t* __restrict__ ulist,
                                                              const int* __restrict__ ucnt,
                                                              int capu, int k,
                                                              const float* __restrict__ tau0,
                                                              float* __restrict__ taub) {
  __shared__ SelState s_sel;
  __shared__ __align__(16) int hist[kHistBins];
  __shared__ uint32_t coll[256];
  const int64_t q = blockIdx.x;
  if (tau0[q] == __int_as_float(0xff800000)) return;  // known (bucket_tau0_kernel)
  const int n = min(ucnt[q], capu);
  float tau = __int_as_float(0x7f800000);
  if (n >= k) {
    const uint32_t* u = ulist + q * capu;
    int rem, eq;
    tau = key_float(hist_select(n, k, s_sel, hist, coll, 256, rem, eq,
                                [u](int i) { return __ldg(u + i); }));
  }
  if (threadIdx.x == 0) taub[q] = tau;
}

// ------------------------------------------------------------------ the scan
// Roles of the CTA (14 warps): warps 0-7 epilogue in two groups (group g
// drains TMEM accumulator g, warp w of a group its lanes 32 (w % 4) ..),
// warps 8-11 operand A (code bits expanded to E4M3 bytes, one code row per
// thread), warp 12 one thread that copies operand B (the item's pair rows,
// one bulk copy) and issues the MMAs, warp 13 takes the work items and
// gathers their per-pair constants, an item ahead of the others (four
// dependent loads: an item of a few small tiles takes no longer than they).
//
// Epilogue. A lane owns a code row (its factors in registers) and walks the
// item's pairs. Per (code, pair) the exact bound costs ten rounded FP32
// operations; instead a prefilter evaluates a fused form of it with packed
// FMAs, two pairs at a time:
//   u = A acc + c0,  x = B G + u,  v = F1 - F2 x,  w = v + F3 E'
// and drops the pair when w > tau - add. Both forms approximate the same real
// value with fewer than 20 roundings of magnitudes bounded by M = |F1| +
// |add| + F2 (A sum(q_u) + |B| D') + F3 E + |tau|; the constants carry a
// slack of 2^-18 of every term of M (c0, E', F1 and the threshold), more
// than three times that error, and the threshold 1e-36 more for what underflows
// (the smallest step is 1.4e-45), so no pair the exact bound keeps is dropped.
// The few that pass are queued per lane (no votes, no cross-lane traffic)
// and decided by the exact form, lane-parallel, when a queue fills and at
// the end of the tile.
struct ItemInfo {
  int c, beg, rows, slot0, cols, t0, nt;
};

struct __align__(16) ColMeta {
  ulonglong2 pre[kGN / 2][3];  // per two pairs: {A, c0}, {B, E'}, {thr, -}
  float4 ex[kGN];              // A, B, E, add
  float2 pt[kGN];              // sum(q_u), tau
  int q[kGN];
  int2 lr[kGN];                // pass 2: lrow
};

__host__ __device__ inline size_t bucket_smem_bytes(int nt, int dpad) {
  return (size_t)kGStages * kGStageBytes + (size_t)nt * dpad + 2 * sizeof(ColMeta) +
         (size_t)kGEpiWarps * kGQueue * 32 * sizeof(uint32_t);
}

template <int MODE>  // 1: upper bounds <= tau; 2: candidates LB <= tau
__global__ void __launch_bounds__(kGThreads, 2) bucket_scan_kernel(BucketParams P) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(8) uint64_t s_fullA[kGStages], s_emptyA[kGStages], s_fullB, s_doneB,
      s_mfull[2], s_mempty[2], s_tfull[2], s_tempty[2];
  __shared__ volatile int s_fail;
  __shared__ ItemInfo s_info[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t* sA = smem;
  uint8_t* sB = sA + kGStages * kGStageBytes;
  ColMeta* s_col = reinterpret_cast<ColMeta*>(sB + (size_t)P.nt * P.dpad);
  uint32_t* s_queue = reinterpret_cast<uint32_t*>(s_col + 2);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_taddr)),
                 "r"(2 * kGN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kGStages; ++i) {
      mbar_init(&s_fullA[i], kGProdWarps * 32);
      mbar_init(&s_emptyA[i], 1);
    }
    mbar_init(&s_fullB, 1);
    mbar_init(&s_doneB, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_mfull[i], 32);
      mbar_init(&s_mempty[i], (kGEpiWarps + kGProdWarps) * 32 + 1);
      mbar_init(&s_tfull[i], 1);
      mbar_init(&s_tempty[i], 128);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = s_taddr;
  const int nch = (P.dpad + kGChunk - 1) / kGChunk;

  if (warp == kGItemWarp) {
    // ---- the items and their per-pair constants, up to one item ahead
    const int total = *P.nitems;
    bool ok = true;
    int next = 0;
    if (lane == 0) next = atomicAdd(P.work, 1);
    for (uint32_t it = 0;; ++it) {
      const uint32_t buf = it & 1u;
      ItemInfo x;
      x.c = -1;
      next = __shfl_sync(kFull, next, 0);
      if (next < total) {
        const int4 e = __ldg(P.items + next);
        x.c = e.x;
        x.beg = __ldg(P.bucket_off + e.x);
        x.rows = __ldg(P.bucket_off + e.x + 1) - x.beg;
        x.slot0 = __ldg(P.boff + e.x) + e.y;
        x.cols = min(P.nt, __ldg(P.bcnt + e.x) - e.y);
        x.t0 = e.z;
        x.nt = e.w;
        if (lane == 0) next = atomicAdd(P.work, 1);
      }
      const int padded = x.c < 0 ? 0 : (x.cols + kGPad - 1) / kGPad * kGPad;
      float4 m[kGN / 32];
      float ps[kGN / 32], tau[kGN / 32];
      int q[kGN / 32];
      int2 lr[kGN / 32];
#pragma unroll
      for (int u = 0; u < kGN / 32; ++u) {
        const int j = u * 32 + lane;
        m[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        ps[u] = 0.0f;
        q[u] = 0;
        if (x.c >= 0 && j < x.cols) {
          m[u] = __ldg(P.smeta + x.slot0 + j);
          ps[u] = __ldg(P.spsum + x.slot0 + j);
          q[u] = __ldg(P.sq + x.slot0 + j);
        }
      }
#pragma unroll
      for (int u = 0; u < kGN / 32; ++u) {
        const bool in = x.c >= 0 && u * 32 + lane < x.cols;
        tau[u] = in ? __ldg(P.tau + q[u]) : __int_as_float(0xff800000);
        if (MODE == 2) lr[u] = in ? __ldg(P.lrow + q[u]) : make_int2(0, 0);
      }
      if (it >= 2) ok = __all_sync(kFull, pd_wait(smem_u32(&s_mempty[buf]), ((it >> 1) - 1) & 1u, &s_fail));
      if (!ok) {
        s_fail = 1;
        break;
      }
      if (lane == 0) s_info[buf] = x;
      ColMeta& M = s_col[buf];
#pragma unroll
      for (int u = 0; u < kGN / 32; ++u) {
        const int j = u * 32 + lane;
        if (j >= padded) continue;
        const bool none = j >= x.cols;
        const float thr = none ? __int_as_float(0xff800000)
                               : (tau[u] - m[u].w) + (kGSlack * (fabsf(m[u].w) + fabsf(tau[u])) + 1e-36f);
        M.ex[j] = m[u];
        M.pt[j] = make_float2(ps[u], tau[u]);
        M.q[j] = q[u];
        if (MODE == 2) M.lr[j] = lr[u];
        const float xmax = m[u].x * ps[u] + fabsf(m[u].y) * (float)P.dpad;
        float* pre = reinterpret_cast<float*>(M.pre[j >> 1]) + (j & 1);
        pre[0] = m[u].x;
        pre[2] = kGSlack * xmax - m[u].x * ps[u];
        pre[4] = m[u].y;
        pre[6] = (MODE == 1 ? m[u].z : -m[u].z) - kGSlack * m[u].z;
        pre[8] = thr;
      }
      mbar_arrive(&s_mfull[buf]);
      if (x.c < 0) break;
    }
  } else if (warp >= kGEpiWarps && warp < kGMmaWarp) {
    // ---- operand A
    const int pt = tid - kGEpiWarps * 32;
    uint32_t sa = 0;
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      const uint32_t buf = it & 1u;
      ok = pd_wait(smem_u32(&s_mfull[buf]), (it >> 1) & 1u, &s_fail);
      if (!ok) break;
      const ItemInfo x = s_info[buf];
      if (x.c < 0) break;
      for (int t = 0; t < x.nt && ok; ++t) {
        const int r = (x.t0 + t) * kGM + pt;
        const bool live = r < x.rows;
        const uint64_t* code = P.codes + (int64_t)(x.beg + r) * P.W;
        for (int ch = 0; ch < nch; ++ch, ++sa) {
          const uint32_t slot = sa % kGStages;
          const uint64_t w0 = live ? __ldg(code + 2 * ch) : 0ull;
          const uint64_t w1 = live && 2 * ch + 1 < P.W ? __ldg(code + 2 * ch + 1) : 0ull;
          if (sa >= (uint32_t)kGStages &&
              !pd_wait(smem_u32(&s_emptyA[slot]), (sa / kGStages - 1) & 1u, &s_fail)) {
            ok = false;
            break;
          }
          // code bit i of a 32-bit group to bit 6 of byte 4 (i % 8) + i / 8:
          // the E4M3 value 2
          uint8_t* dst = sA + slot * kGStageBytes + core_off(pt, 0, kGM);
          constexpr int kChunkStep = (kGM / 8) * 128;
          const uint32_t wv[4] = {(uint32_t)w0, (uint32_t)(w0 >> 32), (uint32_t)w1,
                                  (uint32_t)(w1 >> 32)};
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const uint32_t v = wv[g];
            constexpr uint32_t kBit = 0x40404040u;
            *reinterpret_cast<uint4*>(dst + (2 * g) * kChunkStep) =
                make_uint4((v << 6) & kBit, (v << 5) & kBit, (v << 4) & kBit, (v << 3) & kBit);
            *reinterpret_cast<uint4*>(dst + (2 * g + 1) * kChunkStep) =
                make_uint4((v << 2) & kBit, (v << 1) & kBit, v & kBit, (v >> 1) & kBit);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive(&s_fullA[slot]);
        }
      }
      if (ok) mbar_arrive(&s_mempty[buf]);
    }
    if (!ok) s_fail = 1;
  } else if (warp == kGMmaWarp) {
    // ---- operand B and the MMAs
    if (lane == 0) {
      constexpr uint32_t lboA = (kGM / 8) * 128;
      const uint32_t sbA = smem_u32(sA), sbB = smem_u32(sB);
      uint32_t sa = 0, tc = 0, commits = 0;
      bool ok = true;
      for (uint32_t it = 0; ok; ++it) {
        const uint32_t buf = it & 1u;
        if (!(ok = pd_wait(smem_u32(&s_mfull[buf]), (it >> 1) & 1u, &s_fail))) break;
        const ItemInfo x = s_info[buf];
        if (x.c < 0) break;
        const int nr = (x.cols + kGPad - 1) / kGPad * kGPad;
        // the previous item's MMAs have read operand B
        if (it > 0 && !(ok = pd_wait(smem_u32(&s_doneB), (it - 1) & 1u, &s_fail))) break;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                         smem_u32(&s_fullB)),
                     "r"((uint32_t)(nr * P.dpad))
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
            ::"r"(sbB), "l"(P.qop + (int64_t)x.slot0 * P.dpad), "r"((uint32_t)(nr * P.dpad)),
            "r"(smem_u32(&s_fullB))
            : "memory");
        ok = mbar_wait(smem_u32(&s_fullB), it & 1u);  // (not cut short: the copy must land)
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t idesc = make_idesc_f8(kGM, nr);
        for (int t = 0; t < x.nt && ok; ++t, ++tc) {
          const uint32_t b = tc & 1u;
          if (tc >= 2 && !(ok = pd_wait(smem_u32(&s_tempty[b]), ((tc >> 1) - 1) & 1u, &s_fail)))
            break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t dt = taddr + b * (uint32_t)kGN;
          for (int ch = 0; ch < nch; ++ch, ++sa) {
            const uint32_t slot = sa % kGStages;
            if (!(ok = pd_wait(smem_u32(&s_fullA[slot]), (sa / kGStages) & 1u, &s_fail))) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const int nk = min(kGChunk, P.dpad - ch * kGChunk) / 32;
            for (int i = 0; i < nk; ++i) {
              const uint64_t da =
                  make_desc(sbA + slot * kGStageBytes + (uint32_t)(2 * i) * lboA, lboA, 128);
              const uint64_t db = make_desc(sbB + (uint32_t)(ch * 8 + 2 * i) * 128u, 128u,
                                            (uint32_t)P.dpad * 8u);
              asm volatile(
                  "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                  "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}" ::"r"(dt),
                  "l"(da), "l"(db), "r"(idesc), "r"((ch | i) ? 1u : 0u));
            }
            tc_commit(&s_emptyA[slot]);
          }
          if (!ok) break;
          tc_commit(&s_tfull[b]);
        }
        tc_commit(&s_doneB);
        ++commits;
        mbar_arrive(&s_mempty[buf]);
      }
      if (!ok) s_fail = 1;
      // every MMA issued completes before the CTA frees its TMEM
      if (commits) mbar_wait(smem_u32(&s_doneB), (commits - 1) & 1u);
    }
    __syncwarp();
  } else {
    // ---- epilogue
    const int group = warp >> 2, quarter = warp & 3;
    uint32_t* queue = s_queue + (size_t)warp * kGQueue * 32 + lane;
    const uint32_t queue0 = smem_u32(queue);
    const uint32_t src = taddr + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(group * kGN);
    uint32_t tbase = 0;
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      const uint32_t buf = it & 1u;
      ok = __all_sync(kFull, pd_wait(smem_u32(&s_mfull[buf]), (it >> 1) & 1u, &s_fail));
      if (!ok) break;
      const ItemInfo x = s_info[buf];
      if (x.c < 0) break;
      const ColMeta& M = s_col[buf];
      // a row past the bucket's end: a huge score, and never past the exact test
      auto factors_of = [&](int t) {
        const int r = (x.t0 + t) * kGM + quarter * 32 + lane;
        return t < x.nt && r < x.rows ? __ldg(P.factors + x.beg + r)
                                      : make_float4(3e38f, 0.0f, 0.0f, 0.0f);
      };
      float4 fnext = factors_of((int)((tbase & 1u) == (uint32_t)group ? 0 : 1));
      for (int t = 0; t < x.nt; ++t) {
        const uint32_t tc = tbase + (uint32_t)t;
        if ((int)(tc & 1u) != group) continue;
        const int r = (x.t0 + t) * kGM + quarter * 32 + lane;
        const bool live = r < x.rows;
        const int pos = x.beg + r;
        const float4 f = fnext;
        fnext = factors_of(t + 2);
        const uint64_t F1 = pack2(f.x - kGSlack * fabsf(f.x), f.x - kGSlack * fabsf(f.x));
        const uint64_t NF2 = pack2(-f.y, -f.y), F3 = pack2(f.z, f.z), G2 = pack2(f.w, f.w);
        uint32_t qp = queue0;  // next queue slot of this lane
        auto flush = [&]() {
          asm volatile("" ::: "memory");  // (the queue's stores are opaque)
          const int n = (int)((qp - queue0) >> 7);
          for (int i0 = 0; __any_sync(kFull, i0 < n); i0 += 4) {
            float lb[4], est[4], ub[4];
            int qq[4], slot[4];
            int2 lr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              qq[u] = -1;
              lr[u] = make_int2(0, P.cap);
              lb[u] = est[u] = ub[u] = 0.0f;
              if (i0 + u < n) {
                const uint32_t e = queue[(i0 + u) * 32];
                const int col = (int)(e & 127u);
                const float acc = __uint_as_float(e & ~127u);  // 2 <x_b, q_u>
                const float4 m = M.ex[col];
                const float2 pt = M.pt[col];
                // estimator (§3.3.2 + Theorem 3.2) and its bound, fixed FP32 order
                const float t1 = __fsub_rn(acc, pt.x);
                const float xq = __fadd_rn(__fmul_rn(m.x, t1), __fmul_rn(m.y, f.w));
                const float dist = __fsub_rn(__fadd_rn(f.x, m.w), __fmul_rn(f.y, xq));
                const float er = __fmul_rn(f.z, m.z);
                const float bound = MODE == 1 ? __fadd_rn(dist, er) : __fsub_rn(dist, er);
                if (live && col < x.cols && bound <= pt.y) {
                  qq[u] = M.q[col];
                  lb[u] = bound;
                  est[u] = dist;
                  if (MODE == 2) {
                    ub[u] = __fadd_rn(dist, er);
                    lr[u] = M.lr[col];
                  }
                }
              }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) slot[u] = qq[u] >= 0 ? atomicAdd(P.cnt + qq[u], 1) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              if (qq[u] >= 0 && slot[u] < lr[u].y) {
                if (MODE == 1)
                  P.ulist[(int64_t)qq[u] * P.cap + slot[u]] = float_key(lb[u]);
                else
                  P.list[lr[u].x + slot[u]] = make_int4(pos, __float_as_int(lb[u]),
                                                        __float_as_int(est[u]),
                                                        __float_as_int(ub[u]));
              }
            }
          }
          qp = queue0;
        };
        ok = __all_sync(kFull, pd_wait(smem_u32(&s_tfull[group]), (tc >> 1) & 1u, &s_fail));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int c0 = 0; c0 < x.cols; c0 += 16) {
          uint32_t v[16];
          __syncwarp();
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,"
              "%13,%14,%15}, [%16];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
                "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(src + (uint32_t)c0));
          asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const ulonglong2* pre = M.pre[(c0 >> 1) + i];
            const ulonglong2 k0 = pre[0], k1 = pre[1];
            const uint64_t k2 = pre[2].x;
            uint64_t w2 = fma2(pack2u(v[2 * i], v[2 * i + 1]), k0.x, k0.y);
            w2 = fma2(k1.x, G2, w2);
            w2 = fma2(NF2, w2, F1);
            w2 = fma2(F3, k1.y, w2);
            float wa, wb, ta, tb;
            unpack2(w2, wa, wb);
            unpack2(k2, ta, tb);
            queue_unless_above(qp, wa, ta, v[2 * i] | (uint32_t)(c0 + 2 * i));
            queue_unless_above(qp, wb, tb, v[2 * i + 1] | (uint32_t)(c0 + 2 * i + 1));
          }
          if (__any_sync(kFull, qp - queue0 > kGQueueFlush * 128u)) flush();
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        mbar_arrive(&s_tempty[group]);
        flush();
      }
      if (!ok) break;
      tbase += (uint32_t)x.nt;
      mbar_arrive(&s_mempty[buf]);
    }
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && s_fail) atomicExch(P.err, kErrScanWait);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(2 * kGN));
}

// ------------------------------------------------------- bounds of exact scores
// The re-rank needs the exact score of few of its rows: tau1 is decided by
// the k smallest pilot scores, and of the other survivors only those that can
// beat tau1 matter. Every row also has an 8-bit copy x~ = o + s c (c the
// bytes, o and s per row), with ||x~||^2 and rho >= ||x - x~||, in one record
// of row_stride(d) bytes (a quarter of the row); a query is rounded to 16
// bits, q~ = t (256 h + l). From <q~, x~> (integer dot products of the bytes)
// come rigorous bounds lo <= score <= hi of the canonical FP32 score:
//   squared distance: |  ||q - x|| - ||q~ - x~||  | <= rho + rho_q
//   inner product:    | <q,x> - <q~,x~> | <= rho_q ||x~|| + ||q|| rho
// widened by the rounding of the FP32 steps that form them ((d + 16) 2^-23 of
// ||q~||^2 + ||x~||^2 for the norms, (d / 32 + 40) 2^-23 of ||q~|| sqrt(d)
// (|o| + 255 s) for the product, whose terms that bounds; 1e-33 for what
// underflows), of rho (2^-22 sqrt(d) (|o| + 255 s)) and of the canonical fold
// ((d + 8) 2^-23, relative for the distance). Where a norm overflows there is
// no bound. A row is scored exactly unless its lo is above the k-th smallest
// hi (pilot) or tau1 (the rest).
__host__ __device__ inline int64_t row_stride(int d) {
  return (16 + (int64_t)(d + 15) / 16 * 16 + 31) / 32 * 32;
}

// One warp per row (bucket order).
__global__ void __launch_bounds__(256) pack_rows_kernel(const float* __restrict__ x, int64_t n, int d,
                                                        int64_t stride, uint8_t* __restrict__ out) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  const float* v = x + r * d;
  float mn = __int_as_float(0x7f800000), mx = __int_as_float(0xff800000);
  for (int i = lane; i < d; i += 32) {
    const float t = __ldg(v + i);
    mn = fminf(mn, t);
    mx = fmaxf(mx, t);
  }
  mn = warp_min_f(mn);
  mx = warp_max_f(mx);
  const float step = (mx - mn) / 255.0f;
  const float inv = step > 0.0f ? 1.0f / step : 0.0f;
  uint8_t* rec = out + r * stride;
  float ee = 0.0f, tt = 0.0f;
  const int dc = (d + 15) / 16 * 16;
  for (int i = lane; i < dc; i += 32) {
    int c = 0;
    if (i < d) {
      const float t = __ldg(v + i);
      c = min(255, max(0, __float2int_rn((t - mn) * inv)));
      const float a = fmaf(step, (float)c, mn), e = t - a;
      ee = fmaf(e, e, ee);
      tt = fmaf(a, a, tt);
    }
    rec[16 + i] = (uint8_t)c;
  }
  ee = warp_sum_f(ee);
  tt = warp_sum_f(tt);
  if (lane == 0) {
    const float rho = sqrtf(ee) * (1.0f + (float)(d + 8) * 0x1.0p-23f) +
                      0x1.0p-22f * sqrtf((float)d) * (fabsf(mn) + 255.0f * step) + 1e-20f;
    *reinterpret_cast<float4*>(rec) = make_float4(mn, step, tt, rho);
  }
}

// A query's 16-bit form: consts {t, sum(q~), ||q~||^2, rho_q}, then the high
// bytes (signed) and the low bytes. One warp per query.
__host__ __device__ inline int64_t query_stride(int d) { return 16 + 2 * ((int64_t)(d + 15) / 16 * 16); }

__global__ void __launch_bounds__(256) pack_queries_kernel(const float* __restrict__ Q, int64_t nq,
                                                           int d, uint8_t* __restrict__ out) {
  const int64_t q = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (q >= nq) return;
  const float* v = Q + q * d;
  float mx = 0.0f;
  for (int i = lane; i < d; i += 32) mx = fmaxf(mx, fabsf(__ldg(v + i)));
  mx = warp_max_f(mx);
  const float t = mx / 32767.0f, inv = t > 0.0f ? 1.0f / t : 0.0f;
  const int dc = (d + 15) / 16 * 16;
  uint8_t* rec = out + q * query_stride(d);
  float sq = 0.0f, s2 = 0.0f, ee = 0.0f;
  for (int i = lane; i < dc; i += 32) {
    int a = 0;
    if (i < d) {
      const float x = __ldg(v + i);
      a = min(32767, max(-32767, __float2int_rn(x * inv)));
      const float y = t * (float)a, e = x - y;
      sq += y;
      s2 = fmaf(y, y, s2);
      ee = fmaf(e, e, ee);
    }
    rec[16 + i] = (uint8_t)(a >> 8);
    rec[16 + dc + i] = (uint8_t)(a & 255);
  }
  sq = warp_sum_f(sq);
  s2 = warp_sum_f(s2);
  ee = warp_sum_f(ee);
  if (lane == 0) {
    const float rho = sqrtf(ee) * (1.0f + (float)(d + 8) * 0x1.0p-23f) + 0x1.0p-21f * sqrtf(s2) +
                      1e-20f;
    *reinterpret_cast<float4*>(rec) = make_float4(t, sq, s2, rho);
  }
}

__device__ __forceinline__ int dp4a_su(uint32_t a, uint32_t b, int c) {
  int r;
  asm("dp4a.s32.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

struct QueryBounds {  // per-query constants of row_bounds
  float t, sum, q2, rho, qn, cd, fold, pf;
  int dc4;            // 16-byte chunks of a record
};

// lo and hi of one row's canonical score by a group of G lanes (a power of
// two; lane g of the group), each with up to four 16-byte pieces of the
// record in flight; every lane of the warp calls it. qh: the query's high
// then low bytes in shared memory.
template <bool IP>
__device__ __forceinline__ void row_bounds(const uint8_t* __restrict__ rec, const uint4* qh,
                                           const QueryBounds& B, int G, int g, float& lo,
                                           float& hi) {
  const uint4* r4 = reinterpret_cast<const uint4*>(rec);
  const uint4 m4 = __ldg(r4);
  const uint4* ql = qh + B.dc4;
  int sh = 0;
  uint32_t sl = 0u;
  for (int c0 = g; c0 < B.dc4; c0 += 4 * G) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = c0 + u * G < B.dc4 ? __ldg(r4 + 1 + c0 + u * G) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = min(c0 + u * G, B.dc4 - 1);
      const uint4 h = qh[c], l = ql[c];
      sh = dp4a_su(h.x, v[u].x, sh);
      sh = dp4a_su(h.y, v[u].y, sh);
      sh = dp4a_su(h.z, v[u].z, sh);
      sh = dp4a_su(h.w, v[u].w, sh);
      sl = __dp4a(l.x, v[u].x, sl);
      sl = __dp4a(l.y, v[u].y, sl);
      sl = __dp4a(l.z, v[u].z, sl);
      sl = __dp4a(l.w, v[u].w, sl);
    }
  }
  __syncwarp();
  for (int o = G >> 1; o > 0; o >>= 1) {
    sh += __shfl_xor_sync(kFull, sh, o);
    sl += __shfl_xor_sync(kFull, sl, o);
  }
  const float o = __uint_as_float(m4.x), s = __uint_as_float(m4.y), x2 = __uint_as_float(m4.z),
              rho = __uint_as_float(m4.w);
  const float dot = fmaf(256.0f, (float)sh, (float)sl);
  const float p = fmaf(s * B.t, dot, o * B.sum);
  const float pe = B.pf * B.qn * fmaf(255.0f, s, fabsf(o));
  if (IP) {
    const float xn = sqrtf(x2) * 1.001f + 1e-20f;
    const float e = B.rho * xn + (B.qn + B.rho) * rho + pe +
                    B.fold * (B.qn + B.rho) * (xn + rho) + 1e-33f;
    const bool ok = e < 1e30f;
    lo = ok ? -p - e : __int_as_float(0xff800000);
    hi = ok ? -p + e : __int_as_float(0x7f800000);
  } else {
    const float d2 = (B.q2 + x2) - 2.0f * p;
    const float e = B.cd * (B.q2 + x2) + 2.0f * pe + 1e-33f;
    const float rr = rho + B.rho;
    const bool ok = e + rr < 1e30f;
    const float a = fmaxf(sqrtf(fmaxf(d2 - e, 0.0f)) * (1.0f - 0x1.0p-20f) - rr, 0.0f);
    const float b = sqrtf(fmaxf(d2 + e, 0.0f)) * (1.0f + 0x1.0p-20f) + rr;
    lo = ok ? a * a * (1.0f - B.fold) : 0.0f;
    hi = ok ? b * b * (1.0f + B.fold) : __int_as_float(0x7f800000);
  }
}

// ------------------------------------------------------------------ the tail
constexpr int kTailSurv = 1536;  // survivors gathered before they are bounded
constexpr int kTailKeys = 4096;  // estimate keys kept in shared memory

struct TailParams {
  FusedParams P;
  int4* list;            // {position, LB, estimate, UB}
  const int* lcnt;
  const int2* lrow;      // a query's first entry and capacity
  const int* ucnt;
  int capu;
  const float* taub;
  int* next;             // query counter
  const uint8_t* qrec;   // packed queries (null: every row is scored exactly)
  const uint8_t* rows;   // 8-bit rows
  int64_t rstride;
  int sk;                // estimate keys in shared memory
};

// Per query: its candidates (every code with LB <= tau_ub) -> pilot, tau1,
// survivors, top-k by the rule of finish_query. CTAs take queries from a
// counter. A query whose candidate list overflowed goes to the redo list;
// one whose upper-bound list did has a tau above tau_ub, and its tau_ub is
// the k-th smallest upper bound of its candidates.
template <bool IP>
__global__ void __launch_bounds__(kThreads, 4) bucket_tail_kernel(TailParams T) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ SelState s_sel;
  __shared__ int s_scratch[kCompactU * kThreads / 32];
  __shared__ int s_q, s_cnt, s_pilot, s_top, s_surv, s_ex;
  __shared__ unsigned long long s_T1;
  const FusedParams& P = T.P;
  const int tid = threadIdx.x;
  const int k = P.k, m = P.m, d = P.d;
  const int dc4 = (d + 15) / 16;
  // lanes per 8-bit row: at most four pieces each, up to 16
  int G = 1;
  while (G < 16 && 4 * G < dc4) G *= 2;
  const int g = tid & (G - 1);
  unsigned long long* topk = reinterpret_cast<unsigned long long*>(smem);   // ct
  uint32_t* estk = reinterpret_cast<uint32_t*>(topk + P.ct);                // sk
  uint32_t* pil = estk + T.sk;                                              // ce: pilot positions
  uint32_t* plo = pil + P.ce;                                               // ce: lo bounds
  uint32_t* phi = plo + P.ce;                                               // ce: keys of hi
  uint32_t* surv = phi + P.ce;                                              // kTailSurv + kThreads
  uint32_t* exl = surv + kTailSurv + kThreads;                              // kTailSurv + kThreads
  float* qv = reinterpret_cast<float*>(exl + kTailSurv + kThreads);         // d
  uint4* qh = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(qv) + align_up(sizeof(float) * d, 16));
  int* hist = reinterpret_cast<int*>(topk);                                 // while topk is free
  uint32_t* coll = reinterpret_cast<uint32_t*>(topk) + kHistBins;
  const int coll_cap = 2 * P.ct - kHistBins;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      s_q = atomicAdd(T.next, 1);
      s_pilot = s_top = s_surv = s_ex = 0;
    }
    __syncthreads();
    const int64_t q = s_q;
    if (q >= P.nq) break;
    int n = T.lcnt[q];
    const int2 lr = T.lrow[q];
    if (n > lr.y) {
      if (tid == 0) P.redo[atomicAdd(P.redo_cnt, 1)] = (int32_t)q;
      continue;
    }
    int4* L = T.list + lr.x;
    for (int i = tid; i < d; i += kThreads) qv[i] = P.queries[q * d + i];
    QueryBounds B;
    if (T.qrec) {
      const uint4* rec = reinterpret_cast<const uint4*>(T.qrec + q * query_stride(d));
      const uint4 c = __ldg(rec);
      B.t = __uint_as_float(c.x);
      B.sum = __uint_as_float(c.y);
      B.q2 = __uint_as_float(c.z);
      B.rho = __uint_as_float(c.w);
      B.qn = sqrtf(B.q2) * 1.001f;
      B.cd = (float)(d + 16) * 0x1.0p-23f;
      B.fold = (float)(d + 8) * 0x1.0p-23f;
      B.pf = (float)(d / 32 + 40) * 0x1.0p-23f * sqrtf((float)d);
      B.dc4 = dc4;
      for (int i = tid; i < 2 * dc4; i += kThreads) qh[i] = __ldg(rec + 1 + i);
    }
    float tau_ub = T.taub[q];
    if (T.ucnt[q] > T.capu && n >= k) {
      int rem, eq;
      tau_ub = key_float(hist_select(n, k, s_sel, hist, coll, coll_cap, rem, eq, [L](int i) {
        return float_key(__int_as_float(L[i].w));
      }));
      if (tid == 0) s_cnt = n;
      __syncthreads();  // (compact_cand reads the count first)
      compact_cand(L, &s_cnt, lr.y, s_scratch,
                   [tau_ub](const int4& e) { return __int_as_float(e.y) <= tau_ub; });
      n = s_cnt;
    }
    // pilot: the m smallest (estimate, id)
    const bool staged = n <= T.sk;
    const bool pilot_all = n <= m;
    if (staged)
      for (int i = tid; i < n; i += kThreads) estk[i] = float_key(__int_as_float(L[i].z));
    __syncthreads();
    uint32_t T_e = 0xffffffffu, T_id = 0xffffffffu;
    if (!pilot_all) {
      auto key_of = [&](int i) { return staged ? estk[i] : float_key(__int_as_float(L[i].z)); };
      int ties = 0, eqn = 0;
      T_e = hist_select(n, m, s_sel, hist, coll, coll_cap, ties, eqn, key_of);
      if (eqn > ties)
        T_id = block_select_f<uint32_t>(n, ties, s_sel, [&](int i) {
          return key_of(i) == T_e ? (uint32_t)__ldg(P.perm + L[i].x) : 0xffffffffu;
        });
    }
    for (int b0 = 0; b0 < n; b0 += kThreads) {
      const int i = b0 + tid;
      bool in = false;
      int pos = 0;
      if (i < n) {
        const uint32_t ek = staged ? estk[i] : float_key(__int_as_float(L[i].z));
        in = pilot_all || ek <= T_e;
        if (in) {
          pos = L[i].x;
          if (!pilot_all && ek == T_e) in = (uint32_t)__ldg(P.perm + pos) <= T_id;
        }
      }
      const int slot = warp_reserve(in, &s_pilot);
      if (in) {
        pil[slot] = (uint32_t)pos;
        // marked: not among the survivors (no key of an estimate is all ones)
        if (staged) estk[i] = 0xffffffffu; else L[i].x = pos | (int)0x80000000;
      }
    }
    __syncthreads();
    const int pilot = s_pilot;
    // the pilot rows that can decide tau1
    const bool bounds = T.qrec != nullptr && pilot > k;
    uint32_t ucut = 0xffffffffu;
    if (bounds) {
      for (int b0 = 0; b0 < pilot * G; b0 += kThreads) {
        const int i = (b0 + tid) / G;
        float lo, hi;
        row_bounds<IP>(T.rows + (int64_t)pil[min(i, pilot - 1)] * T.rstride, qh, B, G, g, lo, hi);
        if (i < pilot && g == 0) {
          plo[i] = float_key(lo);
          phi[i] = float_key(hi);
        }
      }
      __syncthreads();
      int rem, eq;
      ucut = hist_select(pilot, k, s_sel, hist, coll, coll_cap, rem, eq,
                         [phi](int i) { return phi[i]; });
    }
    // exact scores of rows idx[0..cnt): keys at most kmax join the top list
    auto score_rows = [&](const uint32_t* idx, int cnt, unsigned long long kmax) {
      const int row_bytes = d * (int)sizeof(float);
      for (int i = tid; i < min(cnt, 2 * kThreads); i += kThreads) {
        const char* x = reinterpret_cast<const char*>(P.data_b + (int64_t)idx[i] * d);
        for (int o = 0; o < row_bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + o));
      }
      for (int r0 = 0; r0 < cnt; r0 += kThreads) {
        const int i = r0 + tid;
        unsigned long long key = ~0ull;
        if (i < cnt) {
          const uint32_t pos = idx[i];
          const uint32_t id = (uint32_t)__ldg(P.perm + pos);
          const float v = row_score<IP>(P.data_b + (int64_t)pos * d, qv, d);
          key = ((unsigned long long)float_key(v) << 32) | id;
        }
        const bool take = i < cnt && key <= kmax;
        const int slot = warp_reserve(take, &s_top);
        if (take) topk[slot] = key;
        __syncthreads();
        const int tc = s_top;
        __syncthreads();
        if (tc > P.ct - kThreads) select_keep_dk(topk, &s_top, k, s_sel);
      }
    };
    if (bounds) {
      for (int b0 = 0; b0 < pilot; b0 += kThreads) {
        const int i = b0 + tid;
        const bool in = i < pilot && plo[i] <= ucut;
        const int slot = warp_reserve(in, &s_ex);
        if (in) exl[slot] = pil[i];
      }
      __syncthreads();
      const int nx = s_ex;
      score_rows(exl, nx, ~0ull);
    } else {
      score_rows(pil, pilot, ~0ull);
    }
    __syncthreads();
    // T1: the k-th smallest of the pilot's keys. Few keys (the usual case)
    // are ranked against each other; the dropped ones do no harm in the list
    // (the end ranks again).
    unsigned long long T1 = ~0ull;
    if (pilot >= k && !pilot_all) {  // (without other candidates T1 is of no use)
      const int nt = s_top;
      if (nt <= kThreads) {
        const unsigned long long mine = tid < nt ? topk[tid] : ~0ull;
        int r = 0;
        for (int j = 0; j < nt; ++j) r += topk[j] < mine ? 1 : 0;
        if (tid < nt && r == k - 1) s_T1 = mine;
        __syncthreads();
        T1 = s_T1;
      } else {
        T1 = select_keep_dk(topk, &s_top, k, s_sel);
      }
    }
    const uint32_t T1d = (uint32_t)(T1 >> 32);
    const float tau1 = (pilot >= k) ? key_float(T1d) : __int_as_float(0x7f800000);
    const float tau = fminf(tau_ub, tau1);
    // the other survivors, LB <= tau: bounded and scored kTailSurv at a time
    auto drain = [&]() {
      __syncthreads();
      const int ns = s_surv;
      if (tid == 0) s_ex = 0;
      __syncthreads();
      if (T.qrec) {
        for (int b0 = 0; b0 < ns * G; b0 += kThreads) {
          const int i = (b0 + tid) / G;
          float lo, hi;
          row_bounds<IP>(T.rows + (int64_t)surv[min(i, ns - 1)] * T.rstride, qh, B, G, g, lo, hi);
          const bool in = i < ns && g == 0 && float_key(lo) <= T1d;
          const int slot = warp_reserve(in, &s_ex);
          if (in) exl[slot] = surv[i];
        }
        __syncthreads();
        const int nx = s_ex;
        score_rows(exl, nx, T1);
      } else {
        score_rows(surv, ns, T1);
      }
      __syncthreads();
      if (tid == 0) s_surv = 0;
      __syncthreads();
    };
    if (!pilot_all) {
      constexpr int U = 4;  // entries per thread in flight
      for (int b0 = 0; b0 < n; b0 += U * kThreads) {
        int2 e[U];
        bool in[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = b0 + u * kThreads + tid;
          e[u] = i < n ? *reinterpret_cast<const int2*>(L + i) : make_int2(-1, 0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = b0 + u * kThreads + tid;
          in[u] = e[u].x >= 0 && __int_as_float(e[u].y) <= tau &&
                  !(staged && estk[i] == 0xffffffffu);
          const int slot = warp_reserve(in[u], &s_surv);
          if (in[u]) surv[slot] = (uint32_t)e[u].x;
        }
        __syncthreads();
        const int sc = s_surv;
        if (sc > kTailSurv - U * kThreads) drain(); else __syncthreads();
      }
      drain();
    }
    __syncthreads();
    const int n_top = s_top;
    int got = n_top;
    if (n_top > kThreads) {
      select_keep_dk(topk, &s_top, k, s_sel);
      got = min(s_top, k);
    }
    if (got <= kThreads) {  // rank each key against all (distinct keys)
      const bool has = tid < got;
      const unsigned long long mine = has ? topk[tid] : 0ull;
      int r = 0;
      if (has)
        for (int j = 0; j < got; ++j) r += topk[j] < mine ? 1 : 0;
      if (has && r < k) {
        P.out_ids[q * k + r] = (int64_t)(mine & 0xffffffffu);
        const float v = key_float((uint32_t)(mine >> 32));
        P.out_dist[q * k + r] = IP ? -v : v;
      }
    }
    for (int j = got + tid; j < k; j += kThreads) {
      P.out_ids[q * k + j] = -1;
      P.out_dist[q * k + j] = IP ? __int_as_float(0xff800000) : __int_as_float(0x7f800000);
    }
  }
}

// Shared memory of the tail for ct top keys, ce pilot rows and sk staged keys.
size_t tail_smem_bytes(int ct, int ce, int sk, int d) {
  return sizeof(unsigned long long) * ct + sizeof(uint32_t) * ((size_t)sk + 3 * ce + 2 * (kTailSurv + kThreads)) +
         align_up(sizeof(float) * d, 16) + 32 * (size_t)((d + 15) / 16);
}

typedef void (*Tau0Fn)(FusedParams, int, ListPool, float*, float*, int*, int*, int2*, int4*);
Tau0Fn pick_tau0(int W, int bq) {
  if (bq == 4) {
    if (W == 2) return bucket_tau0_kernel<2, 4>;
    if (W == 4) return bucket_tau0_kernel<4, 4>;
    if (W == 16) return bucket_tau0_kernel<16, 4>;
  }
  return bucket_tau0_kernel<0, 0>;
}

// Codes the first threshold looks at, the capacity of the upper-bound lists and
// the even share of the candidate lists' pool.
int tau0_codes(int k) { return std::min(4096, std::max(512, 10 * k)) + 15 & ~15; }
int cap_upper(int k) { return k <= 32 ? 4096 : 8192; }
int list_share(const SearchArgs& a) {
  const int64_t codes = std::min<int64_t>(
      a.X->n, (int64_t)std::min(a.nprobe, a.X->K) * std::max(a.X->max_bucket, 1));
  return (int)std::min<int64_t>(a.k <= 32 ? 8192 : 32768, codes);
}

int pairs_per_item(int dpad) {
  return std::max(kGPad, std::min(kGN, 32768 / dpad / kGPad * kGPad));
}

struct BucketScratch {
  int32_t *bcnt, *bfill, *boff;
  int4* items;
  // [0] items, [16] the levels' sums (64-bit), [32] [64] work counters of the
  // passes, [96] tail counter, [120] pool entries taken, [124] runs
  int* ctl;
  uint8_t* qop;
  float4* smeta;
  float* spsum;
  int32_t* sq;
  float *tau0, *taub;
  int *ucnt, *lcnt;
  int2* lrow;
  uint32_t* ulist;
  int4* list;
  int2* runs;  // {query, first probe}
  int* redo;  // [0] count, [32] the redo launch's work counter, list from [64]
  uint8_t* qrec;
  size_t bytes;
};

BucketScratch bucket_carve(const SearchArgs& a, int64_t nq, unsigned char* base) {
  const rabitq_index* X = a.X;
  const int64_t np = nq * std::min(a.nprobe, X->K);
  const int64_t slots = np + (int64_t)kGPad * std::min<int64_t>(X->K, np);
  const int nt = pairs_per_item(X->dpad);
  const int64_t runs = ((X->max_bucket + kGM - 1) / kGM + kGTilesPerItem - 1) / kGTilesPerItem;
  const int64_t items = (np / nt + std::min<int64_t>(X->K, np)) * std::max<int64_t>(runs, 1);
  BucketScratch b;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base + o;
    o = align_up(o + bytes, 256);
    return p;
  };
  // (the counters that each batch clears lie together)
  b.bcnt = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * (2 * X->K + 192 + nq)));
  b.bfill = b.bcnt + X->K;
  b.ctl = b.bfill + X->K;
  b.redo = b.ctl + 128;
  b.boff = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * (X->K + 1)));
  b.items = reinterpret_cast<int4*>(take(sizeof(int4) * items));
  b.qop = take((size_t)slots * X->dpad);
  b.smeta = reinterpret_cast<float4*>(take(sizeof(float4) * slots));
  b.spsum = reinterpret_cast<float*>(take(sizeof(float) * slots));
  b.sq = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * slots));
  b.tau0 = reinterpret_cast<float*>(take(sizeof(float) * nq));
  b.taub = reinterpret_cast<float*>(take(sizeof(float) * nq));
  b.ucnt = reinterpret_cast<int*>(take(sizeof(int) * nq));
  b.lcnt = reinterpret_cast<int*>(take(sizeof(int) * nq));
  b.lrow = reinterpret_cast<int2*>(take(sizeof(int2) * nq));
  const bool counts = a.pred || a.per_query_nprobe;
  b.runs = reinterpret_cast<int2*>(
      take(counts ? sizeof(int2) * nq * ((std::min(a.nprobe, X->K) + kQJ - 1) / kQJ) : 0));
  b.ulist = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * nq * cap_upper(a.k)));
  b.list = reinterpret_cast<int4*>(take(sizeof(int4) * nq * list_share(a)));
  b.qrec = take((size_t)nq * query_stride(X->d));
  b.bytes = o;
  return b;
}

// Most queries scanned together: bounds the lists and the operand rows to
// about 6 and 2 GiB.
int64_t bucket_batch(const SearchArgs& a) {
  const int64_t lists = (int64_t)list_share(a) * 16 + (int64_t)cap_upper(a.k) * 4;
  const int64_t rows = (int64_t)std::min(a.nprobe, a.X->K) * (a.X->dpad + 32);
  return std::max<int64_t>(1, std::min((int64_t(6) << 30) / lists, (int64_t(2) << 30) / rows));
}

inline unsigned blocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// The 8-bit copy of the rows (once everything else of the index is made).
// Without memory for it the re-rank scores every row exactly; so that it never
// costs a search or another index theirs, it is made only where a sixteenth of
// the device's memory (18 GB) stays free beside it.
int pack_rows(rabitq_index* X, cudaStream_t s) {
  const int64_t stride = row_stride(X->d);
  size_t room = 0, total = 0;
  RBQ_CUDA(cudaMemGetInfo(&room, &total));
  if ((size_t)(X->n * stride) + total / 16 > room) return RABITQ_OK;
  if (cudaMalloc(reinterpret_cast<void**>(&X->rows8), (size_t)(X->n * stride)) != cudaSuccess) {
    cudaGetLastError();
    X->rows8 = nullptr;
    return RABITQ_OK;
  }
  pack_rows_kernel<<<blocks(X->n * 32, 256), 256, 0, s>>>(X->data_b, X->n, X->d, stride, X->rows8);
  RBQ_CUDA(cudaGetLastError());
  return RABITQ_OK;
}

bool bucket_applies(const SearchArgs& a, int64_t nq) {
  if (!a.allow_bucket || a.trace || a.bq > 4 || a.k > 256 || a.cand_cap < 65536) return false;
  if (a.layout != RABITQ_LAYOUT_AUTO || a.bulk_asked || a.bucket_tuned == 2) return false;
  // Measured against the per-query scan on eight indexes (100k x 96 to 2M x 256,
  // D' 128 to 1024, L2 and inner products), k 1 to 256, 320 to 10k queries, 4 to
  // 128 probes. Below about four pairs per bucket the tiles are mostly padding.
  // Beyond that, what the scan saves has to pay for the further launches and for
  // the tail (its first threshold, pilot and top-k cost more the larger k is):
  // the batch's codes, counted in 128-bit units, for k + 128 times 36000, and
  // four times that for inner products, where the per-query scan prunes better.
  // Of the 500 points with 1000 queries and more, this rule leaves 12 with over
  // 3% and at most 10% against the per-query scan (four pairs alone: 80, up to
  // 59%: 1000 queries x 4 probes, 100k x 96, k = 100: 0.174 ms per query, 0.262
  // so). The limit of a thousand queries is older than the one on the codes: below
  // it 121 of 260 points are slower (the tail's last wave is mostly idle), but of
  // the 93 that the latter admits only 3 (at most 16%), so it could come down.
  const double pairs = (double)nq * a.mean_probes;
  if (nq < 1000 || pairs < 4.0 * a.X->K) return false;
  const double work = pairs * a.X->n / a.X->K * a.X->dpad / 128.0;
  return work >= 36000.0 * (a.k + 128) * (a.X->metric != RABITQ_METRIC_L2 ? 4.0 : 1.0);
}

void expect_probes(SearchArgs& a) {
  const float most = (float)std::min(a.nprobe, a.X->K);
  a.mean_probes = a.pred ? std::min(most, a.pred->mean_nprobe()) : most;
}

size_t bucket_bytes(const SearchArgs& a, int64_t nq) {
  return bucket_carve(a, std::min(nq, bucket_batch(a)), nullptr).bytes;
}

// Scan, prune and re-rank of P.nq queries whose probe lists and rotations are
// in P. fn / grid / smem: the per-query kernel for the queries handed back.
int bucket_search(const SearchArgs& a, const FusedParams& P0, unsigned char* scratch,
                  void (*fn)(FusedParams), unsigned grid, size_t fn_smem, cudaStream_t s) {
  const rabitq_index* X = a.X;
  const int64_t nb = std::max<int64_t>(1, (P0.nq + bucket_batch(a) - 1) / bucket_batch(a));
  const int64_t per = (P0.nq + nb - 1) / nb;
  const BucketScratch b = bucket_carve(a, per, scratch);
  const int K = X->K, nt = pairs_per_item(X->dpad), want = tau0_codes(a.k);
  const int capu = cap_upper(a.k), share = list_share(a);
  int dev = 0, sms = 0, optin = 0;
  RBQ_CUDA(cudaGetDevice(&dev));
  RBQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  RBQ_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const Tau0Fn t0 = pick_tau0(X->W, a.bq);
  const size_t t0_smem = sizeof(uint64_t) * kGTau0Probes * a.bq * X->W + sizeof(uint32_t) * want +
                         sizeof(int) * kHistBins + sizeof(uint32_t) * 256 + sizeof(float2) * want;
  RBQ_CUDA(cudaFuncSetAttribute(t0, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
  const size_t scan_smem = bucket_smem_bytes(nt, X->dpad);
  RBQ_CUDA(cudaFuncSetAttribute(bucket_scan_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                160 * 1024));
  RBQ_CUDA(cudaFuncSetAttribute(bucket_scan_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                160 * 1024));
  // the tail
  const bool ip = X->metric != RABITQ_METRIC_L2;
  void (*tail)(TailParams) = ip ? bucket_tail_kernel<true> : bucket_tail_kernel<false>;
  TailParams T;
  T.rows = X->rows8;
  T.rstride = row_stride(X->d);
  T.qrec = X->rows8 ? b.qrec : nullptr;
  int ce = 1;
  while (ce < 4 * a.k) ce *= 2;
  T.sk = a.k <= 32 ? 2048 : kTailKeys;
  const size_t tail_smem = tail_smem_bytes(1024, ce, T.sk, X->d);
  RBQ_CUDA(cudaFuncSetAttribute(tail, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024));
  int tail_per_sm = 1;
  RBQ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&tail_per_sm, tail, kThreads, tail_smem));
  for (int64_t q0 = 0; q0 < P0.nq; q0 += per) {
    FusedParams P = P0;
    P.nq = std::min(per, P0.nq - q0);
    P.queries += q0 * P.d;
    P.rq += q0 * P.dpad;
    P.probe_ids += q0 * P.nprobe;
    P.probe_dist += q0 * P.nprobe;
    if (P.probe_nq2) P.probe_nq2 += q0 * P.nprobe;
    if (P.nprobe_q) P.nprobe_q += q0;
    P.q_offset += q0;
    P.out_ids += q0 * P.k;
    P.out_dist += q0 * P.k;
    P.order = nullptr;
    RBQ_CUDA(cudaMemsetAsync(b.bcnt, 0, sizeof(int32_t) * (2 * K + 192), s));  // counts, ctl, redo
    ListPool lp;
    lp.sum = reinterpret_cast<unsigned long long*>(b.ctl + 16);
    lp.used = reinterpret_cast<unsigned*>(b.ctl + 120);
    lp.size = (unsigned)(per * share);
    lp.share = share;
    bucket_count_kernel<<<blocks(P.nq * 32, 256), 256, 0, s>>>(
        P, share, want, b.bcnt, reinterpret_cast<unsigned long long*>(b.ctl + 16), b.lcnt,
        b.ctl + 124, b.runs);
    bucket_plan_kernel<<<1, 1024, 0, s>>>(b.bcnt, X->bucket_off, K, nt, b.boff, b.items, b.ctl);
    if (P.nprobe_q)
      bucket_quant_kernel<true><<<(unsigned)(4 * sms), 256, 0, s>>>(
          P, b.lcnt, b.ctl + 124, b.runs, b.boff, b.bfill, b.qop, b.smeta, b.spsum, b.sq);
    else
      bucket_quant_kernel<false><<<blocks(P.nq * quant_runs(P.nprobe) * 32, 256), 256, 0, s>>>(
          P, b.lcnt, nullptr, nullptr, b.boff, b.bfill, b.qop, b.smeta, b.spsum, b.sq);
    t0<<<(unsigned)P.nq, kThreads, t0_smem, s>>>(P, want, lp, b.tau0, b.taub, b.ucnt, b.lcnt, b.lrow,
                                                  b.list);
    RBQ_CUDA(cudaGetLastError());
    BucketParams B;
    B.codes = X->codes;
    B.factors = X->factors;
    B.bucket_off = X->bucket_off;
    B.W = X->W;
    B.dpad = X->dpad;
    B.nt = nt;
    B.boff = b.boff;
    B.bcnt = b.bcnt;
    B.items = b.items;
    B.nitems = b.ctl;
    B.qop = b.qop;
    B.smeta = b.smeta;
    B.spsum = b.spsum;
    B.sq = b.sq;
    B.err = P.err;
    B.ulist = b.ulist;
    B.list = b.list;
    B.lrow = b.lrow;
    B.work = b.ctl + 32;
    B.tau = b.tau0;
    B.cnt = b.ucnt;
    B.cap = capu;
    bucket_scan_kernel<1><<<(unsigned)(2 * sms), kGThreads, scan_smem, s>>>(B);
    bucket_tau_kernel<<<(unsigned)P.nq, kThreads, 0, s>>>(b.ulist, b.ucnt, capu, a.k, b.tau0,
                                                               b.taub);
    B.work = b.ctl + 64;
    B.tau = b.taub;
    B.cnt = b.lcnt;
    bucket_scan_kernel<2><<<(unsigned)(2 * sms), kGThreads, scan_smem, s>>>(B);
    RBQ_CUDA(cudaGetLastError());
    if (T.qrec)
      pack_queries_kernel<<<blocks(P.nq * 32, 256), 256, 0, s>>>(P.queries, P.nq, P.d, b.qrec);
    T.P = P;
    T.P.m = 4 * a.k;
    T.P.ce = ce;
    T.P.ct = 1024;
    T.P.redo = b.redo + 64;
    T.P.redo_cnt = b.redo;
    T.list = b.list;
    T.lcnt = b.lcnt;
    T.lrow = b.lrow;
    T.ucnt = b.ucnt;
    T.capu = capu;
    T.taub = b.taub;
    T.next = b.ctl + 96;
    tail<<<(unsigned)std::min<int64_t>(P.nq, (int64_t)sms * std::max(tail_per_sm, 1)), kThreads,
           tail_smem, s>>>(T);
    RBQ_CUDA(cudaGetLastError());
    FusedParams R = P;  // the queries handed back
    R.order = b.redo + 64;
    R.nq_dev = b.redo;
    R.next = b.redo + 32;
    R.split = 1;
    fn<<<grid, kThreads, fn_smem, s>>>(R);
    RBQ_CUDA(cudaGetLastError());
  }
  return RABITQ_OK;
}

}  // namespace rbq
