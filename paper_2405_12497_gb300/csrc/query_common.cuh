// query_common.cuh -- device parts shared by the query-phase kernels
// (kernels_search.cu, kernels_bucket.cu): the randomized query quantization,
// block-wide selections, candidate-list compaction, exact re-rank and the
// per-query end of a search.
#pragma once

#include <stddef.h>

#include "common.cuh"
#include "internal.h"

namespace rbq {

// Arguments of the per-query kernels (host-built, passed by value).
struct FusedParams {
  const float* queries;     // nq x d
  const float* rq;          // nq x dpad
  const int32_t* probe_ids; // nq x nprobe
  const float* probe_dist;  // nq x nprobe: centroid scores, the estimator's additive term
  const float* probe_nq2;   // nq x nprobe ||q_r - c||^2 (IP metric), null = probe_dist
  const int32_t* nprobe_q;  // nq or null
  const float* ptc;         // K x dpad
  const uint64_t* codes;    // n x W (bucket order)
  const float4* factors;    // n (bucket order)
  const float* data_b;      // n x d (bucket order)
  const int32_t* perm;      // n: position -> id
  const int32_t* inv_perm;  // n: id -> position
  const int32_t* bucket_off;
  int64_t nq, q_offset;
  int d, dpad, W, bq, k, m, nprobe, pch, cu, ce, ct;
  float eps0;
  uint64_t seed;
  int cand_cap;
  int metric;               // 0: squared distance; 1: inner product (score -<o_r, q_r>)
  int4* cand;               // gridDim.x x cand_cap: {pos, LB, estimate, -}
  int64_t* out_ids;
  float* out_dist;
  int* err;
  rabitq_trace tr;
  // query scheduling: CTAs take the next query from *next (zeroed before the
  // launch) in the order `order` (null = ascending); next == null = static
  // striding by gridDim.x
  const int32_t* order;
  int* next;
  int scap;  // shared-memory capacity for the tail's candidate list (0 = none)
  // Split mode (split > 1, for batches too small to fill the GPU): work item
  // i scans probe slice i % split of query i / split into candidate region i
  // and writes the slice's k smallest upper-bound keys to ub_out[i k ...] and
  // {keys written, candidates} to slice_cnt[2 i ...]; split_merge_kernel
  // then finishes each query from its slices. cand2: one merged-list region
  // of cand_cap entries per query.
  int split;
  uint32_t* ub_out;
  int* slice_cnt;
  int4* cand2;
  // Warp-per-query kernel: candidate region of capw entries per warp; a
  // query whose list outgrows it goes to redo[*redo_cnt++]. The CTA kernel
  // redoing them reads its query count from *nq_dev when that is set.
  int4* candw;
  int capw;
  int32_t* redo;
  int* redo_cnt;
  const int* nq_dev;
};

namespace {

constexpr int kThreads = 256;

// ------------------------------------------------------ fused query kernel
// Shared state of the block radix select.
struct SelState {
  int hist[256];
  int bin, rem, tie_taken;
  int warp_cnt[kThreads / 32];
  unsigned long long wmin[kThreads / 32], wmax[kThreads / 32];
};

struct FusedSmem {
  uint64_t* planes;  // pch x bq x W
  float4* pmeta;     // pch: A, B, E, nq2
  int* psum;         // pch
  int* pbeg;         // pch
  int* pref;         // pch + 1
  float* qv;         // d
  SelState* sel;     // radix-select scratch
  uint32_t* ubk;     // cu: upper-bound keys
  unsigned long long* estk;  // ce: the pilot list, (id << 32) | position
  unsigned long long* topk;  // ct: (exact distance key << 32) | id
  int4* scand;               // scap: the candidate list staged for the tail
};

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__host__ __device__ inline size_t fused_smem_bytes(int pch, int bq, int W, int d, int cu, int ce,
                                                   int ct, int nwarps,
                                                   size_t* off /* 10 entries or null */,
                                                   int scap = 0) {
  size_t o = 0, offs[10];
  (void)nwarps;
  offs[0] = o; o = align_up(o + sizeof(uint64_t) * pch * bq * W, 16);
  offs[1] = o; o = align_up(o + sizeof(float4) * pch, 16);
  offs[2] = o; o = align_up(o + sizeof(int) * pch, 16);
  offs[3] = o; o = align_up(o + sizeof(int) * pch, 16);
  offs[4] = o; o = align_up(o + sizeof(int) * (pch + 1), 16);
  offs[5] = o; o = align_up(o + sizeof(float) * d, 16);
  offs[6] = o; o = align_up(o + sizeof(uint32_t) * cu, 16);
  offs[7] = o; o = align_up(o + sizeof(unsigned long long) * ce, 16);
  offs[8] = o; o = align_up(o + sizeof(unsigned long long) * ct, 16);
  offs[9] = o; o = align_up(o + sizeof(int4) * scap, 16);
  if (off)
    for (int i = 0; i < 10; ++i) off[i] = offs[i];
  return o;
}

// Randomized B_q-bit quantization of q' for one probed cluster with one warp
// (§3.3.1): qd = rq - P^T c, v_l = min qd, v_r = max qd, Delta = (v_r -
// v_l)/(2^B_q - 1), q_u[k] = min(floor((qd[k] - v_l)/Delta + u_k), 2^B_q - 1)
// with u_k from Philox(seed; k/4, query, cluster, 3). Lane l holds elements
// k = 128 i + 4 l + r (r = 0..3), so the four u_k of one Philox call belong to
// one lane; emit(i, k0, qu) receives them block by block (warp-uniform).
// Returns sum(q_u) in every lane; writes v_l and Delta.
template <class Emit>
__device__ __forceinline__ int quant_core(const float* rq, const float* pc, int dpad, int bq,
                                          uint64_t seed, uint64_t gq, int c, float* vl_out,
                                          float* delta_out, Emit emit) {
  const int lane = threadIdx.x & 31;
  const int nblk = (dpad + 127) >> 7;
  float vl = __int_as_float(0x7f800000), vr = __int_as_float(0xff800000);
  for (int kk = lane; kk < dpad; kk += 32) {
    const float v = __fsub_rn(rq[kk], pc[kk]);
    vl = fminf(vl, v);
    vr = fmaxf(vr, v);
  }
  vl = warp_min_f(vl);
  vr = warp_max_f(vr);
  const int qmax = (1 << bq) - 1;
  const float delta = __fdiv_rn(__fsub_rn(vr, vl), (float)qmax);
  int sum = 0;
  for (int i = 0; i < nblk; ++i) {
    const int k0 = 128 * i + 4 * lane;
    int qu[4] = {0, 0, 0, 0};
    if (delta > 0.0f && k0 < dpad) {
      float qd[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) qd[r] = (k0 + r < dpad) ? __fsub_rn(rq[k0 + r], pc[k0 + r]) : 0.0f;
      const U4 w = philox4x32_10(seed, (uint32_t)(k0 >> 2), (uint32_t)gq, (uint32_t)c, kTagQuant);
      const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (k0 + r < dpad) {
          const float u = __fmul_rn(__uint2float_rn(ws[r] >> 8), 0x1.0p-24f);
          const float x = __fdiv_rn(__fsub_rn(qd[r], vl), delta);
          const int v = __float2int_rd(__fadd_rn(x, u));
          qu[r] = v > qmax ? qmax : v;
        }
      }
    }
    sum += qu[0] + qu[1] + qu[2] + qu[3];
    emit(i, k0, qu);
  }
  *vl_out = vl;
  *delta_out = delta;
  return warp_sum_i(sum);
}

// Per-(query, cluster) constants of the estimator: A = Delta/sqrt(D'),
// B = v_l/sqrt(D'), E = ||q_r - c|| 2 eps0/sqrt(D'-1) and the additive term
// add: ||q_r - c||^2 for distances, -<q_r, c> for inner products (§6).
__device__ __forceinline__ float4 quant_meta(float delta, float vl, float nq2, float add,
                                             float eps0, int dpad) {
  const float sqd = __fsqrt_rn((float)dpad);
  const float keps = __fdiv_rn(__fmul_rn(2.0f, eps0), __fsqrt_rn((float)(dpad - 1)));
  const float n_q = __fsqrt_rn(nq2);
  return make_float4(__fdiv_rn(delta, sqd), __fdiv_rn(vl, sqd), __fmul_rn(n_q, keps), add);
}

// Quantize for the popcount scan: B_q bit-planes of q_u into shared memory.
__device__ __forceinline__ void quantize_probe(const FusedParams& P, const FusedSmem& S, int64_t q,
                                               int j, int jg, int c, float nq2, float add) {
  const int lane = threadIdx.x & 31;
  const int dpad = P.dpad, W = P.W, bq = P.bq;
  uint64_t* planes = S.planes + (size_t)j * bq * W;
  float vl, delta;
  const int sum = quant_core(
      P.rq + q * dpad, P.ptc + (int64_t)c * dpad, dpad, bq, P.seed, (uint64_t)(P.q_offset + q), c,
      &vl, &delta, [&](int i, int, const int* qu) {
        // the nibble of lane l sits at bits 4l..4l+3 of the 128-bit block
        for (int b = 0; b < bq; ++b) {
          const uint32_t nib = ((qu[0] >> b) & 1) | (((qu[1] >> b) & 1) << 1) |
                               (((qu[2] >> b) & 1) << 2) | (((qu[3] >> b) & 1) << 3);
          const uint32_t part = nib << (4 * (lane & 7));
          const uint32_t q0 = __reduce_or_sync(kFull, lane < 8 ? part : 0u);
          const uint32_t q1 = __reduce_or_sync(kFull, (lane >= 8 && lane < 16) ? part : 0u);
          const uint32_t q2 = __reduce_or_sync(kFull, (lane >= 16 && lane < 24) ? part : 0u);
          const uint32_t q3 = __reduce_or_sync(kFull, lane >= 24 ? part : 0u);
          if (lane == 0) {
            const int w0 = 2 * i;
            if (w0 < W) planes[b * W + w0] = ((uint64_t)q1 << 32) | q0;
            if (w0 + 1 < W) planes[b * W + w0 + 1] = ((uint64_t)q3 << 32) | q2;
          }
        }
      });
  if (lane == 0) {
    const float4 m = quant_meta(delta, vl, nq2, add, P.eps0, dpad);
    S.pmeta[j] = m;
    S.psum[j] = sum;
    S.pbeg[j] = P.bucket_off[c];
    S.pref[j + 1] = P.bucket_off[c + 1] - P.bucket_off[c];  // length; prefix-summed later
    if (P.tr.sum_qu) P.tr.sum_qu[q * P.nprobe + jg] = sum;
    if (P.tr.meta) {
      float* tm = P.tr.meta + (q * P.nprobe + jg) * 4;
      tm[0] = m.x; tm[1] = m.y; tm[2] = m.z; tm[3] = m.w;
    }
  }
  __syncwarp();
  if (P.tr.planes) {
    uint64_t* tp = P.tr.planes + (q * P.nprobe + jg) * (int64_t)bq * W;
    for (int t = lane; t < bq * W; t += 32) tp[t] = planes[t];
  }
}

// Warp-aggregated slot reservation: lanes with `want` get consecutive slots
// from one atomicAdd per warp (shared-memory counters are hot).
__device__ __forceinline__ int warp_reserve(bool want, int* counter) {
  const unsigned m = __ballot_sync(kFull, want);
  if (m == 0) return -1;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(m) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(counter, __popc(m));
  base = __shfl_sync(kFull, base, leader);
  return want ? base + __popc(m & ((1u << lane) - 1u)) : -1;
}


// ---------------------------------------------------------- block select
// The want-th smallest (1-based, want <= n) of the n keys a[0..n) by an
// MSD radix select, 8 bits per pass; histogram updates are aggregated per
// warp by digit. On return st.rem = how many keys equal to the result are
// among the `want` smallest. Whole block; synchronized on return.
template <class K, class F>
__device__ K block_select_f(int n, int want, SelState& st, F keyf) {
  constexpr int NB = (int)sizeof(K) * 8;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // The leading bits where the smallest and the largest key agree are common
  // to every key and need no histogram pass: one min/max pass finds them.
  K kmin = ~(K)0, kmax = 0;
  for (int i = tid; i < n; i += blockDim.x) {
    const K key = keyf(i);
    kmin = key < kmin ? key : kmin;
    kmax = key > kmax ? key : kmax;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const K a = __shfl_xor_sync(kFull, kmin, o), b = __shfl_xor_sync(kFull, kmax, o);
    kmin = a < kmin ? a : kmin;
    kmax = b > kmax ? b : kmax;
  }
  if (lane == 0) {
    st.wmin[wid] = kmin;
    st.wmax[wid] = kmax;
  }
  __syncthreads();
  kmin = ~(K)0;
  kmax = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    kmin = (K)st.wmin[w] < kmin ? (K)st.wmin[w] : kmin;
    kmax = (K)st.wmax[w] > kmax ? (K)st.wmax[w] : kmax;
  }
  if (kmin == kmax) {  // all keys equal: the answer, with every key a tie
    __syncthreads();
    if (tid == 0) {
      st.bin = (int)(kmin & 255);
      st.hist[st.bin] = n;
      st.rem = want;
    }
    __syncthreads();
    return kmin;
  }
  const K diff = kmin ^ kmax;
  const int top = NB - 1 - (sizeof(K) == 8 ? __clzll((long long)diff) : __clz((int)diff));
  const int start = (top / 8) * 8;  // the byte holding the highest differing bit
  K mask = start + 8 >= NB ? (K)0 : ~(((K)1 << (start + 8)) - 1);
  K prefix = kmin & mask;
  int rem = want;
  for (int shift = start; shift >= 0; shift -= 8) {
    for (int i = tid; i < 256; i += blockDim.x) st.hist[i] = 0;
    __syncthreads();
    for (int b0 = 0; b0 < n; b0 += blockDim.x) {
      const int i = b0 + tid;
      K key = 0;
      bool v = false;
      if (i < n) {
        key = keyf(i);
        v = (key & mask) == prefix;
      }
      const int dig = v ? (int)((key >> shift) & 255) : 256 + lane;
      const unsigned grp = __match_any_sync(kFull, dig);
      if (v && lane == __ffs(grp) - 1) atomicAdd(&st.hist[dig], __popc(grp));
    }
    __syncthreads();
    if (tid < 32) {
      int c[8], sum = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        c[u] = st.hist[lane * 8 + u];
        sum += c[u];
      }
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(kFull, incl >= rem);
      if (lane == __ffs(hit) - 1) {
        int cum = incl - sum;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (cum + c[u] >= rem) {
            st.bin = lane * 8 + u;
            st.rem = rem - cum;
            break;
          }
          cum += c[u];
        }
      }
    }
    __syncthreads();
    prefix |= (K)st.bin << shift;
    mask |= (K)255 << shift;
    rem = st.rem;
    __syncthreads();
  }
  return prefix;
}

template <class K>
__device__ K block_select(const K* a, int n, int want, SelState& st) {
  return block_select_f<K>(n, want, st, [a](int i) { return a[i]; });
}

// The want-th smallest (1-based, want <= n) of n 32-bit keys: a histogram of
// at most kHistBins bins of a power-of-two width over [min, max] (bin = (key -
// min) >> shift, monotone in the key; equal-width bins by a 64-bit division
// cost some hundred instructions per key and pass), repeated inside the bin
// that holds the result while that bin has more keys than threads (scores
// whose range spans many powers of two crowd into few bins at first), then
// the bin's keys are collected into coll and ranked. rem = how many keys
// equal to the result are among the want smallest, eq = how many keys equal
// it in all. hist: kHistBins ints; coll: coll_cap keys. Whole block (kThreads
// threads); synchronized on return.
constexpr int kHistBits = 10, kHistBins = 1 << kHistBits;
template <class F>
__device__ uint32_t hist_select(int n, int want, SelState& st, int* hist, uint32_t* coll,
                                int coll_cap, int& rem, int& eq, F keyf) {
  static_assert(kHistBins == 4 * kThreads, "four bins per thread");
  __shared__ int s_hs[5];  // boundary bin, keys below it, fill, rem, eq
  __shared__ uint32_t s_T;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  for (int i = tid; i < n; i += blockDim.x) {
    const uint32_t key = keyf(i);
    kmin = key < kmin ? key : kmin;
    kmax = key > kmax ? key : kmax;
  }
  kmin = __reduce_min_sync(kFull, kmin);
  kmax = __reduce_max_sync(kFull, kmax);
  if (lane == 0) {
    st.wmin[wid] = kmin;
    st.wmax[wid] = kmax;
  }
  for (int i = tid; i < kHistBins; i += blockDim.x) hist[i] = 0;
  if (tid == 0) s_hs[2] = 0;
  __syncthreads();
  kmin = 0xffffffffu;
  kmax = 0u;
  for (int w = 0; w < nw; ++w) {
    kmin = (uint32_t)st.wmin[w] < kmin ? (uint32_t)st.wmin[w] : kmin;
    kmax = (uint32_t)st.wmax[w] > kmax ? (uint32_t)st.wmax[w] : kmax;
  }
  if (kmin == kmax) {  // all keys equal
    rem = want;
    eq = n;
    __syncthreads();
    return kmin;
  }
  uint32_t lo = kmin, span = kmax - kmin;  // the result is in [lo, lo + span]
  int want_b = want, shift, B, nB;
  for (;;) {
    shift = max(0, 32 - __clz((int)span) - kHistBits);
    for (int i = tid; i < n; i += blockDim.x) {
      const uint32_t off = keyf(i) - lo;
      if (off <= span) atomicAdd(&hist[off >> shift], 1);
    }
    __syncthreads();
    // the bin holding the want_b-th key of the range: four bins per thread
    const int4 c4 = reinterpret_cast<const int4*>(hist)[tid];
    const int c[4] = {c4.x, c4.y, c4.z, c4.w};
    const int sum = c4.x + c4.y + c4.z + c4.w;
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) st.warp_cnt[wid] = incl;
    __syncthreads();
    for (int w = 0; w < wid; ++w) incl += st.warp_cnt[w];
    const int excl = incl - sum;
    if (excl < want_b && incl >= want_b) {  // exactly one thread
      int cum = excl;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (cum + c[u] >= want_b) {
          s_hs[0] = 4 * tid + u;
          s_hs[1] = cum;
          s_hs[3] = c[u];
          break;
        }
        cum += c[u];
      }
    }
    __syncthreads();
    B = s_hs[0];
    want_b -= s_hs[1];
    nB = s_hs[3];
    if (shift == 0 || nB <= min(coll_cap, (int)blockDim.x)) break;
    lo += (uint32_t)B << shift;
    span = (1u << shift) - 1u;
    for (int i = tid; i < kHistBins; i += blockDim.x) hist[i] = 0;
    __syncthreads();
  }
  if (shift == 0) {  // the bin is one key value
    rem = want_b;
    eq = nB;
    __syncthreads();
    return lo + (uint32_t)B;
  }
  for (int b0 = 0; b0 < n; b0 += blockDim.x) {
    const int i = b0 + tid;
    uint32_t key = 0u;
    bool in = false;
    if (i < n) {
      key = keyf(i);
      const uint32_t off = key - lo;
      in = off <= span && (int)(off >> shift) == B;
    }
    const int slot = warp_reserve(in, &s_hs[2]);
    if (in) coll[slot] = key;
  }
  __syncthreads();
  if (tid < nB) {  // rank each key of the bin against the others
    const uint32_t mine = coll[tid];
    int lt = 0, le = 0;
    for (int j = 0; j < nB; ++j) {
      const uint32_t v = coll[j];
      lt += v < mine ? 1 : 0;
      le += v <= mine ? 1 : 0;
    }
    if (lt < want_b && want_b <= le) {  // the threads holding the result
      s_T = mine;
      s_hs[3] = want_b - lt;
      s_hs[4] = le - lt;
    }
  }
  __syncthreads();
  const uint32_t T = s_T;
  rem = s_hs[3];
  eq = s_hs[4];
  __syncthreads();
  return T;
}

// In place, keep the keys below T and `ties` of the keys equal to T; returns
// the new count (whole block; synchronized on return).
template <class K>
__device__ int block_keep_below(K* a, int n, K T, int ties, SelState& st) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) st.tie_taken = 0;
  __syncthreads();
  int out = 0;
  for (int b0 = 0; b0 < n; b0 += blockDim.x) {
    const int i = b0 + tid;
    K key = 0;
    bool keep = false;
    if (i < n) {
      key = a[i];
      keep = key < T || (key == T && atomicAdd(&st.tie_taken, 1) < ties);
    }
    const unsigned bal = __ballot_sync(kFull, keep);
    if (lane == 0) st.warp_cnt[wid] = __popc(bal);
    __syncthreads();
    int before = out, tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      if (w < wid) before += st.warp_cnt[w];
      tot += st.warp_cnt[w];
    }
    if (keep) a[before + __popc(bal & ((1u << lane) - 1u))] = key;
    out += tot;
    __syncthreads();
  }
  return out;
}

// Keep the `keep` smallest of the *cnt keys (no order); returns the
// keep-th smallest key (or ~0 if there are fewer than keep keys).
template <class K>
__device__ K select_keep(K* a, int* cnt, int keep, SelState& st) {
  const int n = *cnt;
  if (n < keep) {
    __syncthreads();
    return ~(K)0;
  }
  const K T = block_select<K>(a, n, keep, st);
  const int kept = block_keep_below<K>(a, n, T, st.rem, st);
  if (threadIdx.x == 0) *cnt = kept;
  __syncthreads();
  return T;
}

// select_keep for 32-bit keys by the histogram select (hist, coll: shared
// memory the caller has free at this point).
__device__ uint32_t select_keep_h(uint32_t* a, int* cnt, int keep, SelState& st, int* hist,
                                  uint32_t* coll, int coll_cap) {
  const int n = *cnt;
  if (n < keep) {
    __syncthreads();
    return 0xffffffffu;
  }
  int rem = 0, eq = 0;
  const uint32_t T =
      hist_select(n, keep, st, hist, coll, coll_cap, rem, eq, [a](int i) { return a[i]; });
  const int kept = block_keep_below<uint32_t>(a, n, T, rem, st);
  if (threadIdx.x == 0) *cnt = kept;
  __syncthreads();
  return T;
}

// Keep the `keep` smallest of the *cnt distinct (distance key << 32 | id)
// keys of a: a 32-bit select on the distance half (by the histogram select
// when hist/coll are given, else the radix select), then -- only when more
// keys share the boundary distance than are kept -- one on the id half of
// those. Returns the keep-th smallest key (~0 if there are fewer than keep).
// Whole block; synchronized on return.
__device__ unsigned long long select_keep_dk(unsigned long long* a, int* cnt, int keep,
                                             SelState& st, int* hist = nullptr,
                                             uint32_t* coll = nullptr, int coll_cap = 0) {
  const int n = *cnt;
  if (n < keep) {
    __syncthreads();
    return ~0ull;
  }
  uint32_t Td;
  int ties = 0, eqn = 0;
  if (hist) {
    Td = hist_select(n, keep, st, hist, coll, coll_cap, ties, eqn,
                     [a](int i) { return (uint32_t)(a[i] >> 32); });
  } else {
    Td = block_select_f<uint32_t>(n, keep, st, [a](int i) { return (uint32_t)(a[i] >> 32); });
    ties = st.rem;
    eqn = st.hist[st.bin];
  }
  uint32_t Tid = 0xffffffffu;
  if (eqn > ties)
    Tid = block_select_f<uint32_t>(n, ties, st, [a, Td](int i) {
      return (uint32_t)(a[i] >> 32) == Td ? (uint32_t)(a[i] & 0xffffffffu) : 0xffffffffu;
    });
  unsigned long long T = ((unsigned long long)Td << 32) | Tid;
  if (Tid == 0xffffffffu) {  // every key at the boundary distance is kept
    T = ((unsigned long long)Td << 32) | 0xffffffffu;
  }
  const int kept = block_keep_below<unsigned long long>(a, n, T, 1, st);
  if (threadIdx.x == 0) *cnt = kept;
  __syncthreads();
  if (Tid == 0xffffffffu) {
    // the keep-th smallest key itself: the largest kept key
    __shared__ unsigned long long s_max;
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    unsigned long long mx = 0;
    for (int i = threadIdx.x; i < kept; i += blockDim.x) mx = a[i] > mx ? a[i] : mx;
    atomicMax(&s_max, mx);
    __syncthreads();
    T = s_max;
    __syncthreads();
  }
  return T;
}

// Sort the first pow2(keep) slots of a shared key buffer holding *cnt <=
// keep keys (padded with the maximum key). Whole block; synchronized on return.
__device__ __forceinline__ void sort_kept_u64(unsigned long long* a, int cnt, int keep) {
  int n = 1;
  while (n < keep) n <<= 1;
  for (int i = cnt + threadIdx.x; i < n; i += blockDim.x) a[i] = ~0ull;
  __syncthreads();
  block_bitonic_sort_u64(a, n);
  __syncthreads();
}

// In-place, order-keeping compaction of the candidate list with predicate f:
// blocks of kCompactU x blockDim entries (kCompactU loads in flight per
// thread, two barriers per block); every read of a block precedes its
// writes, which land below the block's end. scratch: kCompactU x
// (blockDim / 32) ints. (Two entries per thread: four cost the fused kernel
// register spills that outweighed the fewer barriers.)
constexpr int kCompactU = 2;
template <class F>
__device__ __forceinline__ void compact_cand(int4* cand, int* cnt, int cap, int* scratch, F keep_f) {
  const int n = min(*cnt, cap);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  int out = 0;
  __syncthreads();
  for (int b = 0; b < n; b += kCompactU * blockDim.x) {
    int4 e[kCompactU];
    bool keep[kCompactU];
#pragma unroll
    for (int u = 0; u < kCompactU; ++u) {
      const int i = b + u * blockDim.x + threadIdx.x;
      e[u] = make_int4(0, 0, 0, 0);
      keep[u] = false;
      if (i < n) {
        e[u] = cand[i];
        keep[u] = keep_f(e[u]);
      }
    }
    unsigned bal[kCompactU];
#pragma unroll
    for (int u = 0; u < kCompactU; ++u) {
      bal[u] = __ballot_sync(kFull, keep[u]);
      if (lane == 0) scratch[u * nw + wid] = __popc(bal[u]);
    }
    __syncthreads();
    // entry (u, thread) follows every kept entry of sub-blocks < u and of
    // the warps before it in sub-block u
#pragma unroll
    for (int u = 0; u < kCompactU; ++u) {
      int before = out, tot = 0;
      for (int w = 0; w < nw; ++w) {
        const int c = scratch[u * nw + w];
        if (w < wid) before += c;
        tot += c;
      }
      if (keep[u]) cand[before + __popc(bal[u] & below)] = e[u];
      out += tot;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *cnt = out;
  __syncthreads();
}

// One term of the canonical exact score: squared distance, fold of
// (q - x)^2; inner product, fold of q x (negated at the end).
template <bool IP>
__device__ __forceinline__ float score_step(float acc, float q, float x) {
  if (IP) return __fmaf_rn(q, x, acc);
  const float t = __fsub_rn(q, x);
  return __fmaf_rn(t, t, acc);
}

// Canonical exact score of row x against the query qv (shared memory), in
// ascending dimension order: ||q - x||^2, or -<q, x> for inner products.
// 32-byte loads, four in flight, when d is a multiple of 8 (rows, in
// cudaMalloc'ed arrays, then start on 32-byte boundaries); 16-byte loads,
// eight in flight, when d is a multiple of 4.
template <bool IP>
__device__ __forceinline__ float row_score(const float* __restrict__ x, const float* qv, int d) {
  float acc = 0.0f;
  if ((d & 7) == 0) {
    // (qv: 16-byte aligned shared memory, read as float4)
    const float4* q4 = reinterpret_cast<const float4*>(qv);
    auto fold8 = [&](const unsigned long long (&v)[4], int c) {
      const float4 qa = q4[c >> 2], qb = q4[(c >> 2) + 1];
      const float qq[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        acc = score_step<IP>(acc, qq[e], __int_as_float((int)(uint32_t)(v[e >> 1] >> (32 * (e & 1)))));
    };
    int c = 0;
    for (; c + 32 <= d; c += 32) {
      unsigned long long v[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
                     : "=l"(v[u][0]), "=l"(v[u][1]), "=l"(v[u][2]), "=l"(v[u][3])
                     : "l"(x + c + 8 * u));
#pragma unroll
      for (int u = 0; u < 4; ++u) fold8(v[u], c + 8 * u);
    }
    for (; c < d; c += 8) {
      unsigned long long v[4];
      asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
                   : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
                   : "l"(x + c));
      fold8(v, c);
    }
  } else if ((d & 3) == 0) {
    const float4* x4 = reinterpret_cast<const float4*>(x);
    const float4* q4 = reinterpret_cast<const float4*>(qv);
    int c = 0;
    for (; c + 8 <= (d >> 2); c += 8) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldg(x4 + c + u);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float4 qq = q4[c + u];
        acc = score_step<IP>(acc, qq.x, v[u].x);
        acc = score_step<IP>(acc, qq.y, v[u].y);
        acc = score_step<IP>(acc, qq.z, v[u].z);
        acc = score_step<IP>(acc, qq.w, v[u].w);
      }
    }
    for (; c < (d >> 2); ++c) {
      const float4 vv = __ldg(x4 + c), qq = q4[c];
      acc = score_step<IP>(acc, qq.x, vv.x);
      acc = score_step<IP>(acc, qq.y, vv.y);
      acc = score_step<IP>(acc, qq.z, vv.z);
      acc = score_step<IP>(acc, qq.w, vv.w);
    }
  } else {
    for (int dd = 0; dd < d; ++dd) acc = score_step<IP>(acc, qv[dd], __ldg(x + dd));
  }
  return IP ? -acc : acc;
}

// row_score of row c of a rotated copy (rabitq_index::cent_rot, ld columns):
// the fold over the padded columns adds exact zeros (qv: ld floats, zeros past
// d). Lanes of a warp reading their own rows at the same column would all
// want the same quarter of the L1 cache's banks; the rotation spreads them
// (probe selection of 10k queries, 62 of 4096 centroids in 128 dimensions:
// 102 to 84 us; 128 of 4096 in 256 dimensions: 372 to 301 us).
template <bool IP>
__device__ __forceinline__ float row_score_rot(const float* __restrict__ rot, int c, const float* qv,
                                               int ld) {
  const float* x = rot + (int64_t)c * ld;
  const float4* q4 = reinterpret_cast<const float4*>(qv);
  float acc = 0.0f;
  for (int k = 0; k < ld; k += 32) {
    unsigned long long v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
                   : "=l"(v[u][0]), "=l"(v[u][1]), "=l"(v[u][2]), "=l"(v[u][3])
                   : "l"(x + k + 8 * ((u + c) & 3)));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4 qa = q4[(k + 8 * u) >> 2], qb = q4[((k + 8 * u) >> 2) + 1];
      const float qq[8] = {qa.x, qa.y, qa.z, qa.w, qb.x, qb.y, qb.z, qb.w};
#pragma unroll
      for (int e = 0; e < 8; ++e)
        acc = score_step<IP>(acc, qq[e],
                             __int_as_float((int)(uint32_t)(v[u][e >> 1] >> (32 * (e & 1)))));
    }
  }
  return IP ? -acc : acc;
}

// Exact scores of a list of rows: each lane streams its own row (a warp has
// 256 rows' worth of loads outstanding) and folds it in ascending dimension
// order. Keys (score, id) go to the top-k buffer.
// SRC 0: the pilot (ids in S.estk); SRC 1: the candidate list (positions).
// kmax: keys above it cannot enter the result and are not kept (the rest
// of the re-rank set, once the pilot's k smallest keys are known).
template <int SRC>
__device__ void rerank_rows(const FusedParams& P, const FusedSmem& S, int64_t q, int count,
                            const int4* cand, int* top_cnt, int* surv_cnt,
                            unsigned long long kmax = ~0ull) {
  const int d = P.d;
  // Ask L2 for the rows of the first two rounds (no registers held, no
  // waiting): their loads then find most rows in L2 instead of waiting on
  // DRAM four loads at a time. (Asking for a whole set of thousands of rows
  // at once, or two rounds ahead every round, measured slower.)
  const int row_bytes = d * (int)sizeof(float);
  for (int i = threadIdx.x; i < min(count, 2 * (int)blockDim.x); i += blockDim.x) {
    const int pos = SRC == 0 ? (int)(S.estk[i] & 0xffffffffu) : (cand[i].x & 0x7fffffff);
    const char* x = reinterpret_cast<const char*>(P.data_b + (int64_t)pos * d);
    for (int o = 0; o < row_bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + o));
  }
  for (int r0 = 0; r0 < count; r0 += blockDim.x) {
    const int i = r0 + threadIdx.x;
    const bool valid = i < count;
    int pos = 0, id = 0;
    if (valid) {
      if (SRC == 0) {
        const unsigned long long e = S.estk[i];
        id = (int)(e >> 32);
        pos = (int)(e & 0xffffffffu);
      } else {
        pos = cand[i].x & 0x7fffffff;
        id = P.perm[pos];
      }
    }
    float acc = 0.0f;
    if (valid) {
      const float* x = P.data_b + (int64_t)pos * d;
      acc = P.metric ? row_score<true>(x, S.qv, d) : row_score<false>(x, S.qv, d);
    }
    const unsigned long long key = ((unsigned long long)float_key(acc) << 32) | (uint32_t)id;
    const bool take = valid && key <= kmax;
    const int slot = warp_reserve(take, top_cnt);
    if (take) S.topk[slot] = key;
    if (valid) {
      const int si = i + (SRC == 0 ? 0 : *surv_cnt);
      if (P.tr.surv_ids && si < P.tr.surv_cap) P.tr.surv_ids[q * P.tr.surv_cap + si] = id;
    }
    __syncthreads();
    const int tc = *top_cnt;  // read between barriers (see the scan's upkeep)
    __syncthreads();
    if (tc > P.ct - (int)blockDim.x) select_keep_dk(S.topk, top_cnt, P.k, *S.sel);
  }
  __syncthreads();
  if (threadIdx.x == 0) *surv_cnt += count;
  __syncthreads();
}

// Shared counters the per-query finishing step works with.
struct TailShared {
  int* cand_cnt;
  int* top_cnt;
  int* surv;
  int* scratch;  // kCompactU x kThreads / 32 ints
};

// The per-query end of the search (§4, reading R1): given the list of
// candidates {position, LB, estimate, UB} that contains every code with
// LB <= tau_ub, keep LB <= tau_ub; pilot = the m smallest (estimate, id);
// exact distances of the pilot give tau1; tau = min(tau_ub, tau1); exact
// distances of the other codes with LB <= tau; top-k by (distance, id).
// The pilot mark is bit 31 of the position. Whole block.
__device__ void finish_query(const FusedParams& P, const FusedSmem& S, int64_t q, int4* cand,
                             int cand_cap, float tau_ub, const TailShared& ts,
                             bool filtered = false) {
  const int tid = threadIdx.x;
  const int k = P.k, m = P.m;
  if (tid == 0) {
    *ts.top_cnt = 0;
    *ts.surv = 0;
  }
  __syncthreads();
  if (!filtered)  // (a list staged with LB <= tau_ub is already filtered)
    compact_cand(cand, ts.cand_cnt, cand_cap, ts.scratch,
                 [tau_ub](const int4& e) { return __int_as_float(e.y) <= tau_ub; });
  // pilot: the m smallest (estimate, id) of the list
  const int nl = *ts.cand_cnt;
  const bool pilot_all = nl <= m;
  uint32_t T_e = 0xffffffffu, T_id = 0xffffffffu;
  if (!pilot_all) {
    // the top-k buffer is free until the pilot's re-rank: histogram and
    // boundary-bin keys go there
    int ties = 0, eqn = 0;
    T_e = hist_select(nl, m, *S.sel, reinterpret_cast<int*>(S.topk),
                      reinterpret_cast<uint32_t*>(S.topk) + kHistBins, 2 * P.ct - kHistBins, ties,
                      eqn, [cand](int i) { return float_key(__int_as_float(cand[i].z)); });
    // among the list entries whose estimate equals the m-th one, the
    // `ties` smallest ids belong to the pilot; when all of them belong (the
    // usual case: one entry) no id selection is needed
    if (eqn > ties)
      T_id = block_select_f<uint32_t>(nl, ties, *S.sel, [cand, T_e, &P](int i) {
        const int4 e = cand[i];
        return float_key(__int_as_float(e.z)) == T_e ? (uint32_t)__ldg(P.perm + e.x) : 0xffffffffu;
      });
  }
  // write the pilot's (id, position) pairs to the pilot list, mark them
  __shared__ int s_pilot;
  if (tid == 0) s_pilot = 0;
  __syncthreads();
  for (int b0 = 0; b0 < nl; b0 += blockDim.x) {
    const int i = b0 + tid;
    bool in = false;
    int4 e = make_int4(0, 0, 0, 0);
    if (i < nl) {
      e = cand[i];
      const uint32_t ek = float_key(__int_as_float(e.z));
      in = pilot_all || ek < T_e || (ek == T_e && (uint32_t)__ldg(P.perm + e.x) <= T_id);
    }
    const int slot = warp_reserve(in, &s_pilot);
    if (in) {
      S.estk[slot] = (uint32_t)e.x;
      cand[i].x = e.x | (int)0x80000000;
    }
  }
  __syncthreads();
  const int pilot = s_pilot;
  // the pilot's ids, all loads in flight together
  for (int i = tid; i < pilot; i += blockDim.x) {
    const unsigned long long e = S.estk[i];
    S.estk[i] = ((unsigned long long)(uint32_t)__ldg(P.perm + (uint32_t)e) << 32) | e;
  }
  __syncthreads();
  // exact distances of the pilot; tau1 = k-th smallest of them
  rerank_rows<0>(P, S, q, pilot, cand, ts.top_cnt, ts.surv);
  // tau1: the k-th smallest exact distance of the pilot; only the k smallest
  // pilot keys can be in the result, so the rest are dropped here
  // (the pilot list is free now and holds the histogram when large enough;
  // the upper-bound buffer, free since tau_ub, holds the boundary keys)
  const bool hsel = 2 * P.ce >= kHistBins && P.cu >= 256;
  const unsigned long long T1 =
      (pilot >= k) ? select_keep_dk(S.topk, ts.top_cnt, k, *S.sel,
                                    hsel ? reinterpret_cast<int*>(S.estk) : nullptr, S.ubk, P.cu)
                   : ~0ull;
  const float tau1 = (pilot >= k) ? key_float((uint32_t)(T1 >> 32)) : __int_as_float(0x7f800000);
  const float tau = fminf(tau_ub, tau1);
  // the rest of the re-rank set: LB <= tau, outside the pilot
  compact_cand(cand, ts.cand_cnt, cand_cap, ts.scratch,
               [tau](const int4& e) { return e.x >= 0 && __int_as_float(e.y) <= tau; });
  // with k pilot keys kept, a key above the k-th of them cannot be in the
  // result (keys are distinct): such keys are not kept
  rerank_rows<1>(P, S, q, *ts.cand_cnt, cand, ts.top_cnt, ts.surv, T1);
  const int n_top = *ts.top_cnt;
  if (n_top <= (int)blockDim.x) {
    // few keys (the usual case): each thread ranks its key against all of
    // them (distinct keys, so the ranks are a permutation) and writes it to
    // its place in the result
    const bool has = tid < n_top;
    const unsigned long long mine = has ? S.topk[tid] : 0ull;
    int r = 0;
    if (has)
      for (int j2 = 0; j2 < n_top; ++j2) r += S.topk[j2] < mine ? 1 : 0;
    if (has && r < k) {
      P.out_ids[q * k + r] = (int64_t)(mine & 0xffffffffu);
      const float v = key_float((uint32_t)(mine >> 32));
      P.out_dist[q * k + r] = P.metric ? -v : v;  // inner products: <o_r, q_r>
    }
    for (int j2 = n_top + tid; j2 < k; j2 += blockDim.x) {
      P.out_ids[q * k + j2] = -1;
      P.out_dist[q * k + j2] = P.metric ? __int_as_float(0xff800000) : __int_as_float(0x7f800000);
    }
  } else {
    select_keep_dk(S.topk, ts.top_cnt, k, *S.sel);
    const int got = min(*ts.top_cnt, k);
    sort_kept_u64(S.topk, got, k);
    for (int j2 = tid; j2 < k; j2 += blockDim.x) {
      const bool ok = j2 < got;
      P.out_ids[q * k + j2] = ok ? (int64_t)(S.topk[j2] & 0xffffffffu) : -1;
      const float v = ok ? key_float((uint32_t)(S.topk[j2] >> 32)) : __int_as_float(0x7f800000);
      P.out_dist[q * k + j2] = P.metric ? -v : v;  // inner products: <o_r, q_r>, -inf pads
    }
  }
  if (tid == 0) {
    if (P.tr.tau_ub) P.tr.tau_ub[q] = tau_ub;
    if (P.tr.tau1) P.tr.tau1[q] = tau1;
    if (P.tr.tau) P.tr.tau[q] = tau;
    if (P.tr.n_surv) P.tr.n_surv[q] = *ts.surv;
  }
  __syncthreads();
}

// Code words of one code held in registers (WT > 0: compile-time length,
// loaded as 16-byte vectors; WT = 0: generic length, read in place).
template <int WT>
struct CodeRegs {
  uint64_t c[WT > 0 ? WT : 1];
};

template <int WT>
__device__ __forceinline__ void load_code(CodeRegs<WT>& r, const uint64_t* __restrict__ code) {
  if constexpr (WT == 4) {  // one 32-byte load (codes are 32-byte aligned)
    asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
                 : "=l"(r.c[0]), "=l"(r.c[1]), "=l"(r.c[2]), "=l"(r.c[3])
                 : "l"(code));
  } else if constexpr (WT > 0) {
    if constexpr (WT % 2 == 0) {
#pragma unroll
      for (int w = 0; w < WT; w += 2) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(code) + w / 2);
        r.c[w] = ((uint64_t)v.y << 32) | v.x;
        r.c[w + 1] = ((uint64_t)v.w << 32) | v.z;
      }
    } else {
#pragma unroll
      for (int w = 0; w < WT; ++w) r.c[w] = __ldg(code + w);
    }
  }
}

// <x_b, q_u> of one code against the bit-planes of its probe (§3.3.2):
// sum_j 2^j popcount(x_b AND q_u^(j)), unrolled for a compile-time code length
// (WT words) and B_q (BQT planes); WT = 0 / BQT = 0 use the runtime values.
template <int WT, int BQT>
__device__ __forceinline__ int code_ip(const CodeRegs<WT>& r, const uint64_t* __restrict__ code,
                                       const uint64_t* pl, int W, int bq) {
  if constexpr (WT > 0 && BQT > 0) {
    int ip = 0;
#pragma unroll
    for (int b = 0; b < BQT; ++b) {
      uint64_t pw[WT];
      if constexpr (WT % 2 == 0) {
#pragma unroll
        for (int w = 0; w < WT; w += 2) {
          const uint4 v = *reinterpret_cast<const uint4*>(pl + b * WT + w);
          pw[w] = ((uint64_t)v.y << 32) | v.x;
          pw[w + 1] = ((uint64_t)v.w << 32) | v.z;
        }
      } else {
#pragma unroll
        for (int w = 0; w < WT; ++w) pw[w] = pl[b * WT + w];
      }
      int pb = 0;
#pragma unroll
      for (int w = 0; w < WT; ++w) pb += __popcll(r.c[w] & pw[w]);
      ip += pb << b;
    }
    return ip;
  } else {
    int ip = 0;
    for (int b = 0; b < bq; ++b) {
      int pb = 0;
      for (int w = 0; w < W; ++w) pb += __popcll(code[w] & pl[b * W + w]);
      ip += pb << b;
    }
    return ip;
  }
}

// <x_b, q_u> of two codes of the same probe: each plane word is read from
// shared memory once for both (D' = 128 / 256, B_q = 4).
template <int WT>
__device__ __forceinline__ void code_ip2(const CodeRegs<WT>& r0, const CodeRegs<WT>& r1,
                                         const uint64_t* pl, int& i0, int& i1) {
  i0 = 0;
  i1 = 0;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    uint64_t pw[WT];
#pragma unroll
    for (int w = 0; w < WT; w += 2) {
      const uint4 v = *reinterpret_cast<const uint4*>(pl + b * WT + w);
      pw[w] = ((uint64_t)v.y << 32) | v.x;
      pw[w + 1] = ((uint64_t)v.w << 32) | v.z;
    }
    int p0 = 0, p1 = 0;
#pragma unroll
    for (int w = 0; w < WT; ++w) {
      p0 += __popcll(r0.c[w] & pw[w]);
      p1 += __popcll(r1.c[w] & pw[w]);
    }
    i0 += p0 << b;
    i1 += p1 << b;
  }
}


}  // namespace
}  // namespace rbq
