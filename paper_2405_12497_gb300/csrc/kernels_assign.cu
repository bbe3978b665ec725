// kernels_assign.cu -- the k-means assignment (§4): the nearest centroid of
// every row, exactly as a scan of all canonical squared distances finds it
// (ties to the lower id), from tensor-core products.
//
// Rows and centroids are moved by a common point mu (distances do not change;
// the bound below shrinks with the norms), scaled by powers of two (each row
// by its own, the centroids by one) so that the largest magnitude lies in
// [2^13, 2^14), and rounded to FP16: the same 11 significant bits as TF32 at
// twice its rate and half its bytes. What falls under FP16's smallest normal
// is off by at most 2^-38 of the largest element, far inside the bound's 5%.
// The products <x, c>~ give s_c = ||c||^2 - 2 <x, c>~, which differs from the
// canonical score less ||x||^2 (the same for every c) by at most eps_c
// (ProbeEps: operand rounding, accumulation, the canonical fold's own error,
// the FP32 operations). With eps at the largest ||c||, the canonical argmin
// has s_c <= min s + 2 eps. assign_dot_kernel keeps, per row and list of
// columns, the smallest s_c under the running limit (four per list, three per
// tile; what is dropped lies above the last); assign_pick_kernel
// takes the entries under the final one (mostly one, which is the answer) and
// scores them canonically where there are several or the distance is wanted.
// A row with a list that may have dropped an entry, or out of the scaled
// range, goes on a list of rows for the canonical scan.
//
// Measured (GB300), the canonical tiles -> dot, pick and scan: 400k x 128, 2048
// centroids 8.4 -> 0.48 ms; 50k x 960, 512 centroids 3.9 -> 0.3 ms. The first is
// bound by the epilogue's minima (half-rate instructions, four and a half per
// column of a warp's 32 rows; sorted insertion under the running limit took
// 0.61 ms, five two-input minima 0.46, pairs with three-input ones 0.39), the
// second by the operands' way from L2.
#include <cuda_fp16.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "query_common.cuh"
#include "tc_util.cuh"

namespace rbq {
namespace {

constexpr int kAsM = 128, kAsN = 256, kAsStages = 4, kAsEl = 64;
constexpr int kAsA = kAsM * 128, kAsB = kAsN * 128;  // bytes of one K stage (64 FP16 per row)
constexpr int kAsEpiG = 8, kAsEpi = 2 * kAsEpiG;     // epilogue warps: a group per accumulator
constexpr int kAsThreads = (kAsEpi + 2) * 32;
constexpr int kAsCols = kAsN / 2;                    // columns per epilogue half
constexpr int kAsTop = 4;                            // entries kept per row and list
constexpr float kAsFar = 0x1.0p126f;                 // above every score in range
constexpr size_t kAsSmem = (size_t)kAsStages * (kAsA + kAsB);

// Row block r / R, K stage k / 64, row r % R, element k % 64 of a tiled FP16
// operand, in bytes.
__device__ __forceinline__ int64_t tile_at(int64_t r, int k, int R, int nks) {
  return ((r / R) * nks + k / kAsEl) * (int64_t)(R * 128) +
         core_off((int)(r % R), (k % kAsEl) >> 3, R) + (k & 7) * 2;
}

// 2^e with the largest magnitude m scaled into [2^13, 2^14); NaN where m is
// outside [2^-50, 2^60] (the row or set is then scanned canonically).
__device__ __forceinline__ float scale_of(float m) {
  if (m == 0.0f) return 1.0f;
  if (!(m >= 0x1.0p-50f && m <= 0x1.0p60f)) return __int_as_float(0x7fffffff);
  return __uint_as_float((uint32_t)(127 + 13 - ilogbf(m)) << 23);
}

// mu: the mean of the centroids, any point near them would do (one block per
// 32 dimensions).
__global__ void __launch_bounds__(1024) assign_mean_kernel(const float* __restrict__ C, int K,
                                                           int d, float* __restrict__ mu) {
  __shared__ float part[32][33];
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
  float s = 0.0f;
  if (i < d)
    for (int c = w; c < K; c += 32) s = __fadd_rn(s, __ldg(C + (int64_t)c * d + i));
  part[w][threadIdx.x & 31] = s;
  __syncthreads();
  if (w == 0 && i < d) {
    for (int u = 1; u < 32; ++u) s = __fadd_rn(s, part[u][threadIdx.x & 31]);
    mu[i] = s / (float)K;
  }
}

// Warp per centroid: ||c - mu||^2; stat[0] the largest norm, stat[1] the
// largest magnitude, both as bits (non-negative; a NaN is the largest).
__global__ void __launch_bounds__(256) assign_stat_kernel(const float* __restrict__ C, int K,
                                                          int d, const float* __restrict__ mu,
                                                          float* __restrict__ cn2,
                                                          uint32_t* __restrict__ stat) {
  const int c = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (c >= K) return;
  float s = 0.0f;
  uint32_t m = 0;
  for (int i = lane; i < d; i += 32) {
    const float v = __fsub_rn(__ldg(C + (int64_t)c * d + i), __ldg(mu + i));
    s = __fmaf_rn(v, v, s);
    m = max(m, __float_as_uint(v) & 0x7fffffffu);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s = __fadd_rn(s, __shfl_xor_sync(kFull, s, o));
    m = max(m, __shfl_xor_sync(kFull, m, o));
  }
  if (lane == 0) {
    cn2[c] = s;
    atomicMax(stat, __float_as_uint(__fsqrt_rn(s)) & 0x7fffffffu);
    atomicMax(stat + 1, m);
  }
}

// Rows (R = kAsM: each with its own scale, ||x - mu||^2 and scale stored) or
// centroids (R = kAsN: the scale of the set) as FP16 tiles. A warp takes 8
// rows, 4 lanes each: a core matrix of 8 x 16 bytes is one coalesced store.
template <int R>
__global__ void __launch_bounds__(256) assign_tile_kernel(
    const float* __restrict__ X, int64_t M, int d, int nks, int64_t rows,
    const float* __restrict__ mu, const uint32_t* __restrict__ stat, uint8_t* __restrict__ tiles,
    float* __restrict__ xn2, float* __restrict__ xscale) {
  const int64_t r = ((blockIdx.x * 256 + (int64_t)threadIdx.x) >> 5) * 8 + ((threadIdx.x & 31) >> 2);
  const int q = threadIdx.x & 3;
  if (r >= rows) return;  // (whole warps: rows is a multiple of 8)
  const bool live = r < M;
  const float* row = X + (live ? r : 0) * d;
  auto at = [&](int k) {
    return live && k < d ? __fsub_rn(__ldg(row + k), __ldg(mu + k)) : 0.0f;
  };
  float sc;
  if (R == kAsM) {
    float s = 0.0f;
    uint32_t m = 0;
#pragma unroll 4
    for (int k = 2 * q; k < d; k += 8) {
      const float a = at(k), b = at(k + 1);
      s = __fmaf_rn(a, a, s);
      s = __fmaf_rn(b, b, s);
      m = max(m, max(__float_as_uint(a) & 0x7fffffffu, __float_as_uint(b) & 0x7fffffffu));
    }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      s = __fadd_rn(s, __shfl_xor_sync(kFull, s, o));
      m = max(m, __shfl_xor_sync(kFull, m, o));
    }
    sc = scale_of(__uint_as_float(m));
    if (q == 0) {
      xn2[r] = s;
      xscale[r] = sc;
    }
  } else {
    sc = scale_of(__uint_as_float(stat[1]));
  }
#pragma unroll 4
  for (int k = 2 * q; k < nks * kAsEl; k += 8)
    *reinterpret_cast<__half2*>(tiles + tile_at(r, k, R, nks)) =
        __floats2half2_rn(at(k) * sc, at(k + 1) * sc);
}


// A row's scores s are kept times w, its scale and the centroids' over two
// (powers of two), with their column in the low seven bits: |s| <= ||c||
// (||c|| + 2 ||x||) moves by at most 2^-16 of itself. e2 = 2 eps w. NaN outside
// the scaled range.
__device__ __forceinline__ void row_limit(const uint32_t* __restrict__ stat, float xn2, float xs,
                                          int d, float& w, float& e2) {
  w = 0.5f * xs * scale_of(__uint_as_float(__ldg(stat + 1)));
  const float nx = __fsqrt_rn(xn2), nc = __uint_as_float(__ldg(stat));
  const ProbeEps eps(0, nx, d);
  e2 = 2.0f * (eps(nc) + 0x1.01p-16f * (nc * (nc + 2.0f * nx)));
  if (!(nc * (nc + 2.0f * nx) * w < 0x1.0p120f)) w = __int_as_float(0x7fffffff);
  // so small that the canonical products round at the subnormal spacing
  e2 = e2 > 1e-36f ? e2 * w : __int_as_float(0x7fffffff);
}

__device__ __forceinline__ float limit_of(float lo, float e2) {
  return __fadd_ru(__fadd_ru(lo, e2), __fmul_ru(0x1.0p-20f, __fadd_ru(fabsf(lo), e2)));
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// One list entry array: lists x rows of kAsTop scores, then as many ids.
// Item i: row block i / parts, part i % parts of the column tiles. List
// (part, group g, half h): the tiles of the part with parity g, their columns
// [128 h, 128 h + 128).
__global__ void __launch_bounds__(kAsThreads, 1) assign_dot_kernel(
    const uint8_t* __restrict__ xt, const uint8_t* __restrict__ ct, const float* __restrict__ cn2,
    const uint32_t* __restrict__ stat, const float* __restrict__ xn2,
    const float* __restrict__ xscale, int64_t rows, int N, int d, int nks, int ntn, int parts,
    int64_t items, float4* __restrict__ top_s, int4* __restrict__ top_id, int* err) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(8) uint64_t s_full[kAsStages], s_empty[kAsStages], s_tfull[2], s_tempty[2];
  __shared__ volatile int s_fail;
  __shared__ __align__(16) float s_cn2[2][kAsN];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&s_taddr)),
                 "r"(2 * kAsN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    for (int i = 0; i < kAsStages; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[i])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_empty[i])), "r"(1));
    }
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_tfull[i])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_tempty[i])),
                   "r"(kAsEpiG * 32));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    s_fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = s_taddr, sbase = smem_u32(smem);
  auto slot_a = [&](uint32_t slot) { return sbase + slot * (uint32_t)(kAsA + kAsB); };
  auto slot_b = [&](uint32_t slot) { return slot_a(slot) + (uint32_t)kAsA; };
  // tiles [t0, t1) of an item's part
  auto part_of = [&](int64_t i, int& t0, int& t1) {
    const int p = (int)(i % parts);
    t0 = (int)((int64_t)ntn * p / parts);
    t1 = (int)((int64_t)ntn * (p + 1) / parts);
  };

  if (warp == kAsEpi) {  // producer: one lane issues every stage's two bulk copies
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int64_t i = blockIdx.x; i < items && ok; i += gridDim.x) {
        int t0, t1;
        part_of(i, t0, t1);
        const uint8_t* a_src = xt + i / parts * nks * (int64_t)kAsA;
        for (int t = t0; t < t1 && ok; ++t) {
          const uint8_t* b_src = ct + (int64_t)t * nks * kAsB;
          for (int ks = 0; ks < nks; ++ks, ++it) {
            const uint32_t slot = it % kAsStages;
            if (it >= (uint32_t)kAsStages &&
                !pd_wait(smem_u32(&s_empty[slot]), ((it / kAsStages) - 1) & 1u, &s_fail)) {
              ok = false;
              break;
            }
            const uint32_t fb = smem_u32(&s_full[slot]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb),
                         "r"((uint32_t)(kAsA + kAsB))
                         : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                ::"r"(slot_a(slot)), "l"(a_src + (int64_t)ks * kAsA), "r"((uint32_t)kAsA), "r"(fb)
                : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                ::"r"(slot_b(slot)), "l"(b_src + (int64_t)ks * kAsB), "r"((uint32_t)kAsB), "r"(fb)
                : "memory");
          }
        }
      }
      if (!ok) {
        s_fail = 1;
        // the copies already issued land before the CTA exits
        for (uint32_t j = it > (uint32_t)kAsStages ? it - kAsStages : 0; j < it; ++j)
          mbar_wait(smem_u32(&s_full[j % kAsStages]), (j / kAsStages) & 1u);
      }
    }
    __syncwarp();
  } else if (warp == kAsEpi + 1) {  // MMA issue
    if (lane == 0) {
      const uint32_t idesc = make_idesc(0u, kAsM, kAsN);
      constexpr uint32_t lboA = (kAsM / 8) * 128, lboB = (kAsN / 8) * 128;
      uint32_t it = 0, tc = 0;
      bool ok = true, issued = false;
      for (int64_t i = blockIdx.x; i < items && ok; i += gridDim.x) {
        int t0, t1;
        part_of(i, t0, t1);
        for (int t = t0; t < t1 && ok; ++t, ++tc) {
          const uint32_t buf = tc & 1u;
          if (tc >= 2 && !pd_wait(smem_u32(&s_tempty[buf]), ((tc / 2) - 1) & 1u, &s_fail)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint32_t dt = taddr + buf * (uint32_t)kAsN;
          for (int ks = 0; ks < nks; ++ks, ++it) {
            const uint32_t slot = it % kAsStages;
            if (!pd_wait(smem_u32(&s_full[slot]), (it / kAsStages) & 1u, &s_fail)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t a0 = slot_a(slot), b0 = slot_b(slot);
            const int steps = min(kAsEl / 16, (d - ks * kAsEl + 15) / 16);  // 16 elements each
            for (int sI = 0; sI < steps; ++sI) {
              const uint64_t da = make_desc(a0 + (uint32_t)(2 * sI) * lboA, lboA, 128);
              const uint64_t db = make_desc(b0 + (uint32_t)(2 * sI) * lboB, lboB, 128);
              const uint32_t acc = (ks > 0 || sI > 0) ? 1u : 0u;
              asm volatile(
                  "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                  "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dt),
                  "l"(da), "l"(db), "r"(idesc), "r"(acc));
            }
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    smem_u32(&s_empty[slot]))
                : "memory");
            issued = true;
          }
          if (!ok) break;
          asm volatile(
              "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                  smem_u32(&s_tfull[buf]))
              : "memory");
        }
      }
      if (!ok) {
        s_fail = 1;
        if (issued) {  // the last MMAs issued complete before the CTA exits
          const uint32_t j = it - 1;
          mbar_wait(smem_u32(&s_empty[j % kAsStages]), (j / kAsStages) & 1u);
        }
      }
    }
    __syncwarp();
  } else {
    // epilogue: group g takes the CTA's tiles of parity g (TMEM buffer g);
    // its warp w reads the lanes 32 (w % 4) .. (rows) and the columns of half
    // (w / 4) % 2. A lane keeps its row's kAsTop smallest scores of the item.
    const int group = warp / kAsEpiG, quarter = warp & 3, half = (warp >> 2) & 1;
    const int ht = tid & 127;
    const uint32_t bar_id = 1u + 2u * (uint32_t)group + (uint32_t)half;
    float* cn = s_cn2[group] + half * kAsCols;
    const float inf = __int_as_float(0x7f800000);
    uint32_t tc = 0;
    bool stop = false;
    for (int64_t i = blockIdx.x; i < items && !stop; i += gridDim.x) {
      int t0, t1;
      part_of(i, t0, t1);
      const int64_t row = i / parts * kAsM + quarter * 32 + lane;
      float w, e2;
      row_limit(stat, __ldg(xn2 + row), __ldg(xscale + row), d, w, e2);
      float s[kAsTop], thr = 0.5f * kAsFar, drop = inf;
      int id[kAsTop];
#pragma unroll
      for (int u = 0; u < kAsTop; ++u) {
        s[u] = inf;
        id[u] = -1;
      }
      for (int t = t0; t < t1; ++t, ++tc) {
        if ((int)(tc & 1u) != group) continue;
        const int h0 = t * kAsN + half * kAsCols;
        const float n2 = h0 + ht < N ? __ldg(cn2 + h0 + ht) : 0.0f;
        const bool ok = pd_wait(smem_u32(&s_tfull[group]), (tc / 2) & 1u, &s_fail);
        uint32_t gave_up;  // one decision for the whole half; the previous tile is read
        asm volatile(
            "{\n.reg .pred p, q;\nsetp.eq.u32 q, %1, 0;\nbar.red.or.pred p, %2, 128, q;\n"
            "selp.u32 %0, 1, 0, p;\n}"
            : "=r"(gave_up)
            : "r"((uint32_t)ok), "r"(bar_id)
            : "memory");
        if (gave_up) {
          s_fail = 1;
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        cn[ht] = n2;
        asm volatile("bar.sync %0, 128;" ::"r"(bar_id));
        const uint32_t src = taddr + ((uint32_t)(quarter * 32) << 16) +
                             (uint32_t)(group * kAsN + half * kAsCols);
        const int cols = N - h0;
        float m1 = kAsFar, m2 = kAsFar, m3 = kAsFar;
        auto scan = [&](auto whole) {
          for (int c0 = 0; c0 < kAsCols; c0 += 16) {
            uint32_t r[16];
            __syncwarp();
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,"
                "%12,%13,%14,%15}, [%16];"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                  "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                  "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                : "r"(src + (uint32_t)c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
            for (int e4 = 0; e4 < 4; ++e4) {
              const float4 n4 = reinterpret_cast<const float4*>(cn + c0)[e4];
              const float nn[4] = {n4.x, n4.y, n4.z, n4.w};
              float x[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int j = 4 * e4 + e;
                const float v = __fmaf_rn(nn[e], w, -__uint_as_float(r[j]));
                x[e] = __uint_as_float((__float_as_uint(v) & ~127u) | (uint32_t)(c0 + j));
                if (!decltype(whole)::value && c0 + j >= cols) x[e] = kAsFar;
              }
#pragma unroll
              for (int e = 0; e < 4; e += 2) {  // the three smallest of both
                const float lo = fminf(x[e], x[e + 1]), hi = fmaxf(x[e], x[e + 1]);
                m3 = min3(m3, fmaxf(m2, lo), fmaxf(m1, hi));
                m2 = min3(m2, fmaxf(m1, lo), hi);
                m1 = fminf(m1, lo);
              }
            }
          }
        };
        if (cols >= kAsCols)
          scan(std::true_type{});
        else
          scan(std::false_type{});
        // into the list's entries, ascending; what the tile may have dropped
        // lies at m3 or above
        drop = fminf(drop, m3);
        const float m[3] = {m1, m2, m3};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if (m[j] <= thr && m[j] < s[kAsTop - 1]) {
            float x = m[j];
            int xi = h0 + (int)(__float_as_uint(x) & 127u);
#pragma unroll
            for (int u = 0; u < kAsTop; ++u)
              if (x < s[u]) {
                const float y = s[u];
                const int yi = id[u];
                s[u] = x;
                id[u] = xi;
                x = y;
                xi = yi;
              }
            thr = limit_of(s[0], e2);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&s_tempty[group]))
                     : "memory");
      }
      if (stop) break;
      const int64_t at = ((i % parts) * 4 + group * 2 + half) * rows + row;
      top_s[at] = make_float4(s[0], s[1], s[2], fminf(s[3], drop));
      top_id[at] = make_int4(id[0], id[1], id[2], id[3]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && s_fail) atomicExch(err, 2);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                 "r"(2 * kAsN));
}

__device__ __forceinline__ float canon_sqdist(const float* __restrict__ x,
                                              const float* __restrict__ c, int d) {
  float acc = 0.0f;
  int i = 0;
  if ((d & 3) == 0 && (((uintptr_t)x | (uintptr_t)c) & 15) == 0) {  // (rows: the caller's)
    for (; i + 16 <= d; i += 16) {
      float4 a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = __ldg(reinterpret_cast<const float4*>(x + i) + u);
        b[u] = __ldg(reinterpret_cast<const float4*>(c + i) + u);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        acc = score_step<false>(acc, a[u].x, b[u].x);
        acc = score_step<false>(acc, a[u].y, b[u].y);
        acc = score_step<false>(acc, a[u].z, b[u].z);
        acc = score_step<false>(acc, a[u].w, b[u].w);
      }
    }
  }
  for (; i < d; ++i) acc = score_step<false>(acc, __ldg(x + i), __ldg(c + i));
  return acc;
}

// One thread per row: the entries under the limit, canonical scores where
// needed. redo: count, then the rows left to the canonical scan.
__global__ void __launch_bounds__(256) assign_pick_kernel(
    const float* __restrict__ A, int64_t lda, int64_t M, int64_t rows, int d,
    const float* __restrict__ C, const uint32_t* __restrict__ stat, const float* __restrict__ xn2,
    const float* __restrict__ xscale, int nlists, const float4* __restrict__ top_s,
    const int4* __restrict__ top_id, int32_t* __restrict__ assign, float* __restrict__ dist,
    int* __restrict__ redo) {
  const int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (m >= M) return;
  float lo = __int_as_float(0x7f800000);
  for (int l = 0; l < nlists; ++l) lo = fminf(lo, __ldg(&top_s[l * rows + m]).x);
  float w, e2;
  row_limit(stat, __ldg(xn2 + m), __ldg(xscale + m), d, w, e2);
  const float lim = limit_of(lo, e2);
  bool full = !(lim < 1e37f);  // (also NaN)
  int cand[8], n = 0;
  for (int l = 0; l < nlists && !full; ++l) {
    const float4 s = __ldg(&top_s[l * rows + m]);
    if (!(s.x <= lim)) continue;
    const int4 id = __ldg(&top_id[l * rows + m]);
    const float sv[4] = {s.x, s.y, s.z, s.w};
    const int iv[4] = {id.x, id.y, id.z, id.w};
    if (s.w <= lim) full = true;  // more of the quarter may lie under the limit
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (sv[u] <= lim) {
        if (n < 8) cand[n] = iv[u];
        ++n;
      }
  }
  if (full || n == 0 || n > 8) {
    redo[1 + atomicAdd(redo, 1)] = (int)m;
    return;
  }
  int best = cand[0];
  if (n > 1 || dist) {
    float bd = __int_as_float(0x7f800000);
    best = 0x7fffffff;
    for (int u = 0; u < n; ++u) {
      const float v = canon_sqdist(A + m * lda, C + (int64_t)cand[u] * d, d);
      if (v < bd || (v == bd && cand[u] < best)) {
        bd = v;
        best = cand[u];
      }
    }
    if (dist) dist[m] = bd;
  }
  assign[m] = best;
}

// The rows on a short redo list: all canonical distances, a block per row.
__global__ void __launch_bounds__(256) assign_scan_kernel(
    const float* __restrict__ A, int64_t lda, int d, const float* __restrict__ C, int N,
    const int* __restrict__ redo, int most, int32_t* __restrict__ assign,
    float* __restrict__ dist) {
  __shared__ float s_v[8];
  __shared__ int s_i[8];
  const int cnt = *redo;
  if (cnt > most) return;  // left to the tiled kernel
  for (int r = blockIdx.x; r < cnt; r += gridDim.x) {
    const int64_t m = redo[1 + r];
    float v = __int_as_float(0x7f800000);
    int id = 0x7fffffff;
    for (int c = threadIdx.x; c < N; c += blockDim.x) {
      const float a = canon_sqdist(A + m * lda, C + (int64_t)c * d, d);
      if (a < v) {  // (ascending c: ties keep the lower)
        v = a;
        id = c;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float v2 = __shfl_xor_sync(kFull, v, o);
      const int i2 = __shfl_xor_sync(kFull, id, o);
      if (v2 < v || (v2 == v && i2 < id)) {
        v = v2;
        id = i2;
      }
    }
    if ((threadIdx.x & 31) == 0) {
      s_v[threadIdx.x >> 5] = v;
      s_i[threadIdx.x >> 5] = id;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w)
        if (s_v[w] < v || (s_v[w] == v && s_i[w] < id)) {
          v = s_v[w];
          id = s_i[w];
        }
      assign[m] = id == 0x7fffffff ? 0 : id;  // all-infinite row
      if (dist) dist[m] = v;
    }
    __syncthreads();
  }
}

}  // namespace

int AssignWork::alloc(int64_t M, int d, int K, cudaStream_t s) {
  nks = (d + kAsEl - 1) / kAsEl;
  ntn = (K + kAsN - 1) / kAsN;
  // rows of a chunk: at most a GiB of tiles, and no more lists than that
  const int64_t blocks = (M + kAsM - 1) / kAsM;
  chunk = std::min<int64_t>(blocks, std::max<int64_t>(1, (int64_t(1) << 30) / ((int64_t)nks * kAsA))) *
          kAsM;
  // few row blocks: their column tiles in parts
  parts = (int)std::max<int64_t>(1, std::min<int64_t>(ntn, 304 / (chunk / kAsM)));
  RBQ_CHECK(ct.alloc((size_t)ntn * nks * kAsB, s));
  RBQ_CHECK(vec.alloc(sizeof(float) * ((size_t)d + K + 2 * (size_t)chunk + 4), s));
  RBQ_CHECK(xt.alloc((size_t)(chunk / kAsM) * nks * kAsA, s));
  RBQ_CHECK(top.alloc((sizeof(float4) + sizeof(int4)) * 4 * (size_t)parts * chunk, s));
  RBQ_CHECK(redo.alloc(sizeof(int) * (chunk + 2), s));
  RBQ_CUDA(cudaMemsetAsync(redo.p, 0, sizeof(int), s));
  return RABITQ_OK;
}

int AssignWork::check(cudaStream_t s) {
  int h = 0;
  RBQ_CUDA(cudaMemcpyAsync(&h, redo.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  RBQ_CUDA(cudaStreamSynchronize(s));
  if (h) return fail(RABITQ_ETIMEOUT, "a tensor-core wait expired in the k-means assignment");
  return RABITQ_OK;
}

// Smaller problems keep the canonical tiles: below 4096 rows or 64 centroids
// they are under a hundred microseconds and the launches here take most of it.
bool assign_tc_applies(int64_t M, int K) { return M >= 4096 && K >= 64; }

int assign_rows(const float* A, const float* C, const float* Ct, int64_t M, int K, int d,
                AssignWork& w, int32_t* assign, float* dist, cudaStream_t s) {
  int dev = 0, sms = 0;
  RBQ_CUDA(cudaGetDevice(&dev));
  RBQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  RBQ_CUDA(cudaFuncSetAttribute(assign_dot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kAsSmem));
  uint32_t* stat = w.vec.as<uint32_t>();
  float* xn2 = w.vec.as<float>() + 4;
  float* xscale = xn2 + w.chunk;
  float* cn2 = xscale + w.chunk;
  float* mu = cn2 + K;
  uint8_t *xt = w.xt.as<uint8_t>(), *ct = w.ct.as<uint8_t>();
  float4* top_s = w.top.as<float4>();
  int* err = w.redo.as<int>();
  int* redo = err + 1;  // count, rows
  if (!w.ready) assign_mean_kernel<<<(d + 31) / 32, 1024, 0, s>>>(C, K, d, mu);
  RBQ_CUDA(cudaMemsetAsync(stat, 0, 2 * sizeof(uint32_t), s));
  assign_stat_kernel<<<(K + 7) / 8, 256, 0, s>>>(C, K, d, mu, cn2, stat);
  const int64_t crows = (int64_t)w.ntn * kAsN;
  assign_tile_kernel<kAsN><<<(unsigned)(crows / 64), 256, 0, s>>>(C, K, d, w.nks, crows, mu, stat,
                                                                  ct, nullptr, nullptr);
  for (int64_t m0 = 0; m0 < M; m0 += w.chunk) {
    const int64_t m = std::min(w.chunk, M - m0);
    const int64_t rows = (m + kAsM - 1) / kAsM * kAsM;
    const float* a = A + m0 * d;
    float* dm = dist ? dist + m0 : nullptr;
    if (!w.ready || w.chunk < M)  // one chunk: the same tiles serve every call
      assign_tile_kernel<kAsM><<<(unsigned)(rows / 64), 256, 0, s>>>(a, m, d, w.nks, rows, mu, stat,
                                                                     xt, xn2, xscale);
    RBQ_CUDA(cudaMemsetAsync(redo, 0, sizeof(int), s));
    const int64_t items = rows / kAsM * w.parts;
    int4* top_id = reinterpret_cast<int4*>(top_s + 4 * (size_t)w.parts * rows);
    assign_dot_kernel<<<(unsigned)std::min<int64_t>(items, sms), kAsThreads, kAsSmem, s>>>(
        xt, ct, cn2, stat, xn2, xscale, rows, K, d, w.nks, w.ntn, w.parts, items, top_s, top_id,
        err);
    assign_pick_kernel<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(
        a, d, m, rows, d, C, stat, xn2, xscale, 4 * w.parts, top_s, top_id, assign + m0, dm, redo);
    const int most = 8 * sms;
    assign_scan_kernel<<<(unsigned)(2 * sms), 256, 0, s>>>(a, d, d, C, K, redo, most, assign + m0,
                                                           dm);
    RBQ_CUDA(cudaGetLastError());
    RBQ_CHECK(argmin_sqdist_list(a, d, Ct, K, m, K, d, redo, most, assign + m0, dm, s));
  }
  w.ready = true;
  return RABITQ_OK;
}

}  // namespace rbq
