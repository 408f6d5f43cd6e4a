// Tensor-core filter of the search (DC of Section 2.1): the exact distance
// rules are evaluated only for the vectors that can reach a query's top-k.
//
// With y the decoded residual of a vector x of list l (Section 2.1: x is its
// centroid plus y), the ADC distance is, in exact arithmetic,
//   d = D2(q, l) + s_x - 2 <q - mu, y>,   s_x = |y|^2 + 2 <c_l - mu, y>,
// with mu the centroids' mean. The index keeps y in FP16 (one power-of-two
// scale for the whole index) and s_x in FP32; a tcgen05 GEMM of a list's rows
// with the FP16 queries that probe it gives D~ = D2 + s_x - 2 <q~, y~> for
// every pair at 2 D tensor-core operations instead of M table gathers, and
// |D~ - d_rule| <= eps(q, l) where d_rule is the distance the rules define:
// the FP32 rule, or the quantised one, whose eps adds the quantiser's bound
// M Delta / 2 (pair_eps below). Then
//   1. plan:   per pair eps; the pairs grouped by list, up to 128 queries a group;
//   2. GEMM 1: the first kTake vectors of the query's probe sequence: their
//      upper bounds D~ + eps; T = the k-th smallest of them, so at least k
//      vectors have d_rule <= T;
//   3. GEMM 2: every vector of every probed list; those with D~ - eps <= T go
//      to the query's candidate list (every vector of the final top-k does,
//      ties included); a pair on a table of at most 4 bits, whose quantiser
//      bound is too wide to single out vectors, is only marked as alive;
//   4. final:  per query T again over the candidates' upper bounds, then the
//      exact rule for the ones left, and their order by (distance, id).
// The results equal the scanning kernels' bit for bit. A query with more
// candidates than fit (bounds too wide for its data, or values that are not
// finite: every comparison keeps a NaN) is listed for the query-major kernel.
//
// What bounds it: GEMM 2 reads the decoded rows once per group of 128 queries
// (2 D bytes a vector against M for the codes) and is bound by HBM and L2
// reads, its epilogue by issue (about 4 instructions per (vector, query)).
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "scan.cuh"
#include "tc.cuh"

namespace anns {
namespace {

constexpr int kGq = 128;           // queries per group = columns of a tile
constexpr int kTv = 256;           // vectors per tile: two 128-row halves
constexpr int kKE = 64;            // FP16 elements per K chunk (128 bytes, one swizzle row)
constexpr int kFStages = 4;
constexpr int kEpiWarps = 16;
constexpr int kFThreads = 64 + 32 * kEpiWarps;  // warp 0: TMA, warp 1: MMA + TMEM owner, then the epilogue
constexpr uint32_t kYBytes = kTv * 128, kQBytes = kGq * 128, kFStage = kYBytes + kQBytes;
constexpr int kPush = 64;          // staged candidates per epilogue warp
// ring | per epilogue warp: constants of its 64 columns, staged candidates | barriers
constexpr uint32_t kEpiBytes = 64 * 16 + kPush * 12;
constexpr size_t kFilterSmem = 1024 + (size_t)kFStages * kFStage + kEpiWarps * kEpiBytes + 256;
constexpr int kBatch = 4;          // quantised pairs a warp settles at a time
constexpr int kPosBits = 25;       // candidate word: rank << 25 | position in the list
constexpr int kTakeMax = 4096;

struct FItem { int row0, nv_cnt, slot0, pos0; };  // first row, vectors | queries << 16, first slot, position of row0 in its list
// Slots: the pairs of a GEMM list by list, each list's first slot a multiple of 16.

// ---------------------------------------------------------------- the index's part

// FP16 rows of the decoded residuals, s_x, and per list the largest |y|, the
// largest rounding error |y~ - y| and |c - mu| (all rounded upward). One block
// per tile of 32 vectors, one warp per vector.
__global__ void __launch_bounds__(256) decode_kernel(const uint8_t* __restrict__ codes, const float* __restrict__ books,
                                                     const float* __restrict__ cent, const float* __restrict__ mu,
                                                     const int64_t* __restrict__ tile_off,
                                                     const int32_t* __restrict__ list_len, int nlist, int64_t ntiles,
                                                     int dim, int M, int dsub, int nchunk, int W, float up,
                                                     __half* __restrict__ y, float* __restrict__ sx,
                                                     float4* __restrict__ stat) {
  __shared__ int sl;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double down = 1.0 / (double)up;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    if (threadIdx.x == 0) {  // the list whose tiles hold t
      int lo = 0, hi = nlist - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tile_off[mid] <= t) lo = mid; else hi = mid - 1;
      }
      sl = lo;
    }
    __syncthreads();
    const int l = sl;
    const float* c = cent + (int64_t)l * dim;
    for (int i = warp; i < kTileVecs; i += 8) {
      const int64_t row = t * kTileVecs + i;
      double n2 = 0.0, e2 = 0.0, cy = 0.0, cm = 0.0;
      for (int d = lane; d < W; d += 32) {
        __half h = __float2half_rn(0.f);
        if (d < dim) {
          const int m = d / dsub, code = codes[((size_t)t * nchunk + (m >> 4)) * kTileChunkBytes + i * kChunkBytes + (m & 15)];
          const float v = books[((size_t)m * kKsub + code) * dsub + (d - m * dsub)];
          h = __float2half_rn(v * up);
          const double vd = v, cd = (double)c[d] - (double)mu[d], er = (double)__half2float(h) * down - vd;
          n2 += vd * vd;
          e2 += er * er;
          cy += cd * vd;
          cm += cd * cd;
        }
        y[row * W + d] = h;
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        n2 += __shfl_xor_sync(kFull, n2, o);
        e2 += __shfl_xor_sync(kFull, e2, o);
        cy += __shfl_xor_sync(kFull, cy, o);
        cm += __shfl_xor_sync(kFull, cm, o);
      }
      if (lane == 0) {
        sx[row] = (float)(n2 + 2.0 * cy);
        if ((t - tile_off[l]) * kTileVecs + i < list_len[l]) {
          // non-negative floats order like their bit patterns
          float4* s = stat + l;
          atomicMax((int*)&s->x, __float_as_int(__double2float_ru(sqrt(n2) * (1.0 + 1e-9))));
          atomicMax((int*)&s->y, __float_as_int(__double2float_ru(sqrt(e2) * (1.0 + 1e-9))));
          if (i == 0) s->z = __double2float_ru(sqrt(cm) * (1.0 + 1e-9));
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- plan

struct PlanArgs {
  int64_t nq, dim;
  int nprobe, k, M, dsub, Dp, take, nlist;
  int v4;                  // 16-byte loads of Q and the centroids, dsub a multiple of 4
  const int32_t* npq; const int32_t* kpq;
  const int32_t* probes; const float* d2; const uint8_t* bits; const int32_t* list_len;
  const int64_t* tile_off;
  const float* Q; const float* C; const float* ym; const float4* stat; const float* qrows;
  float mu_norm, yscale;   // |mu| (rounded upward), 1 / scale of the decoded rows
  float* eps;              // [nq * nprobe], -1: the pair takes no part
  float* eps0;             // [nq * nprobe] eps without the quantiser's term
  int2* sel;               // [nq * nprobe] GEMM 1: vectors taken, where their bounds go
  uint8_t* in2;            // [nq * nprobe] the pair takes part in GEMM 2
  int* ntake;              // [nq] bounds of the query
  float* thr;              // [nq] T
  uint8_t* alive;          // [nq * nprobe]
  const __half* q16;       // [nq x Dp] the queries' FP16 operand
};

// The pairs of one GEMM regrouped by list.
struct PassArgs {
  int *cnt, *fill;         // [nlist] pairs per list, fill cursors
  int *s0, *i0;            // [nlist + 1] first slot and item of each list
  float2* kc;              // [slots] column constants
  int2* d1;                // GEMM 1: [slots] (vectors taken, destination)
  int* pair;               // GEMM 2: [slots]
  __half* rows;            // [slots x Dp] the queries' rows slot by slot
  FItem* items;
  int tiles;               // vector tiles of a list, at most
};

// eps of a pair: |D~ - d_rule| <= eps. u = 2^-24. With r = |y|max, e = |y~ - y|
// max and cm = |c - mu| of the list, qt = |q~|, qd >= |q~ - (q - mu)| of the
// query, and G = r^2 + 2 (|c| + |q|) r >= the sum over the sub-spaces of
// |y_m|^2 + 2 (|c_m| + |q_m|) |y_m| (Cauchy-Schwarz):
//  - operands: 2 (qd r + qt e);
//  - the tensor cores' FP32 accumulation and the epilogue's FMA: (4 Dp + 24) u
//    qt (r + e), twice the bound the coarse stage's re-rank uses, and 2 u |s_x|;
//  - the FP32 rule's own roundings: P_l and 2 Q_q are sums of dsub products, T'
//    one more operation, M additions and the final one: (dsub + M + 4) u
//    (G + D2); the constant M + dsub + 16 covers s_x's rounding too;
//  - b-bit tables: every level is within 1/2 + 4 u L of its entry and the
//    steps, the offset and the two final roundings add a few u of the sums:
//    M R (1 / (2 L) + 8 u), R >= the largest row range. T'_mc = |y_c - r_m|^2 -
//    |r_m|^2 with r_m the query's residual lies in [-|r_m|^2, (|y_c| + |r_m|)^2
//    - |r_m|^2], so R = max_m (max_c |y_mc| + |r_m|)^2 plus the entries' own
//    rounding.
// 1e-28 covers underflow.
__device__ __forceinline__ float pair_eps(const PlanArgs& a, float qt, float qd, const float4& s, float d2, float& G) {
  const float u = 5.9604645e-8f;
  const float cn = s.z + a.mu_norm, qn = qt + qd + a.mu_norm;
  G = s.x * s.x + 2.f * (cn + qn + s.z) * s.x;
  return 1.01f * (2.f * (qd * s.x + qt * s.y) +
                  u * ((4.f * a.Dp + 24.f) * qt * (s.x + s.y) + (float)(a.M + a.dsub + 16) * (G + d2))) + 1e-28f;
}
__device__ __forceinline__ float quant_eps(int M, int b, float R) {
  const float u = 5.9604645e-8f;
  return 1.01f * (float)M * R * (0.5f / (float)((1 << b) - 1) + 8.f * u);
}

// One block per query: eps of its pairs and the first `take` vectors of its
// probe sequence for GEMM 1, those pairs counted per list.
__global__ void __launch_bounds__(128) plan_kernel(const PlanArgs a, const PassArgs p1) {
  __shared__ int len[ANNS_MAX_NPROBE];
  const int64_t q = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int np = a.npq ? min(max(a.npq[q], 0), a.nprobe) : a.nprobe;
  const int kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  const float qt = __fsqrt_ru(a.qrows[q]) * 1.0001f, qd = a.qrows[a.nq + q];
  const float* qv = a.Q + q * a.dim;
  for (int j = warp; j < a.nprobe; j += 4) {
    const int64_t p = q * a.nprobe + j;
    const int l = j < np && kq > 0 ? a.probes[p] : -1;
    const int n_l = l >= 0 ? a.list_len[l] : 0;
    float eps = -1.f;
    if (n_l > 0) {
      const int b = a.bits[p];
      float rmax = 0.f;
      if (b > 0) {
        const float* cv = a.C + (int64_t)l * a.dim;
        for (int m = lane; m < a.M; m += 32) {
          float s = 0.f;
          if (a.v4) {
            for (int i = 0; i < a.dsub; i += 4) {
              const float4 x = __ldg((const float4*)(qv + m * a.dsub + i)), c = __ldg((const float4*)(cv + m * a.dsub + i));
              const float e0 = x.x - c.x, e1 = x.y - c.y, e2 = x.z - c.z, e3 = x.w - c.w;
              s += e0 * e0 + e1 * e1 + (e2 * e2 + e3 * e3);
            }
          } else {
            for (int i = 0; i < a.dsub; ++i) {
              const float e = qv[m * a.dsub + i] - cv[m * a.dsub + i];
              s += e * e;
            }
          }
          const float v = sqrtf(s) * 1.0001f + a.ym[m];
          rmax = v > rmax || v != v ? v : rmax;  // a NaN stays
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          const float v = __shfl_xor_sync(kFull, rmax, o);
          rmax = v > rmax || v != v ? v : rmax;
        }
      }
      float G;
      eps = pair_eps(a, qt, qd, a.stat[l], a.d2[p], G);
      if (lane == 0) a.eps0[p] = eps;
      if (b > 0) eps += quant_eps(a.M, b, rmax * rmax * 1.0001f + 4.f * (a.dsub + 4) * 5.9604645e-8f * G);
    }
    if (lane == 0) {
      a.eps[p] = eps;
      len[j] = n_l;
    }
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0;
    for (int j0 = 0; j0 < a.nprobe; j0 += 32) {
      const int j = j0 + lane;
      const int n = j < a.nprobe ? len[j] : 0;
      int x = min(n, a.take);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x = min(x + v, a.take);
      }
      const int incl = min(base + x, a.take), excl0 = __shfl_up_sync(kFull, incl, 1);
      const int excl = lane ? excl0 : base, t = incl - excl;
      if (j < a.nprobe) {
        const int64_t p = q * a.nprobe + j;
        a.sel[p] = make_int2(t, (int)(q * a.take) + excl);
        if (t > 0) atomicAdd(p1.cnt + a.probes[p], 1);
      }
      base = __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) a.ntake[q] = base;
  }
}

// One block: exclusive prefixes over the lists of a pass's slots and items
// (totals at [nlist]).
__global__ void __launch_bounds__(1024) plan_scan_kernel(const int32_t* __restrict__ list_len, int nlist,
                                                         const PassArgs w) {
  __shared__ int part[2][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry[2] = {0, 0};
  for (int base = 0; base < nlist; base += 1024) {
    const int l = base + threadIdx.x;
    int v[2] = {0, 0}, x[2];
    if (l < nlist) {
      const int c = w.cnt[l];
      v[0] = (c + 15) & ~15;
      v[1] = (c + kGq - 1) / kGq * min((list_len[l] + kTv - 1) / kTv, w.tiles);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      x[i] = v[i];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x[i], o);
        if (lane >= o) x[i] += y;
      }
      if (lane == 31) part[i][warp] = x[i];
    }
    __syncthreads();
    if (warp < 2) {
      int p = part[warp][lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, p, o);
        if (lane >= o) p += y;
      }
      part[warp][lane] = p;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (l < nlist) (i ? w.i0 : w.s0)[l] = carry[i] + (warp ? part[i][warp - 1] : 0) + x[i] - v[i];
      carry[i] += part[i][31];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    w.s0[nlist] = carry[0];
    w.i0[nlist] = carry[1];
  }
}

// The first `pair_blocks` blocks: each pair of the pass to a slot of its list,
// a warp per pair, which also copies the query's FP16 row there: the GEMM then
// loads a group's rows as plain TMA boxes. (Gathering them in the GEMM by
// tile::gather4 took 0.1 us per four rows, 7.6 us per tile of 128 queries.) The
// other blocks: the items of each list (a warp per list), vector tile by vector
// tile, so that a tile's groups follow one another.
template <int PASS>
__global__ void __launch_bounds__(256) plan_scatter_kernel(const PlanArgs a, const PassArgs w, int pair_blocks) {
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < pair_blocks) {
    const int64_t p0 = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 32;  // 32 pairs a warp
    const int64_t pl = p0 + lane;
    int2 t = make_int2(0, 0);
    bool in = false;
    if (pl < a.nq * a.nprobe) {
      if constexpr (PASS == 1) {
        t = a.sel[pl];
        in = t.x > 0;
      } else {
        in = a.in2[pl] != 0;
      }
    }
    int slot = 0, q = 0;
    if (in) {
      q = (int)(pl / a.nprobe);
      const int l = a.probes[pl];
      const float m2s = -2.f * (a.qrows[2 * a.nq + q] * a.yscale), eps = a.eps[pl], d2 = a.d2[pl];
      slot = w.s0[l] + atomicAdd(w.fill + l, 1);
      if constexpr (PASS == 1) {
        w.kc[slot] = make_float2(__fadd_ru(d2, eps), m2s);
        w.d1[slot] = t;
      } else {
        // D~ - eps <= T  <=>  s_x - 2 dot <= T + eps - D2 (rounded upward)
        w.kc[slot] = make_float2(__fadd_ru(__fadd_ru(a.thr[q], eps), -d2), m2s);
        const int b = a.bits[pl];  // sign bit: only marked, a table of at most 4 bits
        w.pair[slot] = (int)((uint32_t)pl | (b >= 1 && b <= 4 ? 0x80000000u : 0u));
      }
    }
    for (unsigned left = __ballot_sync(kFull, in); left; left &= left - 1u) {
      const int src = __ffs(left) - 1;
      const int qq = __shfl_sync(kFull, q, src), ss = __shfl_sync(kFull, slot, src);
      const uint4* from = (const uint4*)(a.q16 + (size_t)qq * a.Dp);
      uint4* to = (uint4*)(w.rows + (size_t)ss * a.Dp);
      for (int i = lane; i < a.Dp / 8; i += 32) to[i] = __ldg(from + i);
    }
  } else {
    const int l = ((int)blockIdx.x - pair_blocks) * 8 + (threadIdx.x >> 5);
    if (l >= a.nlist) return;
    const int c = w.cnt[l], i0 = w.i0[l], n = w.i0[l + 1] - i0, ng = (c + kGq - 1) / kGq;
    const int n_l = a.list_len[l], row = (int)(a.tile_off[l] * kTileVecs), s0 = w.s0[l];
    for (int i = lane; i < n; i += 32) {
      const int t = i / ng, g = i % ng;
      w.items[i0 + i] = FItem{row + t * kTv, min(kTv, n_l - t * kTv) | (min(kGq, c - g * kGq) << 16), s0 + g * kGq, t * kTv};
    }
  }
}

// ---------------------------------------------------------------- GEMM

struct GemmArgs {
  const FItem* items; const int* nitems;
  const float2* gk;
  const int2* gd; float* ub;                              // GEMM 1
  const int* gp; int nprobe;                              // GEMM 2
  int* qcnt; uint2* cand; int cap; uint8_t* alive;
  const float* sx;
  int nK, ksteps;
  int* status; long long wait_limit;
};

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// One FP32 column of this thread's TMEM lane.
__device__ __forceinline__ float tc_ld1(uint32_t taddr) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=r"(r) : "r"(taddr) : "memory");
  return __uint_as_float(r);
}

__device__ __forceinline__ FItem load_item(const FItem* p) {
  const int4 v = __ldg((const int4*)p);
  return FItem{v.x, v.y, v.z, v.w};
}

// Rows are vectors (256 a tile, two 128-row accumulators), columns the group's
// queries (N = their number rounded up to 16: short groups cost little).
// Persistent, one CTA per SM, items taken round-robin; the ring, the roles and
// the bounded waits are the coarse stage's (coarse_tc.cu).
// MODE 1 writes upper bounds, MODE 2 collects candidates.
template <int MODE>
__global__ void __launch_bounds__(kFThreads, 1) filter_gemm_kernel(const __grid_constant__ CUtensorMap tmY,
                                                                   const __grid_constant__ CUtensorMap tmQ,
                                                                   const GemmArgs a) {
  unsigned char* base = anns_dyn_smem + ((1024u - (smem_addr(anns_dyn_smem) & 1023u)) & 1023u);
  unsigned char* epi = base + (size_t)kFStages * kFStage;
  uint64_t* bars = (uint64_t*)(epi + kEpiWarps * kEpiBytes);
  // full[S] | empty[S] | acc_full[2] | acc_empty[2] | drain, then the TMEM slot and the abort flag
  uint32_t* slot = (uint32_t*)(bars + 2 * kFStages + 5);
  volatile int* abort_flag = (volatile int*)(slot + 1);
  const uint32_t ring = smem_addr(base);
  const uint32_t full0 = smem_addr(bars), empty0 = full0 + 8 * kFStages, accf0 = full0 + 16 * kFStages,
                 acce0 = accf0 + 16, drain = acce0 + 16;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nitems = *a.nitems, stride = gridDim.x;
  if ((int)blockIdx.x >= nitems) return;  // before any barrier or TMEM use

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < kFStages; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(accf0 + 8 * i, 1);
      mbar_init(acce0 + 8 * i, kEpiWarps);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;

  bool ok = true;
  if (warp == 0) {
    // producer: chunk g goes to stage g % S; lane i brings 64 rows of vectors
    // (i < 4) or 32 of queries (i - 4 < 4)
    uint32_t g = 0;
    FItem it = load_item(a.items + blockIdx.x), nx = it, n2 = it;
    if ((int)blockIdx.x + stride < nitems) nx = load_item(a.items + blockIdx.x + stride);
    for (int i = blockIdx.x; i < nitems && ok; i += stride) {
      const int nv = it.nv_cnt & 0xFFFF, cnt = it.nv_cnt >> 16, nbox = (nv + 63) >> 6, qbox = (cnt + 31) >> 5;
      if (i + 2 * stride < nitems) n2 = load_item(a.items + i + 2 * stride);
      for (int k = 0; k < a.nK; ++k, ++g) {
        const uint32_t st = g % kFStages;
        if (g >= kFStages) {
          const bool got = mbar_wait(empty0 + 8 * st, ((g / kFStages) - 1) & 1, a.wait_limit, abort_flag);
          ok = __all_sync(kFull, got);
        }
        if (!ok) break;
        const uint32_t y_dst = ring + st * kFStage, q_dst = y_dst + kYBytes;
        if (lane == 0) mbar_expect_tx(full0 + 8 * st, (uint32_t)nbox * 8192u + (uint32_t)qbox * 4096u);
        __syncwarp();
        if (lane < nbox) tma_load_2d(y_dst + lane * 8192, &tmY, k * kKE, it.row0 + 64 * lane, full0 + 8 * st);
        const int b = lane - 4;
        if (b >= 0 && b < qbox) tma_load_2d(q_dst + b * 4096, &tmQ, k * kKE, it.slot0 + 32 * b, full0 + 8 * st);
      }
      it = nx;
      nx = n2;
    }
    if (lane == 0) {
      if (!ok) {
        *abort_flag = 1;
        atomicExch(a.status, ANNS_DEV_TIMEOUT);
      }
      // Every copy lands before the CTA exits, also where another role gave up
      // after the last one was issued (coarse_tc.cu).
      for (uint32_t st = 0; st < kFStages; ++st) {
        const uint32_t count = g > st ? (g - st + kFStages - 1) / kFStages : 0;
        if (count > 0) mbar_wait(full0 + 8 * st, (count - 1) & 1);
      }
    }
    __syncwarp();
  } else if (tid == 32) {
    // MMA issuer: this CTA's n-th item accumulates into TMEM columns (n & 1) * 256 + 128 * half
    uint32_t g = 0;
    int n = 0;
    FItem it = load_item(a.items + blockIdx.x), nx = it;
    if ((int)blockIdx.x + stride < nitems) nx = load_item(a.items + blockIdx.x + stride);
    for (int i = blockIdx.x; i < nitems && ok; i += stride, ++n) {
      const int nv = it.nv_cnt & 0xFFFF, N = ((it.nv_cnt >> 16) + 15) & ~15;
      it = nx;
      if (i + 2 * stride < nitems) nx = load_item(a.items + i + 2 * stride);
      const uint32_t idesc = (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((128u >> 4) << 24);  // FP16 operands, FP32 sums
      const int b = n & 1, use = n >> 1;
      if (use > 0) ok = mbar_wait(acce0 + 8 * b, (uint32_t)((use - 1) & 1), a.wait_limit, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t d = tmem + (uint32_t)(b * 256);
      for (int k = 0; k < a.nK; ++k, ++g) {
        const uint32_t st = g % kFStages;
        ok = mbar_wait(full0 + 8 * st, (g / kFStages) & 1, a.wait_limit, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t y_addr = ring + st * kFStage, q_addr = y_addr + kYBytes;
        const int ns = min(4, a.ksteps - 4 * k);
        for (int ks = 0; ks < ns; ++ks) {
          const uint32_t acc = (k > 0 || ks > 0) ? 1u : 0u;
          const uint64_t qd = smem_desc_sw128(q_addr + ks * 32);
          mma_f16(d, smem_desc_sw128(y_addr + ks * 32), qd, idesc, acc);
          if (nv > 128) mma_f16(d + 128, smem_desc_sw128(y_addr + 16384 + ks * 32), qd, idesc, acc);
        }
        tc_commit(empty0 + 8 * st);
      }
      if (!ok) break;
      tc_commit(accf0 + 8 * b);
    }
    if (!ok) {
      *abort_flag = 1;
      atomicExch(a.status, ANNS_DEV_TIMEOUT);
    }
    tc_commit(drain);  // arrives once every MMA issued above has completed
    mbar_wait(drain, 0);
  } else if (warp >= 2) {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 of half ((w - 2) / 4)
    // % 2, the 32-column chunks of parity (w - 2) / 8. Two warps a scheduler left
    // two thirds of the issue slots empty (dependent chains of TMEM and shared
    // loads), four fill them better.
    const int quad = warp & 3, half = ((warp - 2) >> 2) & 1, par = (warp - 2) >> 3, r0 = half * 128 + quad * 32;
    unsigned char* mine = epi + (warp - 2) * kEpiBytes;
    float2* ck = (float2*)mine;                       // constants of the warp's columns: chunk c0 at (c0 / 64) * 32
    int2* cd = (int2*)(mine + 64 * 8);                // GEMM 1: (taken, destination); GEMM 2: pair (sign bit: only marked)
    int* sp = (int*)(mine + 64 * 16);                 // staged candidates: pair, position, D~ - D2
    int* spos = sp + kPush;
    float* sv = (float*)(spos + kPush);
    int staged = 0;
    auto flush = [&]() {
      __syncwarp();
      for (int e = lane; e < staged; e += 32) {
        const int p = sp[e], q = p / a.nprobe;
        const int at = atomicAdd(a.qcnt + q, 1);
        if (at < a.cap)
          a.cand[(int64_t)q * a.cap + at] = make_uint2((uint32_t)(p - q * a.nprobe) << kPosBits | (uint32_t)spos[e],
                                                       __float_as_uint(sv[e]));
      }
      staged = 0;
      __syncwarp();
    };
    // The columns of `mask` (bit j: column c0 + j0 + j) one by one: a rolled loop
    // that reads a column again from TMEM (unrolled over the registers it is 32
    // copies of the push, and their instruction fetches cost ten times the work).
    auto push = [&](uint32_t mask, int j0, uint32_t tcol, const float2* kc, const int2* dc, float s, int pos) {
      uint32_t cols = __reduce_or_sync(kFull, mask);
      const int dl = dc[j0 + (lane & 7)].x;  // lane j < 8: column j's pair
      const bool hit = lane < 8 && (cols >> lane & 1u);
      if (hit) a.alive[dl & 0x7FFFFFFF] = 1;
      cols = __ballot_sync(kFull, hit && dl >= 0);  // the others are only marked
      for (; cols; cols &= cols - 1u) {
        const int j = __ffs(cols) - 1;
        const int d = dc[j0 + j].x;
        const unsigned who = __ballot_sync(kFull, mask >> j & 1u);
        const float t = fmaf(tc_ld1(tcol + j0 + j), kc[j0 + j].y, s);
        if (staged > kPush - 32) flush();
        if (mask >> j & 1u) {
          const int e = staged + __popc(who & ((1u << lane) - 1u));
          sp[e] = d;
          spos[e] = pos;
          sv[e] = t;
        }
        staged += __popc(who);
      }
    };
    // the next item's columns are requested while this one is drained, its item
    // one step earlier: a round trip to L2 each, as long as a short tile
    FItem nx = load_item(a.items + blockIdx.x), n2 = nx;
    float2 nk[2] = {};
    int2 nd[2] = {};
    float ns = 0.f;
    auto load_cols = [&](const FItem& f) {  // and the thread's row scalar
      const int nv = f.nv_cnt & 0xFFFF;
      // rows past the list's end hold the next list's vectors: never candidates
      ns = r0 + lane < nv ? __ldg(a.sx + f.row0 + r0 + lane) : INFINITY;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int col = lane + 32 * par + 64 * c, s = f.slot0 + col;
        if (col < (f.nv_cnt >> 16)) {
          nk[c] = __ldg(a.gk + s);
          if constexpr (MODE == 1) {
            nd[c] = __ldg(a.gd + s);
          } else {
            nd[c].x = __ldg(a.gp + s);
          }
        }
      }
    };
    load_cols(nx);
    if ((int)blockIdx.x + stride < nitems) n2 = load_item(a.items + blockIdx.x + stride);
    int n = 0;
    for (int i = blockIdx.x; i < nitems; i += stride, ++n) {
      const FItem it = nx;
      const int nv = it.nv_cnt & 0xFFFF, cnt = it.nv_cnt >> 16, b = n & 1, r = r0 + lane;
      const float s = ns;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        ck[lane + 32 * c] = nk[c];
        cd[lane + 32 * c] = nd[c];
      }
      __syncwarp();
      nx = n2;
      if (i + 2 * stride < nitems) n2 = load_item(a.items + i + 2 * stride);
      if (i + stride < nitems) load_cols(nx);
      // every lane waits; the warp goes on only together (tcgen05.ld is .sync.aligned)
      const bool got = mbar_wait(accf0 + 8 * b, (uint32_t)((n >> 1) & 1), a.wait_limit, abort_flag);
      if (!__all_sync(kFull, got)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (r0 < nv) {
        const int pos = it.pos0 + r;
        for (int c0 = 32 * par; c0 < cnt; c0 += 64) {
          const float2* kc = ck + (c0 >> 6) * 32;
          const int2* dc = cd + (c0 >> 6) * 32;
          float v[32];
          const uint32_t tcol = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * 256 + half * 128 + c0);
          tc_ld32(tcol, v);
          if constexpr (MODE == 1) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              if (c0 + j < cnt) {
                const float2 k = kc[j];
                const int2 d = dc[j];
                if (pos < d.x && r < nv) a.ub[d.y + pos] = __fadd_ru(fmaf(v[j], k.y, s), k.x);
              }
            }
          } else {
            // eight columns at a time: is there a candidate in any lane?
#pragma unroll
            for (int j0 = 0; j0 < 32; j0 += 8) {
              bool any = false;
#pragma unroll
              for (int j = j0; j < j0 + 8; j += 2) {
                const float4 k = *(const float4*)(kc + j);
                v[j] = fmaf(v[j], k.y, s);
                v[j + 1] = fmaf(v[j + 1], k.w, s);
                any = any || !(v[j] > k.x) || !(v[j + 1] > k.z);
              }
              if (!__any_sync(kFull, any)) continue;
              uint32_t mask = 0;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (!(v[j0 + j] > kc[j0 + j].x)) mask |= 1u << j;
              const int left = cnt - c0 - j0;  // columns past the group, rows past the list
              mask &= left >= 8 ? 0xFFu : left > 0 ? (1u << left) - 1u : 0u;
              if (r >= nv) mask = 0;
              push(mask, j0, tcol, kc, dc, s, pos);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * b);
    }
    if (MODE == 2) flush();
    if (!ok && lane == 0) {
      *abort_flag = 1;
      atomicExch(a.status, ANNS_DEV_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ---------------------------------------------------------------- thresholds

// Key order of upper bounds: non-negative floats order like their bit
// patterns, negative values count as 0 and NaN as +inf (both larger bounds).
__device__ __forceinline__ uint32_t bound_key(float u) {
  return u > 0.f ? __float_as_uint(u) : (u <= 0.f ? 0u : 0x7F800000u);
}

// An upper bound of the kq-th smallest of the warp's keys, VPT per lane (absent
// ones all ones): bisection between the smallest and the largest present key
// until the interval is at most 2^8 units of the last place (3e-5 of the
// value, well inside the bounds' own width); +inf when there are fewer keys.
template <int VPT>
__device__ __forceinline__ float warp_kth(const uint32_t (&key)[VPT], int n, int kq) {
  if (n < kq) return INFINITY;
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    lo = min(lo, key[i]);
    hi = max(hi, key[i] == 0xFFFFFFFFu ? 0u : key[i]);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  while (hi - lo > 255u) {  // count(key <= hi) >= kq throughout
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
#pragma unroll
    for (int i = 0; i < VPT; ++i) c += key[i] <= mid ? 1 : 0;
    if ((int)__reduce_add_sync(kFull, c) >= kq) hi = mid;
    else lo = mid + 1u;
  }
  return __uint_as_float(hi);
}

// Which of a query's pairs GEMM 2 takes (lanes over the probe ranks), given T:
//  - none of a pair that no vector can reach T from: the vectors lie within r =
//    |y|max of the centroid, so d >= (sqrt(D2) - r)^2 (with slack for the FP32
//    rule's rounding of D2);
//  - not a pair on a table of at most 4 bits about half of whose vectors would
//    pass (T + eps above the list's expected mean distance, D2 plus the mean of
//    s_x - 2 dot over GEMM 1's vectors): it is scanned anyway.
__device__ __forceinline__ void classify_pairs(const PlanArgs& a, const PassArgs& p2, int64_t q, float T, float mean_t,
                                               int first, int step) {
  for (int j = first; j < a.nprobe; j += step) {
    const int64_t p = q * a.nprobe + j;
    const float eps = a.eps[p];
    bool in = eps != -1.f;
    if (in) {
      const float d2 = a.d2[p];
      const int l = a.probes[p], b = a.bits[p];
      const float away = sqrtf(d2) * (1.f - (2e-5f + 1.3e-7f * (float)a.dim)) - a.stat[l].x;
      if (away > 0.f && away * away * 0.99999f > __fadd_ru(T, eps)) {
        in = false;
      } else if (b >= 1 && b <= 4 && T + eps > d2 + mean_t) {
        a.alive[p] = 1;
        in = false;
      }
      if (in) atomicAdd(p2.cnt + l, 1);
    }
    a.in2[p] = in ? 1 : 0;
  }
}

// One warp per query: T from GEMM 1's bounds, then the pairs of GEMM 2.
// take <= 32 VPT.
template <int VPT>
__global__ void __launch_bounds__(128) threshold_kernel(const PlanArgs a, const PassArgs p2,
                                                        const float* __restrict__ ub) {
  const int64_t q = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (q >= a.nq) return;
  const int n = a.ntake[q], kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  uint32_t key[VPT];
  float sum = 0.f;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int e = lane + 32 * i;
    key[i] = 0xFFFFFFFFu;
    if (e < n) {
      const float u = ub[q * a.take + e];
      key[i] = bound_key(u);
      sum += u;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  const float T = warp_kth<VPT>(key, n, kq);
  if (lane == 0) a.thr[q] = T;
  const float mean_t = n > 0 ? sum / (float)n - (a.d2[q * a.nprobe] + a.eps[q * a.nprobe]) : 0.f;
  classify_pairs(a, p2, q, T, mean_t, lane, 32);
}

// ---------------------------------------------------------------- final

struct FinalArgs {
  int64_t nq, dim;
  int nprobe, k, M, Mp, nchunk, dsub, cap, fin, quantised;  // fin: candidates evaluated by the exact rules, at most
  const int32_t* npq; const int32_t* kpq;
  const int32_t* probes; const float* d2; const uint8_t* bits; const float* eps; const float* eps0;
  const float* thr;
  const int* ntake;
  const int* qcnt; const uint2* cand;
  const float* Q; const float* books; const float* ltab; const float* qt;
  const uint8_t* codes; const int64_t* ids; const int64_t* tile_off; const int64_t* vec_off;
  int fin_warp;
  int32_t* quant_list; int* nquant;              // queries of a mixed batch for final_kernel, or null
  int32_t* over; int* nover; uint8_t* overflag;  // queries for the scanning kernels
  int64_t* over_i; float* over_d;                // their padding, or null
  int64_t* ids_out; float* dists_out;
};

// T'[m][code] of the vector's sub-spaces in ascending m, fed to f(m, T').
// DS: dsub when 2, 4 or 8 (0: any); QT: 2 Q_q from the query's table, else
// formed from the codebook by the table's rule.
template <int DS, bool QT, typename F>
__device__ __forceinline__ void each_entry(const FinalArgs& a, const float* qs, const float* qt, const float* P,
                                           const uint8_t* code, F f) {
  for (int c = 0; c < a.nchunk; ++c, code += kTileChunkBytes) {
    const uint4 w = __ldg((const uint4*)code);
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int m = c * 16 + i;
      if (m < a.M) {
        const int e = m * kKsub + (int)((ww[i >> 2] >> (8 * (i & 3))) & 0xFFu);
        float q2;
        if constexpr (QT) {
          q2 = __ldg(qt + e);
        } else {
          float acc = 0.f;
          if constexpr (DS == 2) {
            const float2 y = __ldg((const float2*)a.books + e);
            acc = add_rn(acc, mul_rn(qs[m * 2], y.x));
            acc = add_rn(acc, mul_rn(qs[m * 2 + 1], y.y));
          } else if constexpr (DS == 4 || DS == 8) {
#pragma unroll
            for (int j = 0; j < DS; j += 4) {
              const float4 y = __ldg((const float4*)(a.books + (size_t)e * DS + j));
              acc = add_rn(acc, mul_rn(qs[m * DS + j], y.x));
              acc = add_rn(acc, mul_rn(qs[m * DS + j + 1], y.y));
              acc = add_rn(acc, mul_rn(qs[m * DS + j + 2], y.z));
              acc = add_rn(acc, mul_rn(qs[m * DS + j + 3], y.w));
            }
          } else {
            for (int j = 0; j < a.dsub; ++j)
              acc = add_rn(acc, mul_rn(qs[m * a.dsub + j], __ldg(a.books + (size_t)e * a.dsub + j)));
          }
          q2 = mul_rn(2.f, acc);
        }
        f(m, sub_rn(__ldg(P + e), q2));
      }
    }
  }
}

constexpr int kFinalThreads = 256, kFinalWarps = kFinalThreads / 32;
size_t final_smem(int64_t dim, int64_t Mp, int fin, int batch) {
  return (size_t)fin * 20 + (size_t)((dim + 3) & ~int64_t(3)) * 4 + (size_t)kFinalWarps * batch * Mp * 4;
}

// Minimum and maximum over the warp (NaN ignored like fminf, fmaxf).
__device__ __forceinline__ float redux_min(float v) {
  float r;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ float redux_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// Row statistics of the tables of n <= N quantised pairs of a query (one warp):
// the row minima to bias[u * Mp + m], and the largest row range of each. One
// pair: two of its rows in flight; four: a row of each, which share the row of 2
// Q_q. What bounds this is L2 reads (1 KB a row and pair, P_l and partly 2 Q_q
// also from HBM) and their latency.
template <int N>
__device__ __forceinline__ void pair_stats(const float* const (&P)[N], int n, const float* qt, int M, int Mp,
                                           float* bias, float (&range)[N]) {
  constexpr int R = N == 1 ? 2 : 1;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < N; ++u) range[u] = 0.f;
  for (int m0 = 0; m0 < M; m0 += R) {
    float qr[R][8], pr[N][R][8];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int m = min(m0 + r, M - 1);
      ldg_row8(qt + m * kKsub, lane, qr[r]);
#pragma unroll
      for (int u = 0; u < N; ++u)
        if (u < n) ldg_row8(P[u] + m * kKsub, lane, pr[u][r]);
    }
#pragma unroll
    for (int u = 0; u < N; ++u) {
      if (u >= n) break;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float lo = sub_rn(pr[u][r][0], qr[r][0]), hi = lo;
#pragma unroll
        for (int e = 1; e < 8; ++e) {
          const float t = sub_rn(pr[u][r][e], qr[r][e]);
          lo = fminf(lo, t);
          hi = fmaxf(hi, t);
        }
        lo = redux_min(lo);
        // max over entries of fl32(t - lo) = fl32(max t - lo): rounding is monotone
        range[u] = fmaxf(range[u], sub_rn(redux_max(hi), lo));
        if (lane == 0) bias[u * Mp + min(m0 + r, M - 1)] = lo;
      }
    }
  }
  __syncwarp();
}

// A warp's batch of pairs, in shared memory.
template <int N>
struct PairBatch {
  int j[N], l[N], c0[N + 1];  // rank, list, first candidate of the batch's list (prefix)
  float s32[N], delta[N], B32[N], reach[N];
};

__device__ __forceinline__ const uint8_t* code_of(const FinalArgs& a, int l, uint32_t pos) {
  return a.codes + (((size_t)a.tile_off[l] + pos / kTileVecs) * a.nchunk) * kTileChunkBytes + (pos % kTileVecs) * kChunkBytes;
}

// The FP32 rule's distance of a vector, and the quantised rule's.
template <int DS>
__device__ __forceinline__ float exact_f32(const FinalArgs& a, const float* qs, const float* P, const uint8_t* code,
                                           float d2) {
  float acc = 0.f;
  each_entry<DS, false>(a, qs, nullptr, P, code, [&](int, float t) { acc = add_rn(acc, t); });
  return add_rn(d2, acc);
}
__device__ __forceinline__ float exact_quant(const FinalArgs& a, const float* qt, const float* P, const uint8_t* code,
                                             const float* bias, float s32, float delta, float B32) {
  int S = 0;
  each_entry<0, true>(a, nullptr, qt, P, code, [&](int m, float t) {
    // rint of a value in [0, 2^22): the low bits of fl32(x + 1.5 * 2^23)
    S += (int)(__float_as_uint(add_rn(mul_rn(sub_rn(t, bias[m]), s32), 12582912.0f)) - 0x4B400000u);
  });
  return add_rn(mul_rn(delta, __int2float_rn(S)), B32);
}

// The statistics and scales of the n pairs in bt (ranks bt.j, lists bt.l): one
// warp; ranges returned for the callers' bounds.
template <int N>
__device__ __forceinline__ void settle_pairs(const FinalArgs& a, int64_t row, int n, const float* qt, float* bias,
                                             PairBatch<N>& bt, float (&range)[N]) {
  const int lane = threadIdx.x & 31;
  const float* P[N];
#pragma unroll
  for (int u = 0; u < N; ++u) P[u] = a.ltab + (size_t)bt.l[u < n ? u : 0] * a.Mp * kKsub;
  pair_stats<N>(P, n, qt, a.M, a.Mp, bias, range);
#pragma unroll
  for (int u = 0; u < N; ++u) {
    if (u >= n) break;
    const int64_t p = row + bt.j[u];
    const float B32 = warp_exact_sum(bias + u * a.Mp, a.M, a.d2[p], true);
    if (lane == 0) {
      const float L = (float)((1 << a.bits[p]) - 1);
      bt.s32[u] = range[u] > 0.f ? __fdiv_rn(L, range[u]) : 0.f;
      bt.delta[u] = range[u] > 0.f ? __fdiv_rn(range[u], L) : 0.f;
      bt.B32[u] = B32;
    }
  }
  __syncwarp();
}

// warp_kth over n keys of f(e), e < n (one warp).
template <typename F>
__device__ __forceinline__ float warp_kth_of(int n, int kq, F f) {
  if (n < kq) return INFINITY;
  const int lane = threadIdx.x & 31;
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
  for (int e = lane; e < n; e += 32) {
    const uint32_t k = f(e);
    lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  while (hi - lo > 255u) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
    for (int e = lane; e < n; e += 32) c += f(e) <= mid ? 1 : 0;
    if ((int)__reduce_add_sync(kFull, c) >= kq) hi = mid;
    else lo = mid + 1u;
  }
  return __uint_as_float(hi);
}

// The same by the whole block, VPT keys per thread (absent ones all ones).
template <int VPT>
__device__ __forceinline__ float block_kth(const uint32_t (&key)[VPT], int kq, int (*wsum)[32]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    lo = min(lo, key[i]);
    hi = max(hi, key[i] == 0xFFFFFFFFu ? 0u : key[i]);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  if (lane == 0) {
    wsum[0][warp] = (int)lo;
    wsum[1][warp] = (int)hi;
  }
  __syncthreads();
  for (int w = 0; w < kFinalWarps; ++w) {
    lo = min(lo, (uint32_t)wsum[0][w]);
    hi = max(hi, (uint32_t)wsum[1][w]);
  }
  __syncthreads();
  for (int step = 0; hi - lo > 255u; ++step) {  // one barrier a step: the sums alternate
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
#pragma unroll
    for (int i = 0; i < VPT; ++i) c += key[i] <= mid ? 1 : 0;
    c = __reduce_add_sync(kFull, c);
    if (lane == 0) wsum[step & 1][warp] = c;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < kFinalWarps; ++w) t += wsum[step & 1][w];
    if (t >= kq) hi = mid;
    else lo = mid + 1u;
  }
  return __uint_as_float(hi);
}

// One block per query: the candidates that can still be in the top-k, their
// distances by the exact rules, and their ranks by (distance, id). FP32 pairs
// take a thread per candidate. Quantised pairs are settled by warps, four at a
// time in probe order and without block barriers: the row statistics of their
// tables, then their candidates, whose bounds now use the pairs' true ranges;
// every finished batch lowers T to the k-th exact distance so far, and a pair
// none of whose candidates reaches T is skipped. `cap` <= VPT * kFinalThreads.
template <int VPT, int DS, int BATCH>
__device__ __forceinline__ void final_query(const FinalArgs& a, const int64_t q) {
  __shared__ int wsum[2][32];
  __shared__ float kj[ANNS_MAX_NPROBE], tj[ANNS_MAX_NPROBE];
  __shared__ int coff[ANNS_MAX_NPROBE + 1], cfill[ANNS_MAX_NPROBE];
  __shared__ int nvalid, next_pair, npairs_s;
  __shared__ PairBatch<BATCH> batch[kFinalWarps];
  __shared__ int T_s;  // T's bits (T >= 0: they order like the value)
  int64_t* cid = (int64_t*)anns_dyn_smem;
  float* cdist = (float*)(cid + a.fin);        // D~ - D2
  float* cex = cdist + a.fin;                  // the exact distance, +inf until it is known (and if it never is)
  uint32_t* cjp = (uint32_t*)(cex + a.fin);
  float* qs = (float*)(cjp + a.fin);
  const int64_t row = q * a.nprobe;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* bias = qs + ((a.dim + 3) & ~int64_t(3)) + warp * BATCH * a.Mp;
  const int kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  const int nc = a.ntake[q] > 0 ? a.qcnt[q] : 0;
  auto leave = [&]() {  // to the scanning kernels
    if (tid == 0) a.over[atomicAdd(a.nover, 1)] = (int32_t)q;
    if (tid == 0) a.overflag[q] = 1;
    if (a.over_i)
      for (int e = tid; e < a.k; e += kFinalThreads) {
        a.over_i[q * a.k + e] = -1;
        a.over_d[q * a.k + e] = INFINITY;
      }
  };
  if (nc > a.cap) {
    leave();
    return;
  }
  if (tid == 0) {
    nvalid = 0;
    next_pair = 0;
    T_s = 0x7F800000;
    if (nc > 0) T_s = (int)bound_key(a.thr[q]);
  }
  for (int d = tid; d < a.dim; d += kFinalThreads) qs[d] = a.Q[q * a.dim + d];
  for (int j = tid; j < a.nprobe; j += kFinalThreads) {
    kj[j] = __fadd_ru(a.d2[row + j], a.eps[row + j]);
    cfill[j] = 0;
  }
  __syncthreads();
  const uint2* cand = a.cand + q * a.cap;
  auto ub_key = [&](int e) {
    const uint2 c = cand[e];
    return bound_key(__fadd_ru(__uint_as_float(c.y), kj[c.x >> kPosBits]));
  };
  if (nc > kq) {
    float T;
    if (nc <= 256) {
      T = warp == 0 ? warp_kth_of(nc, kq, ub_key) : INFINITY;
    } else {
      uint32_t key[VPT];
#pragma unroll
      for (int i = 0; i < VPT; ++i) {
        const int e = tid + kFinalThreads * i;
        key[i] = e < nc ? ub_key(e) : 0xFFFFFFFFu;
      }
      T = block_kth<VPT>(key, kq, wsum);
    }
    if (tid == 0) T_s = min(T_s, (int)bound_key(T));
    __syncthreads();
  }
  // candidates within reach of T, grouped by pair
  {
    const float T = __int_as_float(T_s);
    for (int j = tid; j < a.nprobe; j += kFinalThreads)
      tj[j] = __fadd_ru(__fadd_ru(T, a.eps[row + j]), -a.d2[row + j]);
  }
  __syncthreads();
  for (int e = tid; e < nc; e += kFinalThreads) {
    const uint2 c = cand[e];
    const int j = c.x >> kPosBits;
    if (!(__uint_as_float(c.y) > tj[j])) atomicAdd(&cfill[j], 1);
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0, np = 0;
    for (int j0 = 0; j0 < a.nprobe; j0 += 32) {
      const int j = j0 + lane, v = j < a.nprobe ? cfill[j] : 0;
      np += __popc(__ballot_sync(kFull, v > 0));
      int x = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
      }
      if (j < a.nprobe) {
        coff[j] = base + x - v;
        cfill[j] = base + x - v;
      }
      base += __shfl_sync(kFull, x, 31);
    }
    if (lane == 0) {
      coff[a.nprobe] = base;
      npairs_s = np;
    }
  }
  __syncthreads();
  const int ns = coff[a.nprobe];
  if (ns > a.fin) {
    leave();
    return;
  }
  constexpr uint32_t kPosMask = (1u << kPosBits) - 1u;
  for (int e = tid; e < nc; e += kFinalThreads) {
    const uint2 c = cand[e];
    const int j = c.x >> kPosBits;
    if (!(__uint_as_float(c.y) > tj[j])) {
      const int at = atomicAdd(&cfill[j], 1);
      cjp[at] = c.x;
      cdist[at] = __uint_as_float(c.y);
      cex[at] = INFINITY;
    }
  }
  __syncthreads();
  const float* qt = a.qt + (size_t)q * a.Mp * kKsub;
  // ids, and the distances of the FP32 pairs
  for (int i = tid; i < ns; i += kFinalThreads) {
    const uint32_t w = cjp[i], pos = w & kPosMask;
    const int64_t p = row + (w >> kPosBits);
    const int l = a.probes[p];
    cid[i] = a.ids[a.vec_off[l] + pos];
    if (a.bits[p]) continue;
    cex[i] = exact_f32<DS>(a, qs, a.ltab + (size_t)l * a.Mp * kKsub, code_of(a, l, pos), a.d2[p]);
  }
  if (a.quantised) {
    __syncthreads();
    PairBatch<BATCH>& bt = batch[warp];
    const int most = min(BATCH, max(1, npairs_s / (2 * kFinalWarps)));  // few pairs: spread over the warps
    for (bool more = true; more;) {
      // the next pairs, in probe order, with a candidate within reach of T
      int n = 0;
      while (n < most) {
        int j = 0;
        if (lane == 0) j = atomicAdd(&next_pair, 1);
        j = __shfl_sync(kFull, j, 0);
        if (j >= a.nprobe) {
          more = false;
          break;
        }
        const int c0 = coff[j], c1 = coff[j + 1];
        if (c0 == c1 || a.bits[row + j] == 0) continue;
        const float t0 = __fadd_ru(__fadd_ru(__int_as_float(*(volatile int*)&T_s), a.eps[row + j]), -a.d2[row + j]);
        bool near = false;
        for (int i = c0 + lane; i < c1; i += 32) near = near || !(cdist[i] > t0);
        if (!__any_sync(kFull, near)) continue;
        if (lane == 0) {
          bt.j[n] = j;
          bt.l[n] = a.probes[row + j];
          bt.c0[n + 1] = c1 - c0;
        }
        ++n;
      }
      if (n == 0) break;
      __syncwarp();
      float range[BATCH];
      settle_pairs<BATCH>(a, row, n, qt, bias, bt, range);
      const float T = __int_as_float(*(volatile int*)&T_s);
      if (lane == 0) {
        int at = 0;
        for (int u = 0; u < n; ++u) {  // the pair's true range now bounds its candidates
          const int64_t p = row + bt.j[u];
          bt.reach[u] = __fadd_ru(__fadd_ru(T, a.eps0[p] + quant_eps(a.M, a.bits[p], range[u] * 1.0001f)), -a.d2[p]);
          const int c = bt.c0[u + 1];
          bt.c0[u] = at;
          at += c;
        }
        bt.c0[n] = at;
      }
      __syncwarp();
      bool lower = false;
      for (int e = lane; e < bt.c0[n]; e += 32) {  // the batch's candidates, one per lane
        int u = 0;
        while (e >= bt.c0[u + 1]) ++u;
        const int i = coff[bt.j[u]] + e - bt.c0[u];
        if (cdist[i] > bt.reach[u]) continue;
        const float d = exact_quant(a, qt, a.ltab + (size_t)bt.l[u] * a.Mp * kKsub, code_of(a, bt.l[u], cjp[i] & kPosMask),
                                    bias + u * a.Mp, bt.s32[u], bt.delta[u], bt.B32[u]);
        *(volatile float*)&cex[i] = d;  // other warps may read it: +inf or d, either is a valid bound
        lower = lower || d < T;
      }
      __syncwarp();
      if (__any_sync(kFull, lower)) {
        const float Tn = warp_kth_of(ns, kq, [&](int e) { return bound_key(*(volatile float*)&cex[e]); });
        if (lane == 0) atomicMin(&T_s, (int)bound_key(Tn));
      }
    }
  }
  __syncthreads();
  int64_t* oi = a.ids_out + q * a.k;
  float* od = a.dists_out + q * a.k;
  for (int i = tid; i < ns; i += kFinalThreads) {
    const float d = cex[i];
    if (!(d < INFINITY)) continue;  // +inf and NaN never enter a top-k
    const int64_t id = cid[i];
    int rank = 0;
    for (int e = 0; e < ns; ++e) {
      const float d2 = cex[e];
      rank += d2 < d || (d2 == d && (cid[e] < id || (cid[e] == id && e < i))) ? 1 : 0;
    }
    atomicAdd(&nvalid, 1);
    if (rank < kq) {
      oi[rank] = id;
      od[rank] = d;
    }
  }
  __syncthreads();
  for (int e = min(nvalid, kq) + tid; e < a.k; e += kFinalThreads) {
    oi[e] = -1;
    od[e] = INFINITY;
  }
}

// Block = query; LIST: the blocks walk the *nquant queries of quant_list.
template <int VPT, int DS, int BATCH, bool LIST>
__global__ void __launch_bounds__(kFinalThreads, BATCH == 1 ? 4 : 2) final_kernel(const FinalArgs a) {
  if constexpr (!LIST) {
    final_query<VPT, DS, BATCH>(a, blockIdx.x);
  } else {
    const int n = *a.nquant;
    for (int i = blockIdx.x; i < n; i += gridDim.x) {
      final_query<VPT, DS, BATCH>(a, a.quant_list[i]);
      __syncthreads();  // the next query overwrites the shared state
    }
  }
}

// final_kernel for queries without quantised candidates: one warp per query (a
// few dozen candidates and about k survivors leave most of a block idle, and its
// barriers took half the time). `fin` as there, `fin_warp` of them here. With
// quant_list, a query that has quantised survivors, or too many, goes on to
// final_kernel through that list.
constexpr int kFWarps = 4;
template <int DS>
__global__ void __launch_bounds__(kFWarps * 32) final_fp32_kernel(const FinalArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * kFWarps + warp;
  if (q >= a.nq) return;
  const int64_t row = q * a.nprobe;
  const size_t per = (size_t)a.fin_warp * 16 + (size_t)((a.dim + 3) & ~int64_t(3)) * 4;
  int64_t* cid = (int64_t*)(anns_dyn_smem + warp * per);
  float* cex = (float*)(cid + a.fin_warp);
  uint32_t* cjp = (uint32_t*)(cex + a.fin_warp);  // first the keys of the upper bounds
  float* qs = (float*)(cjp + a.fin_warp);
  const int kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  const int nc = a.ntake[q] > 0 ? a.qcnt[q] : 0;
  const uint2* cand = a.cand + q * a.cap;
  float T = nc > 0 ? a.thr[q] : INFINITY;
  int ns = 0;
  bool over = nc > a.cap, quant = false;
  if (!over) {
    for (int d = lane; d < a.dim; d += 32) qs[d] = a.Q[q * a.dim + d];
    auto ub_key = [&](int e) {
      const uint2 c = cand[e];
      const int64_t p = row + (c.x >> kPosBits);
      return bound_key(__fadd_ru(__uint_as_float(c.y), __fadd_ru(a.d2[p], a.eps[p])));
    };
    if (nc > kq) {
      if (nc <= a.fin_warp) {
        for (int e = lane; e < nc; e += 32) cjp[e] = ub_key(e);
        __syncwarp();
        T = fminf(T, warp_kth_of(nc, kq, [&](int e) { return cjp[e]; }));
        __syncwarp();
      } else {
        T = fminf(T, warp_kth_of(nc, kq, ub_key));
      }
    }
    for (int e0 = 0; e0 < nc; e0 += 32) {
      const int e = e0 + lane;
      uint32_t w = 0;
      bool in = false;
      if (e < nc) {
        const uint2 c = cand[e];
        const int64_t p = row + (c.x >> kPosBits);
        w = c.x;
        in = !(__uint_as_float(c.y) > __fadd_ru(__fadd_ru(T, a.eps[p]), -a.d2[p]));
        quant = quant || (in && a.bits[p] != 0);
      }
      const unsigned m = __ballot_sync(kFull, in);
      const int at = ns + __popc(m & ((1u << lane) - 1u));
      if (in && at < a.fin_warp) cjp[at] = w;
      ns += __popc(m);
    }
    over = ns > a.fin_warp;
    quant = __any_sync(kFull, quant);
  }
  if (a.quant_list && (over || quant)) {
    if (lane == 0) a.quant_list[atomicAdd(a.nquant, 1)] = (int32_t)q;
    return;
  }
  if (over) {
    if (lane == 0) {
      a.over[atomicAdd(a.nover, 1)] = (int32_t)q;
      a.overflag[q] = 1;
    }
    return;
  }
  __syncwarp();
  constexpr uint32_t kPosMask = (1u << kPosBits) - 1u;
  int valid = 0;
  for (int i = lane; i < ns; i += 32) {
    const uint32_t w = cjp[i], pos = w & kPosMask;
    const int64_t p = row + (w >> kPosBits);
    const int l = a.probes[p];
    cid[i] = a.ids[a.vec_off[l] + pos];
    const float d = exact_f32<DS>(a, qs, a.ltab + (size_t)l * a.Mp * kKsub, code_of(a, l, pos), a.d2[p]);
    cex[i] = d;
    valid += d < INFINITY ? 1 : 0;
  }
  valid = __reduce_add_sync(kFull, valid);
  __syncwarp();
  int64_t* oi = a.ids_out + q * a.k;
  float* od = a.dists_out + q * a.k;
  for (int i = lane; i < ns; i += 32) {
    const float d = cex[i];
    if (!(d < INFINITY)) continue;  // +inf and NaN never enter a top-k
    const int64_t id = cid[i];
    int rank = 0;
    for (int e = 0; e < ns; ++e) {
      const float d2 = cex[e];
      rank += d2 < d || (d2 == d && (cid[e] < id || (cid[e] == id && e < i))) ? 1 : 0;
    }
    if (rank < kq) {
      oi[rank] = id;
      od[rank] = d;
    }
  }
  for (int e = min(valid, kq) + lane; e < a.k; e += 32) {
    oi[e] = -1;
    od[e] = INFINITY;
  }
}

// threshold_kernel for batches with quantised tables: the bounds of such pairs
// are wide by the quantiser's term on either side (2 eps between D~ - eps and
// T), so T comes from the exact distances of the vectors with the kq smallest
// bounds instead. One block per query, a warp per pair.
constexpr int kTWarps = 4, kExact = 512;
size_t threshold_smem(int take, int64_t dim, int64_t Mp) {
  return (size_t)take * 4 + (size_t)((dim + 3) & ~int64_t(3)) * 4 + (size_t)kTWarps * Mp * 4;
}
template <int DS>
__global__ void __launch_bounds__(kTWarps * 32) threshold_exact_kernel(const PlanArgs a, const PassArgs p2,
                                                                       const FinalArgs f, const float* __restrict__ ub) {
  __shared__ uint32_t dex[kExact];
  __shared__ int wsum[2][kTWarps], ndex;
  __shared__ float wmean[kTWarps], T_s;
  __shared__ PairBatch<1> batch[kTWarps];
  __shared__ int hits[kTWarps][64];
  uint32_t* key = (uint32_t*)anns_dyn_smem;
  float* qs = (float*)(key + a.take);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* bias = qs + ((a.dim + 3) & ~int64_t(3)) + warp * f.Mp;
  const int64_t q = blockIdx.x, row = q * a.nprobe;
  const int n = a.ntake[q], kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  if (tid == 0) ndex = 0;
  for (int d = tid; d < a.dim; d += kTWarps * 32) qs[d] = a.Q[q * a.dim + d];
  float sum = 0.f;
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
  for (int e = tid; e < n; e += kTWarps * 32) {
    const float u = ub[q * a.take + e];
    const uint32_t k = bound_key(u);
    key[e] = k;
    lo = min(lo, k);
    hi = max(hi, k);
    sum += u;
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  if (lane == 0) {
    wmean[warp] = sum;
    wsum[0][warp] = (int)lo;
    wsum[1][warp] = (int)hi;
  }
  __syncthreads();
  sum = 0.f;
  for (int w = 0; w < kTWarps; ++w) {
    lo = min(lo, (uint32_t)wsum[0][w]);
    hi = max(hi, (uint32_t)wsum[1][w]);
    sum += wmean[w];
  }
  __syncthreads();
  if (n < kq) hi = 0x7F800000u;
  for (int step = 0; n >= kq && hi - lo > 255u; ++step) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
    for (int e = tid; e < n; e += kTWarps * 32) c += key[e] <= mid ? 1 : 0;
    c = __reduce_add_sync(kFull, c);
    if (lane == 0) wsum[step & 1][warp] = c;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < kTWarps; ++w) t += wsum[step & 1][w];
    if (t >= kq) hi = mid;
    else lo = mid + 1u;
  }
  // the exact distances of the vectors whose bounds are <= hi
  const float* qt = f.qt + (size_t)q * f.Mp * kKsub;
  auto keep = [&](float d) {
    const int at = atomicAdd(&ndex, 1);
    if (at < kExact) dex[at] = bound_key(d);
  };
  PairBatch<1>& bt = batch[warp];
  const bool some = n >= kq && hi < 0x7F800000u;
  for (int j = warp; some && j < a.nprobe; j += kTWarps) {
    const int64_t p = row + j;
    const int2 t = a.sel[p];
    if (t.x == 0) continue;
    const int e0 = t.y - (int)(q * a.take), l = a.probes[p], b = a.bits[p];
    const float* P = f.ltab + (size_t)l * f.Mp * kKsub;
    bool settled = false;
    // 32 of the pair's vectors at a time (one by one as they come, a few lanes
    // of a warp would wait out the whole chain of table reads)
    auto settle = [&](int c) {
      if (b > 0 && !settled) {
        if (lane == 0) {
          bt.j[0] = j;
          bt.l[0] = l;
        }
        __syncwarp();
        float range[1];
        settle_pairs<1>(f, row, 1, qt, bias, bt, range);
        settled = true;
      }
      if (lane < c) {
        const uint8_t* code = code_of(f, l, (uint32_t)(hits[warp][lane] - e0));
        keep(b > 0 ? exact_quant(f, qt, P, code, bias, bt.s32[0], bt.delta[0], bt.B32[0])
                   : exact_f32<DS>(f, qs, P, code, a.d2[p]));
      }
      __syncwarp();
    };
    int c = 0;
    for (int eb = e0; eb < e0 + t.x; eb += 32) {
      const int e = eb + lane;
      const bool hit = e < e0 + t.x && key[e] <= hi;
      const unsigned m = __ballot_sync(kFull, hit);
      if (hit) hits[warp][c + __popc(m & ((1u << lane) - 1u))] = e;
      c += __popc(m);
      __syncwarp();
      if (c >= 32) {
        settle(32);
        c -= 32;
        const int rest = lane < c ? hits[warp][32 + lane] : 0;
        __syncwarp();
        if (lane < c) hits[warp][lane] = rest;
        __syncwarp();
      }
    }
    if (c > 0) settle(c);
  }
  __syncthreads();
  if (warp == 0) {
    const float T = warp_kth_of(min(ndex, kExact), kq, [&](int e) { return dex[e]; });
    if (lane == 0) {
      T_s = fminf(T, __uint_as_float(hi));
      a.thr[q] = T_s;
    }
  }
  __syncthreads();
  const float mean_t = n > 0 ? sum / (float)n - (a.d2[row] + a.eps[row]) : 0.f;
  classify_pairs(a, p2, q, T_s, mean_t, tid, kTWarps * 32);
}

// ---------------------------------------------------------------- host side

struct FilterWork {
  size_t bytes = 0, zero_bytes = 0;
  char* base = nullptr;
  template <typename T> T* take(size_t n) {
    T* p = (T*)(base + bytes);
    bytes += (n * sizeof(T) + 255) & ~size_t(255);
    return p;
  }
  int *qcnt, *nover;
  uint8_t *alive, *overflag, *in2;
  int* ntake;
  float *eps, *eps0, *thr, *ub, *qrows;
  int2* sel;
  PassArgs p1{}, p2{};
  uint2* cand;
  int32_t *over, *quant;
  void* Qf;
};

// Vectors of GEMM 1 per query: more of them lower T and with it the candidates
// of GEMM 2, at the cost of reading more rows twice. How much is saved depends on
// the data, what it costs on how many of the rows stay in L2 between the groups
// that share them. Whole plain search, k 10, 10000 queries, 32 probes, 1024 / 2048
// vectors, by the bytes of the rows (L2: 129 MB):
//   D 96, Deep-shaped:  24 MB 636 / 587 us, 96 MB 785 / 742, 192 MB 1102 / 1101,
//                       384 MB 1154 / 885, 576 MB 882 / 941, 960 MB 934 / 1005,
//                       1.9 GB 1162 / 1265
//   D 128, SIFT-shaped: 32 MB 717 / 665, 128 MB 923 / 853, 260 MB 1339 / 947, 512 MB
//                       1616 / 1139, 1 GB 1868 / 1290
//   D 384, embeddings:  768 MB 1401 / 1307 (8 probes 864 / 891); D 768, 1.5 GB 1843 / 1869
// so 2048 up to half a gigabyte, where it was never slower.
int filter_take(const Index& ix, int k) {
  const bool few_rows = (double)ix.ntiles * kTileVecs * ix.fl_w * 2.0 <= 537e6;
  return k <= 16 ? (few_rows ? 2048 : 1024) : k <= 32 ? 2048 : kTakeMax;
}
int filter_fin(int k) { return k <= 32 ? 1024 : 2048; }
int filter_cap(int k) { return k <= 32 ? 2048 : 4096; }

// Upper bounds of the slots and of the items of a GEMM over lists of at most
// `tiles` vector tiles each, `all` in total.
int64_t max_slots(const Index& ix, int64_t P) { return P + 15 * std::min(P, ix.nlist); }
int64_t max_items(const Index& ix, int64_t P, int64_t nq, int64_t tiles) {
  const int64_t all = std::min<int64_t>(ix.fl_tiles, ix.nlist * tiles);
  return std::min(all, P * tiles) + std::min(tiles * (P / kGq), all * (nq / kGq)) + 1;
}

FilterWork filter_work(const Index& ix, int64_t nq, int nprobe, int k, char* base) {
  FilterWork w;
  w.base = base;
  const int64_t P = nq * nprobe, G = max_slots(ix, P), L = ix.nlist, Dp = coarse_tc_dp(ix, ANNS_PREC_FP16);
  const int64_t tiles = (ix.max_list + kTv - 1) / kTv, t1 = std::min<int64_t>(tiles, (filter_take(ix, k) + kTv - 1) / kTv);
  for (PassArgs* p : {&w.p1, &w.p2}) {
    p->cnt = w.take<int>(L);
    p->fill = w.take<int>(L);
  }
  w.qcnt = w.take<int>(nq); w.nover = w.take<int>(2);  // and the count of `quant`
  w.alive = w.take<uint8_t>(P);
  w.overflag = w.take<uint8_t>(nq);
  w.zero_bytes = w.bytes;
  for (PassArgs* p : {&w.p1, &w.p2}) {
    p->tiles = (int)(p == &w.p1 ? t1 : tiles);
    p->s0 = w.take<int>(L + 1);
    p->i0 = w.take<int>(L + 1);
    p->kc = w.take<float2>(G);
    if (p == &w.p1) p->d1 = w.take<int2>(G);
    else p->pair = w.take<int>(G);
    p->rows = w.take<__half>(G * Dp);
    p->items = w.take<FItem>(max_items(ix, P, nq, p->tiles));
  }
  w.ntake = w.take<int>(nq); w.in2 = w.take<uint8_t>(P);
  w.eps = w.take<float>(P); w.eps0 = w.take<float>(P); w.thr = w.take<float>(nq); w.ub = w.take<float>(nq * filter_take(ix, k));
  w.sel = w.take<int2>(P);
  w.cand = w.take<uint2>(nq * filter_cap(k));
  w.over = w.take<int32_t>(nq); w.quant = w.take<int32_t>(nq);
  w.qrows = w.take<float>(3 * nq);
  w.Qf = w.take<__half>(nq * Dp);
  return w;
}

// Four pairs to a warp share the reading of a query's table rows, one pair to a
// warp keeps twice the blocks resident. Four pay where a query has candidates in
// most of many probes of wide tables, and cost a quarter on narrow ones (whole
// search, fixed 8 bits, 2000 queries, 1M vectors, one / four pairs a warp):
//   M 96, D 768 (embeddings): k 64, 16, 32, 64 probes 2816 / 2984, 3709 / 3527, 5450 /
//     4229 us; k 100, 64 probes 6028 / 4578; k 40, 64 probes 4906 / 3917; k 10 2336 / 2916
//   M 120, D 960 (GIST-shaped): 64 probes, k 64 11322 / 11711, k 100 14018 / 14406
//   M 48, D 96: 64 probes, k 64 751 / 999, k 128 1216 / 1514; M 32, D 128: k 64 1162 / 1432
template <int VPT>
cudaError_t run_final_ds(const FinalArgs& a, cudaStream_t s) {
  const int batch = a.Mp >= 96 && a.k >= 64 && a.nprobe >= 48 && !a.npq && !a.quant_list ? kBatch : 1;
  auto go = [&](auto kern) {
    const size_t sm = final_smem(a.dim, a.Mp, a.fin, batch);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    // of a list usually a part of the batch: blocks for a few waves
    kern<<<(unsigned)(a.quant_list ? std::min<int64_t>(a.nq, 2048) : a.nq), kFinalThreads, sm, s>>>(a);
    note_launch();
    return cudaGetLastError();
  };
  auto pick = [&](auto ds) {
    constexpr int DS = decltype(ds)::value;
    if (a.quant_list) return go(final_kernel<VPT, DS, 1, true>);
    if constexpr (VPT == 16) {  // k > 32
      if (batch > 1) return go(final_kernel<VPT, DS, kBatch, false>);
    }
    return go(final_kernel<VPT, DS, 1, false>);
  };
  switch (a.dsub) {
    case 2: return pick(std::integral_constant<int, 2>{});
    case 4: return pick(std::integral_constant<int, 4>{});
    case 8: return pick(std::integral_constant<int, 8>{});
    default: return pick(std::integral_constant<int, 0>{});
  }
}

cudaError_t run_final_fp32(const FinalArgs& a, cudaStream_t s) {
  auto go = [&](auto kern) {
    const size_t sm = kFWarps * ((size_t)a.fin_warp * 16 + (size_t)((a.dim + 3) & ~int64_t(3)) * 4);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((a.nq + kFWarps - 1) / kFWarps), kFWarps * 32, sm, s>>>(a);
    note_launch();
    return cudaGetLastError();
  };
  switch (a.dsub) {
    case 2: return go(final_fp32_kernel<2>);
    case 4: return go(final_fp32_kernel<4>);
    case 8: return go(final_fp32_kernel<8>);
    default: return go(final_fp32_kernel<0>);
  }
}

template <int MODE>
cudaError_t run_gemm(const Index& ix, const CUtensorMap& tmY, const CUtensorMap& tmQ, const GemmArgs& a, int64_t most,
                     cudaStream_t s) {
  int sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ix.device);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(filter_gemm_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFilterSmem);
  if (e != cudaSuccess) return e;
  filter_gemm_kernel<MODE><<<(unsigned)std::min<int64_t>(sms, most), kFThreads, kFilterSmem, s>>>(tmY, tmQ, a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

struct FilterRows {
  void* p[4] = {};
  ~FilterRows() {
    for (void* x : p)
      if (x) cudaFree(x);
  }
};

// The index's part of the filter: decoded FP16 rows and their scalars. Left
// out (the search then scans) for values that are not finite, and where the
// rows would take more than a quarter of the free device memory.
int prepare_filter(Index& ix, const std::vector<float>& cent, const std::vector<float>& books) {
  ix.fl_w = 0;
  if (ix.n == 0 || ix.max_list >= ((int64_t)1 << kPosBits) || ix.ntiles * kTileVecs > (int64_t)INT32_MAX - kTv ||
      ix.dim > 4096)
    return ANNS_OK;
  float big = 0.f;
  for (float v : cent)
    if (!std::isfinite(v)) return ANNS_OK;
  for (float v : books) {
    if (!std::isfinite(v)) return ANNS_OK;
    big = std::max(big, std::fabs(v));
  }
  int ex = 0;
  if (big > 0.f) {
    std::frexp(big, &ex);               // big in [2^(ex-1), 2^ex)
    ex = std::min(std::max(14 - ex, -100), 100);  // scaled: at most 2^14
  }
  const float up = std::ldexp(1.f, ex);
  std::vector<float> ym(ix.M);
  for (int64_t m = 0; m < ix.M; ++m) {
    double most = 0.0;
    for (int c = 0; c < kKsub; ++c) {
      double s = 0.0;
      for (int64_t j = 0; j < ix.dsub; ++j) {
        const double v = books[((size_t)m * kKsub + c) * ix.dsub + j];
        s += v * v;
      }
      most = std::max(most, s);
    }
    ym[m] = (float)(std::sqrt(most) * (1.0 + 1e-6));
  }
  std::vector<float> mu(ix.dim);
  const int W = (int)((ix.dim + 7) & ~int64_t(7));
  const int64_t rows = ix.ntiles * kTileVecs;
  const size_t yb = (size_t)rows * W * sizeof(__half);
  size_t free_b = 0, total_b = 0;
  cudaError_t e = cudaMemGetInfo(&free_b, &total_b);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemGetInfo");
  if (yb + (size_t)rows * 4 > free_b / 4) return ANNS_OK;
  auto hold = std::make_shared<FilterRows>();
  const size_t bytes[4] = {yb, (size_t)rows * sizeof(float), (size_t)ix.nlist * sizeof(float4), (size_t)ix.M * sizeof(float)};
  for (int i = 0; i < 4 && e == cudaSuccess; ++i) e = cudaMalloc(&hold->p[i], bytes[i]);
  if (e == cudaErrorMemoryAllocation) {  // no room: the index works without
    cudaGetLastError();
    return ANNS_OK;
  }
  if (e != cudaSuccess) return cuda_fail(e, "filter arrays");
  ix.fl_hold = hold;
  ix.fl_y = hold->p[0];
  ix.fl_s = (float*)hold->p[1];
  ix.fl_stat = hold->p[2];
  ix.fl_ym = (float*)hold->p[3];
  if (e == cudaSuccess) e = cudaMemcpy(ix.fl_ym, ym.data(), ix.M * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(mu.data(), ix.tc_mu, ix.dim * sizeof(float), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemset(ix.fl_stat, 0, (size_t)ix.nlist * sizeof(float4));
  if (e != cudaSuccess) return cuda_fail(e, "filter tables");
  double mu2 = 0.0;
  for (float v : mu) mu2 += (double)v * v;
  const unsigned grid = (unsigned)std::min<int64_t>(ix.ntiles, 1 << 20);
  decode_kernel<<<grid, 256>>>(ix.codes, ix.codebooks, ix.centroids, ix.tc_mu, ix.tile_off, ix.list_len, (int)ix.nlist,
                               ix.ntiles, (int)ix.dim, (int)ix.M, (int)ix.dsub, (int)ix.nchunk, W, up, (__half*)ix.fl_y,
                               ix.fl_s, (float4*)ix.fl_stat);
  note_launch();
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return cuda_fail(e, "filter rows");
  ix.fl_tiles = 0;
  for (int64_t l = 0; l < ix.nlist; ++l) ix.fl_tiles += (ix.h_list_len64[l] + kTv - 1) / kTv;
  ix.fl_w = W;
  ix.fl_yscale = std::ldexp(1.f, -ex);
  ix.fl_mu = (float)(std::sqrt(mu2) * (1.0 + 1e-6));
  return ANNS_OK;
}

void free_filter(Index& ix) {
  ix.fl_hold.reset();
  ix.fl_y = ix.fl_stat = nullptr;
  ix.fl_s = ix.fl_ym = nullptr;
  ix.fl_w = 0;
}

int restore_filter(Index& ix) {
  std::vector<float> cent((size_t)ix.nlist * ix.dim), books((size_t)ix.M * kKsub * ix.dsub);
  cudaError_t e = cudaMemcpy(cent.data(), ix.centroids, cent.size() * sizeof(float), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(books.data(), ix.codebooks, books.size() * sizeof(float), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "filter rows");
  return prepare_filter(ix, cent, books);
}

bool filter_possible(const Index& ix, const anns_precision_policy& P, int64_t nq, int nprobe, int k) {
  if (ix.fl_w == 0) return false;
  if (P.lut_mode == ANNS_LUT_FIXED_BITS && P.fixed_bits < 5) return false;  // every pair would be scanned anyway
  if (nibble_possible(P) && !grouped_supported(ix, k)) return false;
  const int64_t pairs = nq * nprobe, tiles = (ix.max_list + kTv - 1) / kTv;
  if (pairs > INT32_MAX / 2 || nq * kTakeMax > INT32_MAX || max_slots(ix, pairs) > INT32_MAX ||
      max_items(ix, pairs, nq, tiles) > ((int64_t)1 << 26))
    return false;
  return (int64_t)filter_workspace_bytes(ix, nq, nprobe, k) <= ix.opt_filter_bytes;
}

size_t filter_workspace_bytes(const Index& ix, int64_t nq, int nprobe, int k) {
  return filter_work(ix, nq, nprobe, k, nullptr).bytes;
}

cudaError_t launch_search_filter(const Index& ix, const float* Q, const float* qt, int64_t nq, int nprobe,
                                 const int32_t* nprobe_per_q, int k, const int32_t* k_per_q, const int32_t* probes,
                                 const float* probe_d2, const uint8_t* bits, void* ws, const void* q16,
                                 const float* q16_rows, bool quantised, bool exact_threshold, bool mixed, int64_t* ids_out, float* dists_out,
                                 int64_t* over_i, float* over_d, FilterResult* out, cudaStream_t s) {
  FilterWork w = filter_work(ix, nq, nprobe, k, (char*)ws);
  cudaError_t e = cudaMemsetAsync(w.base, 0, w.zero_bytes, s);
  if (e == cudaSuccess && !q16) {
    e = launch_center_fp16(ix, Q, nq, w.Qf, w.qrows, s);
    q16 = w.Qf;
    q16_rows = w.qrows;
  }
  if (e != cudaSuccess) return e;
  const int Dp = coarse_tc_dp(ix, ANNS_PREC_FP16);
  PlanArgs p{};
  p.nq = nq; p.dim = ix.dim; p.nprobe = nprobe; p.k = k; p.M = (int)ix.M; p.dsub = (int)ix.dsub; p.Dp = Dp;
  p.v4 = ix.dsub % 4 == 0 && ((uintptr_t)Q & 15u) == 0; p.take = filter_take(ix, k); p.nlist = (int)ix.nlist; p.npq = nprobe_per_q; p.kpq = k_per_q; p.probes = probes;
  p.d2 = probe_d2; p.bits = bits; p.list_len = ix.list_len; p.tile_off = ix.tile_off; p.Q = Q; p.C = ix.centroids;
  p.ym = ix.fl_ym; p.stat = (const float4*)ix.fl_stat; p.qrows = q16_rows; p.mu_norm = ix.fl_mu;
  p.yscale = ix.fl_yscale; p.eps = w.eps; p.eps0 = w.eps0; p.sel = w.sel; p.in2 = w.in2; p.ntake = w.ntake;
  p.thr = w.thr; p.alive = w.alive; p.q16 = (const __half*)q16;
  const int64_t P = nq * nprobe, slots = max_slots(ix, P);
  const int pair_blocks = (int)((P + 255) / 256);
  const unsigned scatter_grid = (unsigned)(pair_blocks + (ix.nlist + 7) / 8);
  CUtensorMap tmY, tmQ;
  e = make_tmap(&tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ix.fl_y, ix.ntiles * kTileVecs, ix.fl_w, kKE, 64);
  if (e != cudaSuccess) return e;
  GemmArgs g{};
  g.sx = ix.fl_s; g.nK = Dp / kKE; g.ksteps = (int)((ix.dim + 15) / 16); g.status = ix.dev_status;
  g.wait_limit = ix.opt_wait_cycles > 0 ? ix.opt_wait_cycles : kWaitCycles;
  g.nprobe = nprobe; g.ub = w.ub; g.qcnt = w.qcnt; g.cand = w.cand; g.cap = filter_cap(k);
  g.alive = w.alive;
  auto pass = [&](auto mode, const PassArgs& w1) {
    constexpr int MODE = decltype(mode)::value;
    plan_scan_kernel<<<1, 1024, 0, s>>>(ix.list_len, (int)ix.nlist, w1); note_launch();
    plan_scatter_kernel<MODE><<<scatter_grid, 256, 0, s>>>(p, w1, pair_blocks); note_launch();
    cudaError_t e1 = cudaGetLastError();
    if (e1 == cudaSuccess) e1 = make_tmap(&tmQ, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, w1.rows, slots, Dp, kKE, 32);
    if (e1 != cudaSuccess) return e1;
    g.items = w1.items; g.nitems = w1.i0 + ix.nlist; g.gk = w1.kc; g.gd = w1.d1; g.gp = w1.pair;
    return run_gemm<MODE>(ix, tmY, tmQ, g, max_items(ix, P, nq, w1.tiles), s);
  };
  plan_kernel<<<(unsigned)nq, 128, 0, s>>>(p, w.p1); note_launch();
  if ((e = pass(std::integral_constant<int, 1>{}, w.p1)) != cudaSuccess) return e;
  FinalArgs f{};
  f.nq = nq; f.dim = ix.dim; f.nprobe = nprobe; f.k = k; f.M = (int)ix.M; f.Mp = (int)ix.Mp; f.nchunk = (int)ix.nchunk;
  f.dsub = (int)ix.dsub; f.cap = g.cap; f.fin = filter_fin(k); f.npq = nprobe_per_q; f.kpq = k_per_q; f.probes = probes; f.d2 = probe_d2;
  f.bits = bits; f.eps = w.eps; f.eps0 = w.eps0; f.thr = w.thr; f.quantised = quantised ? 1 : 0; f.ntake = w.ntake; f.qcnt = w.qcnt; f.cand = w.cand; f.Q = Q;
  f.books = ix.codebooks; f.ltab = ix.ltab; f.qt = qt; f.codes = ix.codes; f.ids = ix.ids; f.tile_off = ix.tile_off;
  f.vec_off = ix.vec_off; f.over = w.over; f.nover = w.nover; f.ids_out = ids_out; f.dists_out = dists_out;
  f.overflag = w.overflag; f.over_i = over_i; f.over_d = over_d;
  if (exact_threshold) {
    auto go = [&](auto kern) {
      const size_t sm = threshold_smem(p.take, ix.dim, ix.Mp);
      const cudaError_t e1 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (e1 != cudaSuccess) return e1;
      kern<<<(unsigned)nq, kTWarps * 32, sm, s>>>(p, w.p2, f, w.ub);
      note_launch();
      return cudaGetLastError();
    };
    switch (ix.dsub) {
      case 2: e = go(threshold_exact_kernel<2>); break;
      case 4: e = go(threshold_exact_kernel<4>); break;
      case 8: e = go(threshold_exact_kernel<8>); break;
      default: e = go(threshold_exact_kernel<0>); break;
    }
  } else {
    const unsigned tb = (unsigned)((nq + 3) / 4);
    switch (p.take / 32) {
      case 32: threshold_kernel<32><<<tb, 128, 0, s>>>(p, w.p2, w.ub); break;
      case 64: threshold_kernel<64><<<tb, 128, 0, s>>>(p, w.p2, w.ub); break;
      default: threshold_kernel<128><<<tb, 128, 0, s>>>(p, w.p2, w.ub); break;
    }
    note_launch();
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  if ((e = pass(std::integral_constant<int, 2>{}, w.p2)) != cudaSuccess) return e;
  // a mixed batch settles the queries whose candidates are all on FP32 tables (a
  // predictor keeps those for the nearest lists) a warp each first (Deep-shaped,
  // learned widths: 383 us in blocks, 156 + 188 us so)
  f.fin_warp = k <= 32 ? 256 : 512;
  f.quant_list = quantised && mixed ? w.quant : nullptr;
  f.nquant = w.nover + 1;
  if (!quantised || mixed) e = run_final_fp32(f, s);
  if (e == cudaSuccess && quantised) e = f.cap == 2048 ? run_final_ds<8>(f, s) : run_final_ds<16>(f, s);
  out->over = w.over;
  out->nover = w.nover;
  out->alive = w.alive;
  out->overflag = w.overflag;
  out->thr = w.thr;
  return e;
}

}  // namespace anns
