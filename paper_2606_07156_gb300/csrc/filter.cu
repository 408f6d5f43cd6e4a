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
constexpr int kPosBits = 25;       // candidate word: rank << 25 | position in the list
constexpr int kTakeMax = 4096;
constexpr size_t kFilterWorkspaceMax = (size_t)32 << 30;  // larger batches scan

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
  const int32_t* npq; const int32_t* kpq;
  const int32_t* probes; const float* d2; const uint8_t* bits; const int32_t* list_len;
  const int64_t* tile_off;
  const float* Q; const float* C; const float* ym; const float4* stat; const float* qrows;
  float mu_norm, yscale;   // |mu| (rounded upward), 1 / scale of the decoded rows
  float* eps;              // [nq * nprobe], -1: the pair takes no part
  float* eps0;             // [nq * nprobe] eps without the quantiser's term
  int2* sel;               // [nq * nprobe] GEMM 1: vectors taken, where their bounds go
  int* ntake;              // [nq] bounds of the query
  int *c1, *c2, *f1, *f2;  // [nlist] pairs per list in GEMM 1 and 2, fill cursors
  int *g1, *g2, *i1, *i2;  // [nlist + 1] first slot and item of each list
  float2 *k1, *k2;         // [slots] column constants
  int2* d1;                // [slots] GEMM 1: (vectors taken, destination)
  int* p2;                 // [slots] GEMM 2: pair of each slot
  const __half* q16;       // [nq x Dp] the queries' FP16 operand
  __half *r1, *r2;         // [slots x Dp] its rows slot by slot
  int* slot2;              // [nq * nprobe] slot of each pair, -1: none
  FItem *it1, *it2;
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

// One block per query: eps of its pairs, the first `take` vectors of its probe
// sequence for GEMM 1, and the pairs counted per list.
__global__ void __launch_bounds__(128) plan_kernel(const PlanArgs a) {
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
          for (int i = 0; i < a.dsub; ++i) {
            const float e = qv[m * a.dsub + i] - cv[m * a.dsub + i];
            s += e * e;
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
      if (lane == 0) {
        a.eps0[p] = eps;
        atomicAdd(a.c2 + l, 1);
      }
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
        if (t > 0) atomicAdd(a.c1 + a.probes[p], 1);
      }
      base = __shfl_sync(kFull, incl, 31);
    }
    if (lane == 0) a.ntake[q] = base;
  }
}

// One block: exclusive prefixes over the lists of the slots and the items of
// both GEMMs (totals at [nlist]).
__global__ void __launch_bounds__(1024) plan_scan_kernel(const PlanArgs a) {
  __shared__ int part[4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry[4] = {0, 0, 0, 0};
  int* out[4] = {a.g1, a.i1, a.g2, a.i2};
  for (int base = 0; base < a.nlist; base += 1024) {
    const int l = base + threadIdx.x;
    int v[4] = {0, 0, 0, 0}, x[4];
    if (l < a.nlist) {
      const int tiles = (a.list_len[l] + kTv - 1) / kTv;
      v[0] = (a.c1[l] + 15) & ~15;
      v[1] = (a.c1[l] + kGq - 1) / kGq * min(tiles, (a.take + kTv - 1) / kTv);
      v[2] = (a.c2[l] + 15) & ~15;
      v[3] = (a.c2[l] + kGq - 1) / kGq * tiles;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = v[i];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x[i], o);
        if (lane >= o) x[i] += y;
      }
      if (lane == 31) part[i][warp] = x[i];
    }
    __syncthreads();
    if (warp < 4) {
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
    for (int i = 0; i < 4; ++i) {
      if (l < a.nlist) out[i][l] = carry[i] + (warp ? part[i][warp - 1] : 0) + x[i] - v[i];
      carry[i] += part[i][31];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int i = 0; i < 4; ++i) out[i][a.nlist] = carry[i];
}

// The first `pair_blocks` blocks: each pair to a slot of its list, a warp per
// pair, which also copies the query's FP16 row there: the GEMM then loads a
// group's rows as plain TMA boxes. (Gathering them in the GEMM by tile::gather4
// took 0.1 us per four rows, 7.6 us per 128-query tile where the whole tile now
// takes under 2.) The other blocks: the items of each list (a warp per list),
// vector tile by vector tile, so that a tile's groups follow one another.
__global__ void __launch_bounds__(256) plan_scatter_kernel(const PlanArgs a, int pair_blocks) {
  const int lane = threadIdx.x & 31;
  if ((int)blockIdx.x < pair_blocks) {
    const int64_t p = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (p >= a.nq * a.nprobe) return;
    const float eps = a.eps[p];
    if (eps == -1.f) {
      if (lane == 0) a.slot2[p] = -1;
      return;
    }
    const int q = (int)(p / a.nprobe), l = a.probes[p];
    const int2 t = a.sel[p];
    int s1 = 0, s2 = 0;
    if (lane == 0) {
      const float m2s = -2.f * (a.qrows[2 * a.nq + q] * a.yscale);
      s2 = a.g2[l] + atomicAdd(a.f2 + l, 1);
      a.p2[s2] = (int)p;
      a.slot2[p] = s2;
      a.k2[s2].y = m2s;
      if (t.x > 0) {
        s1 = a.g1[l] + atomicAdd(a.f1 + l, 1);
        a.k1[s1] = make_float2(__fadd_ru(a.d2[p], eps), m2s);
        a.d1[s1] = t;
      }
    }
    s1 = __shfl_sync(kFull, s1, 0);
    s2 = __shfl_sync(kFull, s2, 0);
    const uint4* src = (const uint4*)(a.q16 + (size_t)q * a.Dp);
    uint4* dst2 = (uint4*)(a.r2 + (size_t)s2 * a.Dp);
    uint4* dst1 = (uint4*)(a.r1 + (size_t)s1 * a.Dp);
    for (int i = lane; i < a.Dp / 8; i += 32) {
      const uint4 v = __ldg(src + i);
      dst2[i] = v;
      if (t.x > 0) dst1[i] = v;
    }
  } else {
    const int l = ((int)blockIdx.x - pair_blocks) * 8 + (threadIdx.x >> 5);
    if (l >= a.nlist) return;
    const int n_l = a.list_len[l], row = (int)(a.tile_off[l] * kTileVecs);
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int c = w ? a.c2[l] : a.c1[l], g0 = w ? a.g2[l] : a.g1[l], i0 = w ? a.i2[l] : a.i1[l];
      const int ng = (c + kGq - 1) / kGq, n = (w ? a.i2[l + 1] : a.i1[l + 1]) - i0;
      FItem* out = (w ? a.it2 : a.it1) + i0;
      for (int i = lane; i < n; i += 32) {
        const int t = i / ng, g = i % ng;
        out[i] = FItem{row + t * kTv, min(kTv, n_l - t * kTv) | (min(kGq, c - g * kGq) << 16), g0 + g * kGq, t * kTv};
      }
    }
  }
}

// ---------------------------------------------------------------- GEMM

struct GemmArgs {
  const FItem* items; const int* nitems;
  const float2* gk;
  const int2* gd; float* ub;                              // GEMM 1
  const int* gp; const uint8_t* bits; int nprobe;         // GEMM 2
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
    FItem it = load_item(a.items + blockIdx.x), nx = it;
    for (int i = blockIdx.x; i < nitems && ok; i += stride) {
      const int nv = it.nv_cnt & 0xFFFF, cnt = it.nv_cnt >> 16, nbox = (nv + 63) >> 6, qbox = (cnt + 31) >> 5;
      if (i + stride < nitems) nx = load_item(a.items + i + stride);
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
    }
    if (!ok) {
      if (lane == 0) {
        *abort_flag = 1;
        atomicExch(a.status, ANNS_DEV_TIMEOUT);
        // the copies already issued land before the CTA exits (coarse_tc.cu)
        for (uint32_t st = 0; st < kFStages; ++st) {
          const uint32_t count = g > st ? (g - st + kFStages - 1) / kFStages : 0;
          if (count > 0) mbar_wait(full0 + 8 * st, (count - 1) & 1);
        }
      }
      __syncwarp();
    }
  } else if (tid == 32) {
    // MMA issuer: this CTA's n-th item accumulates into TMEM columns (n & 1) * 256 + 128 * half
    uint32_t g = 0;
    int n = 0;
    FItem it = load_item(a.items + blockIdx.x);
    for (int i = blockIdx.x; i < nitems && ok; i += stride, ++n) {
      const int nv = it.nv_cnt & 0xFFFF, N = ((it.nv_cnt >> 16) + 15) & ~15;
      if (i + stride < nitems) it = load_item(a.items + i + stride);
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
    int2* cd = (int2*)(mine + 64 * 8);                // GEMM 1: (taken, destination); GEMM 2: (pair, marked only)
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
      for (uint32_t cols = __reduce_or_sync(kFull, mask); cols; cols &= cols - 1u) {
        const int j = __ffs(cols) - 1;
        const int2 d = dc[j0 + j];
        if (lane == 0) a.alive[d.x] = 1;
        if (d.y) continue;
        const unsigned who = __ballot_sync(kFull, mask >> j & 1u);
        const float t = fmaf(tc_ld1(tcol + j0 + j), kc[j0 + j].y, s);
        if (staged > kPush - 32) flush();
        if (mask >> j & 1u) {
          const int e = staged + __popc(who & ((1u << lane) - 1u));
          sp[e] = d.x;
          spos[e] = pos;
          sv[e] = t;
        }
        staged += __popc(who);
      }
    };
    FItem nx = load_item(a.items + blockIdx.x);
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
            const int p = __ldg(a.gp + s), b = a.bits[p];
            nd[c] = make_int2(p, b >= 1 && b <= 4);
          }
        }
      }
    };
    load_cols(nx);
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
      if (i + stride < nitems) nx = load_item(a.items + i + stride);
      // every lane waits; the warp goes on only together (tcgen05.ld is .sync.aligned)
      const bool got = mbar_wait(accf0 + 8 * b, (uint32_t)((n >> 1) & 1), a.wait_limit, abort_flag);
      if (!__all_sync(kFull, got)) {
        ok = false;
        break;
      }
      tc_fence_after();
      if (i + stride < nitems) load_cols(nx);
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

// One warp per query: T, and the column constants of the query's pairs in
// GEMM 2: D~ - eps <= T  <=>  s_x - 2 dot <= T + eps - D2 (rounded upward).
// take <= 32 VPT.
template <int VPT>
__global__ void __launch_bounds__(128) threshold_kernel(const PlanArgs a, const float* __restrict__ ub,
                                                        float* __restrict__ thr) {
  const int64_t q = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (q >= a.nq) return;
  const int n = a.ntake[q], kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  if (n == 0) return;  // no pair takes part
  uint32_t key[VPT];
#pragma unroll
  for (int i = 0; i < VPT; ++i) {
    const int e = lane + 32 * i;
    key[i] = e < n ? bound_key(ub[q * a.take + e]) : 0xFFFFFFFFu;
  }
  const float T = warp_kth<VPT>(key, n, kq);
  if (lane == 0) thr[q] = T;
  for (int j = lane; j < a.nprobe; j += 32) {
    const int64_t p = q * a.nprobe + j;
    const int s2 = a.slot2[p];
    if (s2 >= 0) a.k2[s2].x = __fadd_ru(__fadd_ru(T, a.eps[p]), -a.d2[p]);
  }
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
size_t final_smem(int64_t dim, int64_t Mp, int fin) {
  return (size_t)fin * 20 + (size_t)((dim + 3) & ~int64_t(3)) * 4 + (size_t)kFinalWarps * Mp * 4;
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
// take a thread per candidate. Quantised pairs take a warp per pair, in probe
// order: the row statistics of its table (two rows of P_l and 2 Q_q in flight;
// no block barrier, so the warps' loads overlap), then its candidates, whose
// bound now uses the pair's true range; every finished pair lowers T to the
// k-th exact distance so far, and a pair none of whose candidates reaches T is
// skipped. `cap` <= VPT * kFinalThreads.
template <int VPT, int DS>
__global__ void __launch_bounds__(kFinalThreads) final_kernel(const FinalArgs a) {
  __shared__ int wsum[2][32];
  __shared__ float kj[ANNS_MAX_NPROBE], tj[ANNS_MAX_NPROBE];
  __shared__ int coff[ANNS_MAX_NPROBE + 1], cfill[ANNS_MAX_NPROBE];
  __shared__ int nvalid, next_pair;
  __shared__ int T_s;  // T's bits (T >= 0: they order like the value)
  int64_t* cid = (int64_t*)anns_dyn_smem;
  float* cdist = (float*)(cid + a.fin);        // D~ - D2
  float* cex = cdist + a.fin;                  // the exact distance, +inf until it is known (and if it never is)
  uint32_t* cjp = (uint32_t*)(cex + a.fin);
  float* qs = (float*)(cjp + a.fin);
  const int64_t q = blockIdx.x, row = q * a.nprobe;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* bias = qs + ((a.dim + 3) & ~int64_t(3)) + warp * a.Mp;
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
    int base = 0;
    for (int j0 = 0; j0 < a.nprobe; j0 += 32) {
      const int j = j0 + lane, v = j < a.nprobe ? cfill[j] : 0;
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
    if (lane == 0) coff[a.nprobe] = base;
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
  auto code_of = [&](int l, uint32_t pos) {
    return a.codes + (((size_t)a.tile_off[l] + pos / kTileVecs) * a.nchunk) * kTileChunkBytes + (pos % kTileVecs) * kChunkBytes;
  };
  // ids, and the distances of the FP32 pairs
  for (int i = tid; i < ns; i += kFinalThreads) {
    const uint32_t w = cjp[i], pos = w & kPosMask;
    const int64_t p = row + (w >> kPosBits);
    const int l = a.probes[p];
    cid[i] = a.ids[a.vec_off[l] + pos];
    if (a.bits[p]) continue;
    float acc = 0.f;
    each_entry<DS, false>(a, qs, qt, a.ltab + (size_t)l * a.Mp * kKsub, code_of(l, pos),
                          [&](int, float t) { acc = add_rn(acc, t); });
    cex[i] = add_rn(a.d2[p], acc);
  }
  if (a.quantised) {
    __syncthreads();
    for (;;) {
      int j = 0;
      if (lane == 0) j = atomicAdd(&next_pair, 1);
      j = __shfl_sync(kFull, j, 0);
      if (j >= a.nprobe) break;
      const int c0 = coff[j], c1 = coff[j + 1];
      if (c0 == c1) continue;
      const int64_t p = row + j;
      const int b = a.bits[p];
      if (b == 0) continue;
      const float d2 = a.d2[p];
      float T = __int_as_float(*(volatile int*)&T_s);
      bool near = false;
      const float t0 = __fadd_ru(__fadd_ru(T, a.eps[p]), -d2);
      for (int i = c0 + lane; i < c1; i += 32) near = near || !(cdist[i] > t0);
      if (!__any_sync(kFull, near)) continue;  // out of reach
      const int l = a.probes[p];
      const float* P = a.ltab + (size_t)l * a.Mp * kKsub;
      float range = 0.f;
      for (int m0 = 0; m0 < a.M; m0 += 2) {
        const int m1 = min(m0 + 1, a.M - 1);
        float pr[2][8], qr[2][8];
        ldg_row8(P + m0 * kKsub, lane, pr[0]);
        ldg_row8(qt + m0 * kKsub, lane, qr[0]);
        ldg_row8(P + m1 * kKsub, lane, pr[1]);
        ldg_row8(qt + m1 * kKsub, lane, qr[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          float lo = sub_rn(pr[u][0], qr[u][0]), hi = lo;
#pragma unroll
          for (int e = 1; e < 8; ++e) {
            const float t = sub_rn(pr[u][e], qr[u][e]);
            lo = fminf(lo, t);
            hi = fmaxf(hi, t);
          }
          lo = redux_min(lo);
          // max over entries of fl32(t - lo) = fl32(max t - lo): rounding is monotone
          range = fmaxf(range, sub_rn(redux_max(hi), lo));
          if (lane == 0) bias[u ? m1 : m0] = lo;
        }
      }
      __syncwarp();
      const float B32 = warp_exact_sum(bias, a.M, d2, true);
      const float Lf = (float)((1 << b) - 1);
      const float s32 = range > 0.f ? __fdiv_rn(Lf, range) : 0.f, delta = range > 0.f ? __fdiv_rn(range, Lf) : 0.f;
      T = __int_as_float(*(volatile int*)&T_s);
      const float t1 = __fadd_ru(__fadd_ru(T, a.eps0[p] + quant_eps(a.M, b, range * 1.0001f)), -d2);
      bool lower = false;
      for (int i = c0 + lane; i < c1; i += 32) {
        if (cdist[i] > t1) continue;
        int S = 0;
        each_entry<DS, true>(a, qs, qt, P, code_of(l, cjp[i] & kPosMask), [&](int m, float t) {
          // rint of a value in [0, 2^22): the low bits of fl32(x + 1.5 * 2^23)
          S += (int)(__float_as_uint(add_rn(mul_rn(sub_rn(t, bias[m]), s32), 12582912.0f)) - 0x4B400000u);
        });
        const float d = add_rn(mul_rn(delta, __int2float_rn(S)), B32);
        *(volatile float*)&cex[i] = d;  // other warps may read it: +inf or d, either is a valid bound
        lower = lower || d < T;
      }
      __syncwarp();
      if (__any_sync(kFull, lower)) {
        const float Tn = warp_kth_of(ns, kq, [&](int e) {
          return bound_key(*(volatile float*)&cex[e]);
        });
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

// final_kernel for batches without quantised tables: one warp per query (a few
// dozen candidates and about k survivors leave most of a block idle, and its
// barriers took half the time). `fin` as there.
constexpr int kFWarps = 4;
template <int DS>
__global__ void __launch_bounds__(kFWarps * 32) final_fp32_kernel(const FinalArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q = (int64_t)blockIdx.x * kFWarps + warp;
  if (q >= a.nq) return;
  const int64_t row = q * a.nprobe;
  const size_t per = (size_t)a.fin * 16 + (size_t)((a.dim + 3) & ~int64_t(3)) * 4;
  int64_t* cid = (int64_t*)(anns_dyn_smem + warp * per);
  float* cex = (float*)(cid + a.fin);
  uint32_t* cjp = (uint32_t*)(cex + a.fin);  // first the keys of the upper bounds
  float* qs = (float*)(cjp + a.fin);
  const int kq = a.kpq ? min(max(a.kpq[q], 0), a.k) : a.k;
  const int nc = a.ntake[q] > 0 ? a.qcnt[q] : 0;
  const uint2* cand = a.cand + q * a.cap;
  float T = nc > 0 ? a.thr[q] : INFINITY;
  int ns = 0;
  bool over = nc > a.cap;
  if (!over) {
    for (int d = lane; d < a.dim; d += 32) qs[d] = a.Q[q * a.dim + d];
    auto ub_key = [&](int e) {
      const uint2 c = cand[e];
      const int64_t p = row + (c.x >> kPosBits);
      return bound_key(__fadd_ru(__uint_as_float(c.y), __fadd_ru(a.d2[p], a.eps[p])));
    };
    if (nc > kq) {
      if (nc <= a.fin) {
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
      }
      const unsigned m = __ballot_sync(kFull, in);
      const int at = ns + __popc(m & ((1u << lane) - 1u));
      if (in && at < a.fin) cjp[at] = w;
      ns += __popc(m);
    }
    over = ns > a.fin;
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
    const uint8_t* code = a.codes + (((size_t)a.tile_off[l] + pos / kTileVecs) * a.nchunk) * kTileChunkBytes +
                          (pos % kTileVecs) * kChunkBytes;
    float acc = 0.f;
    each_entry<DS, false>(a, qs, nullptr, a.ltab + (size_t)l * a.Mp * kKsub, code,
                          [&](int, float t) { acc = add_rn(acc, t); });
    const float d = add_rn(a.d2[p], acc);
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

// ---------------------------------------------------------------- host side

struct FilterWork {
  size_t bytes = 0, zero_bytes = 0;
  char* base = nullptr;
  template <typename T> T* take(size_t n) {
    T* p = (T*)(base + bytes);
    bytes += (n * sizeof(T) + 255) & ~size_t(255);
    return p;
  }
  int *c1, *c2, *f1, *f2, *qcnt, *nover;
  uint8_t *alive, *overflag;
  int *g1, *g2, *i1, *i2, *ntake, *slot2, *p2;
  float *eps, *eps0, *thr, *ub, *qrows;
  int2 *sel, *d1;
  float2 *k1, *k2;
  FItem *it1, *it2;
  uint2* cand;
  int32_t* over;
  void* Qf;
  __half *r1, *r2;
};

int filter_take(int k) { return k <= 16 ? 1024 : k <= 64 ? 2048 : kTakeMax; }
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
  const int64_t tiles = (ix.max_list + kTv - 1) / kTv, t1 = std::min<int64_t>(tiles, (filter_take(k) + kTv - 1) / kTv);
  w.c1 = w.take<int>(L); w.c2 = w.take<int>(L); w.f1 = w.take<int>(L); w.f2 = w.take<int>(L);
  w.qcnt = w.take<int>(nq); w.nover = w.take<int>(1); w.alive = w.take<uint8_t>(P);
  w.overflag = w.take<uint8_t>(nq);
  w.zero_bytes = w.bytes;
  w.g1 = w.take<int>(L + 1); w.g2 = w.take<int>(L + 1); w.i1 = w.take<int>(L + 1); w.i2 = w.take<int>(L + 1);
  w.ntake = w.take<int>(nq); w.slot2 = w.take<int>(P);
  w.p2 = w.take<int>(G);
  w.eps = w.take<float>(P); w.eps0 = w.take<float>(P); w.thr = w.take<float>(nq); w.ub = w.take<float>(nq * filter_take(k));
  w.sel = w.take<int2>(P); w.d1 = w.take<int2>(G);
  w.k1 = w.take<float2>(G); w.k2 = w.take<float2>(G);
  w.it1 = w.take<FItem>(max_items(ix, P, nq, t1)); w.it2 = w.take<FItem>(max_items(ix, P, nq, tiles));
  w.cand = w.take<uint2>(nq * filter_cap(k));
  w.over = w.take<int32_t>(nq);
  w.qrows = w.take<float>(3 * nq);
  w.Qf = w.take<__half>(nq * Dp); w.r1 = w.take<__half>(G * Dp); w.r2 = w.take<__half>(G * Dp);
  return w;
}

template <int VPT>
cudaError_t run_final_ds(const FinalArgs& a, cudaStream_t s) {
  auto go = [&](auto kern) {
    const size_t sm = final_smem(a.dim, a.Mp, a.fin);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)a.nq, kFinalThreads, sm, s>>>(a);
    note_launch();
    return cudaGetLastError();
  };
  switch (a.dsub) {
    case 2: return go(final_kernel<VPT, 2>);
    case 4: return go(final_kernel<VPT, 4>);
    case 8: return go(final_kernel<VPT, 8>);
    default: return go(final_kernel<VPT, 0>);
  }
}

cudaError_t run_final_fp32(const FinalArgs& a, cudaStream_t s) {
  auto go = [&](auto kern) {
    const size_t sm = kFWarps * ((size_t)a.fin * 16 + (size_t)((a.dim + 3) & ~int64_t(3)) * 4);
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
  e = cudaMalloc(&ix.fl_y, yb);
  if (e == cudaSuccess) e = cudaMalloc(&ix.fl_s, (size_t)rows * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&ix.fl_stat, (size_t)ix.nlist * sizeof(float4));
  if (e == cudaSuccess) e = cudaMalloc(&ix.fl_ym, (size_t)ix.M * sizeof(float));
  if (e == cudaErrorMemoryAllocation) {  // no room: the index works without
    cudaGetLastError();
    free_filter(ix);
    return ANNS_OK;
  }
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
  void* ptrs[] = {ix.fl_y, ix.fl_s, ix.fl_stat, ix.fl_ym};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  ix.fl_y = ix.fl_stat = nullptr;
  ix.fl_s = ix.fl_ym = nullptr;
  ix.fl_w = 0;
}

bool filter_supported(const Index& ix, const anns_precision_policy& P, int64_t nq, int nprobe, int k) {
  if (ix.fl_w == 0 || (ix.opt_kernel != ANNS_KERNEL_AUTO && ix.opt_kernel != ANNS_KERNEL_SPLIT)) return false;
  if (P.lut_mode == ANNS_LUT_FIXED_BITS && P.fixed_bits < 5) return false;  // every pair would be scanned anyway
  // A search of a few short lists is over before the filter's dozen launches
  // (about 100 us) are: a block scans a pair in about Mp (256 + list) / 2000 us,
  // some 400 queries at a time (one query, 8 lists of 312, M = 16: 54 us
  // scanned, 87 us filtered; 777 queries, 19 lists of 150, M = 20, 12 bits: 530
  // and 200 us).
  const double scan_us = (double)nprobe * (double)ix.Mp * (256.0 + (double)ix.n / (double)ix.nlist) / 2000.0 *
                         std::max(1.0, (double)nq / 400.0);
  if (scan_us < 100.0) return false;
  const int64_t pairs = nq * nprobe, tiles = (ix.max_list + kTv - 1) / kTv;
  if (pairs > INT32_MAX / 2 || nq * kTakeMax > INT32_MAX || max_slots(ix, pairs) > INT32_MAX ||
      max_items(ix, pairs, nq, tiles) > ((int64_t)1 << 26))
    return false;
  return filter_workspace_bytes(ix, nq, nprobe, k) <= kFilterWorkspaceMax;
}

size_t filter_workspace_bytes(const Index& ix, int64_t nq, int nprobe, int k) {
  return filter_work(ix, nq, nprobe, k, nullptr).bytes;
}

cudaError_t launch_search_filter(const Index& ix, const float* Q, const float* qt, int64_t nq, int nprobe,
                                 const int32_t* nprobe_per_q, int k, const int32_t* k_per_q, const int32_t* probes,
                                 const float* probe_d2, const uint8_t* bits, void* ws, const void* q16,
                                 const float* q16_rows, bool quantised, int64_t* ids_out, float* dists_out,
                                 int64_t* over_i, float* over_d, FilterResult* out, cudaStream_t s) {
  FilterWork w = filter_work(ix, nq, nprobe, k, (char*)ws);
  cudaError_t e = cudaMemsetAsync(w.c1, 0, w.zero_bytes, s);
  if (e == cudaSuccess && !q16) {
    e = launch_center_fp16(ix, Q, nq, w.Qf, w.qrows, s);
    q16 = w.Qf;
    q16_rows = w.qrows;
  }
  if (e != cudaSuccess) return e;
  const int Dp = coarse_tc_dp(ix, ANNS_PREC_FP16);
  PlanArgs p{};
  p.nq = nq; p.dim = ix.dim; p.nprobe = nprobe; p.k = k; p.M = (int)ix.M; p.dsub = (int)ix.dsub; p.Dp = Dp;
  p.take = filter_take(k); p.nlist = (int)ix.nlist; p.npq = nprobe_per_q; p.kpq = k_per_q; p.probes = probes;
  p.d2 = probe_d2; p.bits = bits; p.list_len = ix.list_len; p.tile_off = ix.tile_off; p.Q = Q; p.C = ix.centroids;
  p.ym = ix.fl_ym; p.stat = (const float4*)ix.fl_stat; p.qrows = q16_rows; p.mu_norm = ix.fl_mu;
  p.yscale = ix.fl_yscale; p.eps = w.eps; p.eps0 = w.eps0; p.sel = w.sel; p.ntake = w.ntake; p.c1 = w.c1; p.c2 = w.c2; p.f1 = w.f1;
  p.f2 = w.f2; p.g1 = w.g1; p.g2 = w.g2; p.i1 = w.i1; p.i2 = w.i2; p.q16 = (const __half*)q16; p.r1 = w.r1; p.r2 = w.r2; p.k1 = w.k1; p.k2 = w.k2;
  p.d1 = w.d1; p.p2 = w.p2; p.slot2 = w.slot2; p.it1 = w.it1; p.it2 = w.it2;
  plan_kernel<<<(unsigned)nq, 128, 0, s>>>(p); note_launch();
  plan_scan_kernel<<<1, 1024, 0, s>>>(p); note_launch();
  const int64_t P = nq * nprobe;
  const int pair_blocks = (int)((P + 7) / 8);
  plan_scatter_kernel<<<(unsigned)(pair_blocks + (ix.nlist + 7) / 8), 256, 0, s>>>(p, pair_blocks); note_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  CUtensorMap tmY, tmQ1, tmQ2;
  e = make_tmap(&tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ix.fl_y, ix.ntiles * kTileVecs, ix.fl_w, kKE, 64);
  const int64_t slots = max_slots(ix, P);
  if (e == cudaSuccess) e = make_tmap(&tmQ1, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, w.r1, slots, Dp, kKE, 32);
  if (e == cudaSuccess) e = make_tmap(&tmQ2, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, w.r2, slots, Dp, kKE, 32);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (ix.max_list + kTv - 1) / kTv, t1 = std::min<int64_t>(tiles, (p.take + kTv - 1) / kTv);
  GemmArgs g{};
  g.sx = ix.fl_s; g.nK = Dp / kKE; g.ksteps = (int)((ix.dim + 15) / 16); g.status = ix.dev_status;
  g.wait_limit = ix.opt_wait_cycles > 0 ? ix.opt_wait_cycles : kWaitCycles;
  g.nprobe = nprobe; g.bits = bits;
  g.items = w.it1; g.nitems = w.i1 + ix.nlist; g.gk = w.k1; g.gd = w.d1; g.ub = w.ub;
  if ((e = run_gemm<1>(ix, tmY, tmQ1, g, max_items(ix, P, nq, t1), s)) != cudaSuccess) return e;
  const unsigned tb = (unsigned)((nq + 3) / 4);
  switch (p.take / 32) {
    case 32: threshold_kernel<32><<<tb, 128, 0, s>>>(p, w.ub, w.thr); break;
    case 64: threshold_kernel<64><<<tb, 128, 0, s>>>(p, w.ub, w.thr); break;
    default: threshold_kernel<128><<<tb, 128, 0, s>>>(p, w.ub, w.thr); break;
  }
  note_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  g.items = w.it2; g.nitems = w.i2 + ix.nlist; g.gk = w.k2; g.gp = w.p2; g.qcnt = w.qcnt; g.cand = w.cand;
  g.cap = filter_cap(k); g.alive = w.alive;
  if ((e = run_gemm<2>(ix, tmY, tmQ2, g, max_items(ix, P, nq, tiles), s)) != cudaSuccess) return e;
  FinalArgs f{};
  f.nq = nq; f.dim = ix.dim; f.nprobe = nprobe; f.k = k; f.M = (int)ix.M; f.Mp = (int)ix.Mp; f.nchunk = (int)ix.nchunk;
  f.dsub = (int)ix.dsub; f.cap = g.cap; f.fin = filter_fin(k); f.npq = nprobe_per_q; f.kpq = k_per_q; f.probes = probes; f.d2 = probe_d2;
  f.bits = bits; f.eps = w.eps; f.eps0 = w.eps0; f.thr = w.thr; f.quantised = quantised ? 1 : 0; f.ntake = w.ntake; f.qcnt = w.qcnt; f.cand = w.cand; f.Q = Q;
  f.books = ix.codebooks; f.ltab = ix.ltab; f.qt = qt; f.codes = ix.codes; f.ids = ix.ids; f.tile_off = ix.tile_off;
  f.vec_off = ix.vec_off; f.over = w.over; f.nover = w.nover; f.ids_out = ids_out; f.dists_out = dists_out;
  f.overflag = w.overflag; f.over_i = over_i; f.over_d = over_d;
  if (quantised) {
    e = f.cap == 2048 ? run_final_ds<8>(f, s) : run_final_ds<16>(f, s);
  } else {
    f.fin = k <= 32 ? 256 : 512;
    e = run_final_fp32(f, s);
  }
  out->over = w.over;
  out->nover = w.nover;
  out->alive = w.alive;
  out->overflag = w.overflag;
  out->thr = w.thr;
  return e;
}

}  // namespace anns
