// The coarse selection of one query by one block (CL, Section 2.1).
#pragma once

#include "common.cuh"

namespace anns {

// The np smallest (D2, id) of a row of `nlist` distances (global or shared
// memory) into probes / probe_d2 (padding -1 / +inf up to nprobe): the np-th
// smallest value's bits by bisection, then the lists up to it (np and those
// equal to the last) ranked by (D2, id) against one another. More than
// kSmallCand of them (many equal distances) go through a warp's sorted list. One
// warp per query takes 38 us for 4096 lists, all of it latency. The results are
// visible to the block after the caller's next barrier.
constexpr int kSmallThreads = 512, kSmallCand = 512;
struct SelectSmem {
  uint32_t ws[2][kSmallThreads / 32];
  float cd[kSmallCand];
  int32_t ci[kSmallCand];
  int total;
};
template <int R>
__device__ __forceinline__ void select_small(const float* row, int64_t nlist, int nprobe, int np, int32_t* probes,
                                             float* probe_d2, SelectSmem& sm) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nw = kSmallThreads / 32;
  for (int e = tid; e < nprobe; e += kSmallThreads) {
    probes[e] = -1;
    probe_d2[e] = INFINITY;
  }
  if (np == 0) return;
  if (tid == 0) sm.total = 0;
  constexpr int V = 16;  // values a thread keeps in registers
  uint32_t key[V];
  uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int64_t l = tid + (int64_t)i * kSmallThreads;
    key[i] = l < nlist ? __float_as_uint(row[l]) : 0xFFFFFFFFu;  // D2 >= 0 (or NaN: above +inf)
    lo = min(lo, key[i]);
    if (l < nlist) hi = max(hi, key[i]);
  }
  for (int64_t l = tid + (int64_t)V * kSmallThreads; l < nlist; l += kSmallThreads) {
    const uint32_t k = __float_as_uint(row[l]);
    lo = min(lo, k);
    hi = max(hi, k);
  }
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
  if (lane == 0) { sm.ws[0][warp] = lo; sm.ws[1][warp] = hi; }
  __syncthreads();
  for (int w = 0; w < nw; ++w) {
    lo = min(lo, sm.ws[0][w]);
    hi = max(hi, sm.ws[1][w]);
  }
  __syncthreads();
  for (int step = 0; lo < hi; ++step) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    int c = 0;
#pragma unroll
    for (int i = 0; i < V; ++i) c += key[i] <= mid ? 1 : 0;
    for (int64_t l = tid + (int64_t)V * kSmallThreads; l < nlist; l += kSmallThreads)
      c += __float_as_uint(row[l]) <= mid ? 1 : 0;
    c = __reduce_add_sync(kFull, c);
    if (lane == 0) sm.ws[step & 1][warp] = (uint32_t)c;
    __syncthreads();
    int t = 0;
    for (int w = 0; w < nw; ++w) t += (int)sm.ws[step & 1][w];
    if (t >= np) hi = mid;
    else lo = mid + 1u;
  }
  auto collect = [&](int64_t l, uint32_t k) {
    if (k <= hi) {
      const int at = atomicAdd(&sm.total, 1);
      if (at < kSmallCand) {
        sm.cd[at] = __uint_as_float(k);
        sm.ci[at] = (int32_t)l;
      }
    }
  };
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const int64_t l = tid + (int64_t)i * kSmallThreads;
    if (l < nlist) collect(l, key[i]);
  }
  for (int64_t l = tid + (int64_t)V * kSmallThreads; l < nlist; l += kSmallThreads) collect(l, __float_as_uint(row[l]));
  __syncthreads();
  const int n = sm.total;
  if (n <= kSmallCand) {
    for (int i = tid; i < n; i += kSmallThreads) {
      const float d = sm.cd[i];
      if (!(d < INFINITY)) continue;  // +inf and NaN are no probes
      int rank = 0;
      for (int e = 0; e < n; ++e) rank += key_less(sm.cd[e], sm.ci[e], d, sm.ci[i]) ? 1 : 0;
      if (rank < np) {
        probes[rank] = sm.ci[i];
        probe_d2[rank] = d;
      }
    }
    return;
  }
  if (warp != 0) return;
  WarpTopK<R, int32_t> top;
  top.init();
  float thd = INFINITY;
  int32_t thi = INT32_MAX;
  for (int64_t b = 0; b < nlist; b += 32) {
    const int64_t l = b + lane;
    const float v = l < nlist ? row[l] : INFINITY;
    const bool c = l < nlist && __float_as_uint(v) <= hi;
    if (__any_sync(kFull, c)) top.offer(c, v, (int32_t)l, np, thd, thi);
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = r * 32 + lane;
    if (e < np && top.d[r] != INFINITY) {
      probes[e] = top.id[r];
      probe_d2[e] = top.d[r];
    }
  }
}

}  // namespace anns
