// Index construction and facts (Section 2.1: IVF lists, PQ codes on residuals
// with one codebook shared by every cluster; covering radius r of Eq. 1).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace anns {

static thread_local std::string g_err;

void set_error(const std::string& msg) { g_err = msg; }
int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}
int cuda_fail(cudaError_t e, const char* what) {
  return fail(e == cudaErrorMemoryAllocation ? ANNS_ERR_OOM : ANNS_ERR_CUDA,
              std::string(what) + ": " + cudaGetErrorString(e));
}

int grow(void** p, size_t* cap, size_t bytes) {
  if (*cap >= bytes && *p) return ANNS_OK;
  if (*p) cudaFree(*p);
  *p = nullptr;
  *cap = 0;
  if (bytes == 0) return ANNS_OK;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) {
    *p = nullptr;
    return cuda_fail(e, "cudaMalloc(workspace)");
  }
  *cap = bytes;
  return ANNS_OK;
}

static void free_index(anns_index* ix) {
  if (!ix) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(ix->device);
  void* ptrs[] = {ix->centroids, ix->codebooks, ix->codes, ix->ids, ix->list_len,
                  ix->vec_off, ix->tile_off, ix->radius, ix->ltab, ix->order, ix->mlp_dev,
                  ix->tc_mu, ix->tc_c[0], ix->tc_c[1], ix->tc_c[2], ix->tc_crows[0], ix->tc_crows[1],
                  ix->tc_crows[2], ix->dev_status, ix->svr_dev};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  free_filter(*ix);
  free_workspace(*ix);
  free_subspaces(*ix);
  for (auto& set : ix->prof_ev)
    for (cudaEvent_t e : set)
      if (e) cudaEventDestroy(e);
  cudaSetDevice(prev);
  delete[] ix->h_list_len64;
  delete[] ix->h_radius;
  delete ix;
}

}  // namespace anns

namespace anns {
namespace index_build {

template <typename T>
int fetch(const T* src, size_t count, bool on_device, std::vector<T>& dst, const char* what) {
  dst.resize(count);
  if (count == 0) return ANNS_OK;
  if (on_device) {
    cudaError_t e = cudaMemcpy(dst.data(), src, count * sizeof(T), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, what);
  } else {
    std::memcpy(dst.data(), src, count * sizeof(T));
  }
  return ANNS_OK;
}

template <typename T>
int upload(T** dst, const T* src, size_t count, const char* what) {
  size_t bytes = std::max<size_t>(count * sizeof(T), 16);
  cudaError_t e = cudaMalloc((void**)dst, bytes);
  if (e != cudaSuccess) return cuda_fail(e, what);
  if (count) {
    e = cudaMemcpy(*dst, src, count * sizeof(T), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, what);
  }
  return ANNS_OK;
}

// A device buffer of one call.
struct Temp {
  void* p = nullptr;
  ~Temp() { if (p) cudaFree(p); }
};

// P_l[m][c] = fl32(yn[m][c] + fl32(2 * <c_lm, y_mc>)) with both inner products
// accumulated in FP32, j ascending, one rounding per operation; rows M..Mp-1
// zero. Block = list, thread = entry c of every row.
__global__ void __launch_bounds__(256) list_tables_kernel(const float* __restrict__ cent, const float* __restrict__ books,
                                                          int64_t dim, int M, int Mp, int dsub, float* __restrict__ out) {
  const int64_t l = blockIdx.x;
  const int c = threadIdx.x;
  const float* cl = cent + l * dim;
  for (int m = 0; m < Mp; ++m) {
    float v = 0.f;
    if (m < M) {
      const float* y = books + ((size_t)m * ANNS_KSUB + c) * dsub;
      float yn = 0.f, acc = 0.f;
      for (int j = 0; j < dsub; ++j) {
        yn = add_rn(yn, mul_rn(y[j], y[j]));
        acc = add_rn(acc, mul_rn(cl[m * dsub + j], y[j]));
      }
      v = add_rn(yn, mul_rn(2.f, acc));
    }
    out[((size_t)l * Mp + m) * ANNS_KSUB + c] = v;
  }
}

// Vector i's codes to its place slot[i] = tile * 32 + lane in the
// warp-interleaved tiles, a thread per 16-byte chunk.
__global__ void pack_codes_kernel(const uint8_t* __restrict__ codes, const int64_t* __restrict__ slot, int64_t n, int M,
                                  int nchunk, uint8_t* __restrict__ packed) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * nchunk) return;
  const int64_t i = t / nchunk;
  const int c = (int)(t - i * nchunk);
  const uint8_t* src = codes + i * M + c * kChunkBytes;
  uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int b = 0; b < kChunkBytes; ++b)
    if (c * kChunkBytes + b < M) w[b >> 2] |= (uint32_t)src[b] << (8 * (b & 3));
  const int64_t s = slot[i];
  *(uint4*)(packed + ((s / kTileVecs) * nchunk + c) * kTileChunkBytes + (s % kTileVecs) * kChunkBytes) =
      make_uint4(w[0], w[1], w[2], w[3]);
}

// Per list the largest squared residual norm: per member the FP64 sum of its
// entries' squared norms, m ascending. Non-negative doubles order like their
// bit patterns; a NaN never counts.
__global__ void radius_kernel(const uint8_t* __restrict__ codes, const int32_t* __restrict__ list_of, int64_t n, int M,
                              const double* __restrict__ yn2, unsigned long long* __restrict__ rmax2) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s = 0.0;
  for (int m = 0; m < M; ++m) s = __dadd_rn(s, yn2[m * ANNS_KSUB + codes[i * M + m]]);
  if (s == s) atomicMax(rmax2 + list_of[i], (unsigned long long)__double_as_longlong(s));
}

// The parts of the index that the GPU forms: code tiles, list tables and
// covering radii (on one host thread the tiles and radii took about 2 ns a code
// byte, the tables a few ns an entry). The codes are read where they are, or
// from a copy on the device.
int pack_index(Index& ix, const anns_build_desc* d, const std::vector<int64_t>& slot, const std::vector<int32_t>& list_of,
               const std::vector<double>& yn2) {
  const int64_t n = ix.n;
  const size_t code_bytes = std::max<size_t>((size_t)ix.ntiles * ix.nchunk * kTileChunkBytes, 16);
  const int64_t step = std::min<int64_t>(n, (int64_t)1 << 24);  // vectors at a time: bounded temporary memory
  Temp codes, slots, lists, norms, rmax;
  cudaError_t e = cudaMalloc((void**)&ix.codes, code_bytes);
  if (e == cudaSuccess) e = cudaMalloc((void**)&ix.ltab, (size_t)ix.nlist * ix.Mp * kKsub * sizeof(float));
  if (e == cudaSuccess) e = cudaMalloc(&slots.p, std::max<size_t>(step * 8, 16));
  if (e == cudaSuccess) e = cudaMalloc(&lists.p, std::max<size_t>(step * 4, 16));
  if (e == cudaSuccess) e = cudaMalloc(&norms.p, yn2.size() * 8);
  if (e == cudaSuccess) e = cudaMalloc(&rmax.p, (size_t)ix.nlist * 8);
  if (e == cudaSuccess && !d->on_device) e = cudaMalloc(&codes.p, std::max<size_t>(step * ix.M, 16));
  if (e == cudaSuccess) e = cudaMemset(ix.codes, 0, code_bytes);
  if (e == cudaSuccess) e = cudaMemset(rmax.p, 0, (size_t)ix.nlist * 8);
  if (e == cudaSuccess) e = cudaMemcpy(norms.p, yn2.data(), yn2.size() * 8, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "index arrays");
  for (int64_t i0 = 0; i0 < n; i0 += step) {
    const int64_t m = std::min(step, n - i0);
    const uint8_t* src = d->codes + i0 * ix.M;
    e = cudaMemcpy(slots.p, slot.data() + i0, m * 8, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(lists.p, list_of.data() + i0, m * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !d->on_device) {
      e = cudaMemcpy(codes.p, src, (size_t)m * ix.M, cudaMemcpyHostToDevice);
      src = (const uint8_t*)codes.p;
    }
    if (e != cudaSuccess) return cuda_fail(e, "index arrays");
    pack_codes_kernel<<<(unsigned)((m * ix.nchunk + 255) / 256), 256>>>(src, (const int64_t*)slots.p, m, (int)ix.M,
                                                                        (int)ix.nchunk, ix.codes);
    note_launch();
    radius_kernel<<<(unsigned)((m + 255) / 256), 256>>>(src, (const int32_t*)lists.p, m, (int)ix.M,
                                                        (const double*)norms.p, (unsigned long long*)rmax.p);
    note_launch();
  }
  list_tables_kernel<<<(unsigned)ix.nlist, 256>>>(ix.centroids, ix.codebooks, ix.dim, (int)ix.M, (int)ix.Mp, (int)ix.dsub,
                                                  ix.ltab);
  note_launch();
  e = cudaGetLastError();
  std::vector<double> r2(ix.nlist);
  if (e == cudaSuccess) e = cudaMemcpy(r2.data(), rmax.p, (size_t)ix.nlist * 8, cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "index kernels");
  for (int64_t l = 0; l < ix.nlist; ++l) ix.h_radius[l] = (float)std::sqrt(r2[l]);
  return ANNS_OK;
}

}  // namespace index_build
}  // namespace anns

using namespace anns;
using namespace anns::index_build;

extern "C" int anns_build_index_from_arrays(const anns_build_desc* d, anns_index** out) {
  set_error("");
  if (!d || !out) return fail(ANNS_ERR_INVALID_ARG, "null desc or out");
  *out = nullptr;
  if (d->n < 0 || d->dim <= 0 || d->nlist <= 0 || d->M <= 0)
    return fail(ANNS_ERR_INVALID_ARG, "n must be >= 0 and dim, nlist, M > 0");
  if (d->ksub != ANNS_KSUB) return fail(ANNS_ERR_INVALID_ARG, "ksub must be 256");
  if (d->dim % d->M) return fail(ANNS_ERR_INVALID_ARG, "dim must be a multiple of M");
  if (d->M > ANNS_MAX_M) return fail(ANNS_ERR_INVALID_ARG, "M must be <= 128");
  if (d->nlist > INT32_MAX || d->n > INT32_MAX)
    return fail(ANNS_ERR_INVALID_ARG, "n and nlist must fit in int32");
  if (!d->centroids || !d->codebooks || (d->n > 0 && (!d->codes || !d->list_of)))
    return fail(ANNS_ERR_INVALID_ARG, "null array");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0)
    return fail(ANNS_ERR_CUDA, "no CUDA device");
  if (d->device < 0 || d->device >= ndev) return fail(ANNS_ERR_INVALID_ARG, "bad device ordinal");
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(d->device);

  const int64_t n = d->n, dim = d->dim, nlist = d->nlist, M = d->M, dsub = dim / M;
  const int64_t Mp = (M + 15) / 16 * 16, nchunk = Mp / 16;
  const bool dev = d->on_device != 0;
  std::vector<float> cent, books;
  std::vector<int32_t> list_of;
  std::vector<int64_t> uids;
  int rc;
  if ((rc = fetch(d->centroids, (size_t)(nlist * dim), dev, cent, "copy centroids")) ||
      (rc = fetch(d->codebooks, (size_t)(M * ANNS_KSUB * dsub), dev, books, "copy codebooks")) ||
      (rc = fetch(d->list_of, (size_t)n, dev, list_of, "copy list_of"))) {
    cudaSetDevice(prev);
    return rc;
  }
  if (d->ids && (rc = fetch(d->ids, (size_t)n, dev, uids, "copy ids"))) {
    cudaSetDevice(prev);
    return rc;
  }
  std::vector<int64_t> cnt(nlist, 0);
  for (int64_t i = 0; i < n; ++i) {
    const int32_t l = list_of[i];
    if (l < 0 || l >= nlist) {
      cudaSetDevice(prev);
      return fail(ANNS_ERR_INVALID_ARG, "list_of value outside [0, nlist)");
    }
    cnt[l]++;
  }
  std::vector<int64_t> voff(nlist + 1, 0), toff(nlist + 1, 0);
  int64_t max_list = 0;
  for (int64_t l = 0; l < nlist; ++l) {
    voff[l + 1] = voff[l] + cnt[l];
    toff[l + 1] = toff[l] + (cnt[l] + kTileVecs - 1) / kTileVecs;
    max_list = std::max(max_list, cnt[l]);
  }
  const int64_t ntiles = toff[nlist];
  // places in the tiles and ids in list order, members in array order
  std::vector<int64_t> pids(n);
  std::vector<int64_t> slot(n);
  {
    std::vector<int64_t> fill(nlist, 0);
    for (int64_t i = 0; i < n; ++i) {
      const int32_t l = list_of[i];
      const int64_t rank = fill[l]++;
      slot[i] = toff[l] * kTileVecs + rank;
      pids[voff[l] + rank] = d->ids ? uids[i] : i;
    }
  }
  // ||y_{m,c}||^2 in FP64 with j ascending
  std::vector<double> yn2((size_t)M * ANNS_KSUB, 0.0);
  for (int64_t m = 0; m < M; ++m)
    for (int c = 0; c < ANNS_KSUB; ++c) {
      double acc = 0.0;
      for (int64_t j = 0; j < dsub; ++j) {
        const double y = (double)books[((size_t)m * ANNS_KSUB + c) * dsub + j];
        const double sq = y * y;
        acc = acc + sq;
      }
      yn2[(size_t)m * ANNS_KSUB + c] = acc;
    }
  anns_index* ix = new anns_index();
  ix->device = d->device;
  ix->n = n; ix->dim = dim; ix->nlist = nlist; ix->M = M; ix->dsub = dsub; ix->Mp = Mp;
  ix->nchunk = nchunk; ix->ntiles = ntiles; ix->max_list = max_list;
  ix->ids32 = std::all_of(pids.begin(), pids.end(),
                          [](int64_t v) { return v >= (int64_t)INT32_MIN && v < (int64_t)INT32_MAX; });
  ix->h_list_len64 = new int64_t[nlist];
  ix->h_radius = new float[nlist];
  std::vector<int32_t> len32(nlist);
  for (int64_t l = 0; l < nlist; ++l) {
    if (n > 0) ix->list_seen += (double)cnt[l] * ((double)cnt[l] / (double)n);
    ix->h_list_len64[l] = cnt[l];
    len32[l] = (int32_t)cnt[l];
  }
  std::vector<int32_t> order(nlist);
  for (int64_t l = 0; l < nlist; ++l) order[l] = (int32_t)l;
  std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return cnt[x] > cnt[y]; });
  if ((rc = upload(&ix->order, order.data(), order.size(), "upload list order")) ||
      (rc = upload(&ix->centroids, cent.data(), cent.size(), "upload centroids")) ||
      (rc = upload(&ix->codebooks, books.data(), books.size(), "upload codebooks")) ||
      (rc = pack_index(*ix, d, slot, list_of, yn2)) ||
      (rc = upload(&ix->ids, pids.data(), pids.size(), "upload ids")) ||
      (rc = upload(&ix->list_len, len32.data(), len32.size(), "upload list_len")) ||
      (rc = upload(&ix->vec_off, voff.data(), voff.size(), "upload vec_off")) ||
      (rc = upload(&ix->tile_off, toff.data(), toff.size(), "upload tile_off")) ||
      (rc = upload(&ix->radius, ix->h_radius, (size_t)nlist, "upload radius")) ||
      (rc = prepare_coarse_tc(*ix, cent)) || (rc = prepare_filter(*ix, cent, books))) {
    free_index(ix);
    cudaSetDevice(prev);
    return rc;
  }
  cudaSetDevice(prev);
  *out = ix;
  return ANNS_OK;
}

extern "C" void anns_free(anns_index* index) { free_index(index); }

extern "C" int anns_get_info(const anns_index* ix, anns_index_info* out) {
  if (!ix || !out) return fail(ANNS_ERR_INVALID_ARG, "null index or out");
  out->n = ix->n; out->dim = ix->dim; out->nlist = ix->nlist; out->M = ix->M;
  out->dsub = ix->dsub; out->Mp = ix->Mp;
  out->code_bytes = ix->ntiles * ix->nchunk * kTileChunkBytes;
  out->max_list = ix->max_list; out->device = ix->device;
  return ANNS_OK;
}

extern "C" int anns_debug_tap(anns_index* ix, int32_t what, void* out, size_t bytes) {
  if (!ix || !out) return fail(ANNS_ERR_INVALID_ARG, "null index or out");
  const void* src = nullptr;
  size_t need = 0;
  bool host = false;
  const size_t pairs = (size_t)(ix->ws_nq * ix->ws_nprobe);
  switch (what) {
    case ANNS_TAP_PROBES: src = ix->ws_probes; need = pairs * 4; break;
    case ANNS_TAP_PROBE_D2: src = ix->ws_probe_d2; need = pairs * 4; break;
    case ANNS_TAP_BITS: src = ix->ws_bits; need = pairs; break;
    case ANNS_TAP_FEATURES: src = ix->ws_feat; need = pairs * kNFeat * 4; break;
    case ANNS_TAP_LIST_SIZES: src = ix->h_list_len64; need = (size_t)ix->nlist * 8; host = true; break;
    case ANNS_TAP_LIST_RADIUS: src = ix->h_radius; need = (size_t)ix->nlist * 4; host = true; break;
    case ANNS_TAP_PACKED_IDS: src = ix->ids; need = (size_t)ix->n * 8; break;
    case ANNS_TAP_COARSE_APPROX:
      if (!ix->ws_tc_valid) return fail(ANNS_ERR_INVALID_ARG, "last search did not use the tensor-core CL");
      src = ix->ws_d2; need = (size_t)ix->ws_tc_nq * ix->nlist * 4; break;
    case ANNS_TAP_COARSE_CANDIDATES: {
      if (!ix->ws_tc_valid) return fail(ANNS_ERR_INVALID_ARG, "last search did not use the tensor-core CL");
      src = coarse_tc_candidates(*ix, ix->ws_tc, ix->ws_tc_nq);
      need = (size_t)ix->ws_tc_nq * 4;
      break;
    }
    case ANNS_TAP_FILTERED:
      if (bytes < 4) return fail(ANNS_ERR_INVALID_ARG, "tap buffer too small");
      *(int32_t*)out = ix->last_filtered ? 1 : 0;
      return ANNS_OK;
    case ANNS_TAP_STATUS: {
      if (bytes < 4) return fail(ANNS_ERR_INVALID_ARG, "tap buffer too small");
      int v = 0;
      cudaError_t e = cudaMemcpy(&v, ix->dev_status, 4, cudaMemcpyDeviceToHost);
      if (e == cudaSuccess) e = cudaMemset(ix->dev_status, 0, 4);
      if (e != cudaSuccess) return cuda_fail(e, "status tap");
      *(int32_t*)out = v;
      return ANNS_OK;
    }
    default: return fail(ANNS_ERR_INVALID_ARG, "unknown tap");
  }
  if (bytes < need) return fail(ANNS_ERR_INVALID_ARG, "tap buffer too small");
  if (need == 0) return ANNS_OK;
  if (!src) return fail(ANNS_ERR_INVALID_ARG, "tap not available (no search yet?)");
  if (host) {
    std::memcpy(out, src, need);
    return ANNS_OK;
  }
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(ix->device);
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(out, src, need, cudaMemcpyDeviceToHost);
  cudaSetDevice(prev);
  if (e != cudaSuccess) return cuda_fail(e, "tap copy");
  return ANNS_OK;
}

extern "C" int anns_sync_status(anns_index* ix, void* stream) {
  if (!ix) return fail(ANNS_ERR_INVALID_ARG, "null index");
  int prev = 0;
  cudaError_t e = cudaGetDevice(&prev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  e = cudaSetDevice(ix->device);
  if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice(index device)");
  int v = 0;
  e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e == cudaSuccess && ix->dev_status) {
    e = cudaMemcpy(&v, ix->dev_status, 4, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && v != 0) e = cudaMemset(ix->dev_status, 0, 4);
  }
  cudaSetDevice(prev);
  if (e != cudaSuccess) return cuda_fail(e, "status read");
  if (v == ANNS_DEV_TIMEOUT) return fail(ANNS_ERR_TIMEOUT, "a bounded wait in a kernel of this index ran out; its output is invalid");
  return ANNS_OK;
}

extern "C" const char* anns_last_error(void) { return anns::g_err.c_str(); }

namespace anns {
namespace {
std::atomic<int64_t> g_launches{0};
}
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
int64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }
}  // namespace anns

extern "C" int64_t anns_kernel_launches(void) { return anns::launch_count(); }
