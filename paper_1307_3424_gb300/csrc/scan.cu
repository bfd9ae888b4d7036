// Device prefix sums and a stable counting sort, used to lay out G.
#include "plan.h"

namespace wproj {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;

// Exclusive block scan of one value per thread; returns the prefix and the block total.
template <class T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *total) {
  __shared__ T warp_tot[kScanThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += n;
  }
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    constexpr int NW = kScanThreads / 32;
    T w = (lane < NW) ? warp_tot[lane] : T(0);
    T wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T n = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += n;
    }
    if (lane < NW) warp_tot[lane] = wi - w;   // exclusive prefix of the warp totals
    if (lane == NW - 1) *total = wi;
  }
  __syncthreads();
  T res = warp_tot[wid] + inc - v;
  __syncthreads();
  return res;
}

template <class Tin, class Tout>
__global__ void k_block_sums(const Tin *__restrict__ in, int64_t n, Tout *__restrict__ sums) {
  __shared__ Tout tot;
  const int64_t base = int64_t(blockIdx.x) * kScanTile + threadIdx.x * kScanPer;
  Tout s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i)
    if (base + i < n) s += Tout(in[base + i]);
  Tout pre = block_exclusive_scan<Tout>(s, &tot);
  (void)pre;
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

// Single-block exclusive scan of `n` values (sequential over tiles; in place is fine).
template <class Tin, class T>
__global__ void k_scan_single(const Tin *in, T *out, int64_t n, T *__restrict__ total) {
  __shared__ T tot;
  T carry = 0;
  for (int64_t t0 = 0; t0 < n; t0 += kScanTile) {
    const int64_t base = t0 + threadIdx.x * kScanPer;
    T v[kScanPer];
    T s = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      v[i] = (base + i < n) ? T(in[base + i]) : T(0);
      s += v[i];
    }
    T pre = block_exclusive_scan<T>(s, &tot) + carry;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      if (base + i < n) out[base + i] = pre;
      pre += v[i];
    }
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

template <class Tin, class Tout>
__global__ void k_scan_apply(const Tin *__restrict__ in, int64_t n, const Tout *__restrict__ offs,
                             Tout *__restrict__ out) {
  __shared__ Tout tot;
  const int64_t base = int64_t(blockIdx.x) * kScanTile + threadIdx.x * kScanPer;
  Tout v[kScanPer];
  Tout s = 0;
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    v[i] = (base + i < n) ? Tout(in[base + i]) : Tout(0);
    s += v[i];
  }
  Tout pre = block_exclusive_scan<Tout>(s, &tot) + offs[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kScanPer; ++i) {
    if (base + i < n) out[base + i] = pre;
    pre += v[i];
  }
}

// The total goes to *total (device) where one is given.  wait: synchronise, so that the
// caller may read the result on the host.
template <class Tin, class Tout>
wproj_status exclusive_scan(const Tin *in, Tout *out, int64_t n, Tout *total, bool wait, cudaStream_t s) {
  if (n <= 0) {
    if (total) WPROJ_CUDA(cudaMemsetAsync(total, 0, sizeof(Tout), s));
    return WPROJ_OK;
  }
  const int64_t nb = (n + kScanTile - 1) / kScanTile;
  if (nb == 1) {
    k_scan_single<Tin, Tout><<<1, kScanThreads, 0, s>>>(in, out, n, total);
    WPROJ_CHECK_LAUNCH("scan");
    if (wait) WPROJ_CUDA(cudaStreamSynchronize(s));
    return WPROJ_OK;
  }
  TmpBuf sums;
  WPROJ_TRY(sums.alloc(sizeof(Tout) * nb));
  k_block_sums<Tin, Tout><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums.as<Tout>());
  WPROJ_CHECK_LAUNCH("scan block sums");
  k_scan_single<Tout, Tout><<<1, kScanThreads, 0, s>>>(sums.as<Tout>(), sums.as<Tout>(), nb, total);
  WPROJ_CHECK_LAUNCH("scan sums");
  k_scan_apply<Tin, Tout><<<(unsigned)nb, kScanThreads, 0, s>>>(in, n, sums.as<Tout>(), out);
  WPROJ_CHECK_LAUNCH("scan apply");
  // a temporary of its own is freed at scope exit: the kernels have to be done with it
  if (wait || sums.own) WPROJ_CUDA(cudaStreamSynchronize(s));
  return WPROJ_OK;
}

// ---- stable counting sort ---------------------------------------------------

__global__ void k_bin_hist(const int32_t *__restrict__ key, int64_t n, int64_t chunk, int n_bins,
                           int n_blocks, int32_t *__restrict__ hist) {
  extern __shared__ int32_t h[];
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x) h[b] = 0;
  __syncthreads();
  const int64_t lo = int64_t(blockIdx.x) * chunk;
  const int64_t hi = min(n, lo + chunk);
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) atomicAdd(&h[key[i]], 1);
  __syncthreads();
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x)
    hist[int64_t(b) * n_blocks + blockIdx.x] = h[b];
}

// The first warp of a block walks its chunk in order (the others only help to load the
// bins' first places); ties inside a group of 32 are
// ranked by lane, so the sort is stable.
__global__ void k_bin_scatter(const int32_t *__restrict__ key, int64_t n, int64_t chunk, int n_bins,
                              int n_blocks, const int64_t *__restrict__ offs,
                              int32_t *__restrict__ out_ids) {
  extern __shared__ int32_t run[];
#pragma unroll 4
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x) run[b] = int32_t(offs[int64_t(b) * n_blocks + blockIdx.x]);
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t lo = int64_t(blockIdx.x) * chunk;
  const int64_t hi = min(n, lo + chunk);
  // the keys of eight groups are loaded together: a group at a time waited for its load
  constexpr int U = 8;
  int next[U];
  auto load = [&](int64_t g0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = g0 + u * 32 + lane;
      next[u] = i < hi ? __ldg(key + i) : -1 - lane;
    }
  };
  load(lo);
  for (int64_t g0 = lo; g0 < hi; g0 += U * 32) {
    int cur[U];
#pragma unroll
    for (int u = 0; u < U; ++u) cur[u] = next[u];
    load(g0 + U * 32);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = cur[u];
      const unsigned peers = __match_any_sync(0xffffffffu, k);
      const int rank = __popc(peers & lt);
      int base = 0;
      if (k >= 0) base = run[k];
      __syncwarp();
      if (k >= 0) {
        out_ids[base + rank] = int32_t(g0 + u * 32 + lane);
        const int leader = 31 - __clz(peers);
        if (lane == leader) run[k] = base + __popc(peers);
      }
      __syncwarp();
    }
  }
}

__global__ void k_bin_ptr(const int64_t *__restrict__ offs, int n_bins, int n_blocks, int64_t n,
                          int64_t *__restrict__ bin_ptr) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < n_bins) bin_ptr[b] = offs[int64_t(b) * n_blocks];
  if (b == n_bins) bin_ptr[b] = n;
}

}  // namespace

wproj_status exclusive_scan_i32_to_i64(const int32_t *in, int64_t *out, int64_t n, cudaStream_t s) {
  return exclusive_scan<int32_t, int64_t>(in, out, n, nullptr, true, s);
}
wproj_status exclusive_scan_i64(const int64_t *in, int64_t *out, int64_t n, cudaStream_t s) {
  return exclusive_scan<int64_t, int64_t>(in, out, n, nullptr, true, s);
}

// exclusive scan of in[0 .. n) with the total in out[n]; does not wait for it
wproj_status exclusive_scan_total(const int32_t *in, int64_t *out, int64_t n, cudaStream_t s) {
  return exclusive_scan<int32_t, int64_t>(in, out, n, out + n, false, s);
}

wproj_status stable_bin_sort(const int32_t *key, int64_t n, int n_bins, int32_t *out_ids,
                             int64_t *bin_ptr, cudaStream_t s, bool wait) {
  if (n >= (int64_t(1) << 31)) return fail(WPROJ_ERR_UNSUPPORTED, "stable_bin_sort: too many items");
  if (n_bins > 16384) return fail(WPROJ_ERR_UNSUPPORTED, "stable_bin_sort: too many bins");
  int n_blocks = (int)std::min<int64_t>(1024, std::max<int64_t>(1, (n + 4095) / 4096));
  int64_t chunk = (n + n_blocks - 1) / n_blocks;
  chunk = std::max<int64_t>(32, (chunk + 31) / 32 * 32);
  n_blocks = (int)std::max<int64_t>(1, (n + chunk - 1) / chunk);
  TmpBuf hist, offs;
  const int64_t nh = int64_t(n_bins) * n_blocks;
  WPROJ_TRY(hist.alloc(sizeof(int32_t) * nh));
  WPROJ_TRY(offs.alloc(sizeof(int64_t) * nh));
  const size_t smem = sizeof(int32_t) * n_bins;
  if (smem > 48 * 1024) {
    WPROJ_CUDA(cudaFuncSetAttribute(k_bin_hist, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    WPROJ_CUDA(cudaFuncSetAttribute(k_bin_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  }
  if (n > 0) {
    k_bin_hist<<<n_blocks, 256, smem, s>>>(key, n, chunk, n_bins, n_blocks, hist.as<int32_t>());
    WPROJ_CHECK_LAUNCH("bin hist");
  } else {
    WPROJ_CUDA(cudaMemsetAsync(hist.ptr, 0, sizeof(int32_t) * nh, s));
  }
  WPROJ_TRY((exclusive_scan<int32_t, int64_t>(hist.as<int32_t>(), offs.as<int64_t>(), nh, nullptr, false, s)));
  if (n > 0) {
    const int thr = std::min(1024, std::max(32, n_bins / 16 / 32 * 32));
    k_bin_scatter<<<n_blocks, thr, smem, s>>>(key, n, chunk, n_bins, n_blocks, offs.as<int64_t>(), out_ids);
    WPROJ_CHECK_LAUNCH("bin scatter");
  }
  k_bin_ptr<<<(n_bins + 1 + 255) / 256, 256, 0, s>>>(offs.as<int64_t>(), n_bins, n_blocks, n, bin_ptr);
  WPROJ_CHECK_LAUNCH("bin ptr");
  if (wait || hist.own || offs.own) WPROJ_CUDA(cudaStreamSynchronize(s));
  return WPROJ_OK;
}

}  // namespace wproj
