// Degridding and gridding of short rows (kernel boxes of at most 64 x 64 cells) from
// interleaved slices: every warp step is 32 consecutive values, 32 consecutive
// 2-byte local indices, 32 gathers from shared memory and four FMAs a lane, with
// no per-entry bookkeeping, no atomics and a fixed order of sums.
//
//  degridding  rows sorted by the grid tile of their visibility and, inside it, by
//              falling length.  A chunk is a run of rows of one tile; their kernels
//              lie in a patch of the grid of at most 96 x 96 cells (66 x 66 on the
//              precision-form workload), which a block holds in shared memory.  A
//              slice is four consecutive rows, eight lanes a row: step j holds the
//              entries 8 j .. 8 j + 7 of each row, so rows of a slice, alike in
//              length, end together.  Index: the cell's place in the patch.
//  gridding    a chunk is a run of one tile's (row, tile) segments (all of them on
//              large grids); a block loads their y into shared memory.  The tile's
//              1024 cells, sorted by falling number of entries, form 32 slices of 32
//              cells, a lane a cell: step j holds the j-th entry of each cell.  Index:
//              the row's place among the chunk's rows.  A lane sums its cell in a
//              register; a tile of one chunk is stored at once, the others' partial
//              tiles are added in chunk order.
// Pads hold the value 0 and the index 0, a shared-memory word that is 0.
//
// What bounds them: the stored bytes, 10 an entry (f32) or 6 (16-bit) plus the pads,
// where a tile holds many entries (N = 1024, M = 2^21, nnz 5.8e8: degridding 1.01 ms
// f32 / 0.75 bf16, gridding 0.94 / 0.70 ms, 86 / 70 % of the copy bandwidth on what is
// stored); the chain of latencies of a block (bounds, patch or y, values) where it
// holds few.  The forms they replace, on the same rows: run descriptors and X from
// L2 1.33 ms, private shared-memory tiles 1.85 ms (f32); 4-byte columns and X from L2
// 1.13 ms, segmented scans over a cell-sorted copy 1.64 ms (bf16), bound by issue and
// latency.  Measured and not taken: no patch, X through L1 (1.7 / 1.25 ms degridding;
// 207 against 190 us on a batch of 64 problems); one group of 8 steps in flight
// instead of two (1.08 / 0.86 ms); a warp's four cell slices one after another
// (gridding 0.97 / 0.75 ms, 204 against 167 us on the batch).
//
// Which plans take them: single plans up to kPatchCellsPerEntry patch cells an entry and
// pads up to the entries.  Rows of 1 to 4 entries take 8 places in the degridding's copy,
// several times the column form's bytes: Phi + Phi^H of 2e6 such rows on a 2048^2 grid
// 252 us on slices and 185 in the column form in bf16 (243 and 984 with run lengths in
// f32, the line's dear side).  Batches have neither line and need less memory on slices
// (64 sparse problems of N = 256: 424 to 514 MB, 508 to 580 without).  64 problems with
// and without slices: N = 64, 40 to 400 rows each, 28 to 38 us and 33 to 46; N = 256,
// 6000 rows of 78 entries, 409 and 443; N = 256, 60 to 600 rows or rows of 1 to 6
// entries, 260 to 336 and 249 to 305: sparse problems on large grids are the dear side.
//
// Chunk sizes: 6 to 24 (degridding) and 8 to 16 (gridding) blocks an SM are within 7 %, 32
// for the gridding up to 80 % slower; at least 4096 entries: 2048 is 20 to 32 % slower on
// 64^2 and 7 to 12 % on 256^2 images; a batch's 16384: 8192 makes its gridding 30 %
// slower; at most 262144: 65536 makes the gridding of 5.8e8 entries 13 to 18 % slower,
// 1048576 is the same.
//
// Building them (262144 rows, 7e7 entries): two stable sorts of the rows, a sort of each
// tile's cells (keys in registers, 15 of the 55 exchanges through shared memory: 0.2 ms)
// and two passes that place the values, ~2 ms of a build of 27.9 ms.
#include <algorithm>
#include <vector>

#include "plan.h"

namespace wproj {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kLpr = 8;              // degridding: lanes per row
constexpr int kRps = 32 / kLpr;      // rows per slice
constexpr int kMaxRowsChunk = 12288; // rows of a gridding chunk (96 KB of y)
constexpr int kMaxLen = 4096;        // entries of a row (64 x 64)
constexpr int kMaxPatch = 96;        // sides of a patch: a tile's 32 cells and the windows of 64 around them

// odd row stride of the patch in shared memory
__host__ __device__ __forceinline__ int patch_stride(int wv) { return wv | 1; }
__host__ __device__ __forceinline__ int patch_words(int hu, int wv) { return 1 + hu * patch_stride(wv); }

// The operators' limits of dynamic shared memory: a limit belongs to the kernel, which
// plans of other threads launch too, so it is the most that any plan takes (75 and 98 KB)
// and not the plan's own size.
const int kMaxDegridSmem = int(sizeof(float2)) * patch_words(kMaxPatch, kMaxPatch);
constexpr int kMaxGridSmem = int(sizeof(float2)) * (1 + kMaxRowsChunk);

template <int VDT> struct RawVal { using type = unsigned; };
template <> struct RawVal<WPROJ_VAL_F32> { using type = float2; };

template <int VDT>
__device__ __forceinline__ float2 to_f2(typename RawVal<VDT>::type r) {
  if constexpr (VDT == WPROJ_VAL_F32) return r;
  else if constexpr (VDT == WPROJ_VAL_BF16) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&r));
  else return __half22float2(*reinterpret_cast<const __half2 *>(&r));
}

// Ask for [p, p + bytes) in L2 (both multiples of 16), at most kAhead of it: a block's
// values are on their way while it loads its patch or its y.  Small chunks (a batch's
// tiles of ~100 rows, 5 of the warp steps a slice) are otherwise a chain of exposed
// memory latencies.
constexpr int64_t kAhead = 65536;
__device__ __forceinline__ void prefetch_l2(const void *p, int64_t bytes) {
  const uint32_t n = uint32_t(bytes < kAhead ? bytes : kAhead);
  if (n) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// ---- operators -----------------------------------------------------------------------------

__device__ __forceinline__ void cp_async8(float2 *dst, const float2 *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}

// A warp's slices of a chunk are walked as one sequence of groups of U steps; the next
// group's loads are in flight while this one is used, across slice ends too.
template <int VDT, int U>
__global__ void __launch_bounds__(kThreads, 4)
k_slice_degrid(const SliceOps o, const float2 *__restrict__ X, float2 *__restrict__ y) {
  extern __shared__ float2 sh[];
  using Raw = typename RawVal<VDT>::type;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x;
  const int64_t s0 = o.d_slice_base[c], s1 = o.d_slice_base[c + 1];
  if (s0 >= s1) {
    chain_wait();
    return;
  }
  const int4 r = o.rect[c];
  int logG = o.logG;
  if (o.tab) {
    const BProb &P = o.tab[o.d_chunk_prob[c]];
    logG = P.logG;
    X += P.grid_off;
  }
  const int Gm = (1 << logG) - 1, ws = patch_stride(r.w);
  const Raw *__restrict__ val = static_cast<const Raw *>(o.d_val);
  if (threadIdx.x == 0) {
    sh[0] = make_float2(0.f, 0.f);
    const int64_t a = o.slice_ptr[s0] * 32, n = o.slice_ptr[s1] * 32 - a;
    prefetch_l2(val + a, n * int(sizeof(Raw)));
    prefetch_l2(o.d_idx + a, n * 2);
  }
  // lane t holds the bounds of the warp's slice t (of each 32)
  long long pl = 0;
  int nl = 0;
  auto bounds = [&](int64_t s) {
    nl = 0;
    if (s < s1) {
      pl = o.slice_ptr[s];
      nl = int(o.slice_ptr[s + 1] - pl);
    }
  };
  bounds(s0 + w + int64_t(lane) * kWarps);
  chain_wait();
  X = after_wait(X);
  for (int a = w; a < r.z; a += kWarps) {
    const float2 *row = X + (int64_t((r.x + a) & Gm) << logG);
    for (int b = lane; b < r.w; b += 32) cp_async8(&sh[1 + a * ws + b], row + ((r.y + b) & Gm));
  }
  Raw v[U], vn[U];
  uint16_t id[U], idn[U];
  auto load = [&](long long p, int n, int j, Raw(&a)[U], uint16_t(&b)[U]) {
    const Raw *__restrict__ vp = val + (p + j) * 32 + lane;
    const uint16_t *__restrict__ ip = o.d_idx + (p + j) * 32 + lane;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j + u < n) {   // the same in every lane
        a[u] = __ldg(vp + u * 32);
        b[u] = __ldg(ip + u * 32);
      } else {
        a[u] = Raw{};
        b[u] = 0;
      }
    }
  };
  long long p0 = __shfl_sync(kFull, pl, 0);
  int n0 = __shfl_sync(kFull, nl, 0);
  load(p0, n0, 0, v, id);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  chain_next();
  int t = 0;
  for (int64_t s = s0 + w; s < s1; s += kWarps) {
    // the next slice
    long long p1 = 0;
    int n1 = 0;
    if (++t == 32) {
      t = 0;
      bounds(s + kWarps + int64_t(lane) * kWarps);
    }
    p1 = __shfl_sync(kFull, pl, t);
    n1 = s + kWarps < s1 ? __shfl_sync(kFull, nl, t) : 0;
    const int k = (lane & (kLpr - 1)) == 0 ? __ldg(o.srow + s * kRps + lane / kLpr) : -1;
    float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f;
    for (int j = 0; j == 0 || j < n0; j += U) {
      const bool last = j + U >= n0;
      load(last ? p1 : p0, last ? n1 : n0, last ? 0 : j + U, vn, idn);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float2 x = sh[id[u]], g = to_f2<VDT>(v[u]);
        if (u & 1) {
          bx = fmaf(g.x, x.x, bx); bx = fmaf(-g.y, x.y, bx);
          by = fmaf(g.x, x.y, by); by = fmaf(g.y, x.x, by);
        } else {
          ax = fmaf(g.x, x.x, ax); ax = fmaf(-g.y, x.y, ax);
          ay = fmaf(g.x, x.y, ay); ay = fmaf(g.y, x.x, ay);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u] = vn[u];
        id[u] = idn[u];
      }
    }
    p0 = p1;
    n0 = n1;
    ax += bx;
    ay += by;
#pragma unroll
    for (int d = kLpr / 2; d; d >>= 1) {
      ax += __shfl_xor_sync(kFull, ax, d);
      ay += __shfl_xor_sync(kFull, ay, d);
    }
    if (k >= 0) {
      const float f = o.row_scale ? __ldg(o.row_scale + k) : 1.f;
      y[k] = o.row_scale ? make_float2(ax * f, ay * f) : make_float2(ax, ay);
    }
  }
}

template <int VDT>
__global__ void __launch_bounds__(kThreads, 4)
k_slice_grid(const SliceOps o, const float2 *__restrict__ y, float2 *__restrict__ partial, float2 *__restrict__ Xt2) {
  extern __shared__ float2 sh[];   // word 0 is 0, then the chunk's y
  __shared__ float2 cell[1024];
  using Raw = typename RawVal<VDT>::type;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = blockIdx.x;
  chain_wait();   // the first kernel of Phi^H
  y = after_wait(y);
  // The slices are sorted by length: the warps take them to and fro, four each, step
  // by step together, so that tiles of a few entries a cell still have loads in
  // flight.  The first steps are asked for before the y are gathered.
  constexpr int NQ = 32 / kWarps, U = 2;
  const uint32_t *__restrict__ slp = o.g_slp + int64_t(c) * 33;
  const uint32_t lo_l = __ldg(slp + lane), hi_l = __ldg(slp + lane + 1);
  const int64_t base = o.g_base[c] * 32 + lane;
  const Raw *__restrict__ val = static_cast<const Raw *>(o.g_val) + base;
  const uint16_t *__restrict__ idx = o.g_idx + base;
  uint32_t p0[NQ];
  int n[NQ], nmax = 0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int sl = q * kWarps + ((q & 1) ? kWarps - 1 - w : w);
    p0[q] = __shfl_sync(kFull, lo_l, sl);
    n[q] = int(__shfl_sync(kFull, hi_l, sl) - p0[q]);
    nmax = max(nmax, n[q]);
  }
  Raw v[NQ][U];
  uint16_t id[NQ][U];
  auto load = [&](int j) {
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (j + u < n[q]) {   // the same in every lane
          const int64_t at = int64_t(p0[q] + uint32_t(j + u)) * 32;
          v[q][u] = __ldg(val + at);
          id[q][u] = __ldg(idx + at);
        } else {
          v[q][u] = Raw{};
          id[q][u] = 0;
        }
  };
  load(0);
  const int64_t rb = o.g_row_base[c];
  const int nrow = int(o.g_row_base[c + 1] - rb);
  if (threadIdx.x == 0) sh[0] = make_float2(0.f, 0.f);
  for (int i = threadIdx.x; i < nrow; i += kThreads) {
    const int k = __ldg(o.g_rows + rb + i);
    float2 t = y[k];
    if (o.row_scale) t = cscale(t, __ldg(o.row_scale + k));
    sh[1 + i] = t;
  }
  __syncthreads();
  float2 acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) acc[q] = make_float2(0.f, 0.f);
  for (int j = 0; j < nmax; j += U) {
    Raw g0[NQ][U];
    uint16_t i0[NQ][U];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        g0[q][u] = v[q][u];
        i0[q][u] = id[q][u];
      }
    load(j + U);
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float2 t = sh[i0[q][u]], g = to_f2<VDT>(g0[q][u]);   // conj(g) y
        acc[q].x = fmaf(g.x, t.x, acc[q].x); acc[q].x = fmaf(g.y, t.y, acc[q].x);
        acc[q].y = fmaf(g.x, t.y, acc[q].y); acc[q].y = fmaf(-g.y, t.x, acc[q].y);
      }
  }
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const int sl = q * kWarps + ((q & 1) ? kWarps - 1 - w : w);
    cell[__ldg(o.g_perm + int64_t(c) * 1024 + sl * 32 + lane)] = acc[q];
  }
  chain_next();
  __syncthreads();
  int tile = o.g_chunk_tile[c], logG = o.logG, t0 = 0;
  if (o.tab) {
    const BProb &P = o.tab[o.g_chunk_prob[c]];
    logG = P.logG;
    t0 = int(P.tile_off);
    Xt2 += P.grid_off;
  }
  const bool single = o.tile_chunk_ptr[t0 + tile + 1] - o.tile_chunk_ptr[t0 + tile] == 1;
  const int tu = tile >> (logG - 5), tv = tile & ((1 << (logG - 5)) - 1);
  for (int e = threadIdx.x; e < 1024; e += kThreads) {
    if (single) Xt2[(int64_t(tu * 32 + (e >> 5)) << logG) + tv * 32 + (e & 31)] = cell[e];
    else partial[int64_t(c) * 1024 + e] = cell[e];
  }
}

// the tiles of several chunks (multi): partial tiles added in chunk order (block: 32
// cells, 8 chunk lanes)
__global__ void __launch_bounds__(256)
k_slice_reduce(const SliceOps o, const float2 *__restrict__ partial, float2 *__restrict__ Xt2) {
  __shared__ float2 red[8][32];
  chain_next();
  int tile = o.multi[blockIdx.x], logG = o.logG;
  const int c0 = o.tile_chunk_ptr[tile], c1 = o.tile_chunk_ptr[tile + 1];
  if (o.tab) {
    const BProb &P = o.tab[o.tile_prob[tile]];
    logG = P.logG;
    tile -= int(P.tile_off);
    Xt2 += P.grid_off;
  }
  const int e = blockIdx.y * 32 + (threadIdx.x & 31), j = threadIdx.x >> 5;
  chain_wait();
  partial = after_wait(partial);
  float2 s = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int c = c0 + j; c < c1; c += 8) s = cadd(s, partial[int64_t(c) * 1024 + e]);
  red[j][threadIdx.x & 31] = s;
  __syncthreads();
  if (j == 0) {
#pragma unroll
    for (int q = 1; q < 8; ++q) s = cadd(s, red[q][threadIdx.x]);
    const int tu = tile >> (logG - 5), tv = tile & ((1 << (logG - 5)) - 1);
    Xt2[(int64_t(tu * 32 + (e >> 5)) << logG) + tv * 32 + (e & 31)] = s;
  }
}

// ---- building the degridding slices from the column form -------------------------------------

__device__ __forceinline__ int axis_tile_of(int j, int Gm) { return (j & Gm) >> 5; }

// sort keys (tile of the visibility's cell; 4096 - length), the extent of a row's
// support from its window origin (j0 - S/2): u0 | u1 << 8 | v0 << 16 | v1 << 24, and its
// runs of consecutive columns, cut at tile edges.  Warp per row.
__global__ void __launch_bounds__(256)
k_row_keys(int64_t m, const int64_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
           const int2 *__restrict__ j0, const int32_t *__restrict__ Sk, int logG, int32_t *__restrict__ key,
           int32_t *__restrict__ tile, uint32_t *__restrict__ ext, int32_t *__restrict__ row_runs) {
  const int lane = threadIdx.x & 31, Gm = (1 << logG) - 1;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t k = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; k < m; k += nw) {
    const int64_t e0 = row_ptr[k], e1 = row_ptr[k + 1];
    const int2 j = j0[k];
    const int h = Sk[k] / 2, au = (j.x - h) & Gm, av = (j.y - h) & Gm;
    int nu = 255, xu = 0, nv = 255, xv = 0, nr = 0;
    for (int64_t e = e0 + lane; e < e1; e += 32) {
      const int q = __ldg(col + e);
      nr += e == e0 || (q & 31) == 0 || __ldg(col + e - 1) != q - 1;
      const int du = ((q >> logG) - au) & Gm, dv = ((q & Gm) - av) & Gm;
      nu = min(nu, du); xu = max(xu, du);
      nv = min(nv, dv); xv = max(xv, dv);
    }
    nu = __reduce_min_sync(kFull, nu); xu = __reduce_max_sync(kFull, xu);
    nv = __reduce_min_sync(kFull, nv); xv = __reduce_max_sync(kFull, xv);
    nr = __reduce_add_sync(kFull, nr);
    if (lane == 0) {
      row_runs[k] = nr;
      key[k] = kMaxLen - int(min(int64_t(kMaxLen), e1 - e0));
      tile[k] = (axis_tile_of(j.x, Gm) << (logG - 5)) | axis_tile_of(j.y, Gm);
      ext[k] = uint32_t(nu) | (uint32_t(xu) << 8) | (uint32_t(nv) << 16) | (uint32_t(xv) << 24);
    }
  }
}

__global__ void k_pick_i32(int64_t n, const int32_t *__restrict__ idx, const int32_t *__restrict__ src,
                           int32_t *__restrict__ dst) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[idx[i]];
}

// the sorted rows and their entries
__global__ void k_sorted_len(int64_t m, const int32_t *__restrict__ idx, const int32_t *__restrict__ src,
                             const int64_t *__restrict__ row_ptr, int32_t *__restrict__ perm,
                             int32_t *__restrict__ len) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const int k = src[idx[i]];
  perm[i] = k;
  len[i] = int32_t(row_ptr[k + 1] - row_ptr[k]);
}

// Block per chunk: its patch (the smallest rectangle that holds its rows' supports,
// the whole axis where that would be as long), the patch's cells and its slices.
__global__ void __launch_bounds__(128)
k_chunk_patch(const int32_t *__restrict__ chunk_tile, const int64_t *__restrict__ chunk_lo,
              const int64_t *__restrict__ chunk_hi, const int32_t *__restrict__ perm, const int32_t *__restrict__ len,
              const int2 *__restrict__ j0, const int32_t *__restrict__ Sk, const uint32_t *__restrict__ ext, int logG,
              int4 *__restrict__ rect, int32_t *__restrict__ cells, int32_t *__restrict__ slices,
              int *__restrict__ max_words) {
  __shared__ int mn[2], mx[2];
  const int c = blockIdx.x, G = 1 << logG, Gm = G - 1, nT = G >> 5;
  const int64_t lo = chunk_lo[c], hi = chunk_hi[c];
  if (threadIdx.x < 2) { mn[threadIdx.x] = 1 << 20; mx[threadIdx.x] = -1; }
  __syncthreads();
  // offsets from 32 cells before the tile: window origins lie within [0, 64) of it
  const int bu = ((chunk_tile[c] / nT) * 32 - 32) & Gm, bv = ((chunk_tile[c] % nT) * 32 - 32) & Gm;
  int nu = 1 << 20, xu = -1, nv = 1 << 20, xv = -1;
  for (int64_t i = lo + threadIdx.x; i < hi; i += 128) {
    if (len[i] <= 0) continue;
    const int k = perm[i], h = Sk[k] / 2;
    const int ru = (j0[k].x - h - bu) & Gm, rv = (j0[k].y - h - bv) & Gm;
    const uint32_t e = ext[k];
    nu = min(nu, ru + int(e & 255u)); xu = max(xu, ru + int((e >> 8) & 255u));
    nv = min(nv, rv + int((e >> 16) & 255u)); xv = max(xv, rv + int(e >> 24));
  }
  if (xu >= 0) {
    atomicMin(&mn[0], nu); atomicMax(&mx[0], xu);
    atomicMin(&mn[1], nv); atomicMax(&mx[1], xv);
  }
  __syncthreads();
  if (threadIdx.x) return;
  int4 r = make_int4(0, 0, 0, 0);
  if (mx[0] >= 0) {
    r = make_int4((bu + mn[0]) & Gm, (bv + mn[1]) & Gm, mx[0] - mn[0] + 1, mx[1] - mn[1] + 1);
    if (r.z >= G) { r.x = 0; r.z = G; }
    if (r.w >= G) { r.y = 0; r.w = G; }
  }
  rect[c] = r;
  cells[c] = r.z * r.w;
  slices[c] = int32_t((hi - lo + kRps - 1) / kRps);
  atomicMax(max_words, patch_words(r.z, r.w));
}

// Block per chunk: steps of every slice (its first row is its longest) and its rows
__global__ void __launch_bounds__(128)
k_slice_steps(const int64_t *__restrict__ chunk_lo, const int64_t *__restrict__ chunk_hi,
              const int64_t *__restrict__ slice_base, const int32_t *__restrict__ perm, const int32_t *__restrict__ len,
              int32_t *__restrict__ steps, int32_t *__restrict__ srow) {
  const int c = blockIdx.x;
  const int64_t lo = chunk_lo[c], hi = chunk_hi[c], b = slice_base[c], n = slice_base[c + 1] - b;
  for (int64_t s = threadIdx.x; s < n; s += 128) {
    steps[b + s] = (len[lo + s * kRps] + kLpr - 1) / kLpr;
    for (int r = 0; r < kRps; ++r) {
      const int64_t i = lo + s * kRps + r;
      srow[(b + s) * kRps + r] = i < hi ? perm[i] : -1;
    }
  }
}

// Values and indices of the degridding slices; block per chunk, warp per row (the pads
// of both arrays set beforehand)
__global__ void __launch_bounds__(256)
k_slice_fill(const int64_t *__restrict__ slice_base, const int64_t *__restrict__ slice_ptr,
             const int32_t *__restrict__ srow, const int4 *__restrict__ rect, const int64_t *__restrict__ row_ptr,
             const int32_t *__restrict__ col, const unsigned char *__restrict__ val, int vb, int logG,
             uint16_t *__restrict__ out_idx, unsigned char *__restrict__ out_val) {
  const int c = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5, Gm = (1 << logG) - 1;
  const int4 r = rect[c];
  const int ws = patch_stride(r.w);
  const int64_t q0 = slice_base[c] * kRps, q1 = slice_base[c + 1] * kRps;
  for (int64_t q = q0 + w; q < q1; q += 8) {
    const int k = srow[q];
    if (k < 0) continue;
    const int64_t s = q / kRps, at = slice_ptr[s] * 32 + (q % kRps) * kLpr;
    const int64_t e0 = row_ptr[k];
    const int n = int(min(row_ptr[k + 1] - e0, (slice_ptr[s + 1] - slice_ptr[s]) * kLpr));
    for (int e = lane; e < n; e += 32) {
      const int cl = __ldg(col + e0 + e);
      const int du = ((cl >> logG) - r.x) & Gm, dv = ((cl & Gm) - r.y) & Gm;
      const int64_t d = at + int64_t(e / kLpr) * 32 + (e & (kLpr - 1));
      out_idx[d] = uint16_t(1 + du * ws + dv);
      if (vb == 8) reinterpret_cast<float2 *>(out_val)[d] = reinterpret_cast<const float2 *>(val)[e0 + e];
      else reinterpret_cast<unsigned *>(out_val)[d] = reinterpret_cast<const unsigned *>(val)[e0 + e];
    }
  }
}

// ---- building the gridding slices from the tile-ordered segments -------------------------------

// Block per chunk: entries per cell, the cells sorted by falling count (ties by cell),
// the steps of the 32 slices and the rows (segments holding entries)
__global__ void __launch_bounds__(1024)
k_cell_sort(const int64_t *__restrict__ chunk_lo, const int64_t *__restrict__ chunk_hi,
            const int32_t *__restrict__ chunk_tile, const SegMeta *__restrict__ meta, const int32_t *__restrict__ col,
            int logG, uint16_t *__restrict__ perm, uint32_t *__restrict__ slp, int32_t *__restrict__ chunk_steps,
            int32_t *__restrict__ chunk_rows, int *__restrict__ max_rows) {
  __shared__ int cnt[1024];
  __shared__ uint32_t key[2][1024];
  __shared__ int rows, top[32];
  const int c = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int Gm = (1 << logG) - 1, nT = 1 << (logG - 5);
  const int tu = chunk_tile[c] / nT, tv = chunk_tile[c] % nT;
  if (chunk_lo[c] >= chunk_hi[c]) {   // most tiles of a sparsely covered grid
    perm[int64_t(c) * 1024 + t] = uint16_t(t);
    if (t < 33) slp[int64_t(c) * 33 + t] = 0;
    if (t == 0) chunk_steps[c] = chunk_rows[c] = 0;
    return;
  }
  cnt[t] = 0;
  if (t == 0) rows = 0;
  __syncthreads();
  int mine = 0;
  for (int64_t s = chunk_lo[c] + w; s < chunk_hi[c]; s += 32) {
    const SegMeta m = meta[s];
    const int n = meta_cnt(m);
    mine += n > 0;
    for (int e = lane; e < n; e += 32) {
      const int q = __ldg(col + meta_off(m) + e);
      atomicAdd(&cnt[((((q >> logG) - tu * 32) & 31) << 5) | (((q & Gm) - tv * 32) & 31)], 1);
    }
  }
  if (lane == 0 && mine) atomicAdd(&rows, mine);
  __syncthreads();
  // bitonic, descending: a key a thread, partners of other warps through shared memory
  uint32_t k = (uint32_t(cnt[t]) << 10) | uint32_t(1023 - t);   // counts < 2^22
  if (__syncthreads_or(cnt[t])) {
    int b = 0;
    for (int size = 2; size <= 1024; size <<= 1)
      for (int d = size >> 1; d; d >>= 1) {
        uint32_t o;
        if (d < 32) {
          o = __shfl_xor_sync(kFull, k, d);
        } else {
          key[b][t] = k;
          __syncthreads();
          o = key[b][t ^ d];
          b ^= 1;
        }
        k = ((t & size) == 0) == ((t & d) == 0) ? max(k, o) : min(k, o);
      }
  }
  perm[int64_t(c) * 1024 + t] = uint16_t(1023 - (k & 1023u));
  if (lane == 0) top[w] = int(k >> 10);
  __syncthreads();
  if (w == 0) {
    const int n = top[lane];
    int inc = n;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += v;
    }
    slp[int64_t(c) * 33 + lane] = uint32_t(inc - n);
    if (lane == 31) {
      slp[int64_t(c) * 33 + 32] = uint32_t(inc);
      chunk_steps[c] = inc;
      chunk_rows[c] = rows;
      atomicMax(max_rows, rows);
    }
  }
}

// Values, indices and the row list of the gridding slices; block per chunk, 32
// segments a round, their entries spread over the threads (a warp per segment waited
// for the longest: 2.6 ms for 7e7 entries).  A cell's entries take their places in
// segment order: the segments of a round that hold the cell set a bit each, and an
// entry's rank is the cell's count so far plus the bits below its segment's.
constexpr size_t kFillSmem = sizeof(uint16_t) * 32 * 1024;   // (segment, cell) of a round's entries
__global__ void __launch_bounds__(1024)
k_cell_fill(const int64_t *__restrict__ chunk_lo, const int64_t *__restrict__ chunk_hi,
            const int32_t *__restrict__ chunk_tile, const SegMeta *__restrict__ meta, const int32_t *__restrict__ col,
            const unsigned char *__restrict__ val, int vb, int logG, const uint16_t *__restrict__ perm,
            const uint32_t *__restrict__ slp, const int64_t *__restrict__ base, const int64_t *__restrict__ row_base,
            int32_t *__restrict__ rows, uint16_t *__restrict__ out_idx, unsigned char *__restrict__ out_val) {
  extern __shared__ uint16_t at_cell[];
  __shared__ int cnt[1024];
  __shared__ unsigned mask[2][1024];
  __shared__ uint32_t place[1024];   // first step of the cell's slice << 5 | lane
  const int c = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int Gm = (1 << logG) - 1, nT = 1 << (logG - 5);
  const int tu = chunk_tile[c] / nT, tv = chunk_tile[c] % nT;
  const int64_t b0 = base[c] * 32, lo = chunk_lo[c], hi = chunk_hi[c], rb = row_base[c];
  if (lo >= hi) return;
  cnt[t] = 0;
  mask[0][t] = mask[1][t] = 0;
  place[perm[int64_t(c) * 1024 + t]] = (slp[int64_t(c) * 33 + w] << 5) | uint32_t(lane);
  __syncthreads();
  int nrow = 0, b = 0;   // rows before the round; the masks' buffer
  SegMeta next{};
  if (lo + lane < hi) next = meta[lo + lane];
  for (int64_t s0 = lo; s0 < hi; s0 += 32, b ^= 1) {
    // every warp: segment s0 + lane, its entries and their end in the round
    const SegMeta m = next;
    const int n = s0 + lane < hi ? meta_cnt(m) : 0;
    const int64_t off = meta_off(m);
    if (s0 + 32 + lane < hi) next = meta[s0 + 32 + lane];
    int end = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, end, o);
      if (lane >= o) end += v;
    }
    const int total = __shfl_sync(kFull, end, 31);
    const int64_t src = off - (end - n);   // + the entry's place in the round
    const unsigned some = __ballot_sync(kFull, n > 0);
    if (w == 0 && n > 0) rows[rb + nrow + __popc(some & ((1u << lane) - 1u))] = m.row;
    for (int e0 = w * 32; e0 < total; e0 += 1024) {
      const int e = e0 + lane;
      int sg = 0;   // segments that end at or before e
#pragma unroll
      for (int o = 16; o; o >>= 1)
        if (__shfl_sync(kFull, end, sg + o - 1) <= e) sg += o;
      const int64_t at = __shfl_sync(kFull, src, sg) + e;
      if (e < total) {
        const int q = __ldg(col + at);
        const int cl = ((((q >> logG) - tu * 32) & 31) << 5) | (((q & Gm) - tv * 32) & 31);
        at_cell[e] = uint16_t((sg << 10) | cl);
        atomicOr(&mask[b][cl], 1u << sg);
      }
    }
    __syncthreads();
    for (int e0 = w * 32; e0 < total; e0 += 1024) {
      const int e = e0 + lane;
      const unsigned sc = e < total ? at_cell[e] : 0u;
      const int sg = int(sc >> 10), cl = int(sc & 1023u);
      const int64_t at = __shfl_sync(kFull, src, sg) + e;
      if (e < total) {
        const uint32_t p = place[cl];
        const unsigned lt = (1u << sg) - 1u;
        const int rank = cnt[cl] + __popc(mask[b][cl] & lt);
        const int64_t d = b0 + (int64_t(p >> 5) + rank) * 32 + (p & 31u);
        out_idx[d] = uint16_t(1 + nrow + __popc(some & lt));
        if (vb == 8) reinterpret_cast<float2 *>(out_val)[d] = __ldg(reinterpret_cast<const float2 *>(val) + at);
        else reinterpret_cast<unsigned *>(out_val)[d] = __ldg(reinterpret_cast<const unsigned *>(val) + at);
      }
    }
    nrow += __popc(some);
    __syncthreads();
    cnt[t] += __popc(mask[b][t]);   // read again after the next round's barrier
    mask[b][t] = 0;
  }
}

int clamp_blocks(int64_t n, int per) { return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, per), 152 * 64)); }

template <int VDT>
wproj_status launch_degrid(const SliceOps &o, size_t smem, const float2 *X, float2 *y, cudaStream_t s) {
  constexpr int U = VDT == WPROJ_VAL_F32 ? 6 : 8;   // steps per group (two groups in registers)
  WPROJ_CUDA(cudaFuncSetAttribute(k_slice_degrid<VDT, U>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDegridSmem));
  WPROJ_CUDA(launch_chained(k_slice_degrid<VDT, U>, (unsigned)o.d_chunks, kThreads, smem, s, o, X, y));
  WPROJ_CHECK_LAUNCH("degrid (slices)");
  return WPROJ_OK;
}
template <int VDT>
wproj_status launch_grid(const SliceOps &o, size_t smem, const float2 *y, float2 *partial, float2 *Xt2, cudaStream_t s) {
  WPROJ_CUDA(cudaFuncSetAttribute(k_slice_grid<VDT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxGridSmem));
  WPROJ_CUDA(launch_chained(k_slice_grid<VDT>, (unsigned)o.g_chunks, kThreads, smem, s, o, y, partial, Xt2));
  WPROJ_CHECK_LAUNCH("grid (slices)");
  if (o.n_multi > 0) {
    WPROJ_CUDA(launch_chained(k_slice_reduce, dim3((unsigned)o.n_multi, 32), 256, 0, s, o, partial, Xt2));
    WPROJ_CHECK_LAUNCH("grid (slices) partial tiles");
  }
  return WPROJ_OK;
}

SliceOps plan_ops(const wproj_plan *p) {
  SliceOps o = p->slices.ops();
  o.logG = ilog2(p->g.G);
  o.row_scale = p->g.value_dtype == WPROJ_VAL_F32 ? nullptr : p->row_scale.as<float>();
  return o;
}

wproj_status fill(wproj_plan *p, cudaStream_t s) {
  SliceCopy &c = p->slices;
  const int vb = p->g.value_dtype == WPROJ_VAL_F32 ? 8 : 4, logG = ilog2(p->g.G);
  k_slice_fill<<<(unsigned)c.d_chunks, 256, 0, s>>>(
      c.d_slice_base.as<int64_t>(), c.slice_ptr.as<int64_t>(), c.srow.as<int32_t>(), c.rect.as<int4>(),
      p->row_ptr.as<int64_t>(), p->col.as<int32_t>(), p->val.as<unsigned char>(), vb, logG, c.d_idx.as<uint16_t>(),
      c.d_val.as<unsigned char>());
  WPROJ_CUDA(cudaFuncSetAttribute(k_cell_fill, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFillSmem));
  k_cell_fill<<<(unsigned)c.g_chunks, 1024, kFillSmem, s>>>(
      c.g_chunk_lo.as<int64_t>(), c.g_chunk_hi.as<int64_t>(), c.g_chunk_tile.as<int32_t>(), p->seg_meta.as<SegMeta>(),
      p->col.as<int32_t>(), p->val.as<unsigned char>(), vb, logG, c.g_perm.as<uint16_t>(), c.g_slp.as<uint32_t>(),
      c.g_base.as<int64_t>(), c.g_row_base.as<int64_t>(), c.g_rows.as<int32_t>(), c.g_idx.as<uint16_t>(),
      c.g_val.as<unsigned char>());
  WPROJ_CHECK_LAUNCH("slice values");
  return WPROJ_OK;
}

}  // namespace

SliceOps SliceCopy::ops() const {
  SliceOps o;
  o.d_chunks = d_chunks;
  o.d_slice_base = d_slice_base.as<int64_t>();
  o.slice_ptr = slice_ptr.as<int64_t>();
  o.srow = srow.as<int32_t>();
  o.rect = rect.as<int4>();
  o.d_idx = d_idx.as<uint16_t>();
  o.d_val = d_val.ptr;
  o.g_chunks = g_chunks;
  o.g_chunk_tile = g_chunk_tile.as<int32_t>();
  o.tile_chunk_ptr = tile_chunk_ptr.as<int32_t>();
  o.multi = multi.as<int32_t>();
  o.n_multi = n_multi;
  o.g_base = g_base.as<int64_t>();
  o.g_slp = g_slp.as<uint32_t>();
  o.g_perm = g_perm.as<uint16_t>();
  o.g_row_base = g_row_base.as<int64_t>();
  o.g_rows = g_rows.as<int32_t>();
  o.g_idx = g_idx.as<uint16_t>();
  o.g_val = g_val.ptr;
  return o;
}

// values and indices; bounds and rows of a slice; base and patch of a chunk
int64_t SliceCopy::degrid_bytes(int value_bytes) const {
  return d_steps * 32 * (value_bytes + 2) + d_slices * (8 + 4 * kRps) + d_chunks * (8 + 16);
}
// values and indices; row lists; the cells' order, the slices' and the chunk's bounds
int64_t SliceCopy::grid_bytes(int value_bytes) const {
  return g_steps * 32 * (value_bytes + 2) + g_nrows * 4 + g_chunks * (2 * 1024 + 33 * 4 + 8 + 8 + 4);
}

void SliceCopy::release() {
  use = false;
  for (DevBuf *b : {&d_slice_base, &slice_ptr, &srow, &rect, &d_idx, &d_val, &g_chunk_tile, &g_chunk_lo, &g_chunk_hi,
                    &tile_chunk_ptr, &g_base, &g_slp, &g_perm, &g_row_base, &g_rows, &g_idx, &g_val, &multi, &partial})
    b->release();
  d_chunks = d_slices = d_steps = g_chunks = g_steps = g_nrows = n_multi = 0;
  d_smem = g_smem = 0;
}

// Slices of a plan whose G sits in the column form (p->col / p->val, 32-cell tiles,
// boxes of at most 64 x 64 cells): p->slices.use tells whether the operators take
// them.  tptr / cum: first segment of every tile and entry prefix of the segments
// p->seg_meta in tile order.  row_runs[m] receives an upper bound of each row's runs.
wproj_status build_slices(wproj_plan *p, const int2 *j0, const int32_t *Sk, const int64_t *tptr, const int64_t *cum,
                          int64_t n_seg, int32_t *row_runs, cudaStream_t s) {
  const GridGeom &g = p->g;
  SliceCopy &c = p->slices;
  c.use = false;   // the arrays are kept where the new ones fit
  c.n_multi = 0;
  const int64_t m = p->m;
  const int vb = g.value_dtype == WPROJ_VAL_F32 ? 8 : 4, logG = ilog2(g.G), n_tiles = g.nT * g.nT;
  // ---- degridding: rows by tile, then by falling length
  TmpBuf key, tile, ext, ids, ids2, rtptr, len, rcum, perm, cells, cbase, nsl, steps, stat;
  TmpBuf ctile, clo, chi, ctp;
  WPROJ_TRY(key.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(tile.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(ext.alloc(sizeof(uint32_t) * m));
  WPROJ_TRY(ids.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(ids2.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(perm.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(len.alloc(sizeof(int32_t) * m));
  WPROJ_TRY(rcum.alloc(sizeof(int64_t) * m));
  WPROJ_TRY(rtptr.alloc(sizeof(int64_t) * (std::max(n_tiles, kMaxLen + 1) + 1)));
  WPROJ_TRY(stat.alloc(sizeof(int) * 2));   // words of the largest patch, rows of the largest gridding chunk
  WPROJ_CUDA(cudaMemsetAsync(stat.ptr, 0, sizeof(int) * 2, s));
  k_row_keys<<<clamp_blocks(m, 8), 256, 0, s>>>(m, p->row_ptr.as<int64_t>(), p->col.as<int32_t>(), j0, Sk, logG,
                                                key.as<int32_t>(), tile.as<int32_t>(), ext.as<uint32_t>(), row_runs);
  WPROJ_CHECK_LAUNCH("row keys");
  WPROJ_TRY(stable_bin_sort(key.as<int32_t>(), m, kMaxLen + 1, ids.as<int32_t>(), rtptr.as<int64_t>(), s, false));
  k_pick_i32<<<ceil_div(m, 256), 256, 0, s>>>(m, ids.as<int32_t>(), tile.as<int32_t>(), key.as<int32_t>());
  WPROJ_CHECK_LAUNCH("row tiles");
  WPROJ_TRY(stable_bin_sort(key.as<int32_t>(), m, n_tiles, ids2.as<int32_t>(), rtptr.as<int64_t>(), s, false));
  k_sorted_len<<<ceil_div(m, 256), 256, 0, s>>>(m, ids2.as<int32_t>(), ids.as<int32_t>(), p->row_ptr.as<int64_t>(),
                                                perm.as<int32_t>(), len.as<int32_t>());
  WPROJ_CHECK_LAUNCH("row lengths");
  WPROJ_TRY(exclusive_scan_i32_to_i64(len.as<int32_t>(), rcum.as<int64_t>(), m, s));
  // chunks: about 12 blocks an SM of at least 4096 entries (a batch's other problems
  // fill the GPU: 16384)
  const int64_t least = p->in_batch ? 16384 : 4096;
  WPROJ_TRY(make_tile_chunks(n_tiles, rtptr.as<int64_t>(), rcum.as<int64_t>(), m, p->nnz,
                             std::min<int64_t>(262144, std::max<int64_t>(least, p->nnz / (152 * 12))), ctile, clo, chi,
                             ctp, &c.d_chunks, s));
  WPROJ_TRY(c.rect.reuse(sizeof(int4) * c.d_chunks));
  WPROJ_TRY(c.d_slice_base.reuse(sizeof(int64_t) * (c.d_chunks + 1)));
  WPROJ_TRY(cells.alloc(sizeof(int32_t) * c.d_chunks));
  WPROJ_TRY(cbase.alloc(sizeof(int64_t) * (c.d_chunks + 1)));
  WPROJ_TRY(nsl.alloc(sizeof(int32_t) * c.d_chunks));
  k_chunk_patch<<<(unsigned)c.d_chunks, 128, 0, s>>>(ctile.as<int32_t>(), clo.as<int64_t>(), chi.as<int64_t>(),
                                                     perm.as<int32_t>(), len.as<int32_t>(), j0, Sk, ext.as<uint32_t>(),
                                                     logG, c.rect.as<int4>(), cells.as<int32_t>(), nsl.as<int32_t>(),
                                                     stat.as<int>());
  WPROJ_CHECK_LAUNCH("chunk patches");
  WPROJ_TRY(exclusive_scan_total(nsl.as<int32_t>(), c.d_slice_base.as<int64_t>(), c.d_chunks, s));
  WPROJ_TRY(exclusive_scan_total(cells.as<int32_t>(), cbase.as<int64_t>(), c.d_chunks, s));
  int64_t n_cells = 0;
  int words = 0, max_rows = 0;
  auto read = [&](void *dst, const void *src, size_t n) { return cudaMemcpyAsync(dst, src, n, cudaMemcpyDeviceToHost, s); };
  WPROJ_CUDA(read(&c.d_slices, c.d_slice_base.as<int64_t>() + c.d_chunks, sizeof(int64_t)));
  WPROJ_CUDA(read(&n_cells, cbase.as<int64_t>() + c.d_chunks, sizeof(int64_t)));
  WPROJ_CUDA(read(&words, stat.ptr, sizeof(int)));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  // Worth it while the patches' cells (read from L2 once a pass) and the pads are not
  // many times the entries (single plans only, see above), and a chunk's y fits shared memory.
  const int64_t nnz = std::max<int64_t>(1, p->nnz);
  if (!p->in_batch && n_cells > kPatchCellsPerEntry * nnz) {
    c.release();
    return WPROJ_OK;
  }
  // ---- gridding: chunks of a tile's segments, about 16 blocks an SM
  WPROJ_TRY(make_tile_chunks(n_tiles, tptr, cum, n_seg, p->nnz,
                             std::min<int64_t>(262144, std::max<int64_t>(least, p->nnz / (152 * 16))), c.g_chunk_tile,
                             c.g_chunk_lo, c.g_chunk_hi, c.tile_chunk_ptr, &c.g_chunks, s));
  TmpBuf gsteps, grows;
  WPROJ_TRY(gsteps.alloc(sizeof(int32_t) * c.g_chunks));
  WPROJ_TRY(grows.alloc(sizeof(int32_t) * c.g_chunks));
  WPROJ_TRY(c.g_perm.reuse(sizeof(uint16_t) * 1024 * c.g_chunks));
  WPROJ_TRY(c.g_slp.reuse(sizeof(uint32_t) * 33 * c.g_chunks));
  WPROJ_TRY(c.g_base.reuse(sizeof(int64_t) * (c.g_chunks + 1)));
  WPROJ_TRY(c.g_row_base.reuse(sizeof(int64_t) * (c.g_chunks + 1)));
  k_cell_sort<<<(unsigned)c.g_chunks, 1024, 0, s>>>(
      c.g_chunk_lo.as<int64_t>(), c.g_chunk_hi.as<int64_t>(), c.g_chunk_tile.as<int32_t>(), p->seg_meta.as<SegMeta>(),
      p->col.as<int32_t>(), logG, c.g_perm.as<uint16_t>(), c.g_slp.as<uint32_t>(), gsteps.as<int32_t>(),
      grows.as<int32_t>(), stat.as<int>() + 1);
  WPROJ_CHECK_LAUNCH("cell slices");
  WPROJ_TRY(exclusive_scan_total(gsteps.as<int32_t>(), c.g_base.as<int64_t>(), c.g_chunks, s));
  WPROJ_TRY(exclusive_scan_total(grows.as<int32_t>(), c.g_row_base.as<int64_t>(), c.g_chunks, s));
  WPROJ_CUDA(read(&c.g_steps, c.g_base.as<int64_t>() + c.g_chunks, sizeof(int64_t)));
  WPROJ_CUDA(read(&c.g_nrows, c.g_row_base.as<int64_t>() + c.g_chunks, sizeof(int64_t)));
  WPROJ_CUDA(read(&max_rows, stat.as<int>() + 1, sizeof(int)));
  // ---- the slices' steps
  WPROJ_TRY(steps.alloc(sizeof(int32_t) * std::max<int64_t>(1, c.d_slices)));
  WPROJ_TRY(c.srow.reuse(sizeof(int32_t) * kRps * std::max<int64_t>(1, c.d_slices)));
  WPROJ_TRY(c.slice_ptr.reuse(sizeof(int64_t) * (c.d_slices + 1)));
  k_slice_steps<<<(unsigned)c.d_chunks, 128, 0, s>>>(clo.as<int64_t>(), chi.as<int64_t>(),
                                                     c.d_slice_base.as<int64_t>(), perm.as<int32_t>(),
                                                     len.as<int32_t>(), steps.as<int32_t>(), c.srow.as<int32_t>());
  WPROJ_CHECK_LAUNCH("slice steps");
  WPROJ_TRY(exclusive_scan_total(steps.as<int32_t>(), c.slice_ptr.as<int64_t>(), c.d_slices, s));
  WPROJ_CUDA(read(&c.d_steps, c.slice_ptr.as<int64_t>() + c.d_slices, sizeof(int64_t)));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  if (max_rows > kMaxRowsChunk || (!p->in_batch && (c.d_steps * 32 > 2 * nnz || c.g_steps * 32 > 2 * nnz))) {
    c.release();
    return WPROJ_OK;
  }
  c.d_smem = sizeof(float2) * size_t(words);
  c.g_smem = sizeof(float2) * size_t(1 + max_rows);
  const size_t de = std::max<int64_t>(1, c.d_steps) * 32, ge = std::max<int64_t>(1, c.g_steps) * 32;
  WPROJ_TRY(c.d_idx.reuse(sizeof(uint16_t) * de));
  WPROJ_TRY(c.d_val.reuse(vb * de));
  WPROJ_TRY(c.g_idx.reuse(sizeof(uint16_t) * ge));
  WPROJ_TRY(c.g_val.reuse(vb * ge));
  WPROJ_TRY(c.g_rows.reuse(sizeof(int32_t) * std::max<int64_t>(1, c.g_nrows)));
  std::vector<int32_t> multi;   // lives until its copy has run
  if (c.g_chunks > n_tiles) {
    std::vector<int32_t> tcp(n_tiles + 1);
    WPROJ_CUDA(cudaMemcpy(tcp.data(), c.tile_chunk_ptr.ptr, sizeof(int32_t) * tcp.size(), cudaMemcpyDeviceToHost));
    for (int t = 0; t < n_tiles; ++t)
      if (tcp[t + 1] - tcp[t] > 1) multi.push_back(t);
    c.n_multi = int64_t(multi.size());
    WPROJ_TRY(c.multi.reuse(sizeof(int32_t) * multi.size()));
    WPROJ_CUDA(cudaMemcpyAsync(c.multi.ptr, multi.data(), sizeof(int32_t) * multi.size(), cudaMemcpyHostToDevice, s));
    if (!p->in_batch) WPROJ_TRY(c.partial.reuse(sizeof(float2) * 1024 * c.g_chunks));
  }
  WPROJ_CUDA(cudaMemsetAsync(c.d_idx.ptr, 0, sizeof(uint16_t) * de, s));
  WPROJ_CUDA(cudaMemsetAsync(c.d_val.ptr, 0, vb * de, s));
  WPROJ_CUDA(cudaMemsetAsync(c.g_idx.ptr, 0, sizeof(uint16_t) * ge, s));
  WPROJ_CUDA(cudaMemsetAsync(c.g_val.ptr, 0, vb * ge, s));
  WPROJ_TRY(fill(p, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));   // the sort's scratch is released
  c.use = true;
  return WPROJ_OK;
}

// The stored values changed (same support): refresh the slices' values.
wproj_status rebuild_slices(wproj_plan *p, cudaStream_t s) {
  if (!p->slices.use) return WPROJ_OK;
  WPROJ_TRY(fill(p, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  return WPROJ_OK;
}

wproj_status degrid_slices(wproj_plan *p, const float2 *Xt, float2 *y, cudaStream_t s) {
  const SliceOps o = plan_ops(p);
  switch (p->g.value_dtype) {
    case WPROJ_VAL_F32: return launch_degrid<WPROJ_VAL_F32>(o, p->slices.d_smem, Xt, y, s);
    case WPROJ_VAL_BF16: return launch_degrid<WPROJ_VAL_BF16>(o, p->slices.d_smem, Xt, y, s);
    default: return launch_degrid<WPROJ_VAL_F16>(o, p->slices.d_smem, Xt, y, s);
  }
}

wproj_status grid_slices(wproj_plan *p, const float2 *y, float2 *Xt2, cudaStream_t s) {
  const SliceOps o = plan_ops(p);
  float2 *part = p->slices.partial.as<float2>();
  switch (p->g.value_dtype) {
    case WPROJ_VAL_F32: return launch_grid<WPROJ_VAL_F32>(o, p->slices.g_smem, y, part, Xt2, s);
    case WPROJ_VAL_BF16: return launch_grid<WPROJ_VAL_BF16>(o, p->slices.g_smem, y, part, Xt2, s);
    default: return launch_grid<WPROJ_VAL_F16>(o, p->slices.g_smem, y, part, Xt2, s);
  }
}

wproj_status batch_degrid_slices(const SliceOps &o, size_t smem, const float2 *Xt, float2 *y, cudaStream_t s) {
  return launch_degrid<WPROJ_VAL_F32>(o, smem, Xt, y, s);
}
wproj_status batch_grid_slices(const SliceOps &o, size_t smem, const float2 *y, float2 *partial, float2 *Xt2,
                               cudaStream_t s) {
  return launch_grid<WPROJ_VAL_F32>(o, smem, y, partial, Xt2, s);
}

}  // namespace wproj
