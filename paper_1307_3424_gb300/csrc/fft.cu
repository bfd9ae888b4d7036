// 2-D FFT passes of libwproj.
//
//  * Phi  (F Z A):   row pass over the N image rows with the zero-padding and
//    the KB correction 1/(a(l) a(m)) fused into the load, then a column pass
//    over all G columns that reads only the N non-zero rows.
//  * Phi^H (A Z^H F^H): column pass over the G columns that keeps only the N
//    image rows, then a row pass over those rows that keeps only the N image
//    columns, fused with the correction and Re(.) (or z - Re(.) for the
//    Douglas-Rachford dual step).
//  * The kernel build: batched S x S inverse transforms of the chirp times the
//    KB tap polynomial, with the chirp generated in the first pass's load.
#include <algorithm>

#include "build.cuh"
#include "fft.cuh"
#include "plan.h"

namespace wproj {

namespace {

__global__ void k_twiddles(float2 *tw) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 2 || i >= kTwiddleLen) return;
  const int l = 31 - __clz(i);
  const int n = 1 << l;
  const int k = i - n;
  double sn, cs;
  sincospi(-2.0 * double(k) / double(n), &sn, &cs);
  tw[i] = make_float2(float(cs), float(sn));
}

// Padded position tq + m G / 16 of a length-G axis -> image index: offset p - N/2
// sits at (p - N/2) mod G, N = G / 2, so m < 4 holds the image's upper half, m >= 12
// its lower half and the rest is padding: 8 of a thread's 16 elements, known at
// compile time, are zeros that are never read or are cropped before the store.
__device__ __forceinline__ constexpr bool in_image(int m) { return m < 4 || m >= 12; }
__device__ __forceinline__ int pad_to_img(int m, int P, int G) { return m < 4 ? P + G / 4 : P - G + G / 4; }

// ---- Phi: F Z A --------------------------------------------------------------

// Each pass is a device body (block `blk` of one transform set) called by a
// kernel for one plan and by a kernel for a batch of same-size problems
// (blockIdx.y = problem of the size class, offsets from its BProb entry).
template <int LOGN, class Cfg>
__device__ __forceinline__ void phi_fwd_rows_body(const float *__restrict__ x, const float2 *__restrict__ xc,
                                                  const float *__restrict__ inv_a, int N,
                                                  float2 *__restrict__ inter, const float2 *__restrict__ tw,
                                                  int blk) {
  constexpr int G = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  row_thread<Cfg>(c, tq);
  const int p = blk * Cfg::C + c;
  const bool ok = p < N;
  const float ap = ok ? inv_a[p] : 0.f;
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) {
    v[m] = make_float2(0.f, 0.f);
    if (in_image(m) && ok) {
      const int q = pad_to_img(m, tq + m * Cfg::TN, G);
      const float s = ap * inv_a[q];
      if (xc) v[m] = cscale(xc[int64_t(p) * N + q], s);
      else v[m].x = x[int64_t(p) * N + q] * s;
    }
  }
  float2 *out = inter + int64_t(p) * G;
  fft_run<LOGN, -1>(v, tq, sm + c * Cfg::LD, tw, [&](int, int Q, float2 o) {
    if (ok) out[Q] = o;
  });
}

template <int LOGN>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_phi_fwd_rows(const float *__restrict__ x, const float2 *__restrict__ xc, const float *__restrict__ inv_a, int N,
               float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  chain_wait();
  chain_next();
  phi_fwd_rows_body<LOGN, RowCfg<LOGN>>(after_wait(x), after_wait(xc), inv_a, N, inter, tw, blockIdx.x);
}

template <int LOGN>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_bphi_fwd_rows(const BProb *__restrict__ tab, const int32_t *__restrict__ plist, const float *__restrict__ x,
                const float *__restrict__ inv_a, float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  const BProb P = tab[plist[blockIdx.y]];
  phi_fwd_rows_body<LOGN, RowCfg<LOGN>>(x + P.img_off, nullptr, inv_a + P.inva_off, P.N, inter + P.inter_off, tw, blockIdx.x);
}

template <int LOGN, class Cfg>
__device__ __forceinline__ void phi_fwd_cols_body(const float2 *__restrict__ inter, int N, float2 *__restrict__ Xt,
                                                  float scale, const float2 *__restrict__ tw, int blk) {
  constexpr int G = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  col_thread<Cfg>(c, tq);
  const int Q = blk * Cfg::C + c;
  const bool ok = Q < G;
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) {
    v[m] = make_float2(0.f, 0.f);
    if (in_image(m) && ok) v[m] = inter[int64_t(pad_to_img(m, tq + m * Cfg::TN, G)) * G + Q];
  }
  fft_run<LOGN, -1>(v, tq, sm + c * Cfg::LD, tw, [&](int, int P, float2 o) {
    if (ok) Xt[int64_t(P) * G + Q] = cscale(o, scale);
  });
}

template <int LOGN>
__global__ void __launch_bounds__(ColCfg<LOGN>::T)
k_phi_fwd_cols(const float2 *__restrict__ inter, int N, float2 *__restrict__ Xt, float scale,
               const float2 *__restrict__ tw) {
  chain_next();
  chain_wait();
  phi_fwd_cols_body<LOGN, ColCfg<LOGN>>(after_wait(inter), N, Xt, scale, tw, blockIdx.x);
}

template <int LOGN>
__global__ void __launch_bounds__(ColCfg<LOGN>::T)
k_bphi_fwd_cols(const BProb *__restrict__ tab, const int32_t *__restrict__ plist, const float2 *__restrict__ inter,
                float2 *__restrict__ Xt, const float2 *__restrict__ tw) {
  const BProb P = tab[plist[blockIdx.y]];
  phi_fwd_cols_body<LOGN, ColCfg<LOGN>>(inter + P.inter_off, P.N, Xt + P.grid_off, 1.0f / P.G, tw, blockIdx.x);
}

// ---- Phi^H: A Z^H F^H -----------------------------------------------------------

template <int LOGN, class Cfg>
__device__ __forceinline__ void phi_adj_cols_body(const float2 *__restrict__ Xt2, int N, float2 *__restrict__ inter,
                                                  const float2 *__restrict__ tw, int blk) {
  constexpr int G = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  col_thread<Cfg>(c, tq);
  const int Q = blk * Cfg::C + c;
  const bool ok = Q < G;
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m)
    v[m] = ok ? Xt2[int64_t(tq + m * Cfg::TN) * G + Q] : make_float2(0.f, 0.f);
  fft_run<LOGN, +1>(v, tq, sm + c * Cfg::LD, tw, [&](int m, int P, float2 o) {
    if (in_image(m) && ok) inter[int64_t(pad_to_img(m, P, G)) * G + Q] = o;
  });
}

template <int LOGN>
__global__ void __launch_bounds__(ColCfg<LOGN>::T)
k_phi_adj_cols(const float2 *__restrict__ Xt2, int N, float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  chain_next();
  chain_wait();
  phi_adj_cols_body<LOGN, ColCfg<LOGN>>(after_wait(Xt2), N, inter, tw, blockIdx.x);
}

template <int LOGN>
__global__ void __launch_bounds__(ColCfg<LOGN>::T)
k_bphi_adj_cols(const BProb *__restrict__ tab, const int32_t *__restrict__ plist, const float2 *__restrict__ Xt2,
                float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  const BProb P = tab[plist[blockIdx.y]];
  phi_adj_cols_body<LOGN, ColCfg<LOGN>>(Xt2 + P.grid_off, P.N, inter + P.inter_off, tw, blockIdx.x);
}

// mode 0: x_re = Re(v) s (and x_c = v s when given); mode 1: x_re = z - Re(v) s
template <int LOGN, class Cfg>
__device__ __forceinline__ void phi_adj_rows_body(const float2 *__restrict__ inter, const float *__restrict__ inv_a,
                                                  int N, float scale, float *__restrict__ x_re,
                                                  float2 *__restrict__ x_c, const float *__restrict__ z, int mode,
                                                  const float2 *__restrict__ tw, int blk) {
  constexpr int G = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  row_thread<Cfg>(c, tq);
  const int p = blk * Cfg::C + c;
  const bool ok = p < N;
  const float2 *in = inter + int64_t(p) * G;
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) v[m] = ok ? in[tq + m * Cfg::TN] : make_float2(0.f, 0.f);
  const float ap = ok ? inv_a[p] : 0.f;
  fft_run<LOGN, +1>(v, tq, sm + c * Cfg::LD, tw, [&](int m, int Q, float2 f) {
    if (in_image(m) && ok) {
      const int q = pad_to_img(m, Q, G);
      const float s = ap * inv_a[q] * scale;
      const int64_t o = int64_t(p) * N + q;
      if (mode == 0) {
        if (x_re) x_re[o] = f.x * s;
        if (x_c) x_c[o] = cscale(f, s);
      } else {
        x_re[o] = z[o] - f.x * s;
      }
    }
  });
}

template <int LOGN>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_phi_adj_rows(const float2 *__restrict__ inter, const float *__restrict__ inv_a, int N, float scale,
               float *__restrict__ x_re, float2 *__restrict__ x_c, const float *__restrict__ z, int mode,
               const float2 *__restrict__ tw) {
  chain_next();
  chain_wait();
  phi_adj_rows_body<LOGN, RowCfg<LOGN>>(after_wait(inter), inv_a, N, scale, x_re, x_c, after_wait(z), mode, tw, blockIdx.x);
}

template <int LOGN>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_bphi_adj_rows(const BProb *__restrict__ tab, const int32_t *__restrict__ plist, const float2 *__restrict__ inter,
                const float *__restrict__ inv_a, float *__restrict__ x_re, const float *__restrict__ z, int mode,
                const float2 *__restrict__ tw) {
  const BProb P = tab[plist[blockIdx.y]];
  phi_adj_rows_body<LOGN, RowCfg<LOGN>>(inter + P.inter_off, inv_a + P.inva_off, P.N, 1.0f / P.G, x_re + P.img_off, nullptr,
                          z ? z + P.img_off : nullptr, mode, tw, blockIdx.x);
}

// ---- batches: one launch per pass for all grid sizes up to 1024^2 -------------------
// A launch per size ran the sizes one after another, each with a tail of its own and
// too few blocks to fill the chip (64 problems: 16 launches, 180 us of transforms).

// the size class, problem and block of the problem that blockIdx.x stands for
__device__ __forceinline__ int class_block(const FftClasses &cl, int &prob, int &blk) {
  int c = 0;
  while (c + 1 < cl.n && int(blockIdx.x) >= cl.first[c + 1]) ++c;
  const int q = int(blockIdx.x) - cl.first[c];
  prob = __ldg(cl.plist[c] + q / cl.per[c]);
  blk = q % cl.per[c];
  return cl.logG[c];
}

#define WPROJ_BATCH_LOGN(logn, CALL) \
  switch (logn) {                    \
    case 4: CALL(4); break;          \
    case 5: CALL(5); break;          \
    case 6: CALL(6); break;          \
    case 7: CALL(7); break;          \
    case 8: CALL(8); break;          \
    case 9: CALL(9); break;          \
    default: CALL(10);               \
  }

__global__ void __launch_bounds__(256, 3)
k_bphi_fwd_rows_all(const FftClasses cl, const BProb *__restrict__ tab, const float *__restrict__ x,
                    const float *__restrict__ inv_a, float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  int prob, blk;
  chain_wait();
  chain_next();
  x = after_wait(x);
  const int lg = class_block(cl, prob, blk);
  const BProb P = tab[prob];
#define CALL(L) phi_fwd_rows_body<L, BatchRowCfg<L>>(x + P.img_off, nullptr, inv_a + P.inva_off, P.N, inter + P.inter_off, tw, blk)
  WPROJ_BATCH_LOGN(lg, CALL)
#undef CALL
}
__global__ void __launch_bounds__(256, 3)
k_bphi_fwd_cols_all(const FftClasses cl, const BProb *__restrict__ tab, const float2 *__restrict__ inter,
                    float2 *__restrict__ Xt, const float2 *__restrict__ tw) {
  int prob, blk;
  chain_next();
  const int lg = class_block(cl, prob, blk);
  const BProb P = tab[prob];
  chain_wait();
  inter = after_wait(inter);
#define CALL(L) phi_fwd_cols_body<L, BatchColCfg<L>>(inter + P.inter_off, P.N, Xt + P.grid_off, 1.0f / P.G, tw, blk)
  WPROJ_BATCH_LOGN(lg, CALL)
#undef CALL
}
__global__ void __launch_bounds__(256, 3)
k_bphi_adj_cols_all(const FftClasses cl, const BProb *__restrict__ tab, const float2 *__restrict__ Xt2,
                    float2 *__restrict__ inter, const float2 *__restrict__ tw) {
  int prob, blk;
  chain_next();
  const int lg = class_block(cl, prob, blk);
  const BProb P = tab[prob];
  chain_wait();
  Xt2 = after_wait(Xt2);
#define CALL(L) phi_adj_cols_body<L, BatchColCfg<L>>(Xt2 + P.grid_off, P.N, inter + P.inter_off, tw, blk)
  WPROJ_BATCH_LOGN(lg, CALL)
#undef CALL
}
__global__ void __launch_bounds__(256, 3)
k_bphi_adj_rows_all(const FftClasses cl, const BProb *__restrict__ tab, const float2 *__restrict__ inter,
                    const float *__restrict__ inv_a, float *__restrict__ x_re, const float *__restrict__ z, int mode,
                    const float2 *__restrict__ tw) {
  int prob, blk;
  chain_next();
  const int lg = class_block(cl, prob, blk);
  const BProb P = tab[prob];
  chain_wait();
  inter = after_wait(inter);
  z = after_wait(z);
#define CALL(L)                                                                                                  \
  phi_adj_rows_body<L, BatchRowCfg<L>>(inter + P.inter_off, inv_a + P.inva_off, P.N, 1.0f / P.G, x_re + P.img_off, \
                                       nullptr, z ? z + P.img_off : nullptr, mode, tw, blk)
  WPROJ_BATCH_LOGN(lg, CALL)
#undef CALL
}

// ---- generic batched 2-D FFT (rows then columns) --------------------------------

template <int LOGN, int DIR>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_fft_rows(const float2 *__restrict__ in, float2 *__restrict__ out, int64_t n_rows,
           const float2 *__restrict__ tw) {
  using Cfg = RowCfg<LOGN>;
  constexpr int N = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  row_thread<Cfg>(c, tq);
  const int64_t r = int64_t(blockIdx.x) * Cfg::C + c;
  const bool ok = r < n_rows;
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) v[m] = ok ? in[r * N + tq + m * Cfg::TN] : make_float2(0.f, 0.f);
  fft_run<LOGN, DIR>(v, tq, sm + c * Cfg::LD, tw, [&](int, int i, float2 o) {
    if (ok) out[r * N + i] = o;
  });
}

// columns of `batch` N x N arrays, flattened as batch * N global columns
template <int LOGN, int DIR>
__global__ void __launch_bounds__(BoxColCfg<LOGN>::T)
k_fft_cols(const float2 *__restrict__ in, float2 *__restrict__ out, int64_t n_cols, float scale,
           const float2 *__restrict__ tw) {
  using Cfg = BoxColCfg<LOGN>;
  constexpr int N = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  col_thread<Cfg>(c, tq);
  const int64_t gc = int64_t(blockIdx.x) * Cfg::C + c;
  const bool ok = gc < n_cols;
  const int64_t at = ((gc >> LOGN) << (2 * LOGN)) + (gc & (N - 1));
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) v[m] = ok ? in[at + int64_t(tq + m * Cfg::TN) * N] : make_float2(0.f, 0.f);
  fft_run<LOGN, DIR>(v, tq, sm + c * Cfg::LD, tw, [&](int, int P, float2 o) {
    if (ok) out[at + int64_t(P) * N] = cscale(o, scale);
  });
}

// ---- kernel build: S x S boxes ---------------------------------------------------

// g(x) of the exact chirp's FP32 remainder at every sample of an S x S box: the
// root and the division once per sample position instead of once per box sample.
__global__ void k_g_table(int S, const float *__restrict__ lsq, float *__restrict__ g) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(S) * S) return;
  const float x = lsq[i / S] + lsq[i % S];
  const float n = sqrtf(1.f - x);
  const float d = 1.f + n;
  g[i] = (x * x) / (2.f * d * d);
}

template <int LOGN>
__global__ void __launch_bounds__(RowCfg<LOGN>::T)
k_box_rows(BoxBatch bb, const float2 *__restrict__ tw) {
  using Cfg = RowCfg<LOGN>;
  constexpr int S = 1 << LOGN;
  extern __shared__ float2 sm[];
  int c, tq;
  row_thread<Cfg>(c, tq);
  const int64_t r = int64_t(blockIdx.x) * Cfg::C + c;
  const bool ok = r < int64_t(bb.nb) * S;
  const int b = int(r >> LOGN), P = int(r & (S - 1));
  // a thread's samples go through its own slots of the exchange buffer, so that
  // the chirp's code exists once and not 16 times
  float2 *own = sm + c * Cfg::LD;
#pragma unroll 2
  for (int m = 0; m < kFftE; ++m) {
    const int Q = tq + m * Cfg::TN;
    own[fft_pad(Q)] = ok ? box_value(bb, b, P, Q) : make_float2(0.f, 0.f);
  }
  float2 v[kFftE];
#pragma unroll
  for (int m = 0; m < kFftE; ++m) v[m] = own[fft_pad(tq + m * Cfg::TN)];
  __syncthreads();
  fft_run<LOGN, +1>(v, tq, own, tw, [&](int, int Q, float2 o) {
    if (ok) bb.K[r * S + Q] = o;
  });
}

// ---- separable kernel boxes (linear chirp, Eq. 5) ------------------------------------
// exp(pi i w (l^2 + m^2)) times the separable taps is an outer product Au x Av,
// so its 2-D inverse DFT is the outer product of two 1-D ones: K = (IDFT Au) x
// (IDFT Av) / S^2, two length-S transforms per box instead of an S x S one.
__global__ void k_box_outer(int nb, int S, const float2 *__restrict__ Au, const float2 *__restrict__ Av, float scale,
                            float2 *__restrict__ K) {
  const int64_t n = int64_t(nb) * S * S;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t b = i / (int64_t(S) * S);
    const int P = int((i / S) % S), Q = int(i % S);
    K[i] = cscale(cmul(Au[b * S + P], Av[b * S + Q]), scale);
  }
}

// ---- the paper's upsampling U (Section 2.2): spectral zero-padding -----------------
// F_G U x = P F_N x: the unitary spectrum of the image (pixel offset p - N/2 at
// index (p - N/2) mod N) placed on the G x G grid, frequency k in [-N/2, N/2)
// at index k mod G, zeros elsewhere.  Its adjoint crops and inverts.

__global__ void k_up_in(int N, const float *__restrict__ x, const float2 *__restrict__ xc, float2 *__restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(N) * N) return;
  const int p = int(i / N), q = int(i % N), h = N / 2;
  const float2 v = xc ? xc[i] : make_float2(x[i], 0.f);
  out[int64_t((p - h + N) % N) * N + (q - h + N) % N] = v;
}

__global__ void k_up_scatter(int N, int G, const float2 *__restrict__ spec, float scale, float2 *__restrict__ Xt) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(G) * G) return;
  const int a = int(i / G), b = int(i % G), h = N / 2;
  const int ka = a < G / 2 ? a : a - G, kb = b < G / 2 ? b : b - G;
  float2 v = make_float2(0.f, 0.f);
  if (ka >= -h && ka < h && kb >= -h && kb < h) v = cscale(spec[int64_t((ka + N) % N) * N + (kb + N) % N], scale);
  Xt[i] = v;
}

__global__ void k_up_gather(int N, int G, const float2 *__restrict__ Xt2, float2 *__restrict__ spec) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(N) * N) return;
  const int a = int(i / N), b = int(i % N);
  const int ka = a < N / 2 ? a : a - N, kb = b < N / 2 ? b : b - N;
  spec[i] = Xt2[int64_t((ka + G) % G) * G + (kb + G) % G];
}

// mode 0: x_re = Re(v) (and x_c = v); mode 1: x_re = z - Re(v); v = scale * img
__global__ void k_up_out(int N, const float2 *__restrict__ img, float scale, float *__restrict__ x_re,
                         float2 *__restrict__ x_c, const float *__restrict__ z, int mode) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= int64_t(N) * N) return;
  const int p = int(i / N), q = int(i % N), h = N / 2;
  const float2 v = cscale(img[int64_t((p - h + N) % N) * N + (q - h + N) % N], scale);
  if (mode == 0) {
    if (x_re) x_re[i] = v.x;
    if (x_c) x_c[i] = v;
  } else {
    x_re[i] = z[i] - v.x;
  }
}

// ---- dispatch ------------------------------------------------------------------

template <class K>
wproj_status set_smem(K kern, size_t smem) {
  if (smem > 48 * 1024) {
    WPROJ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  }
  return WPROJ_OK;
}

template <int LOGN>
wproj_status phi_fwd_impl(wproj_plan *p, const float *x, const float2 *xc, float2 *Xt, cudaStream_t s) {
  const int N = p->g.N, G = p->g.G;
  const float2 *tw = p->twiddle.as<float2>();
  float2 *inter = p->inter.as<float2>();
  {
    using Cfg = RowCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_fwd_rows<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_fwd_rows<LOGN>, ceil_div(N, Cfg::C), Cfg::T, Cfg::SMEM, s, x, xc,
                              p->inv_a.as<float>(), N, inter, tw));
    WPROJ_CHECK_LAUNCH("phi fwd rows");
  }
  {
    using Cfg = ColCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_fwd_cols<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_fwd_cols<LOGN>, ceil_div(G, Cfg::C), Cfg::T, Cfg::SMEM, s, inter, N, Xt, 1.0f / G, tw));
    WPROJ_CHECK_LAUNCH("phi fwd cols");
  }
  return WPROJ_OK;
}

// The same two passes with a caller-provided intermediate buffer (N x G float2).
template <int LOGN>
wproj_status phi_fwd_into_impl(wproj_plan *p, const float *x, float2 *inter, float2 *Xt, cudaStream_t s) {
  const int N = p->g.N, G = p->g.G;
  const float2 *tw = p->twiddle.as<float2>();
  {
    using Cfg = RowCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_fwd_rows<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_fwd_rows<LOGN>, ceil_div(N, Cfg::C), Cfg::T, Cfg::SMEM, s, x, nullptr,
                              p->inv_a.as<float>(), N, inter, tw));
    WPROJ_CHECK_LAUNCH("phi fwd rows");
  }
  {
    using Cfg = ColCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_fwd_cols<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_fwd_cols<LOGN>, ceil_div(G, Cfg::C), Cfg::T, Cfg::SMEM, s, inter, N, Xt, 1.0f / G, tw));
    WPROJ_CHECK_LAUNCH("phi fwd cols");
  }
  return WPROJ_OK;
}

template <int LOGN>
wproj_status phi_adj_impl(wproj_plan *p, const float2 *Xt2, float *x_re, float2 *x_c, const float *z,
                          int mode, cudaStream_t s) {
  const int N = p->g.N, G = p->g.G;
  const float2 *tw = p->twiddle.as<float2>();
  float2 *inter = p->inter.as<float2>();
  {
    using Cfg = ColCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_adj_cols<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_adj_cols<LOGN>, ceil_div(G, Cfg::C), Cfg::T, Cfg::SMEM, s, Xt2, N, inter, tw));
    WPROJ_CHECK_LAUNCH("phi adj cols");
  }
  {
    using Cfg = RowCfg<LOGN>;
    WPROJ_TRY(set_smem(k_phi_adj_rows<LOGN>, Cfg::SMEM));
    WPROJ_CUDA(launch_chained(k_phi_adj_rows<LOGN>, ceil_div(N, Cfg::C), Cfg::T, Cfg::SMEM, s, inter,
                              p->inv_a.as<float>(), N, 1.0f / G, x_re, x_c, z, mode, tw));
    WPROJ_CHECK_LAUNCH("phi adj rows");
  }
  return WPROJ_OK;
}

template <int LOGN>
wproj_status fft2d_impl(const float2 *in, float2 *out, int batch, int inverse, const float2 *tw,
                        cudaStream_t s) {
  constexpr int N = 1 << LOGN;
  using RC = RowCfg<LOGN>;
  using CC = BoxColCfg<LOGN>;
  const int64_t rows = int64_t(batch) * N;
  if (inverse) {
    WPROJ_TRY(set_smem(k_fft_rows<LOGN, +1>, RC::SMEM));
    WPROJ_TRY(set_smem(k_fft_cols<LOGN, +1>, CC::SMEM));
    k_fft_rows<LOGN, +1><<<ceil_div(rows, RC::C), RC::T, RC::SMEM, s>>>(in, out, rows, tw);
    k_fft_cols<LOGN, +1><<<ceil_div(rows, CC::C), CC::T, CC::SMEM, s>>>(out, out, rows, 1.f, tw);
  } else {
    WPROJ_TRY(set_smem(k_fft_rows<LOGN, -1>, RC::SMEM));
    WPROJ_TRY(set_smem(k_fft_cols<LOGN, -1>, CC::SMEM));
    k_fft_rows<LOGN, -1><<<ceil_div(rows, RC::C), RC::T, RC::SMEM, s>>>(in, out, rows, tw);
    k_fft_cols<LOGN, -1><<<ceil_div(rows, CC::C), CC::T, CC::SMEM, s>>>(out, out, rows, 1.f, tw);
  }
  WPROJ_CHECK_LAUNCH("fft2d");
  return WPROJ_OK;
}

template <int LOGN>
wproj_status box_fft_impl(wproj_plan *p, const BoxBatch &bb, cudaStream_t s) {
  constexpr int S = 1 << LOGN;
  using RC = RowCfg<LOGN>;
  using CC = BoxColCfg<LOGN>;
  const float2 *tw = p->twiddle.as<float2>();
  const int64_t rows = int64_t(bb.nb) * S;
  WPROJ_TRY(set_smem(k_box_rows<LOGN>, RC::SMEM));
  WPROJ_TRY(set_smem(k_fft_cols<LOGN, +1>, CC::SMEM));
  k_box_rows<LOGN><<<ceil_div(rows, RC::C), RC::T, RC::SMEM, s>>>(bb, tw);
  WPROJ_CHECK_LAUNCH("box rows");
  k_fft_cols<LOGN, +1><<<ceil_div(rows, CC::C), CC::T, CC::SMEM, s>>>(
      bb.K, bb.K, rows, 1.0f / (float(S) * float(S)), tw);
  WPROJ_CHECK_LAUNCH("box cols");
  return WPROJ_OK;
}

#define WPROJ_LOGN_SWITCH(logn, CALL)                    \
  switch (logn) {                                         \
    case 4: return CALL(4);                               \
    case 5: return CALL(5);                               \
    case 6: return CALL(6);                               \
    case 7: return CALL(7);                               \
    case 8: return CALL(8);                               \
    case 9: return CALL(9);                               \
    case 10: return CALL(10);                             \
    case 11: return CALL(11);                             \
    case 12: return CALL(12);                             \
    default: return fail(WPROJ_ERR_UNSUPPORTED, "FFT size out of range"); \
  }

}  // namespace

// ---- batches: one launch per pass for all problems of a size class ---------------

template <int LOGN>
wproj_status bphi_fwd_impl(int np, const int32_t *plist, const BProb *tab, const float *x, const float *inv_a,
                           float2 *inter, float2 *Xt, const float2 *tw, cudaStream_t s) {
  constexpr int G = 1 << LOGN;
  const int N = G / 2;
  {
    using Cfg = RowCfg<LOGN>;
    WPROJ_TRY(set_smem(k_bphi_fwd_rows<LOGN>, Cfg::SMEM));
    k_bphi_fwd_rows<LOGN><<<dim3(ceil_div(N, Cfg::C), np), Cfg::T, Cfg::SMEM, s>>>(tab, plist, x, inv_a, inter, tw);
    WPROJ_CHECK_LAUNCH("batch phi fwd rows");
  }
  {
    using Cfg = ColCfg<LOGN>;
    WPROJ_TRY(set_smem(k_bphi_fwd_cols<LOGN>, Cfg::SMEM));
    k_bphi_fwd_cols<LOGN><<<dim3(ceil_div(G, Cfg::C), np), Cfg::T, Cfg::SMEM, s>>>(tab, plist, inter, Xt, tw);
    WPROJ_CHECK_LAUNCH("batch phi fwd cols");
  }
  return WPROJ_OK;
}

template <int LOGN>
wproj_status bphi_adj_impl(int np, const int32_t *plist, const BProb *tab, const float2 *Xt2, const float *inv_a,
                           float2 *inter, float *x_re, const float *z, int mode, const float2 *tw, cudaStream_t s) {
  constexpr int G = 1 << LOGN;
  const int N = G / 2;
  {
    using Cfg = ColCfg<LOGN>;
    WPROJ_TRY(set_smem(k_bphi_adj_cols<LOGN>, Cfg::SMEM));
    k_bphi_adj_cols<LOGN><<<dim3(ceil_div(G, Cfg::C), np), Cfg::T, Cfg::SMEM, s>>>(tab, plist, Xt2, inter, tw);
    WPROJ_CHECK_LAUNCH("batch phi adj cols");
  }
  {
    using Cfg = RowCfg<LOGN>;
    WPROJ_TRY(set_smem(k_bphi_adj_rows<LOGN>, Cfg::SMEM));
    k_bphi_adj_rows<LOGN><<<dim3(ceil_div(N, Cfg::C), np), Cfg::T, Cfg::SMEM, s>>>(tab, plist, inter, inv_a, x_re,
                                                                                 z, mode, tw);
    WPROJ_CHECK_LAUNCH("batch phi adj rows");
  }
  return WPROJ_OK;
}

// F U x into Xt (G x G); work: 2 N^2 complex
wproj_status up_forward(wproj_plan *p, const float *x, const float2 *xc, float2 *work, float2 *Xt, cudaStream_t s) {
  const int N = p->g.N, G = p->g.G;
  float2 *a = work, *b = work + int64_t(N) * N;
  k_up_in<<<ceil_div(int64_t(N) * N, 256), 256, 0, s>>>(N, x, xc, a);
  WPROJ_CHECK_LAUNCH("upsampling input");
  WPROJ_TRY(fft2d_generic(a, b, N, 1, 0, p->twiddle.as<float2>(), s));
  k_up_scatter<<<ceil_div(int64_t(G) * G, 256), 256, 0, s>>>(N, G, b, 1.0f / N, Xt);
  WPROJ_CHECK_LAUNCH("upsampling scatter");
  return WPROJ_OK;
}

// (F U)^H of Xt2 into the image; work: 2 N^2 complex
wproj_status up_adjoint(wproj_plan *p, const float2 *Xt2, float *x_re, float2 *x_c, const float *z, int mode,
                        float2 *work, cudaStream_t s) {
  const int N = p->g.N, G = p->g.G;
  float2 *a = work, *b = work + int64_t(N) * N;
  k_up_gather<<<ceil_div(int64_t(N) * N, 256), 256, 0, s>>>(N, G, Xt2, a);
  WPROJ_CHECK_LAUNCH("upsampling gather");
  WPROJ_TRY(fft2d_generic(a, b, N, 1, 1, p->twiddle.as<float2>(), s));
  k_up_out<<<ceil_div(int64_t(N) * N, 256), 256, 0, s>>>(N, b, 1.0f / N, x_re, x_c, z, mode);
  WPROJ_CHECK_LAUNCH("upsampling output");
  return WPROJ_OK;
}

wproj_status phi_forward_fft_into(wproj_plan *p, const float *x, float2 *inter, float2 *Xt, cudaStream_t s) {
  if (p->g.upsampling) return up_forward(p, x, nullptr, inter, Xt, s);
#define CALL(L) phi_fwd_into_impl<L>(p, x, inter, Xt, s)
  WPROJ_LOGN_SWITCH(ilog2(p->g.G), CALL)
#undef CALL
}

wproj_status make_twiddles(DevBuf &tw, cudaStream_t s) {
  WPROJ_TRY(tw.alloc(sizeof(float2) * kTwiddleLen));
  k_twiddles<<<kTwiddleLen / 256, 256, 0, s>>>(tw.as<float2>());
  WPROJ_CHECK_LAUNCH("twiddles");
  return WPROJ_OK;
}

wproj_status init_twiddles(wproj_plan *p, cudaStream_t s) { return make_twiddles(p->twiddle, s); }

wproj_status phi_forward_fft(wproj_plan *p, const float *x, const float2 *xc, float2 *Xt, cudaStream_t s) {
  ScopedTimer t(p, TC_FFT, s);
  if (p->g.upsampling) {
    p->launches += 4;
    return up_forward(p, x, xc, p->inter.as<float2>(), Xt, s);
  }
  p->launches += 2;
#define CALL(L) phi_fwd_impl<L>(p, x, xc, Xt, s)
  WPROJ_LOGN_SWITCH(ilog2(p->g.G), CALL)
#undef CALL
}

wproj_status phi_adjoint_fft(wproj_plan *p, const float2 *Xt2, float *x_re, float2 *x_cplx,
                             const float *z, int mode, cudaStream_t s) {
  ScopedTimer t(p, TC_FFT, s);
  if (p->g.upsampling) {
    p->launches += 4;
    return up_adjoint(p, Xt2, x_re, x_cplx, z, mode, p->inter.as<float2>(), s);
  }
  p->launches += 2;
#define CALL(L) phi_adj_impl<L>(p, Xt2, x_re, x_cplx, z, mode, s)
  WPROJ_LOGN_SWITCH(ilog2(p->g.G), CALL)
#undef CALL
}

wproj_status fft2d_generic(const float2 *in, float2 *out, int n, int batch, int inverse,
                           const float2 *tw, cudaStream_t s) {
#define CALL(L) fft2d_impl<L>(in, out, batch, inverse, tw, s)
  WPROJ_LOGN_SWITCH(ilog2(n), CALL)
#undef CALL
}

template <int LOGN>
wproj_status box_fft_separable_impl(wproj_plan *p, const BoxBatch &bb, cudaStream_t s) {
  constexpr int S = 1 << LOGN;
  using RC = RowCfg<LOGN>;
  const float2 *tw = p->twiddle.as<float2>();
  WPROJ_TRY(set_smem(k_fft_rows<LOGN, +1>, RC::SMEM));
  // the per-box tables are rebuilt for every batch, so they are transformed in place
  float2 *Au = const_cast<float2 *>(bb.Au), *Av = const_cast<float2 *>(bb.Av);
  k_fft_rows<LOGN, +1><<<ceil_div(bb.nb, RC::C), RC::T, RC::SMEM, s>>>(Au, Au, bb.nb, tw);
  k_fft_rows<LOGN, +1><<<ceil_div(bb.nb, RC::C), RC::T, RC::SMEM, s>>>(Av, Av, bb.nb, tw);
  const int64_t n = int64_t(bb.nb) * S * S;
  k_box_outer<<<(int)std::min<int64_t>(152 * 32, ceil_div(n, 256)), 256, 0, s>>>(bb.nb, S, Au, Av,
                                                                                1.0f / (float(S) * float(S)), bb.K);
  WPROJ_CHECK_LAUNCH("separable boxes");
  return WPROJ_OK;
}

wproj_status box_g_table(int S, const float *lsq, float *g, cudaStream_t s) {
  k_g_table<<<ceil_div(int64_t(S) * S, 256), 256, 0, s>>>(S, lsq, g);
  WPROJ_CHECK_LAUNCH("chirp remainder table");
  return WPROJ_OK;
}

wproj_status box_fft(wproj_plan *p, const BoxBatch &bb, cudaStream_t s) {
  if (p->g.chirp == WPROJ_CHIRP_LINEAR && !bb.screens) {   // every box is separable (mode 0)
#define CALL(L) box_fft_separable_impl<L>(p, bb, s)
    WPROJ_LOGN_SWITCH(ilog2(bb.S), CALL)
#undef CALL
  }
#define CALL(L) box_fft_impl<L>(p, bb, s)
  WPROJ_LOGN_SWITCH(ilog2(bb.S), CALL)
#undef CALL
}

// blocks of a problem and shared memory of a pass of the joint launches
template <template <int> class Cfg>
void batch_shape(int logG, int lines, int *per, size_t *smem) {
#define CALL(L)                                                      \
  static_assert(Cfg<L>::SMEM <= 48 * 1024, "no attribute is set");   \
  *per = ceil_div(lines, Cfg<L>::C), *smem = std::max(*smem, Cfg<L>::SMEM)
  WPROJ_BATCH_LOGN(logG, CALL)
#undef CALL
}
template <template <int> class Cfg>
int batch_blocks(FftClasses &cl, bool rows, size_t *smem) {
  int n = 0;
  for (int c = 0; c < cl.n; ++c) {
    const int G = 1 << cl.logG[c];
    batch_shape<Cfg>(cl.logG[c], rows ? G / 2 : G, &cl.per[c], smem);
    cl.first[c] = n;
    n += cl.per[c] * cl.np[c];
  }
  return n;
}

wproj_status batch_phi_fwd_all(FftClasses cl, const BProb *tab, const float *x, const float *inv_a, float2 *inter,
                               float2 *Xt, const float2 *tw, cudaStream_t s) {
  size_t smem = 0;
  int n = batch_blocks<BatchRowCfg>(cl, true, &smem);
  WPROJ_CUDA(launch_chained(k_bphi_fwd_rows_all, n, 256, smem, s, cl, tab, x, inv_a, inter, tw));
  smem = 0;
  n = batch_blocks<BatchColCfg>(cl, false, &smem);
  WPROJ_CUDA(launch_chained(k_bphi_fwd_cols_all, n, 256, smem, s, cl, tab, inter, Xt, tw));
  WPROJ_CHECK_LAUNCH("batch phi fwd");
  return WPROJ_OK;
}
wproj_status batch_phi_adj_all(FftClasses cl, const BProb *tab, const float2 *Xt2, const float *inv_a, float2 *inter,
                               float *x_re, const float *z, int mode, const float2 *tw, cudaStream_t s) {
  size_t smem = 0;
  int n = batch_blocks<BatchColCfg>(cl, false, &smem);
  WPROJ_CUDA(launch_chained(k_bphi_adj_cols_all, n, 256, smem, s, cl, tab, Xt2, inter, tw));
  smem = 0;
  n = batch_blocks<BatchRowCfg>(cl, true, &smem);
  WPROJ_CUDA(launch_chained(k_bphi_adj_rows_all, n, 256, smem, s, cl, tab, inter, inv_a, x_re, z, mode, tw));
  WPROJ_CHECK_LAUNCH("batch phi adj");
  return WPROJ_OK;
}

// the sizes above 1024^2, a launch per pass and size
wproj_status batch_phi_fwd(int logG, int np, const int32_t *plist, const BProb *tab, const float *x,
                           const float *inv_a, float2 *inter, float2 *Xt, const float2 *tw, cudaStream_t s) {
  return logG == 11 ? bphi_fwd_impl<11>(np, plist, tab, x, inv_a, inter, Xt, tw, s)
                    : bphi_fwd_impl<12>(np, plist, tab, x, inv_a, inter, Xt, tw, s);
}

wproj_status batch_phi_adj(int logG, int np, const int32_t *plist, const BProb *tab, const float2 *Xt2,
                           const float *inv_a, float2 *inter, float *x_re, const float *z, int mode,
                           const float2 *tw, cudaStream_t s) {
  return logG == 11 ? bphi_adj_impl<11>(np, plist, tab, Xt2, inv_a, inter, x_re, z, mode, tw, s)
                    : bphi_adj_impl<12>(np, plist, tab, Xt2, inv_a, inter, x_re, z, mode, tw, s);
}

}  // namespace wproj
