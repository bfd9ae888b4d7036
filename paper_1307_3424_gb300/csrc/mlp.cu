// The learned-kernel network: an MLP that maps (w, sub-grid offset) to a
// visibility's w-kernel on a fixed 32 x 32 window of grid cells around its cell
// (2048 values: real and imaginary parts) plus a support mask (1024 logits).
// It is trained on kernels from the plain FFT-and-threshold build (Part I), which
// stays the reference and the fallback.
//
//   x0 = (w_c / 2 - 1, 2 du - 1, 2 dv - 1)                     w_c in grid cells
//   h1 = GELU(W1 x0 + b1)   h2 = GELU(W2 h1 + b2)   h3 = GELU(W3 h2 + b3)   (256 each)
//   y  = W4 h3 + b4                                                     (3072)
//   loss = mean_v (y_v - t_v)^2 + mask_weight * mean_m BCE(y_m, t_m)
//
// Layers 2-4 and all their gradients are BF16 GEMMs on the tcgen05 tensor cores
// (gemm.cu) with FP32 accumulation; the 3-wide first layer runs on the FP32
// cores.  Master parameters, Adam moments and the gradients' reductions are FP32,
// the loss is summed to FP64 precision, all in a fixed order.  Activations and the
// gradients fed to GEMMs are rounded to BF16.  GELU is the erf form.
#include <math.h>

#include <chrono>
#include <new>
#include <vector>

#include "plan.h"

namespace wproj {
namespace mlpk {
constexpr int kIn = 3, kH = 256, kOutV = 2048, kOutM = 1024, kOut = kOutV + kOutM, kWin = 32;
constexpr int64_t oW1 = 0, oB1 = oW1 + kH * kIn, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
                  oB3 = oW3 + kH * kH, oW4 = oB3 + kH, oB4 = oW4 + int64_t(kOut) * kH, kParams = oB4 + kOut;
}  // namespace mlpk
}  // namespace wproj

struct wproj_mlp {
  wproj::DevBuf P, Mo, Ve, Gr;          // FP32 parameters, Adam moments, gradients (flat)
  wproj::DevBuf W2b, W3b, W4b;          // BF16 copies [out x in]
  wproj::DevBuf W2t, W3t, W4t;          // BF16 transposes [in x out]
  int64_t step = 0;
  int64_t cap = 0;                      // batch capacity of the activation buffers
  int64_t fcap = 0;                     // rows of the inference buffers (H1 .. H3)
  wproj::DevBuf Z1, Z2, Z3, H1, H2, H3, Y, dY, dYt, Ht, dZt, dH, dZ, part, loss, err;
  wproj::DevBuf split;                  // partial products of the split-K GEMMs
  wproj::DevBuf csum;                   // column-sum partials of 64-row blocks
};

namespace wproj {

namespace {

using namespace mlpk;

__device__ __forceinline__ float gelu_d(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * __expf(-0.5f * z * z);
}

// first layer on the FP32 cores: Z1 = x0 W1^T + b1 (kept when Z1 is given),
// H1 = GELU(Z1).  Thread j of a block holds weights of units 2j, 2j + 1 and walks
// the block's rows, so the weights are read once a block and a warp stores whole
// 128-byte lines (a thread per element read seven words for each BF16 it wrote:
// 49 against 12 us for 65536 rows).
constexpr int kInRows = 32;
__global__ void __launch_bounds__(kH / 2)
k_in_fwd(int64_t B, const float *__restrict__ x0, const float *__restrict__ P, float *__restrict__ Z1,
         __nv_bfloat16 *__restrict__ H1) {
  __shared__ float xs[kInRows * kIn];
  chain_wait();   // the first kernel of a pass
  chain_next();
  x0 = after_wait(x0);
  P = after_wait(P);
  const int64_t b0 = int64_t(blockIdx.x) * kInRows;
  const int nb = int(B - b0 < kInRows ? B - b0 : kInRows);
  for (int i = threadIdx.x; i < nb * kIn; i += blockDim.x) xs[i] = x0[b0 * kIn + i];
  const int j = 2 * threadIdx.x;
  float w[2][kIn], bias[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    bias[u] = P[oB1 + j + u];
#pragma unroll
    for (int c = 0; c < kIn; ++c) w[u][c] = P[oW1 + (j + u) * kIn + c];
  }
  __syncthreads();
#pragma unroll 4
  for (int r = 0; r < nb; ++r) {
    float z[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) z[u] = bias[u] + w[u][0] * xs[3 * r] + w[u][1] * xs[3 * r + 1] + w[u][2] * xs[3 * r + 2];
    const int64_t i = (b0 + r) * kH + j;
    if (Z1) *reinterpret_cast<float2 *>(Z1 + i) = make_float2(z[0], z[1]);
    *reinterpret_cast<__nv_bfloat162 *>(H1 + i) = __floats2bfloat162_rn(gelu(z[0]), gelu(z[1]));
  }
}

// ---- 64 x 64 blocks of a row-major matrix ----------------------------------------
// The backward passes walk 64 x 64 blocks with 256 threads: thread (tx, ty) takes
// columns 4 tx .. 4 tx + 3 of rows ty, ty + 16, ty + 32, ty + 48.  What the GEMMs
// need of a block (BF16 rows, the BF16 transpose, column sums) leaves in one pass.
constexpr int kBlk = 64;
constexpr int kTLd = kBlk + 2;   // transposed rows of 33 words: 2-way store conflicts

struct BlockSmem {
  __nv_bfloat16 t[kBlk][kTLd];
  float red[16][kBlk];
};

// the block's transpose from sm.t to out (leading dimension R) at (c0, r0); every
// thread stores 32 bytes
__device__ __forceinline__ void store_transposed(const BlockSmem &sm, __nv_bfloat16 *__restrict__ out, int64_t R,
                                                 int64_t r0, int64_t c0) {
  const int c = threadIdx.x >> 2, q = (threadIdx.x & 3) * 16;
  const uint32_t *src = reinterpret_cast<const uint32_t *>(&sm.t[c][q]);
  uint4 *dst = reinterpret_cast<uint4 *>(out + (c0 + c) * R + r0 + q);
  dst[0] = make_uint4(src[0], src[1], src[2], src[3]);
  dst[1] = make_uint4(src[4], src[5], src[6], src[7]);
}

__device__ __forceinline__ void put_bf16x4(__nv_bfloat16 *p, __nv_bfloat162 a, __nv_bfloat162 b) {
  uint2 u;
  u.x = *reinterpret_cast<uint32_t *>(&a);
  u.y = *reinterpret_cast<uint32_t *>(&b);
  *reinterpret_cast<uint2 *>(p) = u;
}

// A sum in three floats: every addition keeps its error (Knuth's two-sum), once more in
// the next word, and every square its rounding (fma), so a thread's 16 terms lose nothing
// that FP64 would keep (two words carry 48 bits: up to 117 units of 2^-53 off on 16 equal
// magnitudes, three 0); magnitudes at which that could overflow or underflow, and
// non-finite ones, go to FP64.  FP64 per element (a convert, an FMA and a divide) took
// 263 us for 4096 x 3072 losses.
struct Sum3 {
  float hi = 0.f, lo = 0.f, lo2 = 0.f;
  double wide = 0;
  // s + v -> s, the rounding error returned
  static __device__ __forceinline__ float two_sum(float &s, float v) {
    const float t = __fadd_rn(s, v), z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(v, z));
    s = t;
    return err;
  }
  __device__ __forceinline__ void low(float v) { lo2 = __fadd_rn(lo2, two_sum(lo, v)); }
  __device__ __forceinline__ void add(float v) {
    if (fabsf(v) <= 1e30f) low(two_sum(hi, v));
    else wide += double(v);
  }
  __device__ __forceinline__ void add_square(float a) {
    const float p = __fmul_rn(a, a);
    if (p >= 1e-30f && p <= 1e30f) {
      low(__fmaf_rn(a, a, -p));
      low(two_sum(hi, p));
    } else if (a != 0.f) {
      wide += double(a) * a;
    }
  }
  __device__ __forceinline__ double value() const { return (double(hi) + (double(lo) + double(lo2))) + wide; }
};

// Loss partials and dY = d loss / d y as BF16 rows, its transpose and its column
// sums over the block's 64 rows (bias gradient partials [row block][column]).
// Bound by memory: reads y and the targets, writes dY twice.
__global__ void __launch_bounds__(256)
k_loss(int64_t B, const float *__restrict__ Y, const float *__restrict__ Tv, const float *__restrict__ Tm,
       float mask_weight, __nv_bfloat16 *__restrict__ dY, __nv_bfloat16 *__restrict__ dYt, float *__restrict__ csum,
       double *__restrict__ part) {
  __shared__ BlockSmem sm;
  chain_next();
  chain_wait();
  Y = after_wait(Y);
  const int64_t c0 = int64_t(blockIdx.x) * kBlk, r0 = int64_t(blockIdx.y) * kBlk;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const bool is_val = c0 < kOutV;   // 64 divides kOutV: a block is all values or all mask
  const float s = is_val ? 2.f / float(B * kOutV) : mask_weight / float(B * kOutM);
  const float *T = is_val ? Tv + c0 : Tm + (c0 - kOutV);
  const int ldt = is_val ? kOutV : kOutM;
  Sum3 acc;
  float cs[4] = {0.f, 0.f, 0.f, 0.f};
  float4 yv[4], tv[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = r0 + ty + 16 * i;
    yv[i] = *reinterpret_cast<const float4 *>(Y + r * kOut + c0 + 4 * tx);
    const float *tp = T + r * ldt + 4 * tx;
    tv[i] = (reinterpret_cast<uintptr_t>(tp) & 15) == 0 ? __ldg(reinterpret_cast<const float4 *>(tp))
                                                         : make_float4(tp[0], tp[1], tp[2], tp[3]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float y4[4] = {yv[i].x, yv[i].y, yv[i].z, yv[i].w}, t4[4] = {tv[i].x, tv[i].y, tv[i].z, tv[i].w};
    __nv_bfloat16 g[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float y = y4[q], t = t4[q];
      float gf;
      if (is_val) {
        const float d = y - t;
        acc.add_square(d);
        gf = s * d;
      } else {
        // BCE with logits: max(y, 0) - t y + log(1 + e^{-|y|})
        acc.add(fmaxf(y, 0.f) - t * y + log1pf(__expf(-fabsf(y))));
        gf = s * (1.f / (1.f + __expf(-y)) - t);
      }
      g[q] = __float2bfloat16_rn(gf);
      cs[q] += __bfloat162float(g[q]);
      sm.t[4 * tx + q][ty + 16 * i] = g[q];
    }
    put_bf16x4(dY + (r0 + ty + 16 * i) * kOut + c0 + 4 * tx, __nv_bfloat162(g[0], g[1]), __nv_bfloat162(g[2], g[3]));
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) sm.red[ty][4 * tx + q] = cs[q];
  __syncthreads();
  store_transposed(sm, dYt, B, r0, c0);
  if (threadIdx.x < kBlk) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < 16; ++q) t += sm.red[q][threadIdx.x];
    csum[int64_t(blockIdx.y) * kOut + c0 + threadIdx.x] = t;
  }
  const double t = block_sum_d<256>(acc.value());
  if (threadIdx.x == 0)
    part[int64_t(blockIdx.y) * gridDim.x + blockIdx.x] =
        is_val ? t / double(B * kOutV) : double(mask_weight) * t / double(B * kOutM);
}

__global__ void __launch_bounds__(1024) k_sum_part_d(const double *__restrict__ part, int n, double *__restrict__ out) {
  chain_next();
  chain_wait();
  part = after_wait(part);
  double v = 0;
  for (int i = threadIdx.x; i < n; i += 1024) v += part[i];
  v = block_sum_d<1024>(v);
  if (threadIdx.x == 0) *out = v;
}

// dZ = dH GELU'(Z): BF16 rows and transpose for the next GEMMs and the column sums
// (IN = false); for the first layer (IN = true) only the four column sums of
// dZ (x0, 1), which are its gradients.
template <bool IN>
__global__ void __launch_bounds__(256)
k_gelu_bwd(int64_t B, const float *__restrict__ dH, const float *__restrict__ Z,
           const float *__restrict__ x0, __nv_bfloat16 *__restrict__ dZ, __nv_bfloat16 *__restrict__ dZt,
           float *__restrict__ csum) {
  __shared__ BlockSmem sm;
  constexpr int NV = IN ? 4 : 1;
  chain_next();
  chain_wait();
  dH = after_wait(dH);
  Z = after_wait(Z);
  const int64_t c0 = int64_t(blockIdx.x) * kBlk, r0 = int64_t(blockIdx.y) * kBlk;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float cs[NV][4];
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int q = 0; q < 4; ++q) cs[v][q] = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = r0 + ty + 16 * i, at = r * kH + c0 + 4 * tx;
    const float4 d = *reinterpret_cast<const float4 *>(dH + at);
    const float4 z = *reinterpret_cast<const float4 *>(Z + at);
    const float g[4] = {d.x * gelu_d(z.x), d.y * gelu_d(z.y), d.z * gelu_d(z.z), d.w * gelu_d(z.w)};
    if constexpr (IN) {
      const float a = x0[r * kIn], b = x0[r * kIn + 1], c = x0[r * kIn + 2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        cs[0][q] += g[q] * a;
        cs[1][q] += g[q] * b;
        cs[2][q] += g[q] * c;
        cs[3][q] += g[q];
      }
    } else {
      __nv_bfloat16 h[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        h[q] = __float2bfloat16_rn(g[q]);
        cs[0][q] += __bfloat162float(h[q]);
        sm.t[4 * tx + q][ty + 16 * i] = h[q];
      }
      put_bf16x4(dZ + at, __nv_bfloat162(h[0], h[1]), __nv_bfloat162(h[2], h[3]));
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if (v) __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) sm.red[ty][4 * tx + q] = cs[v][q];
    __syncthreads();
    if (threadIdx.x < kBlk) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < 16; ++q) t += sm.red[q][threadIdx.x];
      csum[(int64_t(blockIdx.y) * NV + v) * kH + c0 + threadIdx.x] = t;
    }
  }
  if constexpr (!IN) store_transposed(sm, dZt, B, r0, c0);
}

// out[i] = sum over p < n of in[p len + i], in order: 8 lanes of partials per 32 elements
__global__ void __launch_bounds__(256)
k_sum_rows(int n, int64_t len, const float *__restrict__ in, float *__restrict__ out) {
  __shared__ float red[8][33];
  chain_next();
  chain_wait();
  in = after_wait(in);
  const int x = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t i = int64_t(blockIdx.x) * 32 + x;
  float t = 0.f;
  if (i < len) {
#pragma unroll 4
    for (int p = g; p < n; p += 8) t += in[int64_t(p) * len + i];
  }
  red[g][x] = t;
  __syncthreads();
  if (g == 0 && i < len) {
#pragma unroll
    for (int q = 1; q < 8; ++q) t += red[q][x];
    out[i] = t;
  }
}

// The same for n <= 8 in 16-byte loads, a thread four elements (len a multiple of 4):
// six partials of 3072 x 256 took 22 us a word at a time.
__global__ void __launch_bounds__(256)
k_sum_few(int n, int64_t len4, const float4 *__restrict__ in, float4 *__restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x;
  chain_next();
  chain_wait();
  in = after_wait(in);
  if (i >= len4) return;
  float4 v[8];
#pragma unroll
  for (int p = 0; p < 8; ++p) v[p] = p < n ? in[p * len4 + i] : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 t = v[0];
#pragma unroll
  for (int p = 1; p < 8; ++p) {
    t.x += v[p].x;
    t.y += v[p].y;
    t.z += v[p].z;
    t.w += v[p].w;
  }
  out[i] = t;
}

// BF16 transposes of the three layers' activations (blockIdx.z), B x kH each
__global__ void __launch_bounds__(256)
k_transpose_h(int64_t B, const __nv_bfloat16 *__restrict__ h1, const __nv_bfloat16 *__restrict__ h2,
              const __nv_bfloat16 *__restrict__ h3, __nv_bfloat16 *__restrict__ out) {
  __shared__ BlockSmem sm;
  chain_next();
  chain_wait();
  const __nv_bfloat16 *in = after_wait(blockIdx.z == 0 ? h1 : (blockIdx.z == 1 ? h2 : h3));
  const int64_t c0 = int64_t(blockIdx.x) * kBlk, r0 = int64_t(blockIdx.y) * kBlk;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint2 u = *reinterpret_cast<const uint2 *>(in + (r0 + ty + 16 * i) * kH + c0 + 4 * tx);
    const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162 *>(&u.x), b = *reinterpret_cast<const __nv_bfloat162 *>(&u.y);
    sm.t[4 * tx][ty + 16 * i] = a.x;
    sm.t[4 * tx + 1][ty + 16 * i] = a.y;
    sm.t[4 * tx + 2][ty + 16 * i] = b.x;
    sm.t[4 * tx + 3][ty + 16 * i] = b.y;
  }
  __syncthreads();
  store_transposed(sm, out + int64_t(blockIdx.z) * B * kH, B, r0, c0);
}

// BF16 copies and transposes of W2, W3 (256 x 256) and W4 (3072 x 256) from the
// FP32 master parameters: block = one 64 x 64 block, W2's 16 first, then W3's, W4's
constexpr int kWBlocks = 2 * (kH / kBlk) * (kH / kBlk) + (kOut / kBlk) * (kH / kBlk);
__global__ void __launch_bounds__(256)
k_weights(const float *__restrict__ P, __nv_bfloat16 *__restrict__ w2, __nv_bfloat16 *__restrict__ w2t,
          __nv_bfloat16 *__restrict__ w3, __nv_bfloat16 *__restrict__ w3t, __nv_bfloat16 *__restrict__ w4,
          __nv_bfloat16 *__restrict__ w4t) {
  __shared__ BlockSmem sm;
  constexpr int kSq = (kH / kBlk) * (kH / kBlk);
  const int which = blockIdx.x < kSq ? 0 : (blockIdx.x < 2 * kSq ? 1 : 2);
  const int b = blockIdx.x - which * kSq, R = which == 2 ? kOut : kH;
  const float *in = P + (which == 0 ? oW2 : (which == 1 ? oW3 : oW4));
  __nv_bfloat16 *o = which == 0 ? w2 : (which == 1 ? w3 : w4), *ot = which == 0 ? w2t : (which == 1 ? w3t : w4t);
  const int64_t r0 = int64_t(b / (kH / kBlk)) * kBlk, c0 = int64_t(b % (kH / kBlk)) * kBlk;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t at = (r0 + ty + 16 * i) * kH + c0 + 4 * tx;
    const float4 v = *reinterpret_cast<const float4 *>(in + at);   // every matrix starts on a multiple of 4 floats
    const __nv_bfloat16 h[4] = {__float2bfloat16_rn(v.x), __float2bfloat16_rn(v.y), __float2bfloat16_rn(v.z),
                                __float2bfloat16_rn(v.w)};
#pragma unroll
    for (int q = 0; q < 4; ++q) sm.t[4 * tx + q][ty + 16 * i] = h[q];
    put_bf16x4(o + at, __nv_bfloat162(h[0], h[1]), __nv_bfloat162(h[2], h[3]));
  }
  __syncthreads();
  store_transposed(sm, ot, R, r0, c0);
}

// first layer gradients from the 4-way column sums of the row blocks
__global__ void k_in_grad(const float *__restrict__ s4, float *__restrict__ G) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  chain_next();
  chain_wait();
  s4 = after_wait(s4);
  if (j >= kH) return;
  G[oW1 + j * kIn] = s4[j];
  G[oW1 + j * kIn + 1] = s4[kH + j];
  G[oW1 + j * kIn + 2] = s4[2 * kH + j];
  G[oB1 + j] = s4[3 * kH + j];
}

__global__ void k_adam(int64_t n, float *__restrict__ P, const float *__restrict__ G, float *__restrict__ M,
                       float *__restrict__ V, float lr, float c1, float c2) {
  constexpr float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float g = G[i];
    const float m = b1 * M[i] + (1.f - b1) * g;
    const float v = b2 * V[i] + (1.f - b2) * g * g;
    M[i] = m;
    V[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
  }
}

int blocks_for(int64_t n) { return (int)std::min<int64_t>(152 * 16, std::max<int64_t>(1, ceil_div(n, 256))); }

wproj_status sum_rows(int n, int64_t len, const float *in, float *out, cudaStream_t s) {
  if (n <= 8 && len % 4 == 0 && ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0)
    WPROJ_CUDA(launch_chained(k_sum_few, ceil_div(len / 4, 256), 256, 0, s, n, len / 4,
                              reinterpret_cast<const float4 *>(in), reinterpret_cast<float4 *>(out)));
  else
    WPROJ_CUDA(launch_chained(k_sum_rows, ceil_div(len, 32), 256, 0, s, n, len, in, out));
  return WPROJ_OK;
}

wproj_status refresh_weights(wproj_mlp *n, cudaStream_t s) {
  k_weights<<<kWBlocks, 256, 0, s>>>(n->P.as<float>(), n->W2b.as<__nv_bfloat16>(), n->W2t.as<__nv_bfloat16>(),
                                     n->W3b.as<__nv_bfloat16>(), n->W3t.as<__nv_bfloat16>(), n->W4b.as<__nv_bfloat16>(),
                                     n->W4t.as<__nv_bfloat16>());
  WPROJ_CHECK_LAUNCH("weights to bf16");
  return WPROJ_OK;
}

// activations of inference, B rows
wproj_status ensure_forward(wproj_mlp *n, int64_t B) {
  if (n->fcap >= B) return WPROJ_OK;
  n->fcap = 0;
  WPROJ_TRY(n->H1.alloc(2 * B * kH));
  WPROJ_TRY(n->H2.alloc(2 * B * kH));
  WPROJ_TRY(n->H3.alloc(2 * B * kH));
  n->fcap = B;
  return WPROJ_OK;
}

wproj_status ensure_batch(wproj_mlp *n, int64_t B) {
  WPROJ_TRY(ensure_forward(n, B));
  if (n->cap >= B) return WPROJ_OK;
  n->cap = 0;
  WPROJ_TRY(n->Z1.alloc(sizeof(float) * B * kH));
  WPROJ_TRY(n->Z2.alloc(sizeof(float) * B * kH));
  WPROJ_TRY(n->Z3.alloc(sizeof(float) * B * kH));
  WPROJ_TRY(n->Y.alloc(sizeof(float) * B * kOut));
  WPROJ_TRY(n->dY.alloc(2 * B * kOut));
  WPROJ_TRY(n->dYt.alloc(2 * B * kOut));
  WPROJ_TRY(n->Ht.alloc(3 * 2 * B * kH));
  WPROJ_TRY(n->dZt.alloc(2 * B * kH));
  WPROJ_TRY(n->dH.alloc(sizeof(float) * B * kH));
  WPROJ_TRY(n->dZ.alloc(2 * B * kH));
  WPROJ_TRY(n->csum.alloc(sizeof(float) * (B / kBlk) * kOut));   // covers 4 x 256 columns too
  WPROJ_TRY(n->part.alloc(sizeof(double) * (B / kBlk) * (kOut / kBlk)));
  n->cap = B;
  return WPROJ_OK;
}

// C = A B^T (+ bias), FP32 and, when H is given, BF16 (GELU) outputs
wproj_status gemm(int M, int N, int K, const void *A, const void *B, const float *bias, float *Z, __nv_bfloat16 *H,
                  wproj_mlp *n, cudaStream_t s) {
  GemmOut o;
  o.bias = bias;
  o.f32 = Z;
  o.bf16 = H;
  o.gelu = H != nullptr;
  return gemm_bf16_tn(M, N, K, static_cast<const __nv_bfloat16 *>(A), static_cast<const __nv_bfloat16 *>(B), o,
                      n->err.as<int>(), s);
}

// Weight gradient C = A B^T in FP32 (K = the batch, few tiles) with K split over the
// idle SMs: partial products in n->split, added in order into C.  The gradients of
// the activations are not split: they are rounded to BF16 for the next layer, and
// another order of their FP32 sum moves some of those roundings.
wproj_status gemm_wgrad(int M, int N, int K, const void *A, const void *B, float *C, wproj_mlp *n, cudaStream_t s) {
  GemmOut o;
  WPROJ_TRY(gemm_splits(M, N, K, &o.splits));
  WPROJ_TRY(n->split.ensure(sizeof(float) * size_t(o.splits) * M * N));
  o.f32 = o.splits > 1 ? n->split.as<float>() : C;
  WPROJ_TRY(gemm_bf16_tn(M, N, K, static_cast<const __nv_bfloat16 *>(A), static_cast<const __nv_bfloat16 *>(B), o,
                         n->err.as<int>(), s));
  return o.splits > 1 ? sum_rows(o.splits, int64_t(M) * N, n->split.as<float>(), C, s) : WPROJ_OK;
}

// forward of B rows (B a multiple of 128) into Y; train: keep Z1 .. Z3 for backward
wproj_status forward(wproj_mlp *n, const float *x0, int64_t B, float *Y, bool train, cudaStream_t s) {
  const float *P = n->P.as<float>();
  auto *H1 = n->H1.as<__nv_bfloat16>(), *H2 = n->H2.as<__nv_bfloat16>(), *H3 = n->H3.as<__nv_bfloat16>();
  WPROJ_CUDA(launch_chained(k_in_fwd, ceil_div(B, kInRows), kH / 2, 0, s, B, x0, P,
                            train ? n->Z1.as<float>() : nullptr, H1));
  WPROJ_TRY(gemm((int)B, kH, kH, H1, n->W2b.ptr, P + oB2, train ? n->Z2.as<float>() : nullptr, H2, n, s));
  WPROJ_TRY(gemm((int)B, kH, kH, H2, n->W3b.ptr, P + oB3, train ? n->Z3.as<float>() : nullptr, H3, n, s));
  return gemm((int)B, kOut, kH, H3, n->W4b.ptr, P + oB4, Y, nullptr, n, s);
}

// loss (device double at *loss_d) and gradients into n->Gr for B rows
wproj_status backward(wproj_mlp *n, const float *x0, const float *Tv, const float *Tm, int64_t B, float mask_weight,
                      double *loss_d, cudaStream_t s) {
  float *G = n->Gr.as<float>(), *csum = n->csum.as<float>();
  auto *Ht = n->Ht.as<__nv_bfloat16>();
  auto *dZ = n->dZ.as<__nv_bfloat16>(), *dZt = n->dZt.as<__nv_bfloat16>();
  const int nrb = int(B / kBlk);
  const dim3 lg(kOut / kBlk, nrb), hg(kH / kBlk, nrb);
  WPROJ_CUDA(launch_chained(k_loss, lg, 256, 0, s, B, n->Y.as<float>(), Tv, Tm, mask_weight, n->dY.as<__nv_bfloat16>(),
                            n->dYt.as<__nv_bfloat16>(), csum, n->part.as<double>()));
  WPROJ_CUDA(launch_chained(k_sum_part_d, 1, 1024, 0, s, n->part.as<double>(), int(lg.x * lg.y), loss_d));
  WPROJ_CUDA(launch_chained(k_transpose_h, dim3(kH / kBlk, nrb, 3), 256, 0, s, B, n->H1.as<__nv_bfloat16>(),
                            n->H2.as<__nv_bfloat16>(), n->H3.as<__nv_bfloat16>(), Ht));
  // layer 4
  float *dH = n->dH.as<float>();
  WPROJ_TRY(sum_rows(nrb, kOut, csum, G + oB4, s));
  WPROJ_TRY(gemm_wgrad(kOut, kH, (int)B, n->dYt.ptr, Ht + 2 * B * kH, G + oW4, n, s));
  WPROJ_TRY(gemm((int)B, kH, kOut, n->dY.ptr, n->W4t.ptr, nullptr, dH, nullptr, n, s));
  // layers 3 and 2
  const __nv_bfloat16 *Wt[2] = {n->W3t.as<__nv_bfloat16>(), n->W2t.as<__nv_bfloat16>()};
  const float *Z[2] = {n->Z3.as<float>(), n->Z2.as<float>()};
  const int64_t oW[2] = {oW3, oW2}, oB[2] = {oB3, oB2};
  for (int l = 0; l < 2; ++l) {
    WPROJ_CUDA(launch_chained(k_gelu_bwd<false>, hg, 256, 0, s, B, dH, Z[l], nullptr, dZ, dZt, csum));
    WPROJ_TRY(sum_rows(nrb, kH, csum, G + oB[l], s));
    WPROJ_TRY(gemm_wgrad(kH, kH, (int)B, dZt, Ht + (1 - l) * B * kH, G + oW[l], n, s));
    WPROJ_TRY(gemm((int)B, kH, kH, dZ, Wt[l], nullptr, dH, nullptr, n, s));
  }
  // layer 1
  WPROJ_CUDA(launch_chained(k_gelu_bwd<true>, hg, 256, 0, s, B, dH, n->Z1.as<float>(), x0, nullptr, nullptr, csum));
  WPROJ_TRY(sum_rows(nrb, 4 * kH, csum, dH, s));   // dH is spent: its first 4 kH floats take the sums
  WPROJ_CUDA(launch_chained(k_in_grad, 1, kH, 0, s, dH, G));
  return WPROJ_OK;
}

wproj_status check_err(wproj_mlp *n, cudaStream_t s) {
  int h = 0;
  WPROJ_CUDA(cudaMemcpyAsync(&h, n->err.ptr, sizeof(int), cudaMemcpyDeviceToHost, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  if (h) return fail(WPROJ_ERR_TIMEOUT, "mlp: a tensor-core wait ran out");
  return WPROJ_OK;
}

// Training targets from a built plan: window cell (a, b) <-> grid cell
// (j0 - 16 + a, j0 - 16 + b) mod G; values scaled by 1 / sqrt(E_kb), E_kb =
// prod_axes sum_t kb(delta - t)^2 over the W taps.
__global__ void k_targets(int64_t m, const double *__restrict__ uvw, const int64_t *__restrict__ row_ptr,
                          const int32_t *__restrict__ col, const float2 *__restrict__ val, int G, double du,
                          double L, int W, double beta, float *__restrict__ x0, float *__restrict__ Tv,
                          float *__restrict__ Tm) {
  const int64_t k = blockIdx.x;
  if (k >= m) return;
  const double gu = uvw[3 * k] / du, gv = uvw[3 * k + 1] / du;
  const double fu = floor(gu), fv = floor(gv);
  const int ju = int(fu), jv = int(fv);
  const double dlu = gu - fu, dlv = gv - fv;
  for (int i = threadIdx.x; i < kOutV; i += blockDim.x) Tv[k * kOutV + i] = 0.f;
  for (int i = threadIdx.x; i < kOutM; i += blockDim.x) Tm[k * kOutM + i] = 0.f;
  double eu = 0, ev = 0;
  for (int t = -W / 2 + 1; t <= W / 2; ++t) {
    const double a = kb_dev(dlu - t, W, beta), b = kb_dev(dlv - t, W, beta);
    eu += a * a;
    ev += b * b;
  }
  const float inv = float(1.0 / sqrt(eu * ev));
  if (threadIdx.x == 0) {
    const double wc = fabs(uvw[3 * k + 2]) * L * L / 2.0;   // h = |w| L^2 = 2 w_c
    x0[k * 3] = float(wc / 2.0 - 1.0);
    x0[k * 3 + 1] = float(2.0 * dlu - 1.0);
    x0[k * 3 + 2] = float(2.0 * dlv - 1.0);
  }
  __syncthreads();
  const int ou = ((ju - kWin / 2) % G + G) % G, ov = ((jv - kWin / 2) % G + G) % G;
  for (int64_t i = row_ptr[k] + threadIdx.x; i < row_ptr[k + 1]; i += blockDim.x) {
    const int q = col[i];
    const int a = ((q / G - ou) % G + G) % G, b = ((q % G - ov) % G + G) % G;
    if (a < kWin && b < kWin) {
      const float2 v = val[i];
      Tv[k * kOutV + 2 * (a * kWin + b)] = v.x * inv;
      Tv[k * kOutV + 2 * (a * kWin + b) + 1] = v.y * inv;
      Tm[k * kOutM + a * kWin + b] = 1.f;
    }
  }
}

// Network input of every row (the x0 of k_targets).
__global__ void k_features(int64_t m, const double *__restrict__ uvw, double du, double L, float *__restrict__ x0) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const double gu = uvw[3 * k] / du, gv = uvw[3 * k + 1] / du;
  const double wc = fabs(uvw[3 * k + 2]) * L * L / 2.0;
  x0[k * 3] = float(wc / 2.0 - 1.0);
  x0[k * 3 + 1] = float(2.0 * (gu - floor(gu)) - 1.0);
  x0[k * 3 + 2] = float(2.0 * (gv - floor(gv)) - 1.0);
}

// Judge the predicted kernels of rows [r0, r0 + nr) against the plain ones and
// take the predicted values where they pass: rel. L2 over the window <= relmax,
// the predicted support holding >= e of the kernel energy (measured on the
// plain kernel), and no plain entry outside the window.  Block per row.
__global__ void __launch_bounds__(256)
k_judge(int64_t r0, const double *__restrict__ uvw, const int64_t *__restrict__ row_ptr,
        const int32_t *__restrict__ col, float2 *__restrict__ val, const float *__restrict__ Y, int G, double du,
        int W, double beta, double e, double relmax, float *__restrict__ row_err, int8_t *__restrict__ pass) {
  __shared__ float2 T[kWin * kWin];
  __shared__ int outside;
  const int64_t k = r0 + blockIdx.x;
  const float *y = Y + int64_t(blockIdx.x) * kOut;
  const double gu = uvw[3 * k] / du, gv = uvw[3 * k + 1] / du;
  const double fu = floor(gu), fv = floor(gv);
  const double dlu = gu - fu, dlv = gv - fv;
  double eu = 0, ev = 0;
  for (int t = -W / 2 + 1; t <= W / 2; ++t) {
    const double a = kb_dev(dlu - t, W, beta), b = kb_dev(dlv - t, W, beta);
    eu += a * a;
    ev += b * b;
  }
  const double ekb = eu * ev;
  const float sc = float(sqrt(ekb));
  for (int i = threadIdx.x; i < kWin * kWin; i += blockDim.x) T[i] = make_float2(0.f, 0.f);
  if (threadIdx.x == 0) outside = 0;
  __syncthreads();
  const int ou = ((int(fu) - kWin / 2) % G + G) % G, ov = ((int(fv) - kWin / 2) % G + G) % G;
  const int64_t lo = row_ptr[k], hi = row_ptr[k + 1];
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const int q = col[i];
    const int a = ((q / G - ou) % G + G) % G, b = ((q % G - ov) % G + G) % G;
    if (a < kWin && b < kWin) T[a * kWin + b] = val[i];
    else outside = 1;
  }
  __syncthreads();
  double d2 = 0, t2 = 0, sup = 0;
  for (int i = threadIdx.x; i < kWin * kWin; i += blockDim.x) {
    const float2 t = T[i];
    const float px = y[2 * i] * sc, py = y[2 * i + 1] * sc;
    d2 += double(px - t.x) * (px - t.x) + double(py - t.y) * (py - t.y);
    const double tt = double(t.x) * t.x + double(t.y) * t.y;
    t2 += tt;
    if (y[kOutV + i] > 0.f) sup += tt;
  }
  d2 = block_sum_d<256>(d2);
  t2 = block_sum_d<256>(t2);
  sup = block_sum_d<256>(sup);
  __shared__ int ok;
  if (threadIdx.x == 0) {
    const double r = t2 > 0 ? sqrt(d2 / t2) : 1.0;
    ok = (!outside && r <= relmax && sup >= e * ekb) ? 1 : 0;
    if (row_err) row_err[k] = float(r);
    pass[k] = int8_t(ok);
  }
  __syncthreads();
  if (!ok) return;
  for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const int q = col[i];
    const int a = ((q / G - ou) % G + G) % G, b = ((q % G - ov) % G + G) % G;
    const int c = a * kWin + b;
    val[i] = make_float2(y[2 * c] * sc, y[2 * c + 1] * sc);
  }
}

__global__ void k_count_pass(int64_t m, const int8_t *__restrict__ pass, const float *__restrict__ err,
                             unsigned long long *__restrict__ n, double *__restrict__ esum) {
  __shared__ double es[256];
  __shared__ unsigned long long ns[256];
  double a = 0;
  unsigned long long c = 0;
  for (int64_t k = threadIdx.x; k < m; k += blockDim.x) {
    c += pass[k];
    a += err[k];
  }
  es[threadIdx.x] = a;
  ns[threadIdx.x] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    unsigned long long u = 0;
    for (int i = 0; i < 256; ++i) { t += es[i]; u += ns[i]; }
    *n = u;
    *esum = t;
  }
}

}  // namespace

int64_t mlp_num_params() { return kParams; }

wproj_status build_learned_impl(wproj_plan *p, wproj_mlp *n, const double *uvw, int64_t m, double e, double relmax,
                                float *row_err, wproj_learned_info *info, cudaStream_t s) {
  auto t0 = std::chrono::steady_clock::now();
  WPROJ_TRY(build_kernels_impl(p, uvw, m, e, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  auto t1 = std::chrono::steady_clock::now();
  if (p->fmt != WPROJ_INDEX_COLUMNS || p->g.value_dtype != WPROJ_VAL_F32)
    return fail(WPROJ_ERR_UNSUPPORTED, "build_kernels_learned: needs complex64 values and column indices");
  const int64_t chunk = 65536;
  DevBuf x0, Y, err, pass, cnt;
  WPROJ_TRY(x0.alloc(sizeof(float) * 3 * (m + 128)));
  WPROJ_TRY(Y.alloc(sizeof(float) * chunk * kOut));
  WPROJ_TRY(pass.alloc(m));
  WPROJ_TRY(cnt.alloc(sizeof(double) * 2));
  float *err_p = row_err;
  if (!err_p) {
    WPROJ_TRY(err.alloc(sizeof(float) * m));
    err_p = err.as<float>();
  }
  WPROJ_CUDA(cudaMemsetAsync(x0.ptr, 0, sizeof(float) * 3 * (m + 128), s));
  k_features<<<ceil_div(m, 256), 256, 0, s>>>(m, uvw, p->g.du, p->g.L, x0.as<float>());
  WPROJ_CHECK_LAUNCH("mlp features");
  WPROJ_TRY(ensure_forward(n, chunk));
  for (int64_t r = 0; r < m; r += chunk) {
    const int64_t nr = std::min(chunk, m - r);
    const int64_t B = (nr + 127) / 128 * 128;   // padded rows read zero features
    WPROJ_TRY(forward(n, x0.as<float>() + 3 * r, B, Y.as<float>(), false, s));
    k_judge<<<(unsigned)nr, 256, 0, s>>>(r, uvw, p->row_ptr.as<int64_t>(), p->col.as<int32_t>(), p->val.as<float2>(),
                                         Y.as<float>(), p->g.G, p->g.du, p->g.W, p->g.beta, e, relmax, err_p,
                                         pass.as<int8_t>());
    WPROJ_CHECK_LAUNCH("mlp judge");
  }
  WPROJ_TRY(check_err(n, s));
  WPROJ_TRY(rebuild_cells(p, s));
  WPROJ_TRY(rebuild_slices(p, s));
  k_count_pass<<<1, 256, 0, s>>>(m, pass.as<int8_t>(), err_p, cnt.as<unsigned long long>(), cnt.as<double>() + 1);
  WPROJ_CHECK_LAUNCH("mlp pass count");
  unsigned long long np_ = 0;
  double es = 0;
  WPROJ_CUDA(cudaMemcpyAsync(&np_, cnt.ptr, sizeof(np_), cudaMemcpyDeviceToHost, s));
  WPROJ_CUDA(cudaMemcpyAsync(&es, cnt.as<double>() + 1, sizeof(double), cudaMemcpyDeviceToHost, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  auto t2 = std::chrono::steady_clock::now();
  p->dr_valid = false;
  if (info) {
    info->rows = m;
    info->learned = int64_t(np_);
    info->rel_l2_mean = es / double(m);
    info->plain_ms = std::chrono::duration<double, std::milli>(t1 - t0).count();
    info->learned_ms = std::chrono::duration<double, std::milli>(t2 - t1).count();
  }
  return WPROJ_OK;
}

wproj_status mlp_create(wproj_mlp *n) {
  WPROJ_TRY(n->P.alloc(sizeof(float) * kParams));
  WPROJ_TRY(n->Mo.alloc(sizeof(float) * kParams));
  WPROJ_TRY(n->Ve.alloc(sizeof(float) * kParams));
  WPROJ_TRY(n->Gr.alloc(sizeof(float) * kParams));
  WPROJ_TRY(n->W2b.alloc(2 * kH * kH));
  WPROJ_TRY(n->W3b.alloc(2 * kH * kH));
  WPROJ_TRY(n->W4b.alloc(2 * int64_t(kOut) * kH));
  WPROJ_TRY(n->W2t.alloc(2 * kH * kH));
  WPROJ_TRY(n->W3t.alloc(2 * kH * kH));
  WPROJ_TRY(n->W4t.alloc(2 * int64_t(kOut) * kH));
  WPROJ_TRY(n->loss.alloc(sizeof(double)));
  WPROJ_TRY(n->err.alloc(sizeof(int)));
  WPROJ_CUDA(cudaMemset(n->P.ptr, 0, sizeof(float) * kParams));
  WPROJ_CUDA(cudaMemset(n->Mo.ptr, 0, sizeof(float) * kParams));
  WPROJ_CUDA(cudaMemset(n->Ve.ptr, 0, sizeof(float) * kParams));
  WPROJ_CUDA(cudaMemset(n->err.ptr, 0, sizeof(int)));
  return WPROJ_OK;
}

wproj_status mlp_set_params(wproj_mlp *n, const float *p, cudaStream_t s) {
  WPROJ_CUDA(cudaMemcpyAsync(n->P.ptr, p, sizeof(float) * kParams, cudaMemcpyDefault, s));
  WPROJ_CUDA(cudaMemsetAsync(n->Mo.ptr, 0, sizeof(float) * kParams, s));
  WPROJ_CUDA(cudaMemsetAsync(n->Ve.ptr, 0, sizeof(float) * kParams, s));
  n->step = 0;
  WPROJ_TRY(refresh_weights(n, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  return WPROJ_OK;
}

wproj_status mlp_get_params(const wproj_mlp *n, float *p, cudaStream_t s) {
  WPROJ_CUDA(cudaMemcpyAsync(p, n->P.ptr, sizeof(float) * kParams, cudaMemcpyDefault, s));
  WPROJ_CUDA(cudaStreamSynchronize(s));
  return WPROJ_OK;
}

wproj_status mlp_forward(wproj_mlp *n, const float *x0, int64_t m, float *y, int64_t chunk, cudaStream_t s) {
  WPROJ_TRY(ensure_forward(n, chunk));
  for (int64_t r = 0; r < m; r += chunk) {
    const int64_t B = std::min<int64_t>(chunk, m - r);
    WPROJ_TRY(forward(n, x0 + 3 * r, B, y + r * kOut, false, s));
  }
  return check_err(n, s);
}

wproj_status mlp_gradients(wproj_mlp *n, const float *x0, const float *Tv, const float *Tm, int64_t B,
                           double mask_weight, double *loss, float *grad, cudaStream_t s) {
  WPROJ_TRY(ensure_batch(n, B));
  WPROJ_TRY(forward(n, x0, B, n->Y.as<float>(), true, s));
  WPROJ_TRY(backward(n, x0, Tv, Tm, B, float(mask_weight), n->loss.as<double>(), s));
  WPROJ_CUDA(cudaMemcpyAsync(loss, n->loss.as<double>(), sizeof(double), cudaMemcpyDeviceToHost, s));
  if (grad) WPROJ_CUDA(cudaMemcpyAsync(grad, n->Gr.ptr, sizeof(float) * kParams, cudaMemcpyDefault, s));
  return check_err(n, s);
}

wproj_status mlp_train(wproj_mlp *n, const float *x0, const float *Tv, const float *Tm, int64_t m, int B, int steps,
                       double lr, double mask_weight, float *losses, cudaStream_t s) {
  WPROJ_TRY(ensure_batch(n, B));
  std::vector<double> hl(steps);
  DevBuf dl;
  WPROJ_TRY(dl.alloc(sizeof(double) * std::max(1, steps)));
  const int64_t nbatch = m / B;
  for (int it = 0; it < steps; ++it) {
    const int64_t r = (it % nbatch) * B;
    WPROJ_TRY(forward(n, x0 + 3 * r, B, n->Y.as<float>(), true, s));
    WPROJ_TRY(backward(n, x0 + 3 * r, Tv + r * kOutV, Tm + r * kOutM, B, float(mask_weight), dl.as<double>() + it, s));
    n->step += 1;
    const float c1 = 1.f - powf(0.9f, float(n->step)), c2 = 1.f - powf(0.999f, float(n->step));
    k_adam<<<blocks_for(kParams), 256, 0, s>>>(kParams, n->P.as<float>(), n->Gr.as<float>(), n->Mo.as<float>(),
                                               n->Ve.as<float>(), float(lr), c1, c2);
    WPROJ_CHECK_LAUNCH("adam");
    WPROJ_TRY(refresh_weights(n, s));
  }
  WPROJ_CUDA(cudaMemcpyAsync(hl.data(), dl.ptr, sizeof(double) * steps, cudaMemcpyDeviceToHost, s));
  WPROJ_TRY(check_err(n, s));
  if (losses)
    for (int i = 0; i < steps; ++i) losses[i] = float(hl[i]);
  return WPROJ_OK;
}

wproj_status mlp_targets(const wproj_plan *p, const double *uvw, float *x0, float *Tv, float *Tm, cudaStream_t s) {
  if (p->fmt != WPROJ_INDEX_COLUMNS || p->g.value_dtype != WPROJ_VAL_F32)
    return fail(WPROJ_ERR_UNSUPPORTED, "mlp_targets: needs a complex64 plan with column indices");
  k_targets<<<(unsigned)p->m, 128, 0, s>>>(p->m, uvw, p->row_ptr.as<int64_t>(), p->col.as<int32_t>(),
                                           p->val.as<float2>(), p->g.G, p->g.du, p->g.L, p->g.W, p->g.beta, x0, Tv,
                                           Tm);
  WPROJ_CHECK_LAUNCH("mlp targets");
  return WPROJ_OK;
}

}  // namespace wproj

// ---- C-ABI ------------------------------------------------------------------------

using namespace wproj;

extern "C" {

int64_t wproj_mlp_num_params(void) { return mlp_num_params(); }

wproj_status wproj_mlp_create(wproj_mlp **out) {
  if (!out) return fail(WPROJ_ERR_INVALID_ARG, "mlp_create: null out");
  *out = nullptr;
  auto *n = new (std::nothrow) wproj_mlp();
  if (!n) return fail(WPROJ_ERR_OOM, "mlp_create: host allocation");
  wproj_status st = mlp_create(n);
  if (st != WPROJ_OK) {
    delete n;
    return st;
  }
  *out = n;
  return WPROJ_OK;
}

wproj_status wproj_mlp_destroy(wproj_mlp *n) {
  delete n;
  return WPROJ_OK;
}

wproj_status wproj_mlp_set_params(wproj_mlp *n, const float *params, void *stream) {
  if (!n || !params) return fail(WPROJ_ERR_INVALID_ARG, "mlp_set_params: null argument");
  return mlp_set_params(n, params, static_cast<cudaStream_t>(stream));
}

wproj_status wproj_mlp_get_params(const wproj_mlp *n, float *params, void *stream) {
  if (!n || !params) return fail(WPROJ_ERR_INVALID_ARG, "mlp_get_params: null argument");
  return mlp_get_params(n, params, static_cast<cudaStream_t>(stream));
}

wproj_status wproj_mlp_targets(const wproj_plan *p, const double *uvw, float *x0, float *tval, float *tmask,
                               void *stream) {
  if (!p || !p->built) return fail(WPROJ_ERR_NOT_BUILT, "mlp_targets: build the plan first");
  if (!uvw || !x0 || !tval || !tmask) return fail(WPROJ_ERR_INVALID_ARG, "mlp_targets: null argument");
  return mlp_targets(p, uvw, x0, tval, tmask, static_cast<cudaStream_t>(stream));
}

wproj_status wproj_mlp_forward(wproj_mlp *n, const float *x0, int64_t m, float *y, void *stream) {
  if (!n || !x0 || !y) return fail(WPROJ_ERR_INVALID_ARG, "mlp_forward: null argument");
  if (m < 128 || m % 128) return fail(WPROJ_ERR_INVALID_ARG, "mlp_forward: m must be a positive multiple of 128");
  return mlp_forward(n, x0, m, y, std::min<int64_t>(m, 65536), static_cast<cudaStream_t>(stream));
}

wproj_status wproj_mlp_gradients(wproj_mlp *n, const float *x0, const float *tval, const float *tmask, int64_t m,
                                 double mask_weight, double *loss, float *grad, void *stream) {
  if (!n || !x0 || !tval || !tmask || !loss) return fail(WPROJ_ERR_INVALID_ARG, "mlp_gradients: null argument");
  if (m < 128 || m % 128 || m > 65536)
    return fail(WPROJ_ERR_INVALID_ARG, "mlp_gradients: m must be a multiple of 128 up to 65536");
  return mlp_gradients(n, x0, tval, tmask, m, mask_weight, loss, grad, static_cast<cudaStream_t>(stream));
}

wproj_status wproj_build_kernels_learned(wproj_plan *p, wproj_mlp *n, const double *uvw, int64_t m, double e,
                                         double rel_l2_max, float *row_err, wproj_learned_info *info, void *stream) {
  if (!p || !n || !uvw) return fail(WPROJ_ERR_INVALID_ARG, "build_kernels_learned: null argument");
  if (m < 1) return fail(WPROJ_ERR_INVALID_ARG, "build_kernels_learned: m >= 1");
  if (!(e > 0.0 && e <= 1.0)) return fail(WPROJ_ERR_INVALID_ARG, "build_kernels_learned: e must lie in (0, 1]");
  if (!(rel_l2_max >= 0.0)) return fail(WPROJ_ERR_INVALID_ARG, "build_kernels_learned: rel_l2_max >= 0");
  return build_learned_impl(p, n, uvw, m, e, rel_l2_max, row_err, info, static_cast<cudaStream_t>(stream));
}

wproj_status wproj_mlp_train(wproj_mlp *n, const float *x0, const float *tval, const float *tmask, int64_t m,
                             int32_t batch, int32_t steps, double lr, double mask_weight, float *losses,
                             void *stream) {
  if (!n || !x0 || !tval || !tmask) return fail(WPROJ_ERR_INVALID_ARG, "mlp_train: null argument");
  if (batch < 128 || batch % 128 || batch > 65536 || m < batch || m % batch || steps < 0 || !(lr > 0))
    return fail(WPROJ_ERR_INVALID_ARG, "mlp_train: batch a multiple of 128 (<= 65536) dividing m, lr > 0");
  return mlp_train(n, x0, tval, tmask, m, batch, steps, lr, mask_weight, losses, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
