// Stockham FFT (radix 4, one radix-2 stage when log2 n is odd) with 16 elements of a
// transform in each thread's registers.
//
// A thread of a length-N transform (N / 16 threads) holds the elements at stride
// N / 16 from its own index: the inputs of 16 / R butterfly groups of radix R =
// R1 R2, two consecutive Stockham stages.  A pass computes both stages in
// registers and the block exchanges the results through shared memory, so a
// transform of 12 stages crosses shared memory twice (3 passes) where a pass per
// stage crossed it six times; the first pass takes its inputs straight from the
// caller's load and the last hands its outputs to the caller's store.  Loads and
// stores of lanes with consecutive indices are consecutive.  Every butterfly and
// twiddle product is that of the plain stage-by-stage form, in the same order,
// so the results do not depend on the pass structure.
//
// Bound by memory for large grids and by the chain of passes (latency) for small
// ones.  4096^2 grid, Phi's column pass (67 MB in, 134 MB out): 130 us stage by stage,
// 72 us so; row pass 50 and 28 us; 128^2: 12.7 + 7.9 and 4.8 + 4.4 us.
//
// Twiddles come from tables tw_n[k] = exp(-2 pi i k / n), k < n, for every power
// of two n (stored at offset n), computed once in double precision and rounded
// to float.
#pragma once

#include "common.cuh"

namespace wproj {

// Twiddle tables for N = 2 .. 4096, table of size N stored at offset N.
constexpr int kMaxLogN = 12;
constexpr int kTwiddleLen = 2 << kMaxLogN;
constexpr int kFftE = 16;   // elements per thread

template <int R, int DIR>
__device__ __forceinline__ void small_dft(float2 (&a)[R]) {
  if constexpr (R == 2) {
    float2 t = a[1];
    a[1] = csub(a[0], t);
    a[0] = cadd(a[0], t);
  } else {
    static_assert(R == 4, "radix");
    float2 t0 = cadd(a[0], a[2]);
    float2 t1 = csub(a[0], a[2]);
    float2 t2 = cadd(a[1], a[3]);
    float2 t3 = csub(a[1], a[3]);
    a[0] = cadd(t0, t2);
    a[2] = csub(t0, t2);
    // forward: X1 = t1 - i t3, X3 = t1 + i t3; inverse swaps them
    float2 m = make_float2(t1.x + t3.y, t1.y - t3.x);   // t1 - i t3
    float2 p = make_float2(t1.x - t3.y, t1.y + t3.x);   // t1 + i t3
    if (DIR < 0) { a[1] = m; a[3] = p; } else { a[1] = p; a[3] = m; }
  }
}

// One stage's butterfly in registers: input r times exp(-+2 pi i k r / n), tw the
// table of length n.
template <int R, int DIR, bool UNIT>
__device__ __forceinline__ void stage_dft(float2 (&a)[R], int k, const float2 *__restrict__ tw) {
  if constexpr (!UNIT) {   // UNIT: k = 0, all twiddles 1
#pragma unroll
    for (int r = 1; r < R; ++r) {
      float2 w = __ldg(&tw[k * r]);
      if (DIR > 0) w.y = -w.y;
      a[r] = cmul(a[r], w);
    }
  }
  small_dft<R, DIR>(a);
}

// Stages R1 (span Ns) and R2 (span Ns R1) of the groups g of thread tq: element
// (r1 R2 + r2) * (16 / R) + g of v goes in as input (r1, r2) of group q = tq + g N / 16
// and comes out as output (r1, r2), whose Stockham position is
//   (q / Ns) Ns R + q mod Ns + r1 Ns + r2 Ns R1.
template <int LOGN, int R1, int R2, int NS, int DIR>
__device__ __forceinline__ void fft_pass(float2 (&v)[kFftE], int tq, const float2 *__restrict__ twtab) {
  constexpr int N = 1 << LOGN, R = R1 * R2, NG = kFftE / R;
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int k1 = (tq + g * (N / kFftE)) & (NS - 1);
#pragma unroll
    for (int r2 = 0; r2 < R2; ++r2) {
      float2 a[R1];
#pragma unroll
      for (int r1 = 0; r1 < R1; ++r1) a[r1] = v[(r1 * R2 + r2) * NG + g];
      stage_dft<R1, DIR, NS == 1>(a, k1, twtab + NS * R1);
#pragma unroll
      for (int r1 = 0; r1 < R1; ++r1) v[(r1 * R2 + r2) * NG + g] = a[r1];
    }
    if constexpr (R2 > 1) {
#pragma unroll
      for (int r1 = 0; r1 < R1; ++r1) {
        float2 a[R2];
#pragma unroll
        for (int r2 = 0; r2 < R2; ++r2) a[r2] = v[(r1 * R2 + r2) * NG + g];
        stage_dft<R2, DIR, false>(a, r1 * NS + k1, twtab + NS * R);
#pragma unroll
        for (int r2 = 0; r2 < R2; ++r2) v[(r1 * R2 + r2) * NG + g] = a[r2];
      }
    }
  }
}

// position p of a transform in the exchange buffer: one element of padding per 16,
// so that lanes storing at stride 16 (or 8) and lanes reading consecutive
// positions both spread over the banks
__host__ __device__ constexpr int fft_pad(int p) { return p + (p >> 4); }

template <int LOGN, int R1, int R2, int NS>
__device__ __forceinline__ void fft_exchange(float2 (&v)[kFftE], int tq, float2 *s) {
  constexpr int N = 1 << LOGN, R = R1 * R2, NG = kFftE / R;
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int q = tq + g * (N / kFftE), k = q & (NS - 1), base = (q - k) * R + k;
#pragma unroll
    for (int r1 = 0; r1 < R1; ++r1)
#pragma unroll
      for (int r2 = 0; r2 < R2; ++r2) s[fft_pad(base + r1 * NS + r2 * NS * R1)] = v[(r1 * R2 + r2) * NG + g];
  }
  __syncthreads();
#pragma unroll
  for (int m = 0; m < kFftE; ++m) v[m] = s[fft_pad(tq + m * (N / kFftE))];
  __syncthreads();
}

// passes from span NS on; `st(m, p, value)`: output position p = (thread's q) + m N / 16
template <int LOGN, int NS, int DIR, class ST>
__device__ __forceinline__ void fft_passes(float2 (&v)[kFftE], int tq, float2 *s, const float2 *__restrict__ tw, ST st) {
  constexpr int N = 1 << LOGN, left = N / NS;
  // radix 2 first when log2 N is odd, then radix 4, two stages a pass
  constexpr int R1 = (NS == 1 && (LOGN & 1)) ? 2 : 4;
  constexpr int R2 = left / R1 >= 4 ? 4 : 1;
  constexpr int R = R1 * R2, NG = kFftE / R;
  fft_pass<LOGN, R1, R2, NS, DIR>(v, tq, tw);
  if constexpr (NS * R < N) {
    fft_exchange<LOGN, R1, R2, NS>(v, tq, s);
    fft_passes<LOGN, NS * R, DIR>(v, tq, s, tw, st);
  } else {   // NS = N / R: output (r1, r2) of group g sits at tq + (g + NG (r1 + R1 r2)) N / 16
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int r1 = 0; r1 < R1; ++r1)
#pragma unroll
        for (int r2 = 0; r2 < R2; ++r2) {
          const int m = g + NG * (r1 + R1 * r2);
          st(m, tq + m * (N / kFftE), v[(r1 * R2 + r2) * NG + g]);
        }
  }
}

// Transform of the 16 elements a thread holds (element m: position tq + m N / 16).
// Every thread of the block calls it (it synchronises); s: the transform's
// exchange buffer of FftCfg::LD elements.  DIR = -1 forward (exp(-2 pi i ...)),
// +1 inverse (unnormalised).
template <int LOGN, int DIR, class ST>
__device__ __forceinline__ void fft_run(float2 (&v)[kFftE], int tq, float2 *s, const float2 *__restrict__ tw, ST st) {
  fft_passes<LOGN, 1, DIR>(v, tq, s, tw, st);
}

// Launch shapes: C transforms of N / 16 threads a block.  Row passes: thread t is
// thread t mod (N / 16) of transform t / (N / 16).  Column passes: consecutive
// threads take consecutive columns (thread t: column t mod C), C = 4 columns for
// large grids (32-byte row segments, whole sectors) and 8 below.  Blocks of the
// small grids are kept small so that a grid of 128^2 still fills 16 blocks.
constexpr int fft_ld(int n, int mod16) {   // exchange buffer length congruent to mod16 mod 16
  int ld = n + n / 16 - 1;   // fft_pad(n - 1) + 1
  while (ld % 16 != mod16) ++ld;
  return ld;
}
template <int LOGN> struct RowCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int TN = N / kFftE;
  static constexpr int T = LOGN <= 7 ? 64 : (LOGN <= 9 ? 128 : 256);
  static constexpr int C = T / TN;
  static constexpr int LD = fft_ld(N, LOGN <= 5 ? 1 : 4);
  static constexpr size_t SMEM = size_t(C) * LD * sizeof(float2);
};
template <int LOGN> struct ColCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int TN = N / kFftE;
  static constexpr int C = LOGN <= 5 ? 32 : (LOGN <= 8 ? 8 : 4);
  static constexpr int T = C * TN;
  static constexpr int LD = fft_ld(N, C >= 16 ? 1 : 16 / C);
  static constexpr size_t SMEM = size_t(C) * LD * sizeof(float2);
};
// Batches: every grid size up to 1024^2 in blocks of 256 threads, so that one launch
// serves all of a batch's sizes.
constexpr int kBatchMaxLog = 10;
template <int LOGN> struct BatchRowCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int TN = N / kFftE;
  static constexpr int T = 256;
  static constexpr int C = T / TN;
  static constexpr int LD = fft_ld(N, LOGN <= 5 ? 1 : 4);
  static constexpr size_t SMEM = size_t(C) * LD * sizeof(float2);
};
template <int LOGN> struct BatchColCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int TN = N / kFftE;
  static constexpr int T = 256;
  static constexpr int C = T / TN;
  static constexpr int LD = fft_ld(N, C >= 16 ? 1 : 16 / C);
  static constexpr size_t SMEM = size_t(C) * LD * sizeof(float2);
};
// columns of the kernel build's boxes: many boxes, so wider row segments
template <int LOGN> struct BoxColCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int TN = N / kFftE;
  static constexpr int C = LOGN <= 8 ? 4096 / N : (LOGN <= 11 ? 8 : 4);
  static constexpr int T = C * TN;
  static constexpr int LD = fft_ld(N, C >= 16 ? 1 : 16 / C);
  static constexpr size_t SMEM = size_t(C) * LD * sizeof(float2);
};

// thread -> (transform of the block, thread of the transform): rows / columns
template <class Cfg> __device__ __forceinline__ void row_thread(int &c, int &tq) {
  c = int(threadIdx.x) / Cfg::TN;
  tq = int(threadIdx.x) % Cfg::TN;
}
template <class Cfg> __device__ __forceinline__ void col_thread(int &c, int &tq) {
  c = int(threadIdx.x) % Cfg::C;
  tq = int(threadIdx.x) / Cfg::C;
}

}  // namespace wproj
