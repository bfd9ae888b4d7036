// Data shared between the kernel-build pipeline and its FFT passes.
#pragma once

#include "common.cuh"

namespace wproj {

// A batch of nb kernel boxes of side S being built.
struct BoxBatch {
  int S = 0;
  int nb = 0;
  const float2 *Au = nullptr;     // [nb][S] per-axis factor: KB tap polynomial x e^{2 pi i w l^2 / 2}
  const float2 *Av = nullptr;     // [nb][S]
  const int8_t *mode = nullptr;   // [nb] 0: separable phase only; 1: + FP32 remainder; 2: FP64 phase
  const float *wf = nullptr;      // [nb] w as float (remainder term)
  const double *wd = nullptr;     // [nb] w (FP64 phase path)
  const float *lsq = nullptr;     // [S] l_P^2 (float)
  const float *gtab = nullptr;    // [S][S] g(l_P^2 + l_Q^2), g(x) = x^2 / (2 (1 + n)^2) (exact chirp)
  const double *lcoord = nullptr; // [S] l_P (after clamping)
  float2 *K = nullptr;            // [nb][S][S] kernel values, natural order (offset s at s mod S)
  // direction-dependent screens (S = G): screens[bsid[b]] multiplies box b's samples;
  // screen index a holds offset a - S/2 (centred), the box sample P offset P or P - S
  const float2 *screens = nullptr;
  const int32_t *bsid = nullptr;
};

// f[P][Q] = Au[P] Av[Q] e^{2 pi i w g(x)}: the chirp (Eq. 4 / Eq. 5) times the KB
// tap polynomial, at box offsets P' = P (P < S/2) or P - S; Au, Av carry the
// separable part of the phase, w (l^2 + m^2) / 2, and the taps.
__device__ __forceinline__ float2 box_value(const BoxBatch &bb, int b, int P, int Q) {
  const float2 a = bb.Au[int64_t(b) * bb.S + P];
  const float2 c = bb.Av[int64_t(b) * bb.S + Q];
  float2 f = cmul(a, c);
  const int mode = bb.mode[b];
  if (mode == 1) {
    // exact chirp: phase w (1 - n) = w x / 2 + w g(x), g = x^2 / (2 (1 + n)^2), the
    // remainder |w g| <= 1/4 cycle so FP32 keeps it to ~1e-7 cycles; g does not
    // depend on the box and comes from a table of the class (k_g_table)
    float sn, cs;
    sincospif(2.f * (bb.wf[b] * __ldg(bb.gtab + int64_t(P) * bb.S + Q)), &sn, &cs);
    f = cmul(f, make_float2(cs, sn));
  } else if (mode == 2) {
    // large w: the full phase argument in FP64, reduced mod 1
    const double l = bb.lcoord[P], m = bb.lcoord[Q];
    const double x = l * l + m * m;
    const double ph = bb.wd[b] * x / (1.0 + sqrt(1.0 - x));
    const double fr = ph - floor(ph);
    float sn, cs;
    sincospif(2.f * float(fr), &sn, &cs);
    f = cmul(f, make_float2(cs, sn));
  }
  if (bb.screens) {
    const int S = bb.S, h = S / 2;
    const float2 a = bb.screens[(int64_t(bb.bsid[b]) * S + ((P + h) & (S - 1))) * S + ((Q + h) & (S - 1))];
    f = cmul(f, a);
  }
  return f;
}

}  // namespace wproj
