// Per-bin arithmetic of the spectral solves (Sec. 3.1, Eq. 8-9) and of the
// packed column-0 bins, shared by the forward column pass and the adjoint's
// recomputation of a step.
#pragma once
#include "common.cuh"

namespace gfd {

// Bins (k, 0) and (k, N/2) of a real image's packed half spectrum, from the
// column-0 values Z[k] and Z[-k]: A = (Z[k] + conj Z[-k]) / 2,
// B = (Z[k] - conj Z[-k]) / (2i); and back, Z[k] = A + i B.
GFD_D void unpack_pair(float2 Sk, float2 Smk, float2& A, float2& Bv) {
  const float2 c = cconj(Smk);
  A = cscale(cadd(Sk, c), 0.5f);
  const float2 D = csub(Sk, c);
  Bv = make_float2(0.5f * D.y, -0.5f * D.x);  // D / (2i)
}
GFD_D float2 pack_pair(float2 A, float2 B) { return make_float2(A.x - B.y, A.y + B.x); }

// 1/d for d > 0: the hardware approximation and one residual step (almost
// always the correctly rounded quotient, as __frcp_rn, in three instructions).
GFD_D float rcp_refined(float d) {
  const float q = __fdividef(1.0f, d);
  return fmaf(fmaf(-d, q, 1.0f), q, q);
}

// Eq. 9 (u_p) and Eq. 8 (u_I) at one bin, lambda finite:
//   U_p = (conj(H) Y + lam U_E) / (|H|^2 + lam)
//   U_I = (conj(H) Y + lam D2 U_E) / (|H|^2 + lam D2),  D2 = |F(nabla)|^2.
GFD_D void solve_bin(float2 U, float2 H, float2 Y, float lam, float D2, float2& UI, float2& Up) {
  const float2 HY = __ffma2_rn(make_float2(H.x, H.x), Y, make_float2(H.y * Y.y, -H.y * Y.x));
  const float a = fmaf(H.x, H.x, H.y * H.y);
  Up = cscale(__ffma2_rn(make_float2(lam, lam), U, HY), rcp_refined(a + lam));
  const float lg = lam * D2;
  const float den = a + lg;
  const float2 v = cscale(__ffma2_rn(make_float2(lg, lg), U, HY), rcp_refined(den));
  UI = den > 0.0f ? v : U;
}

}  // namespace gfd
