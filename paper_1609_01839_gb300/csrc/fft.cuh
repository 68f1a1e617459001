// Power-of-two complex FFT on a team of threads, exchanged through shared memory.
//
// The transform X[k] = sum_n x[n] W_L^{nk}, W_L = exp(-2 pi i / L) (forward)
// or with W_L^{-nk} (inverse, unnormalised), is computed by the mixed-radix
// decimation-in-frequency recursion L = r_0 * L_1:
//   X[i + r_0 k1] = sum_{n1} W_{L_1}^{n1 k1} [ W_L^{n1 i} sum_{n2} x[n1 + L_1 n2] W_{r_0}^{n2 i} ].
// Stage s holds prod_{s'<s} r_{s'} independent sub-transforms of length L_s,
// stored contiguously; butterfly (g, jj) takes the r_s elements
// g*L_s + jj + i*L_{s+1}, applies a radix-r_s DFT in registers and the twiddle
// W_{L_s}^{jj i}, and puts them back in place.
//
// A team has T = L/E threads with E elements each.  The first stage takes its
// inputs from registers (the caller loads element n = beta + i*L_1 of
// butterfly beta straight from global memory: consecutive threads, consecutive
// n), and the last stage leaves its outputs in registers: it walks its groups
// in the order of their output index kappa (d_0 fastest), so that butterfly
// kappa yields X[kappa + (L/r) i] and consecutive threads hold consecutive
// k, ready to be stored to global memory.  A transform of two (three) stages
// thus passes through shared memory once (twice), with one (two) barriers.
//
// Three kinds differ in where a thread must hold mirrored elements:
//   FK_COL  complex columns: the last stage has one butterfly of E outputs;
//   FK_C2R  inverse rows: the first stage's butterflies come in mirrored
//           pairs (beta, L_1 - beta), which hold n and L - n of all their
//           elements, so the split of the packed row spectrum needs no exchange;
//   FK_R2C  forward rows: likewise (kappa, L/r - kappa) in the last stage.
// Shared positions are padded (P1 elements per L_1, P2 per L_2) so that every
// access of 16 consecutive threads falls on distinct 8-byte banks (FK_R2C: 1.5
// passes on average; the mirrored order and the two orders before it leave no
// padding that is conflict-free for all three).
#pragma once
#include "common.cuh"

namespace gfd {

enum FftKind { FK_COL = 0, FK_C2R = 1, FK_R2C = 2 };

// Elements per thread.
constexpr int fft_elems(int K, int L) {
  if (K == FK_COL) return L >= 256 ? 16 : (L >= 64 ? 8 : (L >= 16 ? 4 : 2));
  return L >= 64 ? 16 : (L >= 16 ? 8 : 4);
}

// Radix of stage s (1 past the last stage).
constexpr int fft_radix(int K, int L, int s) {
  struct Row {
    int L, r[3];
  };
  constexpr Row col[] = {{8, {2, 2, 2}},    {16, {4, 4, 1}},   {32, {2, 4, 4}},  {64, {8, 8, 1}},
                         {128, {4, 4, 8}},  {256, {16, 16, 1}}, {512, {4, 8, 16}}, {1024, {4, 16, 16}},
                         {2048, {8, 16, 16}}, {4096, {16, 16, 16}}};
  constexpr Row c2r[] = {{4, {2, 2, 1}},   {8, {2, 4, 1}},    {16, {4, 4, 1}},   {32, {4, 8, 1}},
                         {64, {8, 8, 1}},  {128, {8, 16, 1}}, {256, {4, 4, 16}}, {512, {4, 8, 16}},
                         {1024, {8, 8, 16}}, {2048, {8, 16, 16}}};
  constexpr Row r2c[] = {{4, {2, 2, 1}},   {8, {4, 2, 1}},    {16, {4, 4, 1}},  {32, {8, 4, 1}},
                         {64, {8, 8, 1}},  {128, {16, 8, 1}}, {256, {8, 4, 8}}, {512, {8, 8, 8}},
                         {1024, {8, 16, 8}}, {2048, {16, 16, 8}}};
  for (int i = 0; i < 10; ++i) {
    const Row& q = K == FK_COL ? col[i] : (K == FK_C2R ? c2r[i] : r2c[i]);
    if (q.L == L) return s < 3 ? q.r[s] : 1;
  }
  return 1;
}
constexpr int fft_stages(int K, int L) { return fft_radix(K, L, 2) > 1 ? 3 : 2; }
// L_s: length of the sub-transforms of stage s.
constexpr int fft_len(int K, int L, int s) {
  int n = L;
  for (int i = 0; i < s; ++i) n /= fft_radix(K, L, i);
  return n;
}
// Pad elements per L_1 and per L_2 positions.
constexpr int fft_pad1(int K, int L) {
  if (K == FK_COL) return L == 32 ? 0 : 1;
  if (K == FK_C2R) return L <= 4 || L == 256 ? 0 : (L == 512 ? 4 : (L >= 1024 ? 2 : 1));
  return L <= 4 ? 0 : (L == 512 ? 7 : (L >= 1024 ? 5 : 1));
}
constexpr int fft_pad2(int K, int L) {
  if (K == FK_COL) return L == 32 ? 1 : 0;
  return K == FK_C2R && L >= 256 ? 1 : 0;
}

template <int K, int L>
struct FftGeo {
  static constexpr int E = fft_elems(K, L), T = L / E, S = fft_stages(K, L);
  static constexpr int L1 = fft_len(K, L, 1), L2 = S == 3 ? fft_len(K, L, 2) : 1;
  static constexpr int P1 = fft_pad1(K, L), P2 = S == 3 ? fft_pad2(K, L) : 0;
  static constexpr int RF = fft_radix(K, L, 0), RL = fft_radix(K, L, S - 1);
  static constexpr int KL = L / RL;  // butterflies of the last stage
  // padded distances of the elements of a butterfly of stage 0 and of stage 1
  static constexpr int STEP0 = L1 + P1 + (S == 3 ? (L1 / L2) * P2 : 0);
  static constexpr int STEP1 = L2 + P2;  // S == 3
  static constexpr int MIN_SIZE = (RF - 1) * STEP0 + L1 + (S == 3 ? (L1 / L2 - 1) * P2 : 0);
  // float2 elements of one transform's buffer; rows shorter than 256 carry a
  // skew that keeps the teams of a warp on different banks
  static constexpr int SIZE =
      K == FK_COL ? MIN_SIZE
                  : (L == 4 ? 5
                            : (L == 8 ? (K == FK_C2R ? 10 : 14)
                                      : (L == 16 ? 22
                                                 : (L == 32 ? (K == FK_C2R ? 36 : 44)
                                                            : (L == 64 ? 76
                                                                       : (L == 128 ? (K == FK_C2R ? 136 : 152)
                                                                                   : MIN_SIZE))))));
};

// cos / sin of 2 pi m / 16
__device__ constexpr float kCos16[16] = {
    1.0f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
    0.0f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
    -1.0f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f,
    0.0f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f};
__device__ constexpr float kSin16[16] = {
    0.0f, 0.38268343236508977f, 0.70710678118654752f, 0.92387953251128674f,
    1.0f, 0.92387953251128674f, 0.70710678118654752f, 0.38268343236508977f,
    0.0f, -0.38268343236508977f, -0.70710678118654752f, -0.92387953251128674f,
    -1.0f, -0.92387953251128674f, -0.70710678118654752f, -0.38268343236508977f};

// The rounding residuals of kCos16 / kSin16 (value minus its float), so that
// hi + lo carries cos and sin to about 48 bits.  With the floats alone every
// non-trivial constant twiddle has |w| < 1 (all six round towards zero), and
// a transform shrinks every output by ~7e-8 of its magnitude: a bias, not a
// random error, which sums of squares of spectra (the residual of Eq. 10-11)
// inherit in full.
constexpr float kC1 = 2.830748968563057e-08f;   // cos(pi/8) residual
constexpr float kS1 = 6.2233507236442165e-09f;  // sin(pi/8) residual
constexpr float kC2 = 1.2101617485882343e-08f;  // cos(pi/4) residual
__device__ constexpr float kCos16Lo[16] = {0.0f, kC1,  kC2,  kS1,  0.0f, -kS1, -kC2, -kC1,
                                           0.0f, -kC1, -kC2, -kS1, 0.0f, kS1,  kC2,  kC1};
__device__ constexpr float kSin16Lo[16] = {0.0f, kS1,  kC2,  kC1,  0.0f, kC1,  kC2,  kS1,
                                           0.0f, -kS1, -kC2, -kC1, 0.0f, -kC1, -kC2, -kS1};

// v * W_R^k (forward: exp(-2 pi i k/R); inverse: exp(+2 pi i k/R)), R <= 16.
// The product uses the constants' residuals (two more FMAs per component), so
// it is the exact product up to roundings of either sign.
template <int R, int k, bool INV>
GFD_D float2 const_twiddle(float2 v) {
  if constexpr (k == 0) {
    return v;
  } else if constexpr (4 * k == R) {
    return cmul_mi<INV>(v);
  } else {
    constexpr int m = k * (16 / R);
    const float c = kCos16[m], cl = kCos16Lo[m];
    const float s = INV ? kSin16[m] : -kSin16[m];
    const float sl = INV ? kSin16Lo[m] : -kSin16Lo[m];
    const float2 vx = make_float2(v.x, v.x), vy = make_float2(v.y, v.y);
    return __ffma2_rn(vx, make_float2(c, s),
                      __ffma2_rn(vy, make_float2(-s, c),
                                 __ffma2_rn(vx, make_float2(cl, sl),
                                            __fmul2_rn(vy, make_float2(-sl, cl)))));
  }
}

// In-register DFT of length R (natural-order input and output).
template <int R, bool INV>
struct DFT {
  template <int k>
  GFD_D static void combine(float2* x, const float2* e, const float2* o) {
    if constexpr (k < R / 2) {
      const float2 t = const_twiddle<R, k, INV>(o[k]);
      x[k] = cadd(e[k], t);
      x[k + R / 2] = csub(e[k], t);
      combine<k + 1>(x, e, o);
    }
  }
  GFD_D static void run(float2* x) {
    float2 e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
      e[i] = x[2 * i];
      o[i] = x[2 * i + 1];
    }
    DFT<R / 2, INV>::run(e);
    DFT<R / 2, INV>::run(o);
    combine<0>(x, e, o);
  }
};
template <bool INV>
struct DFT<1, INV> {
  GFD_D static void run(float2*) {}
};
template <bool INV>
struct DFT<2, INV> {
  GFD_D static void run(float2* x) {
    const float2 a = x[0], b = x[1];
    x[0] = cadd(a, b);
    x[1] = csub(a, b);
  }
};

// W_{Ls}^m from the per-length tables (tw: all lengths, see tab_off).
template <bool INV>
GFD_D float2 twiddle(const float2* __restrict__ tw, int Ls, int m) {
  float2 w = __ldg(&tw[tab_off(Ls) + m]);
  if (INV) w.y = -w.y;
  return w;
}

// First stage, butterfly beta: x holds its inputs; results go to buf.
template <int K, int L, bool INV>
GFD_D void fft_first(float2 (&x)[FftGeo<K, L>::RF], int beta, float2* buf,
                     const float2* __restrict__ tw) {
  using G = FftGeo<K, L>;
  DFT<G::RF, INV>::run(x);
  float2* o = buf + (beta + (G::S == 3 ? (beta / G::L2) * G::P2 : 0));
  o[0] = x[0];
#pragma unroll
  for (int i = 1; i < G::RF; ++i)
    o[i * G::STEP0] = cmul(x[i], twiddle<INV>(tw, L, beta * i));
}

// Middle stage (three-stage transforms), thread j of the team, in place.
template <int K, int L, bool INV>
GFD_D void fft_mid(float2* buf, int j, const float2* __restrict__ tw) {
  using G = FftGeo<K, L>;
  if constexpr (G::S == 3) {
    constexpr int r = fft_radix(K, L, 1), NB = G::E / r;
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int beta = j + G::T * q;
      const int g = beta / G::L2, jj = beta % G::L2;
      float2* o = buf + (g * G::STEP0 + jj);
      float2 x[r];
#pragma unroll
      for (int i = 0; i < r; ++i) x[i] = o[i * G::STEP1];
      DFT<r, INV>::run(x);
      o[0] = x[0];
#pragma unroll
      for (int i = 1; i < r; ++i)
        o[i * G::STEP1] = cmul(x[i], twiddle<INV>(tw, G::L1, jj * i));
    }
  }
}

// Last stage, butterfly kappa: x[i] = X[kappa + KL * i].
template <int K, int L, bool INV>
GFD_D void fft_last(float2 (&x)[FftGeo<K, L>::RL], int kappa, const float2* buf) {
  using G = FftGeo<K, L>;
  int p;
  if constexpr (G::S == 3)
    p = (kappa % G::RF) * G::STEP0 + (kappa / G::RF) * G::STEP1;
  else
    p = kappa * G::STEP0;
  const float2* in = buf + p;
#pragma unroll
  for (int i = 0; i < G::RL; ++i) x[i] = in[i];
  DFT<G::RL, INV>::run(x);
}

// ---------------------------------------------------------------------------
// Short transforms of few columns (column passes of small problems): 4 elements
// per thread, radix 4 with a last radix-2 stage where log2 M is odd, lengths at
// run time.  A lone 256 x 256 image leaves the chip idle, so what counts is one
// warp's path: its instruction count (a radix-16 pass runs some 2000 a thread,
// this about 400) and its code, which is fetched anew by every launch.
// ---------------------------------------------------------------------------
GFD_HD int short_pos(int p) { return p + (p >> 3); }

// Position of output group kappa of `bits` index bits (an even number): base-4
// digits reversed.
GFD_D int rev4(int kappa, int bits) {
  if (bits == 0) return 0;
  const unsigned r = __brev((unsigned)kappa) >> (32 - bits);
  return (int)(((r & 0x55555555u) << 1) | ((r >> 1) & 0x55555555u));
}

// One butterfly of a stage of length Ls with its twiddles, offset jj.
template <bool INV>
GFD_D void short_butterfly(float2 (&x)[4], int Ls, int jj, const float2* __restrict__ tw) {
  DFT<4, INV>::run(x);
#pragma unroll
  for (int i = 1; i < 4; ++i) x[i] = cmul(x[i], twiddle<INV>(tw, Ls, jj * i));
}

// NS transforms of length M = 2^lg >= 8 side by side: x[n][i] = element j + i M/4
// on entry, X[j + i M/4] on return (thread j of M/4).  buf[n]: their buffers.
// Contains block barriers; the buffers must be free on entry.
template <int NS, bool INV>
GFD_D void short_fft(float2 (&x)[NS][4], float2* const (&buf)[NS], int lg, int j,
                     const float2* __restrict__ tw) {
  int Ln = 1 << (lg - 2), Ls = 4 * Ln;
#pragma unroll
  for (int n = 0; n < NS; ++n) {
    short_butterfly<INV>(x[n], Ls, j, tw);
#pragma unroll
    for (int i = 0; i < 4; ++i) buf[n][short_pos(j + i * Ln)] = x[n][i];
  }
  Ls = Ln;
#pragma unroll 1
  while (Ls > 4) {
    __syncthreads();
    Ln = Ls >> 2;
    const int jj = j & (Ln - 1), base = ((j - jj) << 2) + jj;
#pragma unroll
    for (int n = 0; n < NS; ++n) {
#pragma unroll
      for (int i = 0; i < 4; ++i) x[n][i] = buf[n][short_pos(base + i * Ln)];
      short_butterfly<INV>(x[n], Ls, jj, tw);
#pragma unroll
      for (int i = 0; i < 4; ++i) buf[n][short_pos(base + i * Ln)] = x[n][i];
    }
    Ls = Ln;
  }
  __syncthreads();
  if (Ls == 4) {
    const int base = rev4(j, lg - 2) * 4;
#pragma unroll
    for (int n = 0; n < NS; ++n) {
#pragma unroll
      for (int i = 0; i < 4; ++i) x[n][i] = buf[n][short_pos(base + i)];
      DFT<4, INV>::run(x[n]);
    }
  } else {  // two radix-2 butterflies: kappa = j and j + M/4
    const int b0 = rev4(j, lg - 1) * 2, b1 = rev4(j + (1 << (lg - 2)), lg - 1) * 2;
#pragma unroll
    for (int n = 0; n < NS; ++n) {
      const float2 a0 = buf[n][short_pos(b0)], a1 = buf[n][short_pos(b0 + 1)];
      const float2 c0 = buf[n][short_pos(b1)], c1 = buf[n][short_pos(b1 + 1)];
      x[n][0] = cadd(a0, a1);
      x[n][2] = csub(a0, a1);
      x[n][1] = cadd(c0, c1);
      x[n][3] = csub(c0, c1);
    }
  }
}

// Buffer stride of the B columns of a column pass, whose consecutive threads
// walk B columns x 16/B consecutive elements: 16/B (mod 16) puts them on
// distinct banks.
template <int M>
GFD_HD int col_stride(int B) {
  const int want = B < 16 ? 16 / B : 1, n = FftGeo<FK_COL, M>::SIZE;
  return n + ((want - n) & 15);
}

}  // namespace gfd
