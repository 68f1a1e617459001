// Reverse mode of the unrolled method: gradients of a loss of u^K with
// respect to the observation y, the PSF h and the guided filter's eps.
//
// One backward step undoes one iteration (Sec. 3.1 Steps 1-2), in reverse
// order of the forward step, from its checkpoint u_E^k and the forward
// solve's lambda_k:
//   recompute: U_E = DFT(u_E^k), U_I and U_p by Eq. 8-9, u_I and u_p by the
//     inverse DFT;
//   guided filter (Eq. 3-5; periodic windows, so the box mean is its own
//   adjoint): three tiled passes of compensated window sums
//     1. mu, pbar, sigma^2 + eps, a from (u_I, u_p)
//     2. window sums of a, g_u u_I, g_u -> the pointwise adjoints of Eq. 5, 4, 3
//     3. window sums of those adjoints -> g_uI, g_up
//   DFT of g_uI, g_up; the spectral solves (Eq. 8-9) per bin, with lambda's
//   adjoint summed over the bins; the implicit derivative of lambda through
//   Eq. 11 (dlambda = -(df - dT) / f'(lambda)) as a second per-bin pass; the
//   adjoint DFT back to g_uE = g_u of the previous step.
// H = DFT(embedded h), Y = DFT(y) and T (Eq. 12) collect their gradients over
// the steps; the last kernels map them to g_h, g_y.  Where lambda = inf the
// step is u_I = u_p = u_E and lambda is a constant.
//
// Arithmetic: FP32 per pixel and per bin, as in the forward step; the window
// sums carry their rounding errors (a running FP32 sum plus the exact error of
// every addition and product, summed apart), and the statistics that cancel
// (sigma^2, the covariance, box(g_u I) - mu box(g_u), the combinations of
// pass 3) are formed from them in double-float; sums over all bins or pixels
// are FP64.  No FP64 arithmetic per pixel: this part's FP64 rate is a small
// fraction of its FP32 rate.
//
// Spectra are the library's packed half spectra, row-major (tile width N/2):
// Z[m][l] = X(m, l) for 1 <= l < N/2 and Z[m][0] = X(m, 0) + i X(m, N/2).
// Complex gradients follow g_z = dL/dRe z + i dL/dIm z; a sum over all bins
// counts the interior columns twice (each stands for its mirror bin too).
#include "common.cuh"
#include "df.cuh"
#include "launch.h"
#include "spectral.cuh"

namespace gfd {

constexpr int ADJ_TX = 32, ADJ_TY = 16;   // output pixels of a block
constexpr int ADJ_THREADS = 256;
constexpr int ADJ_ROW = 4, ADJ_COL = 2;   // outputs per thread along a row, down a column

// Compensated sums of two quantities, packed: hi the FP32 running sums, lo the
// sums of the exact rounding errors of their additions (and of the low parts of
// added double-float terms).  hi + lo carries about 2^-48 relative error per
// term; taking a term away again is one more addition.
struct CSum2 {
  float2 hi, lo;
};
GFD_D void csum_add(CSum2& s, float2 v, float2 vlo) {
  const float2 t = cadd(s.hi, v), bb = csub(t, s.hi);
  const float2 e = cadd(csub(s.hi, csub(t, bb)), csub(v, bb));
  s.hi = t;
  s.lo = cadd(s.lo, cadd(e, vlo));
}
GFD_D df val_df(float v) { return df{v, 0.0f}; }

// One compensated FP32 sum (a thread's share of a sum over bins or pixels).
struct CSum {
  float hi = 0.0f, lo = 0.0f;
  GFD_D void add(float v) {
    const df t = two_sum(hi, v);
    hi = t.hi;
    lo += t.lo;
  }
  GFD_D void add(df v) {
    const df t = two_sum(hi, v.hi);
    hi = t.hi;
    lo += t.lo + v.lo;
  }
  GFD_D double get() const { return (double)hi + (double)lo; }
};

// ---------------------------------------------------------------------------
// Tiled window sums: OP stages NS planes of a TX x TY tile plus an r halo in
// shared memory, maps every staged pixel to NQ double-float quantities, and
// gets their compensated window sums (periodic windows) at each output pixel:
// along the tile's rows into shared memory (four outputs per thread, slid), then
// down its columns (two, slid).  Bound by FP32 instructions: a term is one
// compensated addition per quantity, 3.3 along a row and 4.5 down a column per
// output at r = 3 (7 and 7 with a sum of its own per output, in 16 x 16 tiles).
// 16 images of 512^2, w = 7: 128, 122, 136 us for the three passes so, 78, 91, 91 us now.
// ---------------------------------------------------------------------------
template <class OP>
__global__ void __launch_bounds__(ADJ_THREADS)
k_adj_box(const AdjDesc* __restrict__ descs, int M, int N, int rad) {
  extern __shared__ __align__(16) unsigned char adj_sm[];
  constexpr int NS = OP::NS, NQ = OP::NQ, NP = (NQ + 1) / 2;  // NP pairs
  const AdjDesc& d = descs[blockIdx.z];
  const int EX = ADJ_TX + 2 * rad, EY = ADJ_TY + 2 * rad;
  // consecutive threads of the row sums take consecutive rows: odd pitches keep
  // them on different banks
  constexpr int RP = ADJ_TX + 1;
  const int TP = EX | 1;
  float4* rows = reinterpret_cast<float4*>(adj_sm);                   // [NP][EY][RP]: hi, lo
  float* tile = reinterpret_cast<float*>(rows + (size_t)NP * EY * RP);  // [NS][EY][TP]
  const int x0 = blockIdx.x * ADJ_TX, y0 = blockIdx.y * ADJ_TY;
  for (int e = threadIdx.x; e < EY * EX; e += blockDim.x) {
    const int ty = e / EX, tx = e - ty * EX;
    const size_t off = (size_t)((y0 - rad + ty) & (M - 1)) * N + ((x0 - rad + tx) & (N - 1));
#pragma unroll
    for (int c = 0; c < NS; ++c) tile[(c * EY + ty) * TP + tx] = __ldg(&OP::plane(d, c)[off]);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < EY * (ADJ_TX / ADJ_ROW); e += blockDim.x) {
    const int ty = e % EY, tx = (e / EY) * ADJ_ROW;
    CSum2 s[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) s[q].hi = s[q].lo = make_float2(0.0f, 0.0f);
    auto term = [&](int dx, float sg) {
      float v[NS];
#pragma unroll
      for (int c = 0; c < NS; ++c) v[c] = tile[(c * EY + ty) * TP + tx + dx];
      df q[2 * NP];
      q[2 * NP - 1] = val_df(0.0f);
      OP::quantities(v, q);
#pragma unroll
      for (int k = 0; k < NP; ++k)
        csum_add(s[k], make_float2(sg * q[2 * k].hi, sg * q[2 * k + 1].hi),
                 make_float2(sg * q[2 * k].lo, sg * q[2 * k + 1].lo));
    };
#pragma unroll 1
    for (int dx = 0; dx < 2 * rad; ++dx) term(dx, 1.0f);
#pragma unroll
    for (int k = 0; k < ADJ_ROW; ++k) {
      term(k + 2 * rad, 1.0f);
#pragma unroll
      for (int q = 0; q < NP; ++q)
        rows[(q * EY + ty) * RP + tx + k] =
            make_float4(s[q].hi.x, s[q].hi.y, s[q].lo.x, s[q].lo.y);
      if (k + 1 < ADJ_ROW) term(k, -1.0f);
    }
  }
  __syncthreads();
  const int tx = threadIdx.x % ADJ_TX, ty0 = (threadIdx.x / ADJ_TX) * ADJ_COL;
  CSum2 S[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) S[q].hi = S[q].lo = make_float2(0.0f, 0.0f);
  auto row = [&](int ty, float sg) {
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const float4 v = rows[(q * EY + ty) * RP + tx];
      csum_add(S[q], make_float2(sg * v.x, sg * v.y), make_float2(sg * v.z, sg * v.w));
    }
  };
#pragma unroll 1
  for (int dy = 0; dy < 2 * rad; ++dy) row(ty0 + dy, 1.0f);
  const float n = (float)((2 * rad + 1) * (2 * rad + 1));
  float eps_part = 0.0f;
#pragma unroll
  for (int k = 0; k < ADJ_COL; ++k) {
    const int gy = y0 + ty0 + k, gx = x0 + tx;
    row(ty0 + k + 2 * rad, 1.0f);
    df W[2 * NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {  // window sums (|lo| <= |hi| in practice)
      W[2 * q] = quick_two_sum(S[q].hi.x, S[q].lo.x);
      W[2 * q + 1] = quick_two_sum(S[q].hi.y, S[q].lo.y);
    }
    if (gy < M && gx < N) eps_part += OP::output(d, (size_t)gy * N + gx, W, n);
    if (k + 1 < ADJ_COL) row(ty0 + k, -1.0f);
  }
  if (OP::kEps) {  // sum of the pass's eps adjoint over the block (FP64), one atomic
    __shared__ double red[ADJ_THREADS / 32];
    double v = eps_part;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < ADJ_THREADS / 32; ++w) t += red[w];
      atomicAdd(d.g_eps, t);
    }
  }
}

GFD_D float df_float(df a) { return a.hi + a.lo; }

// Pass 1: mu = box(I), pbar = box(p), sigma^2 + eps, a (Eq. 3), with
// sigma^2 = (n S_II - S_I^2) / n^2 and cov = (n S_Ip - S_I S_p) / n^2.
struct AdjStats {
  static constexpr int NS = 2, NQ = 4;
  static constexpr bool kEps = false;
  GFD_D static const float* plane(const AdjDesc& d, int c) { return c == 0 ? d.uI : d.up; }
  GFD_D static void quantities(const float (&v)[NS], df* q) {
    q[0] = val_df(v[0]);
    q[1] = val_df(v[1]);
    q[2] = two_prod(v[0], v[1]);
    q[3] = two_prod(v[0], v[0]);
  }
  GFD_D static float output(const AdjDesc& d, size_t o, const df* S, float n) {
    const float inv_n = 1.0f / n, inv2 = inv_n * inv_n;
    const float mu = df_float(S[0]) * inv_n, pb = df_float(S[1]) * inv_n;
    const float var = df_float(df_sub(df_mul_f(S[3], n), df_mul(S[0], S[0]))) * inv2;
    const float cov = df_float(df_sub(df_mul_f(S[2], n), df_mul(S[0], S[1]))) * inv2;
    const float ve = var + (float)d.eps;  // sigma_k^2 + eps
    d.A[o] = cov / ve;
    d.MU[o] = mu;
    d.PB[o] = pb;
    d.VE[o] = ve;
    return 0.0f;
  }
};

// Pass 2: abar, box(g_u I), box(g_u) -> adjoints of Eq. 5 (u = abar I + bbar),
// Eq. 4 (b = pbar - a mu) and Eq. 3 (a = cov / (var + eps)), and eps's.
struct AdjPoint {
  static constexpr int NS = 3, NQ = 3;
  static constexpr bool kEps = true;
  GFD_D static const float* plane(const AdjDesc& d, int c) {
    return c == 0 ? d.A : (c == 1 ? d.gu : d.uI);
  }
  GFD_D static void quantities(const float (&v)[NS], df* q) {
    q[0] = val_df(v[0]);
    q[1] = two_prod(v[1], v[2]);
    q[2] = val_df(v[1]);
  }
  GFD_D static float output(const AdjDesc& d, size_t o, const df* S, float n) {
    const float inv_n = 1.0f / n;
    const float a = d.A[o], mu = d.MU[o], pb = d.PB[o], ve = d.VE[o];
    const float abar = df_float(S[0]) * inv_n, g_b = df_float(S[2]) * inv_n;
    const float gI0 = d.gu[o] * abar;                                       // u = abar I + bbar
    const float g_a = df_float(df_sub(S[1], df_mul_f(S[2], mu))) * inv_n;  // b = pbar - a mu
    const float iv = 1.0f / ve;
    const float g_cov = g_a * iv, g_var = -g_a * a * iv;                   // a = cov / (var + eps)
    // cov = m_Ip - mu pbar, var = m_II - mu^2
    const float g_mu = -a * g_b - pb * g_cov - 2.0f * mu * g_var;
    const float g_pb = g_b - mu * g_cov;
    d.GI0[o] = gI0;
    d.GCOV[o] = g_cov;
    d.GVAR[o] = g_var;
    d.GMU[o] = g_mu;
    d.GPB[o] = g_pb;
    return g_var;  // d(var + eps)/d eps = 1
  }
};

// Pass 3: window sums of the Eq. 3-4 adjoints -> g_uI, g_up.
struct AdjInputs {
  static constexpr int NS = 4, NQ = 4;
  static constexpr bool kEps = false;
  GFD_D static const float* plane(const AdjDesc& d, int c) {
    return c == 0 ? d.GCOV : (c == 1 ? d.GVAR : (c == 2 ? d.GMU : d.GPB));
  }
  GFD_D static void quantities(const float (&v)[NS], df* q) {
#pragma unroll
    for (int k = 0; k < NQ; ++k) q[k] = val_df(v[k]);
  }
  GFD_D static float output(const AdjDesc& d, size_t o, const df* S, float n) {
    const float inv_n = 1.0f / n;
    const float I = d.uI[o], p = d.up[o];
    // m_Ip, m_II and mu terms: p box(g_cov) + 2 I box(g_var) + box(g_mu)
    const df tI = df_add(df_add(df_mul_f(S[0], p), df_mul_f(S[1], 2.0f * I)), S[2]);
    const df tp = df_add(df_mul_f(S[0], I), S[3]);  // m_Ip and pbar terms
    d.guI[o] = d.GI0[o] + df_float(tI) * inv_n;
    d.gup[o] = df_float(tp) * inv_n;
    return 0.0f;
  }
};

template <class OP>
static size_t adj_box_smem(int rad) {
  const size_t EX = ADJ_TX + 2 * rad, EY = ADJ_TY + 2 * rad;
  return (OP::NQ + 1) / 2 * EY * (ADJ_TX + 1) * sizeof(float4) +
         OP::NS * EY * (EX | 1) * sizeof(float);
}

template <class OP>
static cudaError_t launch_adj_box(const AdjDesc* descs, int n, int M, int N, int rad,
                                  cudaStream_t s) {
  const dim3 grid((N + ADJ_TX - 1) / ADJ_TX, (M + ADJ_TY - 1) / ADJ_TY, n);
  k_adj_box<OP><<<grid, ADJ_THREADS, adj_box_smem<OP>(rad), s>>>(descs, M, N, rad);
  return cudaGetLastError();
}

cudaError_t launch_adj_guided_filter(const AdjDesc* descs, int n, int M, int N, int rad,
                                     cudaStream_t s) {
  cudaError_t e = launch_adj_box<AdjStats>(descs, n, M, N, rad, s);
  if (e == cudaSuccess) e = launch_adj_box<AdjPoint>(descs, n, M, N, rad, s);
  if (e == cudaSuccess) e = launch_adj_box<AdjInputs>(descs, n, M, N, rad, s);
  return e;
}

// ---------------------------------------------------------------------------
// Recomputation of a step's spectra
// ---------------------------------------------------------------------------

// lambda_k of the forward solve becomes the step's lambda.
__global__ void k_adj_set_lambda(const AdjDesc* __restrict__ descs, int n, int k) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) *descs[i].lam = descs[i].lam_hist[k];
}

// U_I, U_p of the step (Eq. 8-9 with the forward's FP32 lambda) into UI, Up.
__global__ void k_adj_solve(const AdjDesc* __restrict__ descs, int M, int N,
                            const float* __restrict__ d2tab) {
  const AdjDesc& d = descs[blockIdx.y];
  const double lamd = __ldcg(d.lam);
  const bool branch = !(lamd < 1e300);
  const float lam = branch ? 0.0f : (float)lamd;
  const int L = N / 2, lg = __ffs(L) - 1;  // powers of two
  const int total = M * L;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += gridDim.x * blockDim.x) {
    const int k = idx >> lg, l = idx & (L - 1);
    const float d2r = __ldg(&d2tab[tab_off(M) + k]);
    float2 UI, Up;
    if (branch) {  // lambda = inf: u_I = u_p = u_E (Sec. 3.2)
      UI = Up = d.UE[idx];
    } else if (l != 0) {
      solve_bin(d.UE[idx], d.H[idx], d.Y[idx], lam, d2r + __ldg(&d2tab[tab_off(N) + l]), UI, Up);
    } else {
      const size_t m = (size_t)((M - k) & (M - 1)) * L;
      float2 EA, EB, HA, HB, YA, YB, IA, IB, PA, PB;
      unpack_pair(d.UE[idx], d.UE[m], EA, EB);
      unpack_pair(d.H[idx], d.H[m], HA, HB);
      unpack_pair(d.Y[idx], d.Y[m], YA, YB);
      solve_bin(EA, HA, YA, lam, d2r, IA, PA);
      solve_bin(EB, HB, YB, lam, d2r + 4.0f, IB, PB);
      UI = pack_pair(IA, IB);
      Up = pack_pair(PA, PB);
    }
    d.UI[idx] = UI;
    d.Up[idx] = Up;
  }
}

static int spec_chunks(int M, int N) {
  const size_t total = (size_t)M * (N / 2);
  int chunks = (int)((total + 256 * 8 - 1) / (256 * 8));
  return chunks > 256 ? 256 : chunks;
}

cudaError_t launch_adj_recompute(const AdjDesc* descs, int n, int M, int N, int k,
                                 const float* d2tab, cudaStream_t s) {
  k_adj_set_lambda<<<(n + 63) / 64, 64, 0, s>>>(descs, n, k);
  k_adj_solve<<<dim3(spec_chunks(M, N), n), 256, 0, s>>>(descs, M, N, d2tab);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Spectral adjoint
// ---------------------------------------------------------------------------

GFD_D float2 cmulf(float2 a, float2 b) {  // a * b
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
GFD_D float2 cmulc(float2 a, float2 b) {  // conj(a) * b
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.x, b.y, -a.y * b.x));
}
GFD_D float redot(float2 a, float2 b) { return fmaf(a.x, b.x, a.y * b.y); }  // Re(conj(a) b)

// Per-bin values of pass A (Eq. 8, 9 reversed) for one full-spectrum bin.
// With e = H U_E - Y: U_E - U_p = conj(H) e / (a + lam) and U_E - U_I =
// conj(H) e / (a + lam D2), so lambda's adjoint is formed without the
// cancellation of U_E - U_p where lam >> a.
struct BinA {
  float2 gUE, gH, gY;
  float glam, fprime;
};
GFD_D BinA adj_bin_a(float2 H, float2 Y, float2 UE, float2 GUI, float2 GUp, float D2, float lam) {
  BinA o;
  const float a = fmaf(H.x, H.x, H.y * H.y);
  const float2 HY = cmulc(H, Y);
  const float ip = __frcp_rn(a + lam);
  const float2 Up = make_float2(fmaf(lam, UE.x, HY.x) * ip, fmaf(lam, UE.y, HY.y) * ip);
  const float2 gNp = cscale(GUp, ip);
  const float gDp = -redot(gNp, Up);  // -Re(conj(g_Up) U_p) / (a + lam)
  const float2 e = csub(cmulf(H, UE), Y);
  const float2 He = cmulc(H, e);
  o.glam = redot(gNp, He) * ip;
  float2 gNI = make_float2(0.0f, 0.0f);
  float gDI = 0.0f;
  const float lg = lam * D2, DI = a + lg;
  if (DI > 0.0f) {
    const float ii = __frcp_rn(DI);
    const float2 UI = make_float2(fmaf(lg, UE.x, HY.x) * ii, fmaf(lg, UE.y, HY.y) * ii);
    gNI = cscale(GUI, ii);
    gDI = -redot(gNI, UI);
    o.glam = fmaf(D2 * ii, redot(gNI, He), o.glam);
  }
  const float2 gN = cadd(gNp, gNI);
  const float gD2 = 2.0f * (gDp + gDI);
  // N = conj(H) Y + ...: g_Y += H g_N, g_H += conj(g_N) Y; D = |H|^2 + ...: g_H += 2 g_D H
  o.gY = cmulf(H, gN);
  const float2 gNY = cmulc(gN, Y);
  o.gH = make_float2(fmaf(gD2, H.x, gNY.x), fmaf(gD2, H.y, gNY.y));
  o.gUE = make_float2(lam * fmaf(D2, gNI.x, gNp.x), lam * fmaf(D2, gNI.y, gNp.y));
  const float s = lam * ip;  // lam / (a + lam)
  o.fprime = redot(e, e) * 2.0f * s * a * ip * ip;  // |e|^2 2 lam a / (a + lam)^3
  return o;
}

// Per-bin values of pass B (the implicit derivative of lambda through Eq. 11):
// f = (1/P) sum lam^2 |e|^2 / (a + lam)^2, e = H U_E - Y; c = -g_lam / f'.
GFD_D void adj_bin_b(float2 H, float2 Y, float2 UE, float lam, float cP, float2& gUE, float2& gH,
                     float2& gY) {
  const float a = fmaf(H.x, H.x, H.y * H.y);
  const float2 e = csub(cmulf(H, UE), Y);
  const float ip = __frcp_rn(a + lam);
  const float s = lam * ip;                         // lam / (a + lam)
  const float ge = 2.0f * cP * s * s;               // g_e = ge e
  const float2 g = cscale(e, ge);
  const float ga = -2.0f * cP * s * s * redot(e, e) * ip;  // -2 lam^2 |e|^2 / (a + lam)^3
  gUE = cmulc(H, g);                                // conj(H) g_e
  const float2 Ug = cmulc(UE, g);                   // conj(U_E) g_e
  gH = make_float2(fmaf(2.0f * ga, H.x, Ug.x), fmaf(2.0f * ga, H.y, Ug.y));
  gY = make_float2(-g.x, -g.y);
}

// Pass A over the packed half spectrum of every image (grid: (chunks, n)).
// Writes g_UE, adds to g_H and g_Y, and sums g_lam and P f'(lam) (FP64).
__global__ void k_adj_spec_a(const AdjDesc* __restrict__ descs, int M, int N,
                             const float* __restrict__ d2tab) {
  const AdjDesc& d = descs[blockIdx.y];
  const double lamd = __ldcg(d.lam);
  const bool branch = !(lamd < 1e300);
  const float lam = branch ? 0.0f : (float)lamd;
  const int L = N / 2, lg = __ffs(L) - 1;  // powers of two
  const int total = M * L;
  const float invP = 1.0f / ((float)M * (float)N);
  CSum cl, cf;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += gridDim.x * blockDim.x) {
    if (branch) {
      d.gUE[idx] = make_float2(0.0f, 0.0f);
      continue;
    }
    const int k = idx >> lg, l = idx & (L - 1);
    const float d2r = __ldg(&d2tab[tab_off(M) + k]);
    if (l != 0) {
      const BinA o = adj_bin_a(d.H[idx], d.Y[idx], d.UE[idx], cscale(d.GUI[idx], invP),
                               cscale(d.GUp[idx], invP), d2r + __ldg(&d2tab[tab_off(N) + l]),
                               lam);
      d.gUE[idx] = o.gUE;
      d.gH[idx] = cadd(d.gH[idx], o.gH);
      d.gY[idx] = cadd(d.gY[idx], o.gY);
      cl.add(2.0f * o.glam);  // the bin and its mirror
      cf.add(2.0f * o.fprime);
    } else {
      const size_t m = (size_t)((M - k) & (M - 1)) * L;
      float2 HA, HB, YA, YB, EA, EB, GIA, GIB, GPA, GPB;
      unpack_pair(d.H[idx], d.H[m], HA, HB);
      unpack_pair(d.Y[idx], d.Y[m], YA, YB);
      unpack_pair(d.UE[idx], d.UE[m], EA, EB);
      unpack_pair(cscale(d.GUI[idx], invP), cscale(d.GUI[m], invP), GIA, GIB);
      unpack_pair(cscale(d.GUp[idx], invP), cscale(d.GUp[m], invP), GPA, GPB);
      const BinA oa = adj_bin_a(HA, YA, EA, GIA, GPA, d2r, lam);
      const BinA ob = adj_bin_a(HB, YB, EB, GIB, GPB, d2r + 4.0f, lam);
      d.gUE[idx] = pack_pair(oa.gUE, ob.gUE);
      d.gH[idx] = cadd(d.gH[idx], pack_pair(oa.gH, ob.gH));
      d.gY[idx] = cadd(d.gY[idx], pack_pair(oa.gY, ob.gY));
      cl.add(oa.glam);
      cl.add(ob.glam);
      cf.add(oa.fprime);
      cf.add(ob.fprime);
    }
  }
  double sl = cl.get(), sf = cf.get();
  __shared__ double red[2][32];
  for (int o = 16; o > 0; o >>= 1) {
    sl += __shfl_xor_sync(0xffffffffu, sl, o);
    sf += __shfl_xor_sync(0xffffffffu, sf, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = sl;
    red[1][threadIdx.x >> 5] = sf;
  }
  __syncthreads();
  if (threadIdx.x == 0 && !branch) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += red[0][w];
      b += red[1][w];
    }
    atomicAdd(&d.acc[0], a);
    atomicAdd(&d.acc[1], b);
  }
}

// Per image: c = -g_lam / f'(lam) and g_T -= c; clears the sums for the next step.
__global__ void k_adj_lambda(const AdjDesc* __restrict__ descs, int n, double P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const AdjDesc& d = descs[i];
  const double lam = *d.lam;
  if (lam < 1e300 && d.acc[1] > 0.0) {
    const double fprime = d.acc[1] / P;
    const double c = -d.acc[0] / fprime;
    d.acc[2] = c;
    d.acc[3] -= c;  // g_T
  } else {
    d.acc[2] = 0.0;
  }
  d.acc[0] = 0.0;
  d.acc[1] = 0.0;
}

// Pass B: the c-weighted gradient of f through e = H U_E - Y and a = |H|^2.
__global__ void k_adj_spec_b(const AdjDesc* __restrict__ descs, int M, int N) {
  const AdjDesc& d = descs[blockIdx.y];
  const double lamd = __ldcg(d.lam);
  if (!(lamd < 1e300)) return;
  const float lam = (float)lamd;
  const float cP = (float)(__ldcg(&d.acc[2]) / ((double)M * N));
  const int L = N / 2, lg = __ffs(L) - 1;  // powers of two
  const int total = M * L;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += gridDim.x * blockDim.x) {
    const int k = idx >> lg, l = idx & (L - 1);
    float2 gUE, gH, gY;
    if (l != 0) {
      adj_bin_b(d.H[idx], d.Y[idx], d.UE[idx], lam, cP, gUE, gH, gY);
    } else {
      const size_t m = (size_t)((M - k) & (M - 1)) * L;
      float2 HA, HB, YA, YB, EA, EB, uA, uB, hA, hB, yA, yB;
      unpack_pair(d.H[idx], d.H[m], HA, HB);
      unpack_pair(d.Y[idx], d.Y[m], YA, YB);
      unpack_pair(d.UE[idx], d.UE[m], EA, EB);
      adj_bin_b(HA, YA, EA, lam, cP, uA, hA, yA);
      adj_bin_b(HB, YB, EB, lam, cP, uB, hB, yB);
      gUE = pack_pair(uA, uB);
      gH = pack_pair(hA, hB);
      gY = pack_pair(yA, yB);
    }
    d.gUE[idx] = cadd(d.gUE[idx], gUE);
    d.gH[idx] = cadd(d.gH[idx], gH);
    d.gY[idx] = cadd(d.gY[idx], gY);
  }
}

// g_u of the previous step is the adjoint DFT of g_UE, written by the inverse
// transform; where lambda = inf (u_I = u_p = u_E) it is g_uI + g_up instead.
__global__ void k_adj_next(const AdjDesc* __restrict__ descs, int M, int N) {
  const AdjDesc& d = descs[blockIdx.y];
  if (__ldcg(d.lam) < 1e300) return;
  const size_t P = (size_t)M * N;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < P;
       i += (size_t)gridDim.x * blockDim.x)
    d.gu[i] = d.guI[i] + d.gup[i];
}

cudaError_t launch_adj_spectral(const AdjDesc* descs, int n, int M, int N, const float* d2tab,
                                cudaStream_t s) {
  const int chunks = spec_chunks(M, N);
  k_adj_spec_a<<<dim3(chunks, n), 256, 0, s>>>(descs, M, N, d2tab);
  k_adj_lambda<<<(n + 63) / 64, 64, 0, s>>>(descs, n, (double)M * N);
  k_adj_spec_b<<<dim3(chunks, n), 256, 0, s>>>(descs, M, N);
  return cudaGetLastError();
}

cudaError_t launch_adj_next(const AdjDesc* descs, int n, int M, int N, cudaStream_t s) {
  const size_t P = (size_t)M * N;
  int chunks = (int)((P + 256 * 8 - 1) / (256 * 8));
  if (chunks > 256) chunks = 256;
  k_adj_next<<<dim3(chunks, n), 256, 0, s>>>(descs, M, N);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Statistics of Eq. 12 and the final gradients of y and h
// ---------------------------------------------------------------------------

// sum y, sum y^2 (FP64) into acc[4], acc[5]; sum |h| into acc[6] (block 0).
__global__ void k_adj_stats(const AdjDesc* __restrict__ descs, int M, int N) {
  const AdjDesc& d = descs[blockIdx.y];
  const size_t P = (size_t)M * N;
  CSum cy, cyy;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < P;
       i += (size_t)gridDim.x * blockDim.x) {
    const float v = __ldg(&d.y[i]);
    cy.add(v);
    cyy.add(two_prod(v, v));
  }
  double sy = cy.get(), syy = cyy.get();
  for (int o = 16; o > 0; o >>= 1) {
    sy += __shfl_xor_sync(0xffffffffu, sy, o);
    syy += __shfl_xor_sync(0xffffffffu, syy, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&d.acc[4], sy);
    atomicAdd(&d.acc[5], syy);
  }
  if (blockIdx.x == gridDim.x - 1) {
    double s, a;
    psf_sums(d.h, d.kh * d.kw, s, a);
    if (threadIdx.x == 0) d.acc[6] = a;
  }
}

// dT/dy and dT/dh through rho (Eq. 12): acc[7] = g_num, acc[8] = g_den (zero
// where rho is clamped to 1); writes g_eps.
__global__ void k_adj_rho(const AdjDesc* __restrict__ descs, int n, double P) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const AdjDesc& d = descs[i];
  const double Sy = d.acc[4], Syy = d.acc[5], h1 = d.acc[6], sig2 = d.sigma * d.sigma;
  const double num = Syy - Sy * Sy / P - P * sig2;
  const double den = h1 * h1 * Syy;
  const double rad = 1.0 - num / den;
  double g_num = 0.0, g_den = 0.0;
  if (rad > 0.0 && rad < 1.0 && d.rho_fixed <= 0.0) {
    const double rho = sqrt(rad);
    const double g_rad = d.acc[3] * P * sig2 / (2.0 * rho);
    g_num = -g_rad / den;
    g_den = g_rad * num / (den * den);
  }
  d.acc[7] = g_num;
  d.acc[8] = g_den;
  *d.g_eps_out = *d.g_eps;
}

// g_y = (adjoint DFT of g_Y, in gtmp) + dT/dy terms.
__global__ void k_adj_final_y(const AdjDesc* __restrict__ descs, int M, int N) {
  const AdjDesc& d = descs[blockIdx.y];
  const size_t P = (size_t)M * N;
  // g_num (2 y - 2 Sy / P) + g_den h1^2 2 y = a y + b, a in double-float
  const double g_num = d.acc[7], g_den = d.acc[8], Sy = d.acc[4], h1 = d.acc[6];
  const df a = df_from_double(2.0 * (g_num + g_den * h1 * h1));
  const df b = df_from_double(-2.0 * g_num * Sy / (double)P);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < P;
       i += (size_t)gridDim.x * blockDim.x) {
    const df v = df_add(df_add(df_mul_f(a, __ldg(&d.y[i])), b), df_make(__ldg(&d.gtmp[i])));
    d.gy_out[i] = v.hi + v.lo;
  }
}

// g_h[i][j] = (adjoint DFT of g_H at the canvas position of h[i][j], in gtmp2)
// + dT/dh (Eq. 12 through sum |h|).
__global__ void k_adj_final_h(const AdjDesc* __restrict__ descs, int M, int N) {
  const AdjDesc& d = descs[blockIdx.y];
  const int rh = d.kh / 2, rw = d.kw / 2;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d.kh * d.kw; e += gridDim.x * blockDim.x) {
    const int i = e / d.kw, j = e - i * d.kw;
    const int ci = ((i - rh) % M + M) % M, cj = ((j - rw) % N + N) % N;
    const double hv = d.h[e];
    const double sgn = hv > 0.0 ? 1.0 : (hv < 0.0 ? -1.0 : 0.0);
    d.gh_out[e] = (float)((double)d.gtmp2[(size_t)ci * N + cj] +
                          d.acc[8] * 2.0 * d.acc[6] * d.acc[5] * sgn);
  }
}

cudaError_t launch_adj_stats(const AdjDesc* descs, int n, int M, int N, cudaStream_t s) {
  const size_t P = (size_t)M * N;
  int chunks = (int)((P + 256 * 16 - 1) / (256 * 16));
  if (chunks > 64) chunks = 64;
  k_adj_stats<<<dim3(chunks, n), 256, 0, s>>>(descs, M, N);
  return cudaGetLastError();
}

cudaError_t launch_adj_final(const AdjDesc* descs, int n, int M, int N, int max_psf,
                             cudaStream_t s) {
  const size_t P = (size_t)M * N;
  int chunks = (int)((P + 256 * 8 - 1) / (256 * 8));
  if (chunks > 256) chunks = 256;
  k_adj_rho<<<(n + 63) / 64, 64, 0, s>>>(descs, n, (double)P);
  k_adj_final_y<<<dim3(chunks, n), 256, 0, s>>>(descs, M, N);
  k_adj_final_h<<<dim3((max_psf + 255) / 256, n), 256, 0, s>>>(descs, M, N);
  return cudaGetLastError();
}

template <class OP>
static cudaError_t configure_adj_box() {
  return cudaFuncSetAttribute(k_adj_box<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)adj_box_smem<OP>(8));
}

cudaError_t configure_adj_kernels() {
  cudaError_t e = configure_adj_box<AdjStats>();
  if (e == cudaSuccess) e = configure_adj_box<AdjPoint>();
  if (e == cudaSuccess) e = configure_adj_box<AdjInputs>();
  return e;
}

}  // namespace gfd
