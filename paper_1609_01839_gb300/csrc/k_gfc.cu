// Guided filter with a colour guidance image (the paper notes the guided
// filter serves colour as well as grey-scale images, Sec. 3.1): guidance I
// with 3 channels (planar [3][M][N]), filtering input p.  Per window k,
//   a_k = (Sigma_k + eps U)^-1 (mean_k(I p) - mu_k pbar_k)   (3-vector, Eq. 3)
//   b_k = pbar_k - a_k . mu_k                                 (Eq. 4)
//   u   = abar . I + bbar                                     (Eq. 5)
// with mu_k, Sigma_k the window mean and covariance of I.
//
// Two tiled passes, each a TX x TY block of output pixels whose input tile
// plus an r-pixel halo is staged in shared memory; window sums run along the
// rows into shared memory (four outputs per thread), then down its columns (two
// outputs per thread).  Neighbouring windows share the sum of what they have in
// common and add their own ends to it: as many additions as sliding takes, but
// nothing is ever taken away again, so a pixel touches the windows that hold it
// and no others, whatever its value (an infinity, a NaN, a bright outlier):
//   1. the 13 window sums (I_c, p, I_c I_d, I_c p), the 3 x 3 solve -> a, b planes;
//   2. the window sums of a and b -> u.
// Windows are periodic or truncated at the canvas edge (means over the
// pixels inside).
//
// Arithmetic.  FP64 runs at 1.5 operations per cycle and SM on this part (70
// cycles latency), so ordinary tiles use none per pixel.  Pass 1 splits each value on
// a grid of the tile, v = c + g m + l with c the grid's point next to a pixel of the
// tile and |m| <= 4096 / (2r+1), as the grey-scale filter does (l is formed from v and c
// themselves, not from their rounded difference): the sums of m and of the
// products m m' are exact in FP32, those of the remainders' parts are small,
// and n S_mm' - S_m S_m' is formed exactly as a double-float.  The normal
// equations are eliminated in double-float (about 48 bits) and a, b rounded
// once.  Pass 2's sums are compensated (an FP32 running sum plus the exact
// error of every addition).  1024 x 1024, w = 9: 1111 us with FP64 sums and
// solves, 135 us as it is, the same error against FP64 (2.5e-8); 128 us with slid
// sums of rounded deviations and no look at the tile, which spread what is not
// finite and lost dark pixels' digits beside bright ones.
//
// With R_I, R_p a tile's ranges the remainders' sums cost the means about 2^-24 R w
// / 4096 and the covariances about 6e-11 R R'.  Held against the rounding of u,
// 2^-24 s with s a low estimate of |p| in the tile, and against eps, that is small
// enough where R_p <= 256 s, R_I R_p <= 2^14 sqrt(eps) s and R_I^2 <= 2^16 eps
// (images of [0, 1] down to eps = 2e-5).  A nearly flat plane's range counts as
// |v| / (256 (2r+1)) at least, which keeps |v| below 2^20 grid steps.  Tiles beyond
// (bright pixels in a dark neighbourhood, tiny eps) and tiles with values that are
// not finite or whose squares leave FP32's range are summed and solved in FP64
// (cgf_ab_exact) at that kernel's price.
#include "common.cuh"
#include "df.cuh"
#include "launch.h"

namespace gfd {

constexpr int CGF_TX = 32, CGF_TY = 16;  // outputs of a block
constexpr int CGF_THREADS = 256;
constexpr int CGF_RMAX = 8;
constexpr int CGF_ROW = 4, CGF_COL = 2;  // outputs per thread along a row, down a column
constexpr int CGF_Q = 13;                // window sums, each a leading and a remainder part

// Row sums [CGF_Q][rows][CGF_RP] float2 and the input tile [rows][pitch] float4.
// Consecutive threads of the row sums take consecutive rows: odd pitches keep
// them on different banks.
constexpr int CGF_RP = CGF_TX + 1;
GFD_HD int cgf_pitch(int rad) { return (CGF_TX + 2 * rad) | 1; }
GFD_HD size_t cgf_smem1(int rad) {
  const int EY = CGF_TY + 2 * rad;
  return (size_t)cgf_pitch(rad) * EY * sizeof(float4) + (size_t)CGF_Q * EY * CGF_RP * sizeof(float2);
}
// pass 2: row sums [2][rows][CGF_RP] float4, the tile [rows][pitch] float4
GFD_HD size_t cgf_smem2(int rad) {
  const int EY = CGF_TY + 2 * rad;
  return (size_t)(cgf_pitch(rad) + 2 * CGF_RP) * EY * sizeof(float4);
}

// Canvas index of tile coordinate v (may lie outside [0, L)); -1 when the
// window is truncated there.
GFD_D int cgf_wrap(int v, int L, bool trunc) {
  if (trunc) return (v >= 0 && v < L) ? v : -1;
  return v & (L - 1);
}

GFD_D int cgf_count(int x, int L, int rad) {
  const int a = x - rad < 0 ? 0 : x - rad;
  const int b = x + rad > L - 1 ? L - 1 : x + rad;
  return b - a + 1;
}

// Stage the tile of 4 planes (origin (y0 - rad, x0 - rad)); out-of-canvas pixels of
// truncated windows are `out`.
GFD_D void cgf_stage(float4* s, const float* p0, const float* p1, const float* p2, const float* p3,
                     float4 out, int M, int N, int y0, int x0, int rad, bool trunc) {
  const int EX = CGF_TX + 2 * rad, EY = CGF_TY + 2 * rad;
  for (int e = threadIdx.x; e < EX * EY; e += blockDim.x) {
    const int ty = e / EX, tx = e - ty * EX;
    const int gy = cgf_wrap(y0 - rad + ty, M, trunc), gx = cgf_wrap(x0 - rad + tx, N, trunc);
    float4 v = out;
    if (gy >= 0 && gx >= 0) {
      const size_t off = (size_t)gy * N + gx;
      v = make_float4(__ldg(p0 + off), __ldg(p1 + off), __ldg(p2 + off), __ldg(p3 + off));
    }
    s[ty * cgf_pitch(rad) + tx] = v;
  }
}

// One plane's split: v - c = g m + l, c = g mc the reference (on the grid, so that
// |l| <= g / 2).
struct CgfGrid {
  float g, ig, mc;
};
constexpr float CGF_MAGIC = 12582912.0f;  // rounds |t| < 2^22 to an integer

// v = g m + l with an integer m; both exact (l has at most 24 bits: |l| < g and v
// is a multiple of 2^-24 |v| or smaller than g).
GFD_D void cgf_split(float v, float g, float ig, float& m, float& l) {
  m = fmaf(v, ig, CGF_MAGIC) - CGF_MAGIC;
  l = fmaf(-g, m, v);
}

// The leading parts (integers, exact) and the remainders' parts of the 13
// sums: 0-3 the values r, g, b, p; 4-9 the products rr, rg, rb, gg, gb, bb;
// 10-12 rp, gp, bp.
struct CgfSums {
  float h[CGF_Q], l[CGF_Q];
  GFD_D void clear() {
#pragma unroll
    for (int q = 0; q < CGF_Q; ++q) h[q] = l[q] = 0.0f;
  }
  // the sums with one pixel more, each handed to out(q, leading, remainder)
  template <class F>
  GFD_D void with(float4 v, const CgfGrid (&G)[4], F out) const {
    const float vs[4] = {v.x, v.y, v.z, v.w};
    float m[4], x[4], xh[4], xl[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      cgf_split(vs[c], G[c].g, G[c].ig, m[c], xl[c]);
      m[c] -= G[c].mc;
      xh[c] = m[c] * G[c].g;
      x[c] = xh[c] + xl[c];
      out(c, h[c] + m[c], l[c] + xl[c]);
    }
    constexpr int qi[9] = {0, 0, 0, 1, 1, 2, 0, 1, 2}, qj[9] = {0, 1, 2, 1, 2, 2, 3, 3, 3};
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const int i = qi[q], j = qj[q];
      // x_i x_j - h_i h_j = x_i l_j + l_i h_j
      out(4 + q, fmaf(m[i], m[j], h[4 + q]), fmaf(x[i], xl[j], fmaf(xl[i], xh[j], l[4 + q])));
    }
  }
  GFD_D void add(float4 v, const CgfGrid (&G)[4]) {
    with(v, G, [&](int q, float hq, float lq) {
      h[q] = hq;
      l[q] = lq;
    });
  }
};

// Calls add(state, i) and put(k, state, i) so that put k gets the sum over
// i = k .. k + 2 rad, its last element i not yet added, for k = 0..3: the
// elements that all four (then two) of them hold are summed once.
template <class S, class ADD, class PUT>
GFD_D void windows4(S zero, int rad, ADD add, PUT put) {
  if (rad == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) put(k, zero, k);
    return;
  }
  S all = zero;  // 3 .. 2 rad
#pragma unroll 1
  for (int i = 3; i <= 2 * rad; ++i) add(all, i);
  S two = all;  // 1 .. 2 rad
  add(two, 1);
  add(two, 2);
  put(0, two, 0);
  put(1, two, 2 * rad + 1);
  add(all, 2 * rad + 1);  // 3 .. 2 rad + 2
  add(all, 2 * rad + 2);
  put(2, all, 2);
  put(3, all, 2 * rad + 3);
}

// n S_xy - S_x S_y of one pair in double-float: the integer parts' difference
// exactly (two exact products), times both grids, plus the remainders' parts
// n L_xy - (H_x l_y + l_x H_y + l_x l_y), H = g S_m.
GFD_D df cgf_cov(float n, float sxy, float lxy, float sx, float lx, float gx, float sy, float ly,
                 float gy) {
  const df a = two_prod(n, sxy), b = two_prod(sx, sy);
  df D = two_sum(a.hi, -b.hi);
  D = quick_two_sum(D.hi, D.lo + (a.lo - b.lo));
  const float Hx = gx * sx, Hy = gy * sy;
  const float lo = fmaf(n, lxy, -fmaf(Hx, ly, (Hy + ly) * lx));
  return df_add(df_mul_f(D, gx * gy), df_make(lo));
}

// Window sums, statistics and solve of a staged tile in FP64 (tiles whose values do
// not suit the split; rows: the block's row sums, as doubles).
__device__ __noinline__ static void cgf_ab_exact(const float4* tile, double* rows, int M, int N,
                                                 int rad, double eps, bool trunc, int x0, int y0,
                                                 float* __restrict__ ab) {
  const int EY = CGF_TY + 2 * rad, TP = cgf_pitch(rad);
  for (int e = threadIdx.x; e < EY * CGF_TX; e += blockDim.x) {
    const int ty = e / CGF_TX, tx = e % CGF_TX;
    double s[CGF_Q] = {};
    for (int dx = 0; dx <= 2 * rad; ++dx) {
      const float4 t = tile[ty * TP + tx + dx];
      const double r = t.x, g = t.y, b = t.z, v = t.w;
      s[0] += r;
      s[1] += g;
      s[2] += b;
      s[3] += v;
      s[4] = fma(r, r, s[4]);
      s[5] = fma(r, g, s[5]);
      s[6] = fma(r, b, s[6]);
      s[7] = fma(g, g, s[7]);
      s[8] = fma(g, b, s[8]);
      s[9] = fma(b, b, s[9]);
      s[10] = fma(r, v, s[10]);
      s[11] = fma(g, v, s[11]);
      s[12] = fma(b, v, s[12]);
    }
#pragma unroll
    for (int q = 0; q < CGF_Q; ++q) rows[(q * EY + ty) * CGF_RP + tx] = s[q];
  }
  __syncthreads();
  const size_t P = (size_t)M * N;
  for (int e = threadIdx.x; e < CGF_TY * CGF_TX; e += blockDim.x) {
    const int ty = e / CGF_TX, tx = e % CGF_TX, gy = y0 + ty, gx = x0 + tx;
    if (gy >= M || gx >= N) continue;
    double S[CGF_Q];
#pragma unroll
    for (int q = 0; q < CGF_Q; ++q) {
      S[q] = 0.0;
      for (int dy = 0; dy <= 2 * rad; ++dy) S[q] += rows[(q * EY + ty + dy) * CGF_RP + tx];
    }
    const double n = trunc ? (double)(cgf_count(gy, M, rad) * cgf_count(gx, N, rad))
                           : (double)((2 * rad + 1) * (2 * rad + 1));
    const double in = 1.0 / n;
    const double mr = S[0] * in, mg = S[1] * in, mb = S[2] * in, mp = S[3] * in;
    // Sigma + eps U (symmetric) and the covariance of I with p
    const double c00 = S[4] * in - mr * mr + eps, c01 = S[5] * in - mr * mg;
    const double c02 = S[6] * in - mr * mb, c11 = S[7] * in - mg * mg + eps;
    const double c12 = S[8] * in - mg * mb, c22 = S[9] * in - mb * mb + eps;
    const double vr = S[10] * in - mr * mp, vg = S[11] * in - mg * mp, vb = S[12] * in - mb * mp;
    // elimination (the system is positive definite)
    const double i0 = 1.0 / c00, l1 = c01 * i0, l2 = c02 * i0;
    const double b11 = c11 - l1 * c01, b12 = c12 - l1 * c02, b22 = c22 - l2 * c02;
    const double w1 = vg - l1 * vr, w2 = vb - l2 * vr;
    const double i1 = 1.0 / b11, m2 = b12 * i1;
    const double a2 = (w2 - m2 * w1) / (b22 - m2 * b12);
    const double a1 = (w1 - b12 * a2) * i1;
    const double a0 = (vr - c01 * a1 - c02 * a2) * i0;
    const size_t o = (size_t)gy * N + gx;
    ab[o] = (float)a0;
    ab[P + o] = (float)a1;
    ab[2 * P + o] = (float)a2;
    ab[3 * P + o] = (float)(mp - (a0 * mr + a1 * mg + a2 * mb));
  }
}

// Pass 1: window statistics and the 3 x 3 solve of Eq. 3; a (3 planes) and b.
__global__ void __launch_bounds__(CGF_THREADS, 2)
k_cgf_ab(const float* __restrict__ I, const float* __restrict__ p, int M, int N, int rad,
         double eps_d, float2 eps, int trunc_i, float* __restrict__ ab) {
  extern __shared__ __align__(16) unsigned char cgf_sm[];
  __shared__ float s_max[5][CGF_THREADS / 32];
  const bool trunc = trunc_i != 0;
  const int EX = CGF_TX + 2 * rad, EY = CGF_TY + 2 * rad, TP = cgf_pitch(rad);
  float4* tile = reinterpret_cast<float4*>(cgf_sm);           // [EY][TP]
  float2* rows = reinterpret_cast<float2*>(tile + TP * EY);   // [13][EY][CGF_RP]
  const size_t P = (size_t)M * N;
  const int x0 = blockIdx.x * CGF_TX, y0 = blockIdx.y * CGF_TY;
  // reference: of each plane the middle one of three pixels (one outlier is passed by)
  float4 c;
  {
    const size_t row = (size_t)((y0 + CGF_TY / 2) & (M - 1)) * N;
    const size_t o0 = row + ((x0 + CGF_TX / 4) & (N - 1)), o1 = row + ((x0 + CGF_TX / 2) & (N - 1));
    const size_t o2 = row + ((x0 + 3 * CGF_TX / 4) & (N - 1));
    auto mid = [&](const float* q) {
      const float u = __ldg(q + o0), v = __ldg(q + o1), t = __ldg(q + o2);
      return fmaxf(fminf(u, v), fminf(fmaxf(u, v), t));
    };
    c = make_float4(mid(I), mid(I + P), mid(I + 2 * P), mid(p));
  }
  cgf_stage(tile, I, I + P, I + 2 * P, p, trunc ? c : make_float4(0.0f, 0.0f, 0.0f, 0.0f), M, N, y0,
            x0, rad, trunc);
  __syncthreads();
  // the tile's largest |deviation| of each plane fixes the grids; with the means of
  // |p| they tell whether the split suits the tile (see the top of the file)
  float4 mx = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float sp = 0.0f, np = 0.0f;
  bool fast = eps.x >= 1e-25f && eps.x <= 1e30f;
  for (int e = threadIdx.x; e < EX * EY; e += blockDim.x) {
    const float4 v = tile[(e / EX) * TP + e % EX];
    const float4 d = make_float4(fabsf(v.x - c.x), fabsf(v.y - c.y), fabsf(v.z - c.z),
                                 fabsf(v.w - c.w));
    // (false for NaN)
    fast = fast && d.x <= 1e15f && d.y <= 1e15f && d.z <= 1e15f && d.w <= 1e15f;
    mx = make_float4(fmaxf(mx.x, d.x), fmaxf(mx.y, d.y), fmaxf(mx.z, d.z), fmaxf(mx.w, d.w));
    sp += fabsf(v.w);
    np += 1.0f;
  }
  mx = make_float4(warp_max(mx.x), warp_max(mx.y), warp_max(mx.z), warp_max(mx.w));
  sp = warp_sum(sp) / warp_sum(np);  // the mean of the warp's pixels (64 or more)
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    s_max[0][w] = mx.x;
    s_max[1][w] = mx.y;
    s_max[2][w] = mx.z;
    s_max[3][w] = mx.w;
    s_max[4][w] = sp;
  }
  fast = __syncthreads_and(fast) != 0;
  CgfGrid G[4];
  {
    const float inv = 1.0f / (float)(4096 / (2 * rad + 1) - 2);
    const float flat = 1.0f / (float)(256 * (2 * rad + 1));
    float cs[4] = {c.x, c.y, c.z, c.w};
    float top = 0.0f, low = s_max[4][0], mean = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float b = 0.0f;
#pragma unroll
      for (int w = 0; w < CGF_THREADS / 32; ++w) {
        b = fmaxf(b, s_max[q][w]);
        if (q == 0) {
          low = fminf(low, s_max[4][w]);
          mean += s_max[4][w] / (float)(CGF_THREADS / 32);
        }
      }
      // |v| <= 2^20 g: a nearly flat plane takes the coarser grid of a larger range (in
      // FP64 such planes, highlights clipped at 1, took 908 us instead of 123)
      b = fmaxf(b, (fabsf(cs[q]) + b) * flat);
      int e = 0;
      float f = 0.5f;
      if (b > 0.0f) f = frexpf(b * inv, &e);
      if (e < -100) e = -100;
      G[q].g = ldexpf(ceilf(8.0f * f) * 0.125f, e);  // 3-bit mantissa: g m is exact
      G[q].ig = 1.0f / G[q].g;
      float lc;
      cgf_split(cs[q], G[q].g, G[q].ig, G[q].mc, lc);
      cs[q] -= lc;  // (exact, as |c| <= 2^20 g)
      if (q < 3) {
        top = fmaxf(top, b);
      } else {  // the lowest of the warps' means (a few bright pixels do not raise it)
        const float sc = fmaxf(low, mean * 0.015625f);
        fast = fast && b <= 256.0f * sc && top * b <= 16384.0f * sqrtf(eps.x) * sc;
      }
      fast = fast && (b == 0.0f || b >= 1e-25f);
    }
    fast = fast && top * top <= 65536.0f * eps.x;
    c = make_float4(cs[0], cs[1], cs[2], cs[3]);
  }
  // pixels outside the canvas of truncated windows count nothing: no deviation, or zero
  if (trunc && (x0 < rad || y0 < rad || x0 + CGF_TX + rad > N || y0 + CGF_TY + rad > M)) {
    const float4 none = fast ? c : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int e = threadIdx.x; e < EX * EY; e += blockDim.x) {
      const int ty = e / EX, tx = e - ty * EX;
      if (cgf_wrap(y0 - rad + ty, M, true) < 0 || cgf_wrap(x0 - rad + tx, N, true) < 0)
        tile[ty * TP + tx] = none;
    }
    __syncthreads();
  }
  if (!fast) {  // the same for the whole block
    cgf_ab_exact(tile, reinterpret_cast<double*>(rows), M, N, rad, eps_d, trunc, x0, y0, ab);
    return;
  }
  // row sums: CGF_ROW neighbouring outputs of a tile row
  for (int e = threadIdx.x; e < EY * (CGF_TX / CGF_ROW); e += blockDim.x) {
    const int ty = e % EY, tx = (e / EY) * CGF_ROW;
    const float4* in = tile + ty * TP + tx;
    CgfSums zero;
    zero.clear();
    windows4(
        zero, rad, [&](CgfSums& s, int i) { s.add(in[i], G); },
        [&](int k, const CgfSums& s, int i) {
          s.with(in[i], G, [&](int q, float hq, float lq) {
            rows[(q * EY + ty) * CGF_RP + tx + k] = make_float2(hq, lq);
          });
        });
  }
  __syncthreads();
  const int tx = threadIdx.x % CGF_TX, ty0 = (threadIdx.x / CGF_TX) * CGF_COL;
  const int gx = x0 + tx;
  float2 C[CGF_Q];  // the rows that both outputs hold
#pragma unroll
  for (int q = 0; q < CGF_Q; ++q) {
    C[q] = make_float2(0.0f, 0.0f);
    const float2* rr = rows + (q * EY + ty0) * CGF_RP + tx;
    for (int dy = 1; dy <= 2 * rad; ++dy) C[q] = cadd(C[q], rr[dy * CGF_RP]);
  }
#pragma unroll 1
  for (int k = 0; k < CGF_COL; ++k) {
    const int gy = y0 + ty0 + k;
    float2 S[CGF_Q];
#pragma unroll
    for (int q = 0; q < CGF_Q; ++q)
      S[q] = cadd(C[q], rows[(q * EY + ty0 + (k == 0 ? 0 : 2 * rad + 1)) * CGF_RP + tx]);
    if (gy < M && gx < N) {
      const float n = trunc ? (float)(cgf_count(gy, M, rad) * cgf_count(gx, N, rad))
                            : (float)((2 * rad + 1) * (2 * rad + 1));
      auto cov = [&](int q, int i, int j) {
        return cgf_cov(n, S[q].x, S[q].y, S[i].x, S[i].y, G[i].g, S[j].x, S[j].y, G[j].g);
      };
      // n^2 (Sigma + eps U) a = n^2 cov(I, p): eliminated in double-float
      const df en = df_mul_f(df_mul_f(df{eps.x, eps.y}, n), n);
      const df A00 = df_add(cov(4, 0, 0), en), A01 = cov(5, 0, 1);
      const df A02 = cov(6, 0, 2), A11 = df_add(cov(7, 1, 1), en);
      const df A12 = cov(8, 1, 2), A22 = df_add(cov(9, 2, 2), en);
      const df v0 = cov(10, 0, 3), v1 = cov(11, 1, 3);
      const df v2 = cov(12, 2, 3);
      const df i0 = df_rcp(A00), l1 = df_mul(A01, i0), l2 = df_mul(A02, i0);
      const df B11 = df_sub(A11, df_mul(l1, A01)), B12 = df_sub(A12, df_mul(l1, A02));
      const df B22 = df_sub(A22, df_mul(l2, A02));
      const df w1 = df_sub(v1, df_mul(l1, v0)), w2 = df_sub(v2, df_mul(l2, v0));
      const df i1 = df_rcp(B11), m2 = df_mul(B12, i1);
      const df C22 = df_sub(B22, df_mul(m2, B12));
      const df a2 = df_mul(df_sub(w2, df_mul(m2, w1)), df_rcp(C22));
      const df a1 = df_mul(df_sub(w1, df_mul(B12, a2)), i1);
      const df a0 = df_mul(df_sub(df_sub(v0, df_mul(A01, a1)), df_mul(A02, a2)), i0);
      // b = pbar - a . mu, the means restored to absolute values
      const float inv_n = 1.0f / n;
      auto mean = [&](int q, float cq) {
        const df s = two_prod(G[q].g, S[q].x);
        const df d = df_add(s, df_make(S[q].y));  // n (mean - c)
        const float r = d.hi * inv_n;             // quotient and its residual
        const float e = fmaf(-r, n, d.hi) + d.lo;
        return df_add(df_make(cq), quick_two_sum(r, e * inv_n));
      };
      df b = mean(3, c.w);
      b = df_sub(b, df_mul(a0, mean(0, c.x)));
      b = df_sub(b, df_mul(a1, mean(1, c.y)));
      b = df_sub(b, df_mul(a2, mean(2, c.z)));
      const size_t o = (size_t)gy * N + gx;
      ab[o] = a0.hi + a0.lo;
      ab[P + o] = a1.hi + a1.lo;
      ab[2 * P + o] = a2.hi + a2.lo;
      ab[3 * P + o] = b.hi + b.lo;
    }
  }
}

// Compensated sums of four planes: hi the FP32 running sums, lo the exact
// errors of their additions.
struct CgfComp {
  float2 hi[2], lo[2];
  GFD_D void clear() {
    hi[0] = hi[1] = lo[0] = lo[1] = make_float2(0.0f, 0.0f);
  }
  GFD_D void add(int i, float2 v, float2 vlo) {  // pair i
    const float2 s = cadd(hi[i], v), bb = csub(s, hi[i]);
    const float2 e = cadd(csub(hi[i], csub(s, bb)), csub(v, bb));
    hi[i] = s;
    lo[i] = cadd(lo[i], cadd(e, vlo));
  }
};

// Pass 2: window means of a and b, u = abar . I + bbar (Eq. 5).
__global__ void __launch_bounds__(CGF_THREADS)
k_cgf_out(const float* __restrict__ I, const float* __restrict__ ab, int M, int N, int rad,
          int trunc_i, float* __restrict__ u) {
  extern __shared__ __align__(16) unsigned char cgf_sm[];
  const bool trunc = trunc_i != 0;
  const int EY = CGF_TY + 2 * rad, TP = cgf_pitch(rad);
  float4* tile = reinterpret_cast<float4*>(cgf_sm);  // [EY][TP]
  float4* rows = tile + TP * EY;                     // [2][EY][CGF_RP]: (hi pair, lo pair)
  const size_t P = (size_t)M * N;
  const int x0 = blockIdx.x * CGF_TX, y0 = blockIdx.y * CGF_TY;
  cgf_stage(tile, ab, ab + P, ab + 2 * P, ab + 3 * P, make_float4(0.0f, 0.0f, 0.0f, 0.0f), M, N, y0,
            x0, rad, trunc);
  __syncthreads();
  for (int e = threadIdx.x; e < EY * (CGF_TX / CGF_ROW); e += blockDim.x) {
    const int ty = e % EY, tx = (e / EY) * CGF_ROW;
    const float4* in = tile + ty * TP + tx;
    CgfComp zero;
    zero.clear();
    auto add = [&](CgfComp& s, int i) {
      const float4 v = in[i];
      s.add(0, make_float2(v.x, v.y), make_float2(0.0f, 0.0f));
      s.add(1, make_float2(v.z, v.w), make_float2(0.0f, 0.0f));
    };
    windows4(zero, rad, add, [&](int k, CgfComp s, int i) {
      add(s, i);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        rows[(h * EY + ty) * CGF_RP + tx + k] =
            make_float4(s.hi[h].x, s.hi[h].y, s.lo[h].x, s.lo[h].y);
    });
  }
  __syncthreads();
  const int tx = threadIdx.x % CGF_TX, ty0 = (threadIdx.x / CGF_TX) * CGF_COL;
  const int gx = x0 + tx;
  CgfComp core;  // the rows that both outputs hold
  core.clear();
  auto add = [&](CgfComp& s, int ty) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 v = rows[(i * EY + ty) * CGF_RP + tx];
      s.add(i, make_float2(v.x, v.y), make_float2(v.z, v.w));
    }
  };
#pragma unroll 1
  for (int dy = 1; dy <= 2 * rad; ++dy) add(core, ty0 + dy);
#pragma unroll
  for (int k = 0; k < CGF_COL; ++k) {
    const int gy = y0 + ty0 + k;
    CgfComp s = core;
    add(s, k == 0 ? ty0 : ty0 + 2 * rad + 1);
    if (gy < M && gx < N) {
      const float n = trunc ? (float)(cgf_count(gy, M, rad) * cgf_count(gx, N, rad))
                            : (float)((2 * rad + 1) * (2 * rad + 1));
      const size_t o = (size_t)gy * N + gx;
      df v = quick_two_sum(s.hi[1].y, s.lo[1].y);
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[0].x, s.lo[0].x), __ldg(&I[o])));
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[0].y, s.lo[0].y), __ldg(&I[P + o])));
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[1].x, s.lo[1].x), __ldg(&I[2 * P + o])));
      const float inv_n = 1.0f / n, q = v.hi * inv_n;  // v / n, rounded once
      float r = fmaf(fmaf(-q, n, v.hi) + v.lo, inv_n, q);
      if (!(fabsf(r) < 1e30f)) {  // near the end of FP32's range, or not finite: in FP64
        double sum[4] = {0.0, 0.0, 0.0, 0.0};
        for (int dy = 0; dy <= 2 * rad; ++dy)
          for (int dx = 0; dx <= 2 * rad; ++dx) {
            const float4 t = tile[(ty0 + k + dy) * TP + tx + dx];
            sum[0] += t.x;
            sum[1] += t.y;
            sum[2] += t.z;
            sum[3] += t.w;
          }
        r = (float)((sum[0] * I[o] + sum[1] * I[P + o] + sum[2] * I[2 * P + o] + sum[3]) / n);
      }
      u[o] = r;
    }
  }
}

cudaError_t launch_guided_filter_color(const float* I, const float* p, int M, int N, int w,
                                       double eps, int boundary, float* ab, float* u,
                                       cudaStream_t s) {
  const int rad = (w - 1) / 2;
  const dim3 grid((N + CGF_TX - 1) / CGF_TX, (M + CGF_TY - 1) / CGF_TY);
  const int trunc = boundary == GFD_BOUNDARY_TRUNCATED ? 1 : 0;
  const float eh = (float)eps;
  const float2 e2 = make_float2(eh, (float)(eps - (double)eh));
  k_cgf_ab<<<grid, CGF_THREADS, cgf_smem1(rad), s>>>(I, p, M, N, rad, eps, e2, trunc, ab);
  k_cgf_out<<<grid, CGF_THREADS, cgf_smem2(rad), s>>>(I, ab, M, N, rad, trunc, u);
  return cudaGetLastError();
}

cudaError_t configure_gfc_kernels() {
  cudaError_t e = cudaFuncSetAttribute(k_cgf_ab, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)cgf_smem1(CGF_RMAX));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k_cgf_out, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)cgf_smem2(CGF_RMAX));
}

}  // namespace gfd
