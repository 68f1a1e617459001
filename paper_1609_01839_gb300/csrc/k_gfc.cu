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
// rows into shared memory (four outputs per thread, slid), then down its
// columns (two outputs per thread):
//   1. the 13 window sums (I_c, p, I_c I_d, I_c p), the 3 x 3 solve -> a, b planes;
//   2. the window sums of a and b -> u.
// Windows are periodic or truncated at the canvas edge (means over the
// pixels inside).
//
// Arithmetic.  FP64 runs at 1.5 operations per cycle and SM on this part (70
// cycles latency), so none is used per pixel.  Pass 1 takes deviations from
// the tile's centre pixel and splits each on a grid, x = g m + x_l with |m| <=
// 4096 / (2r+1), as the grey-scale filter does: the sums of m and of the
// products m m' are exact in FP32, those of the remainders' parts are small,
// and n S_mm' - S_m S_m' is formed exactly as a double-float.  The normal
// equations are eliminated in double-float (about 48 bits) and a, b rounded
// once.  Pass 2's sums are compensated (an FP32 running sum plus the exact
// error of every addition).  1024 x 1024, w = 9: 1111 us with FP64 sums and
// solves, 131 us as it is, the same error against FP64 (2.5e-8).
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

// Stage the tile of 4 planes (origin (y0 - rad, x0 - rad)) minus c;
// out-of-canvas pixels of truncated windows are zero.
GFD_D void cgf_stage(float4* s, const float* p0, const float* p1, const float* p2, const float* p3,
                     float4 c, int M, int N, int y0, int x0, int rad, bool trunc) {
  const int EX = CGF_TX + 2 * rad, EY = CGF_TY + 2 * rad;
  for (int e = threadIdx.x; e < EX * EY; e += blockDim.x) {
    const int ty = e / EX, tx = e - ty * EX;
    const int gy = cgf_wrap(y0 - rad + ty, M, trunc), gx = cgf_wrap(x0 - rad + tx, N, trunc);
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (gy >= 0 && gx >= 0) {
      const size_t off = (size_t)gy * N + gx;
      v = make_float4(__ldg(p0 + off) - c.x, __ldg(p1 + off) - c.y, __ldg(p2 + off) - c.z,
                      __ldg(p3 + off) - c.w);
    }
    s[ty * cgf_pitch(rad) + tx] = v;
  }
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
  // add (sg = 1) or take away (sg = -1) a pixel's deviations
  GFD_D void update(float4 v, float4 g, float4 ig, float sg) {
    constexpr float kMagic = 12582912.0f;  // rounds |t| < 2^22 to an integer
    const float x[4] = {v.x, v.y, v.z, v.w};
    const float gs[4] = {g.x, g.y, g.z, g.w}, is[4] = {ig.x, ig.y, ig.z, ig.w};
    float m[4], xh[4], xl[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      m[c] = fmaf(x[c], is[c], kMagic) - kMagic;
      xh[c] = m[c] * gs[c];
      xl[c] = x[c] - xh[c];
      h[c] = fmaf(sg, m[c], h[c]);
      l[c] = fmaf(sg, xl[c], l[c]);
    }
    constexpr int qi[9] = {0, 0, 0, 1, 1, 2, 0, 1, 2}, qj[9] = {0, 1, 2, 1, 2, 2, 3, 3, 3};
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const int i = qi[q], j = qj[q];
      h[4 + q] = fmaf(sg * m[i], m[j], h[4 + q]);
      // x_i x_j - h_i h_j = x_i l_j + l_i h_j
      l[4 + q] = fmaf(sg * x[i], xl[j], fmaf(sg * xl[i], xh[j], l[4 + q]));
    }
  }
};

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

// Pass 1: window statistics and the 3 x 3 solve of Eq. 3; a (3 planes) and b.
__global__ void __launch_bounds__(CGF_THREADS, 2)
k_cgf_ab(const float* __restrict__ I, const float* __restrict__ p, int M, int N, int rad,
         float2 eps, int trunc_i, float* __restrict__ ab) {
  extern __shared__ __align__(16) unsigned char cgf_sm[];
  __shared__ float s_max[4][CGF_THREADS / 32];
  const bool trunc = trunc_i != 0;
  const int EX = CGF_TX + 2 * rad, EY = CGF_TY + 2 * rad, TP = cgf_pitch(rad);
  float4* tile = reinterpret_cast<float4*>(cgf_sm);           // [EY][TP]
  float2* rows = reinterpret_cast<float2*>(tile + TP * EY);   // [13][EY][CGF_RP]
  const size_t P = (size_t)M * N;
  const int x0 = blockIdx.x * CGF_TX, y0 = blockIdx.y * CGF_TY;
  float4 c;
  {
    const size_t o = (size_t)((y0 + CGF_TY / 2) & (M - 1)) * N + ((x0 + CGF_TX / 2) & (N - 1));
    c = make_float4(__ldg(I + o), __ldg(I + P + o), __ldg(I + 2 * P + o), __ldg(p + o));
  }
  cgf_stage(tile, I, I + P, I + 2 * P, p, c, M, N, y0, x0, rad, trunc);
  __syncthreads();
  // the tile's largest |deviation| of each plane fixes the grids
  float4 mx = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int e = threadIdx.x; e < EX * EY; e += blockDim.x) {
    const float4 v = tile[(e / EX) * TP + e % EX];
    mx = make_float4(fmaxf(mx.x, fabsf(v.x)), fmaxf(mx.y, fabsf(v.y)), fmaxf(mx.z, fabsf(v.z)),
                     fmaxf(mx.w, fabsf(v.w)));
  }
  mx = make_float4(warp_max(mx.x), warp_max(mx.y), warp_max(mx.z), warp_max(mx.w));
  if ((threadIdx.x & 31) == 0) {
    const int w = threadIdx.x >> 5;
    s_max[0][w] = mx.x;
    s_max[1][w] = mx.y;
    s_max[2][w] = mx.z;
    s_max[3][w] = mx.w;
  }
  __syncthreads();
  float4 g, ig;
  {
    float gs[4], is[4];
    const float inv = 1.0f / (float)(4096 / (2 * rad + 1) - 1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float b = 0.0f;
#pragma unroll
      for (int w = 0; w < CGF_THREADS / 32; ++w) b = fmaxf(b, s_max[q][w]);
      int e = 0;
      float f = 0.5f;
      if (b > 0.0f && b < 1e37f) f = frexpf(b * inv, &e);
      if (e < -100) e = -100;
      gs[q] = ldexpf(ceilf(8.0f * f) * 0.125f, e);  // 3-bit mantissa: g m is exact
      is[q] = 1.0f / gs[q];
    }
    g = make_float4(gs[0], gs[1], gs[2], gs[3]);
    ig = make_float4(is[0], is[1], is[2], is[3]);
  }
  // row sums: CGF_ROW neighbouring outputs of a tile row, slid
  for (int e = threadIdx.x; e < EY * (CGF_TX / CGF_ROW); e += blockDim.x) {
    const int ty = e % EY, tx = (e / EY) * CGF_ROW;
    const float4* in = tile + ty * TP + tx;
    CgfSums s;
    s.clear();
#pragma unroll 1
    for (int dx = 0; dx < 2 * rad; ++dx) s.update(in[dx], g, ig, 1.0f);
#pragma unroll 1
    for (int k = 0; k < CGF_ROW; ++k) {
      s.update(in[k + 2 * rad], g, ig, 1.0f);
#pragma unroll
      for (int q = 0; q < CGF_Q; ++q)
        rows[(q * EY + ty) * CGF_RP + tx + k] = make_float2(s.h[q], s.l[q]);
      if (k + 1 < CGF_ROW) s.update(in[k], g, ig, -1.0f);
    }
  }
  __syncthreads();
  const int tx = threadIdx.x % CGF_TX, ty0 = (threadIdx.x / CGF_TX) * CGF_COL;
  const int gx = x0 + tx;
  float2 S[CGF_Q];
#pragma unroll
  for (int q = 0; q < CGF_Q; ++q) {
    S[q] = make_float2(0.0f, 0.0f);
    const float2* rr = rows + (q * EY + ty0) * CGF_RP + tx;
    for (int dy = 0; dy < 2 * rad; ++dy) S[q] = cadd(S[q], rr[dy * CGF_RP]);
  }
#pragma unroll 1
  for (int k = 0; k < CGF_COL; ++k) {
    const int ty = ty0 + k, gy = y0 + ty;
#pragma unroll
    for (int q = 0; q < CGF_Q; ++q)
      S[q] = cadd(S[q], rows[(q * EY + ty + 2 * rad) * CGF_RP + tx]);
    if (gy < M && gx < N) {
      const float n = trunc ? (float)(cgf_count(gy, M, rad) * cgf_count(gx, N, rad))
                            : (float)((2 * rad + 1) * (2 * rad + 1));
      auto cov = [&](int q, int i, int j, float gi, float gj) {
        return cgf_cov(n, S[q].x, S[q].y, S[i].x, S[i].y, gi, S[j].x, S[j].y, gj);
      };
      // n^2 (Sigma + eps U) a = n^2 cov(I, p): eliminated in double-float
      const df en = df_mul_f(df_mul_f(df{eps.x, eps.y}, n), n);
      const df A00 = df_add(cov(4, 0, 0, g.x, g.x), en), A01 = cov(5, 0, 1, g.x, g.y);
      const df A02 = cov(6, 0, 2, g.x, g.z), A11 = df_add(cov(7, 1, 1, g.y, g.y), en);
      const df A12 = cov(8, 1, 2, g.y, g.z), A22 = df_add(cov(9, 2, 2, g.z, g.z), en);
      const df v0 = cov(10, 0, 3, g.x, g.w), v1 = cov(11, 1, 3, g.y, g.w);
      const df v2 = cov(12, 2, 3, g.z, g.w);
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
      auto mean = [&](int q, float gq, float cq) {
        const df s = two_prod(gq, S[q].x);
        const df d = df_add(s, df_make(S[q].y));  // n (mean - c)
        const float r = d.hi * inv_n;             // quotient and its residual
        const float e = fmaf(-r, n, d.hi) + d.lo;
        return df_add(df_make(cq), quick_two_sum(r, e * inv_n));
      };
      df b = mean(3, g.w, c.w);
      b = df_sub(b, df_mul(a0, mean(0, g.x, c.x)));
      b = df_sub(b, df_mul(a1, mean(1, g.y, c.y)));
      b = df_sub(b, df_mul(a2, mean(2, g.z, c.z)));
      const size_t o = (size_t)gy * N + gx;
      ab[o] = a0.hi + a0.lo;
      ab[P + o] = a1.hi + a1.lo;
      ab[2 * P + o] = a2.hi + a2.lo;
      ab[3 * P + o] = b.hi + b.lo;
    }
    if (k + 1 < CGF_COL) {
#pragma unroll
      for (int q = 0; q < CGF_Q; ++q) S[q] = csub(S[q], rows[(q * EY + ty) * CGF_RP + tx]);
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
  const float2 zero = make_float2(0.0f, 0.0f);
  for (int e = threadIdx.x; e < EY * (CGF_TX / CGF_ROW); e += blockDim.x) {
    const int ty = e % EY, tx = (e / EY) * CGF_ROW;
    const float4* in = tile + ty * TP + tx;
    CgfComp s;
    s.clear();
    auto add = [&](float4 v, float sg) {
      s.add(0, make_float2(sg * v.x, sg * v.y), zero);
      s.add(1, make_float2(sg * v.z, sg * v.w), zero);
    };
#pragma unroll 1
    for (int dx = 0; dx < 2 * rad; ++dx) add(in[dx], 1.0f);
#pragma unroll
    for (int k = 0; k < CGF_ROW; ++k) {
      add(in[k + 2 * rad], 1.0f);
#pragma unroll
      for (int i = 0; i < 2; ++i)
        rows[(i * EY + ty) * CGF_RP + tx + k] =
            make_float4(s.hi[i].x, s.hi[i].y, s.lo[i].x, s.lo[i].y);
      if (k + 1 < CGF_ROW) add(in[k], -1.0f);
    }
  }
  __syncthreads();
  const int tx = threadIdx.x % CGF_TX, ty0 = (threadIdx.x / CGF_TX) * CGF_COL;
  const int gx = x0 + tx;
  CgfComp s;
  s.clear();
  auto add = [&](int ty, float sg) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float4 v = rows[(i * EY + ty) * CGF_RP + tx];
      s.add(i, make_float2(sg * v.x, sg * v.y), make_float2(sg * v.z, sg * v.w));
    }
  };
#pragma unroll 1
  for (int dy = 0; dy < 2 * rad; ++dy) add(ty0 + dy, 1.0f);
#pragma unroll
  for (int k = 0; k < CGF_COL; ++k) {
    const int gy = y0 + ty0 + k;
    add(ty0 + k + 2 * rad, 1.0f);
    if (gy < M && gx < N) {
      const float n = trunc ? (float)(cgf_count(gy, M, rad) * cgf_count(gx, N, rad))
                            : (float)((2 * rad + 1) * (2 * rad + 1));
      const size_t o = (size_t)gy * N + gx;
      df v = quick_two_sum(s.hi[1].y, s.lo[1].y);
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[0].x, s.lo[0].x), __ldg(&I[o])));
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[0].y, s.lo[0].y), __ldg(&I[P + o])));
      v = df_add(v, df_mul_f(quick_two_sum(s.hi[1].x, s.lo[1].x), __ldg(&I[2 * P + o])));
      const float inv_n = 1.0f / n, q = v.hi * inv_n;  // v / n, rounded once
      u[o] = fmaf(fmaf(-q, n, v.hi) + v.lo, inv_n, q);
    }
    if (k + 1 < CGF_COL) add(ty0 + k, -1.0f);
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
  k_cgf_ab<<<grid, CGF_THREADS, cgf_smem1(rad), s>>>(I, p, M, N, rad, e2, trunc, ab);
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
