// Guided filter u = guidfilter(u_I, u_p, w, eps) (Sec. 2, Eq. 3-5), r = (w-1)/2,
// with periodic windows (every window holds w^2 pixels) or windows truncated
// at the canvas edge (every mean divided by the number of pixels it covers).
//
// Every warp works alone, down a strip of GFW_COLS input columns (4 per
// lane): no block barriers.  Input rows are loaded to registers one row ahead
// of use (and requested into L2 a few rows ahead); their deviations from the
// reference enter a per-warp ring in shared memory, where the row that leaves
// the windows finds them again.  Each lane touches only its own 4 columns.
// For the item's rows the warp forms, row by row,
//   1. window sums down its columns of J = I - c_I, Q = p - c_p, J^2, J Q
//      (in registers; slid from row to row, and for plain FP32 sums re-formed
//      directly every 4 rows),
//   2. window sums along the row by warp shuffles (the 2r neighbouring
//      columns come from the adjacent lanes) -> mu_k, pbar_k, sigma_k^2 and
//      the covariance -> a_k (Eq. 3), b_k (Eq. 4) for each column,
//   3. window sums of a and b down the columns (a per-warp ring of the last
//      2r+1 rows of a, b in shared memory, each lane touching only its own
//      columns), re-formed every 4 rows and slid in between,
//   4. window sums along the row by shuffles -> abar, bbar ->
//      u = abar I + bbar (Eq. 5), stored as 16-byte vectors.
// The strip's outer 4*ceil(r/2) columns on each side are halo (their sums
// are incomplete); the columns in between are the item's output, so
// neighbouring strips overlap by the halo.  Input rows and columns wrap
// periodically (truncated windows mask the wrapped ones to zero).  Window
// statistics are taken about reference values (c_I, c_p: the item's centre
// pixel): a_k and b_k do not depend on them, and the sums of J^2 and J Q are
// smaller about a nearby reference.
//
// The arithmetic of the window sums of step 1-2 is a policy (GFD_VAR_*):
// double-float running sums (every addition and product error-free), FP64
// accumulators, or plain FP32.  sigma_k^2 and the covariance are then formed
// as (n S_JJ - S_J^2) / n^2 and (n S_JQ - S_J S_Q) / n^2 in that arithmetic
// and rounded to FP32 once.
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "df.cuh"
#include "launch.h"

namespace gfd {

constexpr int GFW_COLS = 128;   // input columns per strip (4 per lane)
constexpr int GFW_SUB = 4;      // rows between direct re-formations of FP32 column sums
constexpr int GFW_WARPS = 4;    // most warps per block
constexpr int GFW_AHEAD = 4;    // input rows requested into L2 ahead of use
constexpr int GF_RMAX = 8;      // w <= 17
constexpr unsigned FULL = 0xffffffffu;

template <int RAD>
struct GfwGeom {
  static constexpr int WIN = 2 * RAD + 1;
  static constexpr int RI = WIN + 1;  // rows of the ring of deviations: the window, the row leaving
  static constexpr int HALO = 4 * ((RAD + 1) / 2);  // >= 2r, multiple of 4
  static constexpr int WOUT = GFW_COLS - 2 * HALO;  // output columns per strip
};

// per-warp shared memory: (a, b) ring of 2r+1 rows, (J, Q) ring of 2r+2 rows
GFD_HD int gfw_ring_floats(int rad) { return 2 * ((2 * rad + 1) + (2 * rad + 2)) * GFW_COLS; }
static int gfw_wout(int rad) { return GFW_COLS - 8 * ((rad + 1) / 2); }

// ---------------------------------------------------------------------------
// Window-sum arithmetic (one policy per GFD_VAR_* mode).  kSub: rows between
// direct re-formations of the column sums (the exact policies only slide).
// ---------------------------------------------------------------------------
struct SumF32 {
  static constexpr int kSub = GFW_SUB;
  float v;
  GFD_D void clear() { v = 0.0f; }
  GFD_D void add(float x) { v += x; }
  GFD_D void add_prod(float x, float y) { v = fmaf(x, y, v); }
};

struct SumF64 {
  static constexpr int kSub = 1 << 30;
  double v;
  GFD_D void clear() { v = 0.0; }
  GFD_D void add(float x) { v += (double)x; }
  GFD_D void add_prod(float x, float y) { v = fma((double)x, (double)y, v); }  // exact product
};

// hi: the FP32-rounded running sum; lo: the exact rounding errors of every
// addition (two-sum) and product (two-product), summed in FP32.
struct SumDF {
  static constexpr int kSub = 1 << 30;
  float hi, lo;
  GFD_D void clear() { hi = lo = 0.0f; }
  GFD_D void add(float x) {
    const df t = two_sum(hi, x);
    hi = t.hi;
    lo += t.lo;
  }
  GFD_D void add_prod(float x, float y) {
    const float p = x * y;
    const float e = fmaf(x, y, -p);
    const df t = two_sum(hi, p);
    hi = t.hi;
    lo += t.lo + e;
  }
};

// Split sums.  Every deviation x (J or Q) is split on a grid g chosen per item
// from a bound on |x|: x = g m + x_l with m = round(x / g), |m| <= split_max(r),
// and x_l = x - g m, both exact in FP32 (g has a 3-bit mantissa).  split_max
// keeps the window sums of m_J^2 and m_J m_Q below 2^24, so the sums of m,
// m_J^2 and m_J m_Q are exact in FP32; n S_mm - S_m^2 and n S_mJmQ - S_mJ S_mQ
// follow with one rounding (the square's error comes from an FMA).  The
// remainders' parts, x_l, J^2 - (g_J m_J)^2 = J J_l + J_l g_J m_J and
// J Q - g_J m_J g_Q m_Q = J Q_l + J_l g_Q m_Q, are summed in FP32, where
// their rounding is about 1 / (2 split_max) of that of plain sums.
// Everything comes in pairs (J, Q), one packed FP32 instruction per pair, in
// the register pairs that the ring's rows load; mixing int32 and FP32 halves
// cost 10 % more instructions.  What bounds the kernel now: over a 4096 x 4096
// image, w = 9 (138 us), the FMA pipe is busy 48 % of the cycles, the data path of
// shared memory and shuffles 55 %, issue 48 %, DRAM 17 %, with 8 to 12 warps per SM
// (rows per item, registers, rings) to overlap them; the wait between dependent
// packed operations is the top stall.  Launches of few items are at 20 to 45 %.  Per
// batched solve of 256 images 14.7 -> 12.2 ms, of which 1.3 by the choice of
// rows per item (gfw_rows).  Fewer registers (128: spills) took 15.3 ms; leaving
// rows re-read through L1 instead of the ring 16.7 ms.
struct SumIG {
  static constexpr int kSub = 1 << 30;
};

GFD_D bool is_finite(float v) { return fabsf(v) <= 3.402823466e38f; }  // false for NaN

// The grids of one item: g and 1/g for (J, Q).
struct IGGrid {
  float2 g, ig;
};

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds |v| < 2^22 to an integer

// Largest |m| of the split for windows of radius r: (2r+1)^2 m^2 <= 2^24.
constexpr int split_max(int rad) {
  const long long n = (long long)(2 * rad + 1) * (2 * rad + 1);
  int m = 2048;
  while (n * m * m > (1LL << 24)) --m;
  return m;
}

static_assert(split_max(2) == 819 && split_max(3) == 585 && split_max(4) == 455 &&
                  split_max(8) == 240 && split_max(0) == 2048,
              "split range per window radius");

// The smallest g with a 3-bit mantissa and bound / g <= split_max - 1.
template <int RAD>
GFD_D void ig_grid(float bound, float& g, float& ig) {
  int e = 0;
  float f = 0.5f;
  if (bound > 0.0f && bound < 1e37f) f = frexpf(bound * (1.0f / (split_max(RAD) - 1)), &e);
  if (e < -100) e = -100;
  g = ldexpf(ceilf(8.0f * f) * 0.125f, e);
  ig = 1.0f / g;
}

// Value of lane (lane + off) (compile-time offset after unrolling).
template <class T>
GFD_D T lane_shift(T v, int off) {
  if (off > 0) return __shfl_down_sync(FULL, v, off);
  if (off < 0) return __shfl_up_sync(FULL, v, -off);
  return v;
}

// e[q] = the value of strip column 4*lane + q - RAD, q < 2 RAD + 4, gathered
// from v[k] = column 4*lane + k of every lane.  Columns beyond the warp's
// edges are not available: lanes within RAD columns of an edge get values
// of other columns (those lanes' sums are halo and never used).
template <int RAD, class T>
GFD_D void gather_row(const T (&v)[4], T (&e)[2 * RAD + 4]) {
#pragma unroll
  for (int q = 0; q < 2 * RAD + 4; ++q) {
    const int c = q - RAD;                           // column offset from 4*lane
    const int lo = c >= 0 ? c / 4 : -((3 - c) / 4);  // floor(c / 4): source lane offset
    e[q] = lane_shift(v[c - 4 * lo], lo);
  }
}

// Window sums of radius RAD along the strip: s[k] = sum of columns
// 4*lane + k - RAD .. 4*lane + k + RAD.
template <int RAD, class T>
GFD_D void row_sums(const T (&e)[2 * RAD + 4], T (&s)[4]) {
  T acc = e[0];
#pragma unroll
  for (int q = 1; q <= 2 * RAD; ++q) acc += e[q];
  s[0] = acc;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    acc += e[k + 2 * RAD] - e[k - 1];
    s[k] = acc;
  }
}

template <int RAD, class T>
GFD_D void hsum4_scalar(const T (&v)[4], T (&s)[4]) {
  T e[2 * RAD + 4];
  gather_row<RAD>(v, e);
  row_sums<RAD>(e, s);
}

template <int RAD>
GFD_D void hsum4(const SumF32 (&v)[4], SumF32 (&s)[4]) {
  const float in[4] = {v[0].v, v[1].v, v[2].v, v[3].v};
  float out[4];
  hsum4_scalar<RAD>(in, out);
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k].v = out[k];
}

template <int RAD>
GFD_D void hsum4(const SumF64 (&v)[4], SumF64 (&s)[4]) {
  const double in[4] = {v[0].v, v[1].v, v[2].v, v[3].v};
  double out[4];
  hsum4_scalar<RAD>(in, out);
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k].v = out[k];
}

// Double-float: the hi parts are added with two-sums (errors kept), the lo
// parts (already the errors of the column sums) plainly.
template <int RAD>
GFD_D void hsum4(const SumDF (&v)[4], SumDF (&s)[4]) {
  constexpr int E = 2 * RAD + 4;
  const float vh[4] = {v[0].hi, v[1].hi, v[2].hi, v[3].hi};
  const float vl[4] = {v[0].lo, v[1].lo, v[2].lo, v[3].lo};
  float eh[E], el[E];
  gather_row<RAD>(vh, eh);
  gather_row<RAD>(vl, el);
  float hi = eh[0], err = 0.0f, lo = el[0];
#pragma unroll
  for (int q = 1; q <= 2 * RAD; ++q) {
    const df t = two_sum(hi, eh[q]);
    hi = t.hi;
    err += t.lo;
    lo += el[q];
  }
  s[0].hi = hi;
  s[0].lo = err + lo;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    df t = two_sum(hi, eh[k + 2 * RAD]);
    err += t.lo;
    t = two_sum(t.hi, -eh[k - 1]);
    hi = t.hi;
    err += t.lo;
    lo += el[k + 2 * RAD] - el[k - 1];
    s[k].hi = hi;
    s[k].lo = err + lo;
  }
}

// Means and (co)variance of a window of n pixels from S = (sum J, sum Q,
// sum J^2, sum J Q):  var = (n S_JJ - S_J^2) / n^2 (sigma_k^2, the
// population variance), cov = (n S_JQ - S_J S_Q) / n^2.
GFD_D void window_stats(const SumF32& s0, const SumF32& s1, const SumF32& s2, const SumF32& s3,
                        float n, float inv_n, const IGGrid&, float& mJ, float& mQ, float& var,
                        float& cov) {
  (void)n;
  mJ = s0.v * inv_n;
  mQ = s1.v * inv_n;
  var = fmaf(-mJ, mJ, s2.v * inv_n);
  cov = fmaf(-mJ, mQ, s3.v * inv_n);
}

GFD_D void window_stats(const SumF64& s0, const SumF64& s1, const SumF64& s2, const SumF64& s3,
                        float n, float inv_n, const IGGrid&, float& mJ, float& mQ, float& var,
                        float& cov) {
  (void)inv_n;
  const double nn = (double)n, inv2 = 1.0 / (nn * nn);
  mJ = (float)(s0.v / nn);
  mQ = (float)(s1.v / nn);
  var = (float)(fma(nn, s2.v, -s0.v * s0.v) * inv2);
  cov = (float)(fma(nn, s3.v, -s0.v * s1.v) * inv2);
}

GFD_D void window_stats(const SumDF& s0, const SumDF& s1, const SumDF& s2, const SumDF& s3,
                        float n, float inv_n, const IGGrid&, float& mJ, float& mQ, float& var,
                        float& cov) {
  const df S0{s0.hi, s0.lo}, S1{s1.hi, s1.lo}, S2{s2.hi, s2.lo}, S3{s3.hi, s3.lo};
  const df v = df_sub(df_mul_f(S2, n), df_mul(S0, S0));
  const df c = df_sub(df_mul_f(S3, n), df_mul(S0, S1));
  const float inv2 = inv_n * inv_n;
  mJ = (s0.hi + s0.lo) * inv_n;
  mQ = (s1.hi + s1.lo) * inv_n;
  var = (v.hi + v.lo) * inv2;
  cov = (c.hi + c.lo) * inv2;
}

// Column-sum update by one input row's deviations (sign +1: the row enters,
// -1: it leaves).
template <class ACC>
GFD_D void col_update(ACC (&V)[4][4], const float (&J)[4], const float (&Q)[4], float sgn,
                      const IGGrid&) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    V[0][k].add(sgn * J[k]);
    V[1][k].add(sgn * Q[k]);
    V[2][k].add_prod(sgn * J[k], J[k]);
    V[3][k].add_prod(sgn * J[k], Q[k]);
  }
}

template <class ACC>
GFD_D void col_clear(ACC (&V)[4][4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) V[q][k].clear();
}
// Row window sums of a pair of quantities (single shuffles, packed additions).
template <int RAD>
GFD_D void hsum4_pair(const float2 (&v)[4], float2 (&s)[4]) {
  float2 e[2 * RAD + 4];
#pragma unroll
  for (int q = 0; q < 2 * RAD + 4; ++q) {
    const int c = q - RAD;
    const int lo = c >= 0 ? c / 4 : -((3 - c) / 4);
    e[q] = make_float2(lane_shift(v[c - 4 * lo].x, lo), lane_shift(v[c - 4 * lo].y, lo));
  }
  float2 acc = e[0];
#pragma unroll
  for (int q = 1; q <= 2 * RAD; ++q) acc = cadd(acc, e[q]);
  s[0] = acc;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    acc = cadd(acc, csub(e[k + 2 * RAD], e[k - 1]));
    s[k] = acc;
  }
}

// The window sums down the strip's columns of one lane and what a row needs of
// them: the means of J and Q, sigma_k^2 and the covariance of the lane's four
// windows.
template <int RAD, class ACC>
struct GfwCols {  // one accumulator per quantity and column
  ACC V[4][4];    // [J, Q, J^2, J Q][column]
  GFD_D void clear() { col_clear(V); }
  GFD_D void update(const float2 (&x)[4], float sgn, const IGGrid& G) {
    const float j[4] = {x[0].x, x[1].x, x[2].x, x[3].x};
    const float q[4] = {x[0].y, x[1].y, x[2].y, x[3].y};
    col_update(V, j, q, sgn, G);
  }
  // whether no column sum holds (or still holds, slid) a value that is not finite
  GFD_D bool finite() const {
    if constexpr (std::is_same<ACC, SumF64>::value) {
      const double t = (V[2][0].v + V[2][1].v) + (V[2][2].v + V[2][3].v) + (V[3][0].v + V[3][1].v) +
                       (V[3][2].v + V[3][3].v);
      return t - t == 0.0;
    } else if constexpr (std::is_same<ACC, SumDF>::value) {
      return is_finite((V[2][0].lo + V[2][1].lo) + (V[2][2].lo + V[2][3].lo) +
                       (V[3][0].lo + V[3][1].lo) + (V[3][2].lo + V[3][3].lo));
    } else {
      return true;  // re-formed every few rows
    }
  }
  template <class F>
  GFD_D void windows(const float (&n)[4], const float (&inv_n)[4], const IGGrid& G, F out) const {
    ACC S0[4], S1[4], S2[4], S3[4];
    hsum4<RAD>(V[0], S0);
    hsum4<RAD>(V[1], S1);
    hsum4<RAD>(V[2], S2);
    hsum4<RAD>(V[3], S3);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      float mJ, mQ, var, cov;
      window_stats(S0[k], S1[k], S2[k], S3[k], n[k], inv_n[k], G, mJ, mQ, var, cov);
      out(k, mJ, mQ, var, cov);
    }
  }
};

// Split sums, in pairs.
template <int RAD>
struct GfwCols<RAD, SumIG> {
  float2 h01[4], h23[4];  // (m_J, m_Q), (m_J^2, m_J m_Q) per column, exact
  float2 l01[4], l23[4];  // the remainders' parts
  GFD_D void clear() {
#pragma unroll
    for (int k = 0; k < 4; ++k) h01[k] = h23[k] = l01[k] = l23[k] = make_float2(0.0f, 0.0f);
  }
  // one input row's deviations enter (sgn 1) or leave (sgn -1; a constant)
  GFD_D void update(const float2 (&x)[4], float sgn, const IGGrid& G) {
    const float2 mag = make_float2(kMagic, kMagic);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 m = csub(__ffma2_rn(x[k], G.ig, mag), mag);
      const float2 xh = __fmul2_rn(m, G.g);
      const float2 xl = csub(x[k], xh);
      const float sm = sgn * m.x, sx = sgn * x[k].x, sl = sgn * xl.x;
      h01[k] = sgn > 0.0f ? cadd(h01[k], m) : csub(h01[k], m);
      h23[k] = __ffma2_rn(make_float2(sm, sm), m, h23[k]);
      l01[k] = sgn > 0.0f ? cadd(l01[k], xl) : csub(l01[k], xl);
      l23[k] = __ffma2_rn(make_float2(sx, sx), xl, __ffma2_rn(make_float2(sl, sl), xh, l23[k]));
    }
  }
  GFD_D bool finite() const {
    const float2 t = cadd(cadd(l23[0], l23[1]), cadd(l23[2], l23[3]));
    return is_finite(t.x + t.y);
  }
  template <class F>
  GFD_D void windows(const float (&n)[4], const float (&inv_n)[4], const IGGrid& G, F out) const {
    float2 S01[4], S23[4], L01[4], L23[4];
    hsum4_pair<RAD>(h01, S01);
    hsum4_pair<RAD>(h23, S23);
    hsum4_pair<RAD>(l01, L01);
    hsum4_pair<RAD>(l23, L23);
    const float2 gg = make_float2(G.g.x * G.g.x, G.g.x * G.g.y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 sJ = make_float2(S01[k].x, S01[k].x), n2 = make_float2(n[k], n[k]);
      // (n S_mm - S_m^2, n S_mJmQ - S_mJ S_mQ): p + e the exact products
      const float2 p = __fmul2_rn(sJ, S01[k]), pn = make_float2(-p.x, -p.y);
      const float2 e = __ffma2_rn(sJ, S01[k], pn);
      const float2 D = csub(__ffma2_rn(n2, S23[k], pn), e);
      const float2 hh = __fmul2_rn(G.g, S01[k]);  // (g_J sum m_J, g_Q sum m_Q)
      const float2 t = __ffma2_rn(hh, make_float2(2.0f, 1.0f), L01[k]);  // 2 h_J + l_J, h_Q + l_Q
      const float2 c = __fmul2_rn(t, make_float2(L01[k].x, L01[k].x));
      const float2 lo = __ffma2_rn(n2, L23[k], make_float2(-c.x, -fmaf(hh.x, L01[k].y, c.y)));
      const float2 m = cscale(cadd(hh, L01[k]), inv_n[k]);
      const float2 vc = cscale(__ffma2_rn(gg, D, lo), inv_n[k] * inv_n[k]);
      out(k, m.x, m.y, vc.x, vc.y);
    }
  }
};

// Pixels of the window of radius RAD about position x in [0, L) that lie in
// [0, L) (truncated windows).
GFD_D int window_count(int x, int L, int RAD) {
  const int a = x - RAD < 0 ? 0 : x - RAD;
  const int b = x + RAD > L - 1 ? L - 1 : x + RAD;
  return b - a + 1;
}

// 1/n for small integers n as floats, the correctly rounded quotient.
GFD_D float rcp_count(float n) {
  const float q = __fdividef(1.0f, n);
  return fmaf(fmaf(-n, q, 1.0f), q, q);
}

template <int RAD, class ACC, bool TRUNC>
GFD_D void gfw_items(const ClassDesc& cd, const ImgDesc* __restrict__ imgs, ImgState* st,
                     int iter, bool shifted, int rows, float* ring, int gwarp, int nwarps) {
  using G = GfwGeom<RAD>;
  constexpr int WIN = G::WIN, HALO = G::HALO, WOUT = G::WOUT, RI = G::RI;
  const int lane = threadIdx.x & 31;
  const int M = cd.M, N = cd.N;
  const int strips = (N + WOUT - 1) / WOUT;
  const int per_img = strips * ((M + rows - 1) / rows);
  const int n_items = cd.n_img * per_img;
  const float n_full = (float)(WIN * WIN);
  const float inv_full = 1.0f / n_full;
  // rings of rows of (a, b) and of (J, Q): this lane's columns 0, 1 of a row at
  // [row], columns 2, 3 half a row on, as (x0, y0, x1, y1)
  float4* const rab = reinterpret_cast<float4*>(ring) + lane;
  constexpr int ROW = GFW_COLS / 2, HALF = ROW / 2;  // float4 per ring row
  float4* const rjq = rab + WIN * ROW;
  // this lane's columns lie in the strip's output part
  const bool out_lane = 4 * lane >= HALO && 4 * lane < HALO + WOUT;

  for (int item = gwarp; item < n_items; item += nwarps) {
    const int li = item / per_img, rem = item - li * per_img;
    const int y0 = (rem / strips) * rows, x0 = (rem % strips) * WOUT;
    const int H = rows < M - y0 ? rows : M - y0;
    const int gi = cd.img0 + li;
    const ImgDesc& d = imgs[gi];
    const float* __restrict__ I = d.uI;
    const float* __restrict__ P = d.up;
    const float* uo = (iter >= 0 && d.isnr_out) ? d.uo : nullptr;
    // this lane's 4 columns (16-byte aligned: x0 and HALO are multiples of 4)
    const int xs = x0 - HALO + 4 * lane;  // unwrapped column of the lane's first value
    const int gx = xs & (N - 1);
    const bool store = out_lane && x0 + 4 * lane - HALO < N;
    // truncated windows: columns outside the canvas hold zero, and every
    // window's pixel count along the row
    float cmask[4] = {1.0f, 1.0f, 1.0f, 1.0f}, ncol[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if constexpr (TRUNC) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int x = xs + k;
        const bool in = x >= 0 && x < N;
        cmask[k] = in ? 1.0f : 0.0f;
        ncol[k] = in ? (float)window_count(x, N, RAD) : 1.0f;
      }
    }
    float cI = 0.0f, cP = 0.0f;
    if (shifted) {
      const size_t c = (size_t)((y0 + H / 2) & (M - 1)) * N + ((x0 + WOUT / 2) & (N - 1));
      cI = __ldg(&I[c]);
      cP = __ldg(&P[c]);
      if (!is_finite(cI)) cI = 0.0f;
      if (!is_finite(cP)) cP = 0.0f;
    }
    const float eps = (float)d.eps;
    IGGrid G{};
    if constexpr (std::is_same<ACC, SumIG>::value) {
      // |J| <= max |u_I| + |c_I| (the bound the inverse row pass recorded)
      const ImgState* S = st + gi;
      ig_grid<RAD>(__uint_as_float(__ldcg(&S->absmax[0])) + fabsf(cI), G.g.x, G.ig.x);
      ig_grid<RAD>(__uint_as_float(__ldcg(&S->absmax[1])) + fabsf(cP), G.g.y, G.ig.y);
    }
    // input row j of the item is image row y0 - 2r + j; it stays in ring slot
    // j % RI until row j + RI enters
    const int nin = H + 4 * RAD;
    auto row_off = [&](int j) { return (unsigned)((y0 - 2 * RAD + j) & (M - 1)) * N + gx; };
    auto load = [&](int j, float4& vi, float4& vp) {
      const unsigned off = row_off(j);
      vi = __ldcg(reinterpret_cast<const float4*>(I + off));
      vp = __ldcg(reinterpret_cast<const float4*>(P + off));
    };
    const float2 cc = make_float2(cI, cP);
    // deviations of input row j about the references (zero outside the canvas
    // for truncated windows), also put into ring slot `slot`
    auto enter = [&](int j, int slot, const float4& vi, const float4& vp, float2 (&x)[4]) {
      x[0] = csub(make_float2(vi.x, vp.x), cc);
      x[1] = csub(make_float2(vi.y, vp.y), cc);
      x[2] = csub(make_float2(vi.z, vp.z), cc);
      x[3] = csub(make_float2(vi.w, vp.w), cc);
      if constexpr (TRUNC) {
        const int yy = y0 - 2 * RAD + j;
        const float rm = (yy >= 0 && yy < M) ? 1.0f : 0.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = cscale(x[k], rm * cmask[k]);
      }
      rjq[slot * ROW] = make_float4(x[0].x, x[0].y, x[1].x, x[1].y);
      rjq[slot * ROW + HALF] = make_float4(x[2].x, x[2].y, x[3].x, x[3].y);
    };
    auto ring_row = [&](int slot, float2 (&x)[4]) {
      const float4 u = rjq[slot * ROW], v = rjq[slot * ROW + HALF];
      x[0] = make_float2(u.x, u.y);
      x[1] = make_float2(u.z, u.w);
      x[2] = make_float2(v.x, v.y);
      x[3] = make_float2(v.z, v.w);
    };
    GfwCols<RAD, ACC> V;
    float2 VA[4];  // (a, b) per column: window sums down the columns
#pragma unroll
    for (int k = 0; k < 4; ++k) VA[k] = make_float2(0.0f, 0.0f);
    float err = 0.0f;
    // the first window's rows but one go to the ring; the next row waits in
    // registers
    float4 nI, nP;
    load(0, nI, nP);
    for (int j = 0; j < 2 * RAD; ++j) {
      float2 x[4];
      const float4 vi = nI, vp = nP;
      load(j + 1, nI, nP);
      enter(j, j, vi, vp, x);
    }
    float2 old[4];  // row s - 1: the guidance of output row s - 1 - 2r, leaving at step s
    // ring slots of input rows s and s + 2r and of stats row s
    int s_cur = 0, s_new = 2 * RAD, s_ab = 0;
    // stats row s (image row y0 - r + s) has its column window on input rows
    // j = s .. s + 2r; output row t = s - 2r needs stats rows t .. t + 2r
    for (int s = 0; s < H + 2 * RAD; ++s) {
      const int t = s - 2 * RAD;  // output row (if >= 0)
      // the reference row of the ISNR sums is requested early (used last)
      float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (uo && store && t >= 0)
        g = __ldg(reinterpret_cast<const float4*>(uo + (size_t)((y0 + t) & (M - 1)) * N + gx));
      float2 x[4];
      enter(s + 2 * RAD, s_new, nI, nP, x);
      if (s + 1 < H + 2 * RAD) load(s + 2 * RAD + 1, nI, nP);
      if (s + 2 * RAD + GFW_AHEAD < nin && (lane & 7) == 0) {  // one request per 128 bytes
        const unsigned off = row_off(s + 2 * RAD + GFW_AHEAD);
        asm volatile("prefetch.global.L2 [%0];" ::"l"(I + off));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(P + off));
      }
      bool direct = s % ACC::kSub == 0;
      if (!direct) {
        V.update(x, 1.0f, G);
        V.update(old, -1.0f, G);
        // A pixel that is not finite cannot be taken away again.  (Only planes of
        // the caller's own can have one here and there.)
        if (iter < 0 && !V.finite()) direct = true;
      }
      if (direct) {
        V.clear();
        int slot = s_cur;
#pragma unroll(ACC::kSub < 1000 ? WIN : 1)
        for (int dd = 0; dd < WIN; ++dd) {
          float2 y[4];
          ring_row(slot, y);
          V.update(y, 1.0f, G);
          slot = slot + 1 == RI ? 0 : slot + 1;
        }
      }
      ring_row(s_cur, old);
      // 2. row window sums -> a_k (Eq. 3), b_k (Eq. 4)
      float n[4], inv_n[4];
      float srow_mask = 1.0f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        n[k] = n_full;
        inv_n[k] = inv_full;
      }
      if constexpr (TRUNC) {
        const int ys = y0 - RAD + s;
        const bool in = ys >= 0 && ys < M;
        srow_mask = in ? 1.0f : 0.0f;
        const float nrow = in ? (float)window_count(ys, M, RAD) : 1.0f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          n[k] = nrow * ncol[k];
          inv_n[k] = rcp_count(n[k]);
        }
      }
      float A[4], B[4];
      V.windows(n, inv_n, G, [&](int k, float mJ, float mQ, float var, float cov) {
        A[k] = __fdividef(cov, var + eps);  // var + eps >= eps > 0
        // b_k about the references: b_k = B_k + c_p - a_k c_I (Eq. 4), and the
        // constant parts are restored in the output below
        B[k] = fmaf(-A[k], mJ, mQ);
        if constexpr (TRUNC) {  // windows centred outside the canvas do not exist
          const float m = srow_mask * cmask[k];
          A[k] *= m;
          B[k] *= m;
        }
      });
      // 3. ring slot s % WIN holds stats row s - WIN until overwritten here
      const bool slide = t > 0 && t % GFW_SUB != 0;
      if (slide) {
        const float4 u = rab[s_ab * ROW], v = rab[s_ab * ROW + HALF];
        VA[0] = cadd(VA[0], csub(make_float2(A[0], B[0]), make_float2(u.x, u.y)));
        VA[1] = cadd(VA[1], csub(make_float2(A[1], B[1]), make_float2(u.z, u.w)));
        VA[2] = cadd(VA[2], csub(make_float2(A[2], B[2]), make_float2(v.x, v.y)));
        VA[3] = cadd(VA[3], csub(make_float2(A[3], B[3]), make_float2(v.z, v.w)));
      }
      rab[s_ab * ROW] = make_float4(A[0], B[0], A[1], B[1]);
      rab[s_ab * ROW + HALF] = make_float4(A[2], B[2], A[3], B[3]);
      s_cur = s_cur + 1 == RI ? 0 : s_cur + 1;
      s_new = s_new + 1 == RI ? 0 : s_new + 1;
      s_ab = s_ab + 1 == WIN ? 0 : s_ab + 1;
      if (t < 0) continue;
      if (!slide) {  // direct: the ring holds stats rows t .. t + 2r
#pragma unroll
        for (int k = 0; k < 4; ++k) VA[k] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int q = 0; q < WIN; ++q) {
          const float4 u = rab[q * ROW], v = rab[q * ROW + HALF];
          VA[0] = cadd(VA[0], make_float2(u.x, u.y));
          VA[1] = cadd(VA[1], make_float2(u.z, u.w));
          VA[2] = cadd(VA[2], make_float2(v.x, v.y));
          VA[3] = cadd(VA[3], make_float2(v.z, v.w));
        }
      }
      // 4. row window sums of a, b -> u = abar I + bbar (Eq. 5); the guidance
      //    at output row t is input row j = t + 2r = s.  With b_k = B_k + c_p
      //    - a_k c_I, u = abar (I - c_I) + Bbar + c_p: no large terms cancel
      //    where I and p are large (small lambda amplifies noise in them)
      float2 SAB[4];
      hsum4_pair<RAD>(VA, SAB);
      float nout = 0.0f;
      if constexpr (TRUNC) nout = (float)window_count(y0 + t, M, RAD);
      float o[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float in = inv_full;
        if constexpr (TRUNC) in = rcp_count(nout * ncol[k]);
        o[k] = fmaf(fmaf(SAB[k].x, old[k].x, SAB[k].y), in, cP);
      }
      if (store) {
        const size_t off = (size_t)((y0 + t) & (M - 1)) * N + gx;
        *reinterpret_cast<float4*>(d.u + off) = make_float4(o[0], o[1], o[2], o[3]);
        if (uo) {
          const float e0 = o[0] - g.x, e1 = o[1] - g.y, e2 = o[2] - g.z, e3 = o[3] - g.w;
          err = fmaf(e0, e0, fmaf(e1, e1, fmaf(e2, e2, fmaf(e3, e3, err))));
        }
      }
    }
    if (uo) {
      // ||u - u_orig||^2 of this item: FP32 in the warp, FP64 across items
      err = warp_sum(err);
      if (lane == 0) {
        ImgState* S = st + gi;
        atomicAdd(&S->err2, (double)err);
        __threadfence();
        const unsigned int prev = atomicAdd(&S->gf_done, 1u);
        if (prev == (unsigned)per_img - 1) {
          __threadfence();
          const double e2 = __ldcg(&S->err2);
          d.isnr_out[iter] = 10.0 * log10(S->den_isnr / e2);
          S->err2 = 0.0;
          S->gf_done = 0;
          __threadfence();
        }
      }
    }
    __syncwarp();
  }
}

// One kernel per window radius: its registers and code are those of the radius.
template <int RAD, class ACC, bool TRUNC>
__global__ void __launch_bounds__(GFW_WARPS * 32)
k_guided_filter(ClassDesc cd, const ImgDesc* __restrict__ imgs, const __grid_constant__ ImgDesc one,
                ImgState* st, int iter, int shifted, int H) {
  extern __shared__ __align__(16) float gsm[];
  const int warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  gfw_items<RAD, ACC, TRUNC>(cd, imgs ? imgs : &one, st, iter, shifted != 0, H,
                             gsm + (size_t)warp * gfw_ring_floats(RAD), blockIdx.x * W + warp,
                             gridDim.x * W);
}

static int gf_sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
  }
  return n;
}

using GfKernel = void (*)(ClassDesc, const ImgDesc*, const ImgDesc, ImgState*, int, int, int);

template <int RAD>
static GfKernel gf_kernel_rad(int var_mode, bool tr) {
  switch (var_mode) {
    case GFD_VAR_FP64:
      return tr ? k_guided_filter<RAD, SumF64, true> : k_guided_filter<RAD, SumF64, false>;
    case GFD_VAR_FP32:
    case GFD_VAR_FP32_RAW:
      return tr ? k_guided_filter<RAD, SumF32, true> : k_guided_filter<RAD, SumF32, false>;
    case GFD_VAR_DOUBLE_FLOAT:
      return tr ? k_guided_filter<RAD, SumDF, true> : k_guided_filter<RAD, SumDF, false>;
    default: return tr ? k_guided_filter<RAD, SumIG, true> : k_guided_filter<RAD, SumIG, false>;
  }
}

static GfKernel gf_kernel(int var_mode, int boundary, int rad) {
  const bool tr = boundary == GFD_BOUNDARY_TRUNCATED;
  switch (rad) {
    case 0: return gf_kernel_rad<0>(var_mode, tr);
    case 1: return gf_kernel_rad<1>(var_mode, tr);
    case 2: return gf_kernel_rad<2>(var_mode, tr);
    case 3: return gf_kernel_rad<3>(var_mode, tr);
    case 4: return gf_kernel_rad<4>(var_mode, tr);
    case 5: return gf_kernel_rad<5>(var_mode, tr);
    case 6: return gf_kernel_rad<6>(var_mode, tr);
    case 7: return gf_kernel_rad<7>(var_mode, tr);
    default: return gf_kernel_rad<GF_RMAX>(var_mode, tr);
  }
}

// Largest |I| and |p| of one image into ImgState::absmax (the bound of the
// split sums when no inverse row pass has recorded it).  Every block leaves its
// maxima in the scratch; the last one to finish (a counter, reset for the next
// call) reduces them, so no launch has to clear anything first.  Bound by DRAM:
// each thread keeps 8 independent 16-byte loads in flight.
__global__ void __launch_bounds__(512)
k_plane_absmax(const float* __restrict__ I, const float* __restrict__ p, int P4, ImgState* st,
               unsigned int* __restrict__ scratch) {
  __shared__ float s_m[2][16];
  __shared__ bool s_last;
  const float4* I4 = reinterpret_cast<const float4*>(I);
  const float4* p4 = reinterpret_cast<const float4*>(p);
  // (values that are not finite have no part in it: fmaxf passes over NaN)
  auto top1 = [](float m, float v) { return is_finite(v) ? fmaxf(m, fabsf(v)) : m; };
  auto top = [&](float m, float4 v) { return top1(top1(top1(top1(m, v.x), v.y), v.z), v.w); };
  float mi = 0.0f, mp = 0.0f;
  const int step = gridDim.x * blockDim.x;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  for (; i + 3 * step < P4; i += 4 * step) {
    float4 a[4], b[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] = __ldg(&I4[i + k * step]);
      b[k] = __ldg(&p4[i + k * step]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      mi = top(mi, a[k]);
      mp = top(mp, b[k]);
    }
  }
  for (; i < P4; i += step) {
    mi = top(mi, __ldg(&I4[i]));
    mp = top(mp, __ldg(&p4[i]));
  }
  mi = warp_max(mi);
  mp = warp_max(mp);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s_m[0][warp] = mi;
    s_m[1][warp] = mp;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < num_warps(); ++w) {
      mi = fmaxf(mi, s_m[0][w]);
      mp = fmaxf(mp, s_m[1][w]);
    }
    scratch[2 * blockIdx.x] = __float_as_uint(mi);
    scratch[2 * blockIdx.x + 1] = __float_as_uint(mp);
    __threadfence();
    s_last = atomicAdd(&scratch[2 * ABSMAX_BLOCKS], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  __threadfence();
  float m[2] = {0.0f, 0.0f};
  for (int q = lane; q < (int)gridDim.x; q += 32) {
    m[0] = fmaxf(m[0], __uint_as_float(__ldcg(&scratch[2 * q])));
    m[1] = fmaxf(m[1], __uint_as_float(__ldcg(&scratch[2 * q + 1])));
  }
  m[0] = warp_max(m[0]);
  m[1] = warp_max(m[1]);
  if (lane == 0) {
    st->absmax[0] = __float_as_uint(m[0]);
    st->absmax[1] = __float_as_uint(m[1]);
    scratch[2 * ABSMAX_BLOCKS] = 0u;
  }
}

cudaError_t launch_plane_absmax(const ClassLaunch& c, unsigned int* scratch, cudaStream_t s) {
  const int P4 = c.cd.M * c.cd.N / 4;
  int blocks = (P4 + 512 * 4 - 1) / (512 * 4);
  if (blocks > ABSMAX_BLOCKS) blocks = ABSMAX_BLOCKS;
  k_plane_absmax<<<blocks, 512, 0, s>>>(c.one->uI, c.one->up, P4, c.st, scratch);
  return cudaGetLastError();
}

// Rows per item (any number; the last item of a strip may have fewer).  A warp
// takes H + 2r + a few row steps for its H output rows; alone on its scheduler a
// step takes about twice its issue time (dependent latencies), so warps up to
// two per scheduler are free and more share it.  Candidates fill one, two, ...
// warps per scheduler and then whole waves of the resident warps, so that no
// wave is left nearly empty: one 4096 x 4096 image, w = 9, has 37 strips, whose
// 64-row items make 1.3 waves.  Few items are cut down to 4 rows to spread over
// the GPU (one 256 x 256 image, w = 7: 20 us with 16 rows, 12 us).
static int gfw_rows(int M, int hmax, int rad, int images, int strips, int resident, int scheds) {
  const long long per_row = (long long)images * strips;
  int best = 0;
  double best_t = 0.0;
  for (int c = 1; c <= 12; ++c) {
    const int per_sched = resident / scheds < 1 ? 1 : resident / scheds;
    const long long target = c < per_sched ? (long long)c * scheds
                                           : (long long)(c - per_sched + 1) * resident;
    long long nb = target / per_row;
    if (nb < 1) nb = 1;
    if (nb > M / 4) nb = M / 4;
    int H = (int)((M + nb - 1) / nb);
    if (H > hmax) H = hmax;
    nb = (M + H - 1) / H;
    const long long items = per_row * nb, active = items < resident ? items : resident;
    const double waves = (double)((items + resident - 1) / resident);
    const double share = (double)((active + scheds - 1) / scheds);
    const double t = waves * (H + 2 * rad + 2 + 0.5 * rad) * (share > 2.0 ? share : 2.0);
    if (best == 0 || t < best_t) {
      best = H;
      best_t = t;
    }
  }
  return best;
}

// Warps per block and resident blocks per SM of a kernel.  Wide windows' rings
// leave room for fewer warps per SM than whole blocks of GFW_WARPS would use:
// blocks shrink to the size that keeps most warps resident (w = 17: 6 instead
// of 4).  The answer is a property of the kernel, looked up once (threads that
// race on the first call store the same value).
static void gfw_block(GfKernel kern, int var_mode, int boundary, int rad, int& W, int& per_sm) {
  static std::atomic<int> known[5][2][GF_RMAX + 1];
  std::atomic<int>& k = known[var_mode][boundary][rad];
  int v = k.load(std::memory_order_relaxed);
  if (v == 0) {
    int bw = GFW_WARPS, bn = 0;
    for (int w = GFW_WARPS; w >= 1; w /= 2) {
      int n = 0;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
              &n, kern, w * 32, (size_t)w * gfw_ring_floats(rad) * sizeof(float)) != cudaSuccess)
        n = 0;
      if (n * w > bn * bw) {
        bw = w;
        bn = n;
      }
    }
    v = bw * 256 + (bn < 1 ? 1 : bn);
    if (bn >= 1) k.store(v, std::memory_order_relaxed);
  }
  W = v >> 8;
  per_sm = v & 255;
}

// One launch per window radius present in the class (the images of a class
// are ordered by radius, so each group is a contiguous range).  Items are
// (image, strip, block of H rows).
cudaError_t launch_guided_filter(const ClassLaunch& c, int iter, int var_mode, int boundary,
                                 cudaStream_t s) {
  const int shifted = var_mode == GFD_VAR_FP32_RAW ? 0 : 1;
  for (int g = 0; g < c.n_rad_groups; ++g) {
    const RadGroup& rg = c.rad_groups[g];
    const GfKernel kern = gf_kernel(var_mode, boundary, rg.rad);
    ClassDesc cd = c.cd;
    cd.img0 = rg.img0;
    cd.n_img = rg.n_img;
    int W, per_sm;
    gfw_block(kern, var_mode, boundary, rg.rad, W, per_sm);
    const size_t smem = (size_t)W * gfw_ring_floats(rg.rad) * sizeof(float);
    const int div = c.grid_div > 1 ? c.grid_div : 1;
    const int blocks = (per_sm * gf_sm_count() + div - 1) / div;
    const int strips = (cd.N + gfw_wout(rg.rad) - 1) / gfw_wout(rg.rad);
    // the tile shape bounds the rule's choice
    const int hmax = c.gf_rows > 0 ? c.gf_rows : DEF_GF_ROWS;
    const int H = gfw_rows(cd.M, hmax, rg.rad, cd.n_img, strips, blocks * W,
                           (4 * gf_sm_count() + div - 1) / div);
    const int n_items = cd.n_img * strips * ((cd.M + H - 1) / H);
    const int need = (n_items + W - 1) / W;
    kern<<<blocks < need ? blocks : need, W * 32, smem, s>>>(cd, c.imgs, one_desc(c), c.st,
                                                             iter, shifted, H);
  }
  return cudaGetLastError();
}

// The kernels of one variance mode and boundary, a context's own: setting an
// attribute loads its kernel.
cudaError_t configure_gf_kernel(int var_mode, int boundary) {
  for (int rad = 0; rad <= GF_RMAX; ++rad) {
    const size_t bytes = GFW_WARPS * gfw_ring_floats(rad) * sizeof(float);
    if (bytes <= DEFAULT_SMEM) continue;
    const cudaError_t e = cudaFuncSetAttribute((const void*)gf_kernel(var_mode, boundary, rad),
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gfd
