// Regularisation parameter by the discrepancy principle (Sec. 3.2).
//
// With a_b = |H_b|^2 and r_b = |H_b U_E,b - Y_b|^2 over all DFT bins b, the
// residual of u_p is f(lambda) = (1/P) sum_b lambda^2 r_b / (a_b + lambda)^2
// (Eq. 10-11 with Parseval's 1/P).  If ||h*u_E - y||^2 = f(inf) <= T the
// estimate is already in K and lambda = inf; otherwise lambda solves
// f(lambda) = T, whose root is unique because f increases (Eq. 11).
//
// GPU procedure (one spectral pass per evaluation, no host round trip):
//   each pass evaluates f at KNODES nodes lambda_j of the current bracket,
//   accumulating the per-bin terms in FP32 per thread and in FP64 across
//   warps and blocks; one warp of the image's last block then updates the
//   bracket.  Wide brackets use geometric nodes and are narrowed to the pair
//   of nodes that straddles T.  Brackets of ratio <= 4 use Chebyshev-
//   Lobatto nodes in t = ln(lambda): as a function of t, f is analytic in
//   the strip |Im t| < pi (its poles lie at lambda = -|H_b|^2 <= 0, i.e.
//   t = ln|H_b|^2 + i pi), whatever the spectrum, so the degree-11
//   interpolant in t through the node values has its root within ~1e-10
//   relative of the true one on a bracket of ratio 4 (~1e-14 on ratio 1.6).
//   Node values are rounded to FP32; their logarithms, formed once in FP64,
//   are the exact abscissae.  The interpolant is evaluated in double-float
//   arithmetic (FP64 is slow on this part), and its root is located by
//   multisection with one trial point per lane, which needs only the sign
//   of the interpolant.
// The first pass of each iteration is fused into the forward column FFT.  In
// iterations 0-2 its bracket is wide or of ratio 4; from iteration 3 on lambda
// moves little and the pass needs no bracket: it expands f about the
// extrapolated lambda c.  With t = c / (a + c) in (0, 1], s = ln(lambda / c) and
// e = tanh(s / 2),
//   lambda / (a + lambda) = t (1 + e) / (1 + e x),   x = 2 t - 1 in (-1, 1],
// so  P f(lambda) = (1 + e)^2 sum_k (k + 1) (-e)^k N_k,  N_k = sum_b r_b t_b^2 x_b^k,
// a series in e whose terms shrink at least as fast as (k + 1) |e|^k whatever
// the spectrum is.  One reciprocal per bin and two operations per moment serve
// all KMOM = 8 moments (12 nodes take a reciprocal and five operations each),
// and on the batched workload |e| <= 0.01 from iteration 5 on: the truncated
// terms are below 1e-15.  The root is accepted where its truncation error is
// below MOM_TOL; otherwise the series at a few |e| on the root's side, as far
// as its sign is certain against the truncated terms, gives the bracket of a
// fallback pass.
#pragma once
#include "common.cuh"
#include "df.cuh"

namespace gfd {

constexpr float INTERP_RATIO = 4.0f;   // largest bracket ratio interpolated
constexpr float MOM_REACH = 0.35f;      // largest |e| searched: lambda within a factor 2.08 of c
constexpr float MOM_TOL = 1e-10f;       // accepted truncation error of the root, relative
constexpr float INITIAL_LO = 1e-8f, INITIAL_HI = 1e4f;
constexpr int MODE_GEOM = 0, MODE_CHEB = 1, MODE_MOM = 2;

// Lanes of the warp that runs a per-image update (threads 0..31 of the
// block): the whole warp, or every thread of a block smaller than a warp
// (the column passes of 8- and 16-row canvases run 16 threads per block).
GFD_D int upd_lanes() { return blockDim.x >= 32 ? 32 : (int)blockDim.x; }
GFD_D unsigned int upd_mask() {
  return blockDim.x >= 32 ? 0xffffffffu : ((1u << blockDim.x) - 1u);
}

// cos(pi j / (n - 1)), j = 0..n-1 (Chebyshev-Lobatto points), n = KNODES
__device__ constexpr float kLobatto[KNODES] = {
    1.0f, 0.9594929736144974f, 0.8412535328311812f, 0.6548607339452851f,
    0.41541501300188644f, 0.14231483827328512f, -0.142314838273285f, -0.4154150130018863f,
    -0.654860733945285f, -0.8412535328311811f, -0.9594929736144974f, -1.0f};

// Node lambda_j (ascending) of a bracket [lo, hi] for the given layout.
GFD_D float bracket_node(float lo, float hi, int mode, int j) {
  if (j == 0) return lo;
  if (j >= KNODES - 1) return hi;
  if (mode == MODE_CHEB)  // Chebyshev-Lobatto in ln(lambda)
    return lo * exp2f(0.5f * (1.0f - kLobatto[j]) * log2f(hi / lo));
  return lo * exp2f((float)j / (KNODES - 1) * log2f(hi / lo));
}

// Chebyshev nodes (interpolated) for narrow brackets, geometric nodes
// (bracketed) otherwise.
GFD_D int bracket_mode(float lo, float hi) {
  return hi <= INTERP_RATIO * lo ? MODE_CHEB : MODE_GEOM;
}

// Set the next pass's bracket (single thread).
GFD_D void set_bracket(ImgState* st, float lo, float hi) {
  const int mode = bracket_mode(lo, hi);
  st->lo = lo;
  st->hi = hi;
  st->mode = mode;
  for (int j = 0; j < KNODES; ++j) st->node[j] = bracket_node(lo, hi, mode, j);
}

// Warp variant: lane j < KNODES writes node j.
GFD_D void set_bracket_warp(ImgState* st, float lo, float hi, int lane) {
  const int mode = bracket_mode(lo, hi);
  if (lane == 0) {
    st->lo = lo;
    st->hi = hi;
    st->mode = mode;
  }
  if (lane < KNODES) st->node[lane] = bracket_node(lo, hi, mode, lane);
  __syncwarp(upd_mask());
}

// The next pass expands f about c (node[0]).
GFD_D void set_center_warp(ImgState* st, float c, int lane) {
  if (lane == 0) {
    st->lo = c;
    st->hi = c;
    st->mode = MODE_MOM;
    st->node[0] = c;
  }
  __syncwarp(upd_mask());
}

// One bin's contribution: wr = (Hermitian weight) * r, a = |H|^2.
// t = lambda / (a + lambda) comes from an approximate reciprocal refined by
// one FMA residual step, which makes it (almost always) the correctly
// rounded quotient.  Without the step, every bin with a << lambda would carry
// the same reciprocal error for a given node: a node-dependent bias of ~1e-7
// in f(lambda_j) that moves the root by ~1e-7 / |d ln f / d ln lambda|,
// i.e. by percents where f is nearly flat in lambda.
// Nodes are taken two at a time (packed FP32 pairs).
struct BinAcc {
  float2 v[KNODES / 2];  // node sums (moments N_0.. in MODE_MOM)
  float w;               // sum of wr
  GFD_D void clear() {
#pragma unroll
    for (int j = 0; j < KNODES / 2; ++j) v[j] = make_float2(0.0f, 0.0f);
    w = 0.0f;
  }
};

GFD_D void accum_bin(float wr, float a, const float2* nodes, BinAcc& acc) {
  acc.w += wr;
  const float2 w2 = make_float2(wr, wr), a2 = make_float2(a, a);
#pragma unroll
  for (int j = 0; j < KNODES / 2; ++j) {
    const float2 n = nodes[j];
    const float2 d = cadd(a2, n);
    const float2 q = make_float2(__fdividef(1.0f, d.x), __fdividef(1.0f, d.y));
    const float2 t0 = __fmul2_rn(n, q);
    const float2 t = __ffma2_rn(__ffma2_rn(make_float2(-t0.x, -t0.y), d, n), q, t0);
    acc.v[j] = __ffma2_rn(w2, __fmul2_rn(t, t), acc.v[j]);
  }
}

// The bin's terms of the moments about c (MODE_MOM), two at a time.
GFD_D void accum_bin_moments(float wr, float a, float c, BinAcc& acc) {
  acc.w += wr;
  const float d = a + c;
  const float q = __fdividef(1.0f, d);
  const float t0 = c * q;
  const float t = fmaf(fmaf(-t0, d, c), q, t0);
  const float p0 = wr * (t * t);
  const float x = fmaf(2.0f, t, -1.0f);
  const float2 xx = make_float2(x * x, x * x);
  float2 p = make_float2(p0, p0 * x);
#pragma unroll
  for (int j = 0; j < KMOM / 2; ++j) {
    acc.v[j] = cadd(acc.v[j], p);
    if (j + 1 < KMOM / 2) p = __fmul2_rn(p, xx);
  }
}

// Long sums of the per-bin terms.  Threads keep FP32 partials over a short
// run of bins (one item); warp_fold adds the warp's total of each partial to
// per-warp double-float accumulators in shared memory (hi + lo, exact
// two-sum) and clears the partials; block_partials_folded turns the per-warp
// accumulators into the block's FP64 sums.  This keeps f(lambda) and
// ||h*u_E - y||^2 accurate to about 1e-10 relative over millions of bins,
// which matters where f is nearly flat in lambda.
struct WarpAcc {
  float hi[16][KNODES + 1];
  float lo[16][KNODES + 1];
};

GFD_D void warp_fold_one(float v, int j, int lane, int warp, WarpAcc* wa) {
  v = warp_sum(v);
  if (lane == 0) {
    const df t = two_sum(wa->hi[warp][j], v);
    wa->hi[warp][j] = t.hi;
    wa->lo[warp][j] += t.lo;
  }
}

// n: the leading sums in use (KNODES, or KMOM in MODE_MOM); the rest are zero.
GFD_D void warp_fold(BinAcc& acc, int n, WarpAcc* wa) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int j = 0; j < KNODES; j += 2) {
    if (j >= n) break;
    warp_fold_one(acc.v[j / 2].x, j, lane, warp, wa);
    warp_fold_one(acc.v[j / 2].y, j + 1, lane, warp, wa);
  }
  warp_fold_one(acc.w, KNODES, lane, warp, wa);
  acc.clear();
}

// Sum over groups of n consecutive lanes (n a power of two <= 32), FP64.  An
// FP64 addition takes 70 cycles here: a tree instead of one thread's chain.
GFD_D double group_sum_dbl(double v, int n) {
  const unsigned int mask = upd_mask();
  for (int o = n >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o);
  return v;
}

// part[j] = sum over warps of hi + lo (FP64); clears the accumulators.
// Synchronises before and after.
GFD_D void block_partials_folded(WarpAcc* wa, double* part) {
  __syncthreads();
  const int nwarp = num_warps();  // a power of two <= 16: one thread per (sum, warp)
  for (int e = threadIdx.x; e < 16 * nwarp; e += blockDim.x) {
    const int j = e / nwarp, w = e - j * nwarp;
    double v = 0.0;
    if (j <= KNODES) {
      v = (double)wa->hi[w][j] + (double)wa->lo[w][j];
      wa->hi[w][j] = 0.0f;
      wa->lo[w][j] = 0.0f;
    }
    v = group_sum_dbl(v, nwarp);
    if (j <= KNODES && w == 0) part[j] = v;
  }
  __syncthreads();
}

// Zero the accumulators (every thread calls; synchronise before use).
GFD_D void warp_acc_clear(WarpAcc* wa) {
  float* p = &wa->hi[0][0];
  for (int i = threadIdx.x; i < 2 * 16 * (KNODES + 1); i += blockDim.x) p[i] = 0.0f;
}

GFD_D double warp_sum_dbl(double v) {
  const unsigned int n = blockDim.x < 32 ? blockDim.x : 32u;
  const unsigned int mask = n == 32 ? 0xffffffffu : ((1u << n) - 1u);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    if ((unsigned)o < n) v += __shfl_xor_sync(mask, v, o);
  return v;
}

// Sum of vals[i * stride + j] over i < n for each j < m, by the whole block
// in FP64 (loads bypass L1: the values were written by other blocks).
// Results land in sums[0..m) (shared), visible to every thread on return.
// Several columns: one warp per column (a single barrier); one column: the
// whole block.
GFD_D void block_sum_columns(const double* vals, int n, int stride, int m, double* red,
                             double* sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarp = num_warps();
  if (m > 1 && (blockDim.x & 31) == 0) {  // whole warps
    for (int j = warp; j < m; j += 2 * nwarp) {  // two columns' chains side by side
      const int j2 = j + nwarp;
      double s = 0.0, t = 0.0;
      for (int i = lane; i < n; i += 32) {
        s += __ldcg(&vals[(size_t)i * stride + j]);
        if (j2 < m) t += __ldcg(&vals[(size_t)i * stride + j2]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        t += __shfl_xor_sync(0xffffffffu, t, o);
      }
      if (lane == 0) {
        sums[j] = s;
        if (j2 < m) sums[j2] = t;
      }
    }
    __syncthreads();
    return;
  }
  for (int j = 0; j < m; ++j) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += __ldcg(&vals[(size_t)i * stride + j]);
    s = warp_sum_dbl(s);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (warp == 0) {
      double t = lane < nwarp ? red[lane] : 0.0;
      if (nwarp > 1) t = group_sum_dbl(t, nwarp);
      if (lane == 0) sums[j] = t;
    }
    __syncthreads();
  }
}

// Called by every block after storing its item's partials: true in exactly
// one block per image and pass (the one finishing last), after all partials
// are visible.
GFD_D bool last_item(unsigned int* counter, unsigned int n_items, int* s_flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned int prev = atomicAdd(counter, 1u);
    *s_flag = (prev == n_items - 1);
  }
  __syncthreads();
  const bool last = *s_flag != 0;
  if (last) __threadfence();
  return last;
}

// Root of the interpolant in t = ln(lambda) through (t_m, g_m), m < KNODES,
// t_m = ln(x_m) of the FP32 node values x_m (ascending; g increasing through
// 0 between x_j and x_{j+1}).  Lane m < KNODES holds (x_m, g_m).  The
// logarithms are formed in FP64 and carried as double-float, as are the
// barycentric weights w_m = 1 / prod_{n != m} (t_m - t_n) of the actual nodes.
// Inside (t_j, t_{j+1}) the interpolant is p(t) = l(t) S(t) with
// l(t) = prod_m (t - t_m), whose sign there is (-1)^(nk-1-j) (nk nodes), and
// S(t) = sum_m w_m g_m / (t - t_m) (the first barycentric form), so the sign
// of p at a point needs S alone, one double-float quotient per node.  The
// root is bracketed by multisection: every lane evaluates the sign at its own
// trial point and the bracket shrinks to the two trial points that straddle
// the root.  After a plain round (one point per lane, spread evenly across
// the bracket; 32 lanes, or the block's threads if fewer) the next
// round's points sit in a window about the secant estimate from p at the
// bracket's ends (window half-width 1/16, then 1/256, then 1/4096 of the
// bracket while the root keeps falling inside it; a round whose window misses
// still leaves a valid bracket, and the next round is plain again).  Returns
// lambda = exp(t_root) at the bracket's midpoint once its width is <= rtol.
GFD_D df df_div_fast(df a, df b) {  // a / b, error ~2^-44 relative
  const float ib = __fdividef(1.0f, b.hi);
  const float q1 = a.hi * ib;
  const df p = two_prod(b.hi, q1);
  const float r = ((a.hi - p.hi) - p.lo + a.lo) - q1 * b.lo;  // a - q1 b
  return quick_two_sum(q1, r * ib);
}

GFD_D double interp_root_warp(float xm, float gm, int j, double rtol, int lane) {
  constexpr int nk = KNODES;
  const bool own = lane < nk;
  const df tm = own ? df_from_double(log((double)xm)) : df_make(0.0f);
  // All abscissa differences are scaled by a power of two ~ 1/(node span):
  // exact, and it keeps the products of 11 differences in FP32 range (the
  // sign of S and the root do not depend on the scale).
  const float t0 = __shfl_sync(upd_mask(), tm.hi, 0);
  const float tK = __shfl_sync(upd_mask(), tm.hi, nk - 1);
  int ex;
  frexpf(tK - t0, &ex);
  const float sc = ldexpf(1.0f, -ex);
  df prod = df_make(1.0f);
  for (int n = 0; n < nk; ++n) {
    const df tn{__shfl_sync(upd_mask(), tm.hi, n), __shfl_sync(upd_mask(), tm.lo, n)};
    if (own && n != lane) {
      const df dd = df_sub(tm, tn);
      prod = df_mul(prod, df{dd.hi * sc, dd.lo * sc});
    }
  }
  const df c = own ? df_mul_f(df_rcp(prod), gm) : df_make(0.0f);  // w_m g_m
  __shared__ df s_t[KNODES], s_c[KNODES];
  __shared__ float s_g[KNODES];
  if (own) {
    s_t[lane] = tm;
    s_c[lane] = c;
    s_g[lane] = gm;
  }
  __syncwarp(upd_mask());
  const float sig = ((nk - 1 - j) & 1) ? -1.0f : 1.0f;  // sign of l(t) in the bracket
  df a = s_t[j], b = s_t[j + 1];
  float pa = s_g[j], pb = s_g[j + 1];  // p at the bracket's ends
  int level = 0;                       // windows in a row that held the root
  const int nl = upd_lanes();  // trial points per round
  const float inv_np1 = 1.0f / (float)(nl + 1);
  const float frac32 = (float)(lane + 1) * inv_np1;
  for (int round = 0; round < 24; ++round) {
    const df width = df_sub(b, a);
    if (df_to_double(width) <= rtol) break;  // absolute in t: relative in lambda
    // trial points: across the bracket, or across a window about the secant
    // estimate of the root
    df wlo = a, ww = width;
    if (level > 0) {
      const float est = pa / (pa - pb);
      if (est > 0.0f && est < 1.0f) {
        const float h = level == 1 ? 0.0625f : (level == 2 ? 0.00390625f : 0.000244140625f);
        const float f0 = fmaxf(est - h, 0.0f), f1 = fminf(est + h, 1.0f);
        wlo = df_add(a, df_mul_f(width, f0));
        ww = df_mul_f(width, f1 - f0);
      } else {
        level = 0;
      }
    }
    const df t = df_add(wlo, df_mul_f(ww, frac32));
    df S0 = df_make(0.0f), S1 = df_make(0.0f);  // two partial sums (shorter chains)
    float ell = 1.0f;
    bool at_node = false;
    float node_g = 0.0f;
    // add node m's term w_m g_m / (t - t_m) to S (t at a node: p(t) = g_m)
    auto term = [&](int m, df& S) {
      const df tmm = s_t[m];
      df d = two_sum(t.hi, -tmm.hi);
      d.lo += t.lo - tmm.lo;
      if (d.hi == 0.0f && d.lo == 0.0f) {
        at_node = true;
        node_g = s_g[m];
        return;
      }
      d = quick_two_sum(d.hi, d.lo);
      d.hi *= sc;
      d.lo *= sc;
      ell *= d.hi;
      const df q = df_div_fast(s_c[m], d);
      const df u = two_sum(S.hi, q.hi);
      S.hi = u.hi;
      S.lo += u.lo + q.lo;
    };
#pragma unroll 2
    for (int m = 0; m < nk; m += 2) {  // registers stay low in the pass kernels
      term(m, S0);
      term(m + 1, S1);
    }
    const df Sv = df_add(quick_two_sum(S0.hi, S0.lo), quick_two_sum(S1.hi, S1.lo));
    const bool neg = at_node ? (node_g < 0.0f) : (sig * Sv.hi < 0.0f);
    const float pv = at_node ? node_g : ell * (Sv.hi + Sv.lo);  // p(t), for the estimate
    const unsigned below = __ballot_sync(upd_mask(), neg);
    // the interpolant increases: trial points below the root form a prefix
    const int nb = __popc(below);  // lanes 0..nb-1 are below the root
    const float p_lo = __shfl_sync(upd_mask(), pv, nb > 0 ? nb - 1 : 0);
    const float p_hi = __shfl_sync(upd_mask(), pv, nb < nl ? nb : nl - 1);
    const bool hit = nb > 0 && nb < nl;  // the root lies between two trial points
    if (nb > 0) {
      a = df_add(wlo, df_mul_f(ww, (float)nb * inv_np1));
      pa = p_lo;
    }
    if (nb < nl) {
      b = df_add(wlo, df_mul_f(ww, (float)(nb + 1) * inv_np1));
      pb = p_hi;
    }
    level = hit ? level + 1 : 0;
  }
  return exp(0.5 * (df_to_double(a) + df_to_double(b)));
}

// Record lambda_k and set up iteration k+1's fused first pass (prev: the last
// finite lambda before it).  lambda jumps
// by a factor of 2..600 from the first iteration (u_E = 0) to the second, and
// mostly falls to 0.2..1.2 of it in the third; the fourth stays within a few
// percent of the third on most images, and later it changes smoothly.  The
// second iteration's bracket has geometric nodes, resolved by one more pass;
// the third's, [0.28, 1.1] lambda_1, is narrow enough (ratio <= 4) for the
// interpolation to resolve it in the fused pass itself; later first passes
// expand f about lambda_2, then about the extrapolation
// lambda_k (lambda_k / lambda_{k-1}) (ratio clamped to [1/2, 2]).
GFD_D void resolve_warp(ImgState* st, double lam, double prev, int iter, double* lam_out,
                        int lane) {
  if (lane == 0) {
    st->lam = lam;
    st->need = 0;
    if (lam_out) lam_out[iter] = lam;
  }
  // lambda = inf (or no finite root) keeps the pending bracket or centre
  if (isfinite(lam) && lam > 0.0) {
    const float l = (float)lam;
    if (iter == 0) {
      set_bracket_warp(st, fmaxf(l, (float)LAMBDA_LO), 150.0f * l, lane);
    } else if (iter == 1) {
      set_bracket_warp(st, fmaxf(0.28f * l, (float)LAMBDA_LO), 1.1f * l, lane);
    } else {
      float c = l;
      if (iter > 2 && isfinite(prev) && prev > 0.0) {
        const df ip = df_rcp(df_from_double(prev));
        c = l * fminf(fmaxf(l * (ip.hi + ip.lo), 0.5f), 2.0f);
      }
      set_center_warp(st, fmaxf(c, (float)LAMBDA_LO), lane);
    }
    if (lane == 0) st->lam_prev = lam;
  }
  __syncwarp(upd_mask());
}

// Root of the moment expansion about c = node[0] (see the top of the file).
// tot[0..KMOM-1] are the sums N_k.  Every lane evaluates the series at a trial
// point of its own in FP32, three rounds; two Newton steps with the series
// in FP64 follow.  Sets lam to the root and returns true if it is accepted;
// otherwise leaves the bracket of the next pass in (lo, hi): up to a point that
// the series has certainly past the root; without one a ratio of 3.95, narrow
// enough to be interpolated, or (wide) the whole range on the root's side.
GFD_D bool moment_root_warp(const double* tot, double scale, float c, float lam_up, bool wide,
                            int lane, double& lam, float& lo, float& hi) {
  static_assert(KMOM == 8, "the series is evaluated by halves of four terms");
  const int nl = upd_lanes();
  const unsigned int mask = upd_mask();
  // a_k = (k + 1) (-1)^k N_k / (P T), one per lane, then to every lane
  double ak = 0.0;
  if (lane < KMOM) ak = tot[lane] * scale * ((lane & 1) ? -(lane + 1) : (lane + 1));
  double a[KMOM];
  float af[KMOM];
#pragma unroll
  for (int k = 0; k < KMOM; ++k) {
    a[k] = __shfl_sync(mask, ak, k);
    af[k] = (float)a[k];
  }
  auto value = [&](float e) {  // f / T - 1
    float p = af[KMOM - 1];
#pragma unroll
    for (int k = KMOM - 2; k >= 0; --k) p = fmaf(p, e, af[k]);
    return fmaf(p, (1.0f + e) * (1.0f + e), -1.0f);
  };
  float e0 = -MOM_REACH, e1 = MOM_REACH;
  const float inv = 1.0f / (float)(nl + 1);
  for (int round = 0; round < 3; ++round) {
    const float w = e1 - e0;
    const unsigned int above = __ballot_sync(mask, !(value(fmaf(w, (lane + 1) * inv, e0)) < 0.0f));
    const int nb = above ? __ffs(above) - 1 : nl;  // leading trial points below the root
    e1 = nb < nl ? fmaf(w, (nb + 1) * inv, e0) : e1;
    e0 = nb > 0 ? fmaf(w, nb * inv, e0) : e0;
  }
  double e = 0.5 * ((double)e0 + (double)e1);
  const float ef = (float)e, g = 1.0f + ef;
  float p = af[KMOM - 1], dp = 0.0f;  // series and its derivative
#pragma unroll
  for (int k = KMOM - 2; k >= 0; --k) {
    dp = fmaf(dp, ef, p);
    p = fmaf(p, ef, af[k]);
  }
  const float slope = g * fmaf(g, dp, 2.0f * p);  // d(f / T) / de
  const float islope = __fdividef(1.0f, slope);
#pragma unroll 1
  for (int it = 0; it < 5; ++it) {
    // the series by halves: four dependent FP64 operations (70 cycles each)
    // instead of seven
    const double e2 = e * e;
    const double q0 = fma(fma(a[3], e, a[2]), e2, fma(a[1], e, a[0]));
    const double q1 = fma(fma(a[7], e, a[6]), e2, fma(a[5], e, a[4]));
    const double F = fma(fma(q1, e2 * e2, q0), fma(2.0, e, e2 + 1.0), -1.0);
    const float step = (float)F * islope;
    e -= (double)step;
    if (!(fabsf(step) > 1e-7f)) break;  // the next would be below 1e-13
  }
  const float er = (float)e;
  // truncated terms, at most (KMOM + 1) |e|^KMOM N_0 (1 + e)^2 / (1 - |e|)^2 in
  // all (N_k <= N_0), over the slope in s: de / ds = (1 - e^2) / 2
  const float x2 = er * er, x4 = x2 * x2, d1 = 1.0f - fabsf(er);
  const float err = (KMOM + 1) * x4 * x4 * af[0] * g * g * islope * 2.0f / ((1.0f - x2) * d1 * d1);
  const float est = c * __fdividef(1.0f + er, 1.0f - er);
  if (slope > 0.0f && err <= MOM_TOL && est > (float)LAMBDA_LO) {
    // c (1 + e) / (1 - e), the reciprocal by two Newton steps from FP32
    const double d = 1.0 - e;
    double q = (double)__fdividef(1.0f, (float)d);
    q = fma(fma(-d, q, 1.0), q, q);
    q = fma(fma(-d, q, 1.0), q, q);
    lam = fma((double)c, e, (double)c) * q;
    return true;
  }
  // The root's side of c by the sign of f(c) - T; along it, the last |e| that
  // the series certainly has before the root and the first certainly past it.
  const bool up = a[0] < 1.0;
  float before = 0.0f, past = 0.0f;
#pragma unroll 1
  for (int i = 0; i < 4; ++i) {
    const float m = i == 0 ? 0.11f : (i == 1 ? 0.18f : (i == 2 ? 0.25f : MOM_REACH));
    const float m2 = m * m, m4 = m2 * m2;
    const float v = up ? value(m) : -value(-m);
    const float r1 = (1.0f + m) / (1.0f - m);
    const float margin = (KMOM + 1) * m4 * m4 * af[0] * r1 * r1 + 2e-7f;
    if (v > margin) past = m;
    if (!(v < -margin)) break;
    before = m;
  }
  const float rb = (1.0f + before) / (1.0f - before), rp = (1.0f + past) / (1.0f - past);
  const float near = 0.99f * rb, far = past > 0.0f ? 1.01f * rp : 3.95f * near;
  lo = up ? c * near : c / far;
  hi = up ? c * far : c / near;
  if (wide && past == 0.0f) {
    if (up)
      hi = fmaxf(lam_up, hi);
    else
      lo = (float)LAMBDA_LO;
  }
  return false;
}

// Consume the totals of the pass that just completed for this image (tot:
// KNODES node sums and the residual sum, visible to the warp).  Run by the
// 32 lanes of one warp of the image's last block; every lane takes the same
// decisions from the same values.  FP64 is limited to a handful of
// operations (the sums themselves are FP64).
__device__ __noinline__ static void lambda_update_warp(ImgState* st, const double* tot, bool primary,
                              bool last_chance, int iter, double* lam_out, double* res_out,
                              int lane) {
  // the state's fields are requested together: they come from L2, one trip
  const double invP = st->invP, T = st->T, invT = st->invT, prev = st->lam_prev;
  const int mode = st->mode, max_pass = st->max_pass;
  const float amax = (float)st->amax, node = lane < KNODES ? st->node[lane] : 0.0f;
  const double resinf = tot[KNODES] * invP;
  if (primary) {
    if (lane == 0) {
      st->res = resinf;
      if (res_out) res_out[iter] = resinf;
    }
    if (!isfinite(resinf)) {
      if (lane == 0) st->status |= ST_NONFINITE;
      resolve_warp(st, INFINITY, prev, iter, lam_out, lane);
      return;
    }
    if (resinf <= T) {  // u_E in K (Sec. 3.2): lambda = inf, u_I = u_p = u_E
      resolve_warp(st, INFINITY, prev, iter, lam_out, lane);
      return;
    }
    if (lane == 0) {
      const float t = sqrtf((float)T / (float)resinf);
      st->lam_up = fminf(1e30f, amax * t / (1.0f - t));
    }
    __syncwarp(upd_mask());
  }
  if (mode == MODE_MOM) {
    const float c = __shfl_sync(upd_mask(), node, 0);
    if (!isfinite(tot[0])) {
      if (lane == 0) st->status |= ST_NONFINITE;
      resolve_warp(st, INFINITY, prev, iter, lam_out, lane);
      return;
    }
    double lam;
    float lo, hi;
    // lambda still jumps in iterations 3 and 4; two passes find a root far above
    // c only if the first of them takes the whole range
    const bool wide = max_pass == 2 && iter < 5;
    if (moment_root_warp(tot, invP * invT, c, st->lam_up, wide, lane, lam, lo, hi)) {
      resolve_warp(st, lam, prev, iter, lam_out, lane);
      return;
    }
    lo = fmaxf(lo, (float)LAMBDA_LO);
    set_bracket_warp(st, lo, fmaxf(hi, 1.05f * lo), lane);
    if (lane == 0) st->need = 1;
    return;
  }
  // g_m = f(lambda_m) / T - 1, increasing in lambda, for the pass's nodes
  constexpr int nk = KNODES;
  const float gm = lane < nk ? (float)((tot[lane] * invP - T) * invT) : 0.0f;
  const float xm = node;
  const float g0 = __shfl_sync(upd_mask(), gm, 0);
  const float gK = __shfl_sync(upd_mask(), gm, nk - 1);
  const float lo = __shfl_sync(upd_mask(), xm, 0);
  const float hi = __shfl_sync(upd_mask(), xm, nk - 1);
  // a missed first bracket whose root is expected close to it
  const bool near = primary && iter == 2 && mode == MODE_CHEB;
  // the second iteration's jump, past its first bracket: seldom far past it.  A
  // root that is takes one pass more than from the whole range, four in all
  // whatever it is: with fewer to go the whole range comes at once.
  const bool jump = primary && iter == 1 && max_pass >= 4;
  bool open = true;
  if (!(g0 <= 0.0f)) {  // root below the bracket (or NaN)
    if (!isfinite(g0)) {
      if (lane == 0) st->status |= ST_NONFINITE;
      resolve_warp(st, INFINITY, prev, iter, lam_out, lane);
      return;
    }
    if (lo <= (float)LAMBDA_LO * 1.000001f) {
      if (lane == 0) st->status |= ST_NONCONVERGED;
      resolve_warp(st, LAMBDA_LO, prev, iter, lam_out, lane);
      return;
    }
    // below the third iteration's first bracket (four passes to go): the
    // ratio-4 bracket just under it; otherwise everything down to the smallest
    // lambda
    const float nlo = near ? fmaxf(0.25f * lo, (float)LAMBDA_LO) : (float)LAMBDA_LO;
    set_bracket_warp(st, nlo, lo, lane);
  } else if (gK < 0.0f) {  // root above the bracket
    // above the third iteration's first bracket: the ratio-4 bracket just
    // over it; above the second's: a ratio-16 bracket, whose intervals are
    // interpolated by the pass after; otherwise up to the bound from res and
    // |H|^2
    set_bracket_warp(st, hi, near ? 4.0f * hi : (jump ? 16.0f * hi : fmaxf(st->lam_up, hi * 4.0f)),
                     lane);
  } else {
    // nodes with g < 0 form a prefix 0..j
    const unsigned below = __ballot_sync(upd_mask(), lane < nk && gm < 0.0f);
    int j = 31 - __clz(below | 1u);
    if (j > nk - 2) j = nk - 2;
    if (mode == MODE_CHEB) {
      const double lam = interp_root_warp(xm, gm, j, st->rtol, lane);
      resolve_warp(st, lam, prev, iter, lam_out, lane);
      open = false;
    } else {
      const float nlo = __shfl_sync(upd_mask(), xm, j), nhi = __shfl_sync(upd_mask(), xm, j + 1);
      set_bracket_warp(st, nlo, nhi, lane);
    }
  }
  if (open) {
    if (lane == 0) st->need = 1;
    if (last_chance) {  // the pass schedule ran out with the bracket still open
      if (lane == 0) st->status |= ST_PASSES_EXHAUSTED;
      const double mid = sqrt((double)st->lo * (double)st->hi);
      __syncwarp(upd_mask());
      resolve_warp(st, mid, prev, iter, lam_out, lane);
    }
  }
}

}  // namespace gfd
