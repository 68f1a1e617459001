// 2-D real DFT passes and the spectral steps of the deblurring solve.
//
// Packed half spectrum (M rows x N/2 complex): S(m, l) = X(m, l) for
// 1 <= l < N/2 and S(m, 0) = X(m, 0) + i X(m, N/2), X the full 2-D DFT.  A
// row pass maps each real row to its packed row DFT; a column pass is a plain
// complex FFT down every packed column (column 0 included, since its two real
// row spectra pack into one complex signal).  Bins (m, 0) and (m, N/2) are
// unpacked where a spectral formula needs them.
//
// Spectra are stored column-tiled: S(m, l) at (l / TB) * M * TB + m * TB +
// l % TB, TB the class's tile width.  A column item (TB columns, all M rows)
// is then one contiguous block of memory, and a row item (rpc rows) writes a
// contiguous run of rpc * TB values per tile.  TB = N/2 is plain row-major.
#include <cooperative_groups.h>

#include "fft.cuh"
#include "lambda.cuh"
#include "spectral.cuh"
#include "launch.h"

namespace gfd {

GFD_D float* real_plane(const ImgDesc& d, int sel) {
  switch (sel) {
    case SEL_Y: return const_cast<float*>(d.y);
    case SEL_U: return d.u;
    case SEL_S: return reinterpret_cast<float*>(d.S);
    case SEL_QI: return reinterpret_cast<float*>(d.QI);
    case SEL_QP: return reinterpret_cast<float*>(d.Qp);
    case SEL_H: return reinterpret_cast<float*>(d.H);
    case SEL_UI: return d.uI;
    case SEL_UP: return d.up;
    default: return reinterpret_cast<float*>(d.Y);
  }
}
GFD_D float2* cplx_plane(const ImgDesc& d, int sel) {
  return reinterpret_cast<float2*>(real_plane(d, sel));
}

// Streaming loads: spectra and images pass through once per launch and stay out
// of L1, which keeps the twiddle tables there.
GFD_D float2 load_stream(const float2* p) { return __ldcg(p); }

// Barrier among the threads of a row team: teams of at most a warp exchange
// inside it.
template <int T>
GFD_D void team_sync(unsigned int mask) {
  if constexpr (T <= 32)
    __syncwarp(mask);
  else
    __syncthreads();
}
GFD_D unsigned int warp_mask() {
  return blockDim.x >= 32 ? 0xffffffffu : ((1u << blockDim.x) - 1u);
}

// ---------------------------------------------------------------------------
// Row passes.  A block takes rpc consecutive rows of one image, a team of T
// threads per row.  Elements go from global memory to registers, through the
// team's buffer in shared memory once or twice, and from registers to global
// memory; the mirrored pairs that the real transform needs sit in one thread
// (fft.cuh).  Teams of a warp or less (rows of up to 1024 reals) run without
// block barriers.  What bounds them is shared memory and the pieces of TB
// values that a row has in each tile (16 to 64 bytes per store): the
// transform that staged its input, every stage and its output in shared memory
// took 4.25 ms (forward) and 7.4 ms (inverse, two planes) per batched solve of
// 256 images, this one 3.0 and 5.3 ms.
// ---------------------------------------------------------------------------

// The slots of a mirrored butterfly pair (A, B) of radix r over positions
// beta + D i (A) and D - beta + D i (B), D r = L: slot t pairs A_t with
// B_{r-1-t}, whose position is L minus that of A_t.  The pair holding beta = 0
// and beta = D/2 mirrors onto itself instead: slots 1..r/2-1 pair A_t with
// A_{r-t}, slots r/2..r-1 pair B_u with B_{r-1-u} (u = t - r/2), and slot 0
// holds positions 0 and L/2, both their own mirrors.
template <int r>
struct MirrorSlots {
  // position of slot t's first element
  GFD_D static int first(bool self, int beta, int D, int t) {
    return (self && t >= r / 2) ? D / 2 + D * (t - r / 2) : beta + D * t;
  }
  // and of its second
  GFD_D static int second(bool self, int beta, int D, int t) {
    return (self && t == 0) ? D * r / 2 : D * r - first(self, beta, D, t);
  }
};

GFD_D float2 select2(bool c, float2 a, float2 b) { return c ? a : b; }

// Which row of the block (of rpc) and which thread of its team a thread is on
// the side of the tiled spectra: TB threads for the columns of a tile's row,
// then the block's rows, whose pieces of TB values lie side by side, so that a
// warp's access is one run of up to rpc * TB values instead of 32 / TB pieces.
// On the side of the image a team is T consecutive threads.
template <int T>
GFD_D void tiled_thread(int TB, int rpc, int& row, int& j) {
  const int w = TB < T ? TB : T, lw = __ffs(w) - 1, lr = __ffs(rpc) - 1;
  const int tid = threadIdx.x;
  row = (tid >> lw) & (rpc - 1);
  j = ((tid >> (lw + lr)) << lw) + (tid & (w - 1));
}

// Forward: real rows -> packed row spectra (tiled).  Each row of N reals is read
// as N/2 complex z[n] = x[2n] + i x[2n+1]; Z = FFT_{N/2}(z); with
// E = (Z[k] + conj Z[-k]) / 2 and O = (Z[k] - conj Z[-k]) / (2i),
// X[k] = E + W_N^k O and X[-k] = conj(E - W_N^k O); X[0], X[N/2] = Re Z[0] +-
// Im Z[0] (packed as X[0] + i X[N/2]).  do_sum: FP64 row sums of the source.
template <int L>
__global__ void __launch_bounds__(256, 3)
k_row_r2c(ClassDesc cd, const ImgDesc* __restrict__ imgs, const __grid_constant__ ImgDesc one,
          const float2* __restrict__ tw, int rpc, int src_sel, int dst_sel, int do_sum) {
  extern __shared__ __align__(16) float2 smem[];
  using G = FftGeo<FK_R2C, L>;
  constexpr int T = G::T, r0 = G::RF, rl = G::RL;
  constexpr int N = 2 * L, KL = G::KL;
  const int TB = cd.TB, M = cd.M;
  const int team = threadIdx.x / T, j = threadIdx.x % T;
  const int row_c = blockIdx.x * rpc + team;
  const ImgDesc& d = imgs ? imgs[cd.img0 + row_c / M] : one;
  const int row = row_c % M;
  const unsigned int mask = warp_mask();
  float2* buf = smem + team * G::SIZE;
  const float* plane = src_sel >= SEL_ITER0 ? d.u_iters + (size_t)(src_sel - SEL_ITER0) * M * N
                                            : real_plane(d, src_sel);
  const float2* src = reinterpret_cast<const float2*>(plane) + (size_t)row * L;
  float part = 0.0f;
#pragma unroll
  for (int q = 0; q < G::E / r0; ++q) {
    const int beta = j + T * q;
    float2 x[r0];
#pragma unroll
    for (int i = 0; i < r0; ++i) x[i] = load_stream(src + beta + i * G::L1);
    if (do_sum) {
#pragma unroll
      for (int i = 0; i < r0; ++i) part += x[i].x + x[i].y;
    }
    fft_first<FK_R2C, L, false>(x, beta, buf, tw);
  }
  if (do_sum) {  // one FP64 sum per row
    __shared__ double red[8];
    if constexpr (T <= 32) {
#pragma unroll
      for (int o = T / 2; o > 0; o >>= 1) part += __shfl_xor_sync(mask, part, o);
      if (j == 0) d.rowsum[row] = (double)part;
    } else {
      part = warp_sum(part);
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = (double)part;
      __syncthreads();
      if (j == 0) {
        double s = 0.0;
        for (int w = 0; w < T / 32; ++w) s += red[(threadIdx.x >> 5) + w];
        d.rowsum[row] = s;
      }
    }
  }
  if constexpr (G::S == 3) {
    team_sync<T>(mask);
    fft_mid<FK_R2C, L, false>(buf, j, tw);
  }
  __syncthreads();  // the last stage's threads are spread over the block's rows
  int trow, tj;
  tiled_thread<T>(TB, rpc, trow, tj);
  const float2* tbuf = smem + trow * G::SIZE;
  // tiled row: column k of tile k / TB (the block's rows are of one image)
  float2* dst = cplx_plane(d, dst_sel) + (size_t)(row - team + trow) * TB;
  const int lg = __ffs(TB) - 1;
  auto put = [&](int k, float2 v) {
    dst[(((size_t)(k >> lg) * M) << lg) + (k & (TB - 1))] = v;
  };
#pragma unroll
  for (int q = 0; q < G::E / rl / 2; ++q) {
    const int kap = tj + T * q;
    const bool self = q == 0 && tj == 0;
    float2 A[rl], B[rl];
    fft_last<FK_R2C, L, false>(A, kap, tbuf);
    fft_last<FK_R2C, L, false>(B, self ? KL / 2 : KL - kap, tbuf);
#pragma unroll
    for (int t = 0; t < rl; ++t) {
      const int k = MirrorSlots<rl>::first(self, kap, KL, t);
      float2 a = A[t], b = B[rl - 1 - t];
      if (q == 0) {
        if (t >= rl / 2) a = select2(self, B[t - rl / 2], a);
        if (t >= rl / 2)
          b = select2(self, B[rl + rl / 2 - 1 - t], b);
        else
          b = select2(self, A[t == 0 ? rl / 2 : rl - t], b);
      }
      const float2 E = cscale(cadd(a, cconj(b)), 0.5f);
      const float2 D = cscale(csub(a, cconj(b)), 0.5f);
      const float2 WO = cmul(__ldg(&tw[tab_off(N) + k]), make_float2(D.y, -D.x));
      float2 u = cadd(E, WO), v = cconj(csub(E, WO));
      if (q == 0 && t == 0 && self) {
        u = make_float2(a.x + a.y, a.x - a.y);  // X[0] + i X[N/2]
        v = cconj(b);                           // X[N/4] = conj Z[L/2]
      }
      put(k, u);
      put(MirrorSlots<rl>::second(self, kap, KL, t), v);
    }
  }
}

// Inverse: packed row spectra (tiled) -> real rows (scaled).  With
// E = R[k] + conj R[L-k] and O = (R[k] - conj R[L-k]) W_N^{-k},
// Z[k] = E + i O and Z[L-k] = conj(E) + i conj(O) (R[0], R[N/2] are the real and
// imaginary parts of the packed entry 0); the unnormalised inverse FFT of Z
// gives x[2n] + i x[2n+1] times N.  Blocks cover spectrum sel0 -> real plane
// dsel0, then sel1 -> dsel1.
template <int L>
__global__ void __launch_bounds__(256, 3)
k_row_c2r(ClassDesc cd, const ImgDesc* __restrict__ imgs, const __grid_constant__ ImgDesc one,
          const float2* __restrict__ tw, int rpc, int sel0, int sel1, int dsel0, int dsel1, float scale, ImgState* st) {
  extern __shared__ __align__(16) float2 smem[];
  using G = FftGeo<FK_C2R, L>;
  constexpr int T = G::T, r0 = G::RF, rl = G::RL;
  constexpr int N = 2 * L;
  const int TB = cd.TB, M = cd.M;
  const int team = threadIdx.x / T, j = threadIdx.x % T;
  const int per_plane = cd.n_img * M / rpc;
  const bool second = (int)blockIdx.x >= per_plane;
  const int row_c = ((int)blockIdx.x - (second ? per_plane : 0)) * rpc + team;
  const int li = row_c / M, row = row_c % M;
  const ImgDesc& d = imgs ? imgs[cd.img0 + li] : one;
  const unsigned int mask = warp_mask();
  float2* buf = smem + team * G::SIZE;
  int trow, tj;
  tiled_thread<T>(TB, rpc, trow, tj);
  float2* tbuf = smem + trow * G::SIZE;
  const float2* src = cplx_plane(d, second ? sel1 : sel0) + (size_t)(row - team + trow) * TB;
  const int lg = __ffs(TB) - 1;
  auto get = [&](int k) {
    return load_stream(src + (((size_t)(k >> lg) * M) << lg) + (k & (TB - 1)));
  };
#pragma unroll
  for (int q = 0; q < G::E / r0 / 2; ++q) {
    const int beta = tj + T * q;
    const bool self = q == 0 && tj == 0;
    float2 u[r0], v[r0];  // Z at the slots' first and second positions
#pragma unroll
    for (int t = 0; t < r0; ++t) {
      u[t] = get(MirrorSlots<r0>::first(self, beta, G::L1, t));
      v[t] = get(MirrorSlots<r0>::second(self, beta, G::L1, t));
    }
#pragma unroll
    for (int t = 0; t < r0; ++t) {
      const int k = MirrorSlots<r0>::first(self, beta, G::L1, t);
      const float2 a = u[t], b = v[t];
      const float2 E = cadd(a, cconj(b)), D = csub(a, cconj(b));
      const float2 O = cmul(D, cconj(__ldg(&tw[tab_off(N) + k])));
      u[t] = make_float2(E.x - O.y, E.y + O.x);
      v[t] = make_float2(E.x + O.y, O.x - E.y);
      if (q == 0 && t == 0 && self) {
        u[t] = make_float2(a.x + a.y, a.x - a.y);
        v[t] = make_float2(2.0f * b.x, -2.0f * b.y);
      }
    }
    float2 A[r0], B[r0];
#pragma unroll
    for (int i = 0; i < r0; ++i) {
      A[i] = u[i];
      B[i] = v[r0 - 1 - i];
      if (q == 0) {
        if (i >= r0 / 2) A[i] = select2(self, i == r0 / 2 ? v[0] : v[r0 - i], A[i]);
        B[i] = select2(self, i < r0 / 2 ? u[i + r0 / 2] : v[r0 + r0 / 2 - 1 - i], B[i]);
      }
    }
    fft_first<FK_C2R, L, true>(A, beta, tbuf, tw);
    fft_first<FK_C2R, L, true>(B, self ? G::L1 / 2 : G::L1 - beta, tbuf, tw);
  }
  __syncthreads();  // back to a team per row
  if constexpr (G::S == 3) {
    fft_mid<FK_C2R, L, true>(buf, j, tw);
    team_sync<T>(mask);
  }
  float2* rowp =
      reinterpret_cast<float2*>(real_plane(d, second ? dsel1 : dsel0)) + (size_t)row * L;
  float amax = 0.0f;
#pragma unroll
  for (int q = 0; q < G::E / rl; ++q) {
    const int kap = j + T * q;
    float2 x[rl];
    fft_last<FK_C2R, L, true>(x, kap, buf);
#pragma unroll
    for (int i = 0; i < rl; ++i) {
      const float2 v = cscale(x[i], scale);
      rowp[kap + i * G::KL] = v;
      amax = fmaxf(amax, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
  }
  // largest |value| of the plane (u_I, u_p): bounds the guided filter's
  // split window sums; non-negative floats order like their bit patterns
  if (st) {
    amax = warp_max(amax);  // the teams of a warp share one image and plane
    if ((threadIdx.x & 31) == 0)
      atomicMax(&st[cd.img0 + li].absmax[second ? 1 : 0], __float_as_uint(amax));
  }
}

// ---------------------------------------------------------------------------
// Column passes.  An item is B adjacent packed columns of one image (B = TB
// in the iteration kernels: one contiguous tile of M x B values), thread
// (b, j) = (threadIdx % B, threadIdx / B) of column b's team.  Consecutive
// threads walk the B columns, then consecutive rows, so every load and store
// of a warp covers whole sectors of the tile.  They are bound by the latency
// of these loads at 16 to 24 warps per SM: inputs come straight from global
// memory to the first stage's registers (no landing tile, which cost a pass
// through shared memory and half the blocks per SM), the next item's tiles are
// prefetched into L2, and the tile width is a compile-time constant, so that
// a thread's rows are immediate offsets.  The prefetch is issued just before the
// last stage: at the start of an item it comes so early that on a batch larger
// than L2 its lines are gone before use (ncu: 329 MB read for 201 MB of
// tiles; the solve pass took 8.6 ms per batched solve, 6.8 ms with the late
// prefetch, 7.1 ms with none).
// ---------------------------------------------------------------------------

// Setup / utility column FFT: plane src -> dst, in place allowed; B columns
// (inside one tile) per block.
template <int M, bool INV>
__global__ void __launch_bounds__(512)
k_col_plain(ClassDesc cd, const ImgDesc* __restrict__ imgs, const __grid_constant__ ImgDesc one,
            const float2* __restrict__ tw, int B, int src_sel, int dst_sel) {
  extern __shared__ __align__(16) float2 smem[];
  using G = FftGeo<FK_COL, M>;
  constexpr int T = G::T, r0 = G::RF;
  const int Lc = cd.N / 2, TB = cd.TB;
  const int cpi = Lc / B;
  const ImgDesc& d = imgs ? imgs[cd.img0 + blockIdx.x / cpi] : one;
  const int c0 = (blockIdx.x % cpi) * B;
  const int b = threadIdx.x & (B - 1), j = threadIdx.x >> (__ffs(B) - 1);
  const size_t off = (size_t)(c0 / TB) * M * TB + (c0 % TB) + b;
  const float2* src = cplx_plane(d, src_sel) + off;
  float2* dst = cplx_plane(d, dst_sel) + off;
  float2* buf = smem + b * col_stride<M>(B);
#pragma unroll
  for (int q = 0; q < G::E / r0; ++q) {
    const int beta = j + T * q;
    float2 x[r0];
#pragma unroll
    for (int i = 0; i < r0; ++i) x[i] = load_stream(src + (size_t)(beta + i * G::L1) * TB);
    fft_first<FK_COL, M, INV>(x, beta, buf, tw);
  }
  __syncthreads();
  if constexpr (G::S == 3) {
    fft_mid<FK_COL, M, INV>(buf, j, tw);
    __syncthreads();
  }
  float2 x[G::E];
  fft_last<FK_COL, M, INV>(x, j, buf);
#pragma unroll
  for (int i = 0; i < G::E; ++i) dst[(size_t)(j + i * T) * TB] = x[i];
}

// Forward column FFT of the iterate's row spectra (in place on S), fused with
// the first evaluation of Eq. 11: node sums, or the moments about the
// extrapolated lambda (lambda.cuh), from the transform's outputs in registers
// and H, Y loaded beside them.  A block takes a contiguous range of items and
// keeps its sums while consecutive items belong to the same image; it
// publishes them (one partial slot, one counter update) only when the image
// changes.  Batched solve of 256 images, 15 iterations: 10.3 ms with staged
// tiles and 12 or 8 nodes per pass, 6.9 ms as it is; 4 images of 4096^2, 30
// iterations: 16.2 -> 9.2 ms (without prefetch, which takes 10.8 ms there: one
// block per SM loads and computes in turn).  Three blocks per SM (80 registers)
// spill and take 8.0 ms.
template <int M, int BT>
__global__ void __launch_bounds__(M >= 4096 ? 512 : 256, M >= 4096 ? 1 : 2)
k_col_fwd_lambda(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st,
                 const float2* __restrict__ tw, int iter, int row_items) {
  extern __shared__ __align__(16) float2 smem[];
  using G = FftGeo<FK_COL, M>;
  constexpr int T = G::T, r0 = G::RF, E = G::E;
  __shared__ float2 s_nodes[KNODES / 2];
  __shared__ int s_mode;
  __shared__ double s_tot[KNODES + 1];
  __shared__ int s_flag;
  __shared__ WarpAcc s_wacc;
  const int B = BT > 0 ? BT : cd.TB;
  const int Lc = cd.N / 2;
  const int cpi = Lc / B;
  const int n_items = cd.n_img * cpi;
  const int per_cta = (n_items + gridDim.x - 1) / gridDim.x;
  const int first = blockIdx.x * per_cta;
  const int stop = min(first + per_cta, n_items);
  if (first >= stop) return;  // the last blocks of a grid that does not divide the items
  const int tile = M * B;
  const int b = threadIdx.x & (B - 1), j = threadIdx.x >> (__ffs(B) - 1);
  float2* buf = smem + b * col_stride<M>(B);
  double* red = reinterpret_cast<double*>(smem + B * col_stride<M>(B));
  auto prefetch = [&](int item) {
    if (item < stop) {
      const ImgDesc& d = imgs[cd.img0 + item / cpi];
      const size_t off = (size_t)(item % cpi) * tile;
      prefetch_l2(d.S + off, (unsigned int)(tile * sizeof(float2)));
      prefetch_l2(d.H + off, (unsigned int)(tile * sizeof(float2)));
      prefetch_l2(d.Y + off, (unsigned int)(tile * sizeof(float2)));
    }
  };
  BinAcc acc;
  acc.clear();
  int cur = -1, slot = 0, count = 0;
  // publish the sums of `count` items of image `cur` (slot = its first tile);
  // the block completing the image's count reduces all slots and updates
  // the image's lambda
  auto flush = [&]() {
    ImgState* S = st + cur;
    const ImgDesc& d = imgs[cur];
    block_partials_folded(&s_wacc, d.part + (size_t)slot * (KNODES + 1));
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned int prev = atomicAdd(&S->cta_done, (unsigned int)count);
      s_flag = (prev + count == (unsigned int)cpi);
    }
    __syncthreads();
    if (s_flag) {
      __threadfence();
      block_sum_columns(d.part, cpi, KNODES + 1, KNODES + 1, red, s_tot);
      for (int q = threadIdx.x; q < cpi * (KNODES + 1); q += blockDim.x) d.part[q] = 0.0;
      if (threadIdx.x < 32)
        lambda_update_warp(S, s_tot, true, false, iter, d.lam_out, d.res_out,
                           threadIdx.x);
      if (threadIdx.x == 0) {
        S->cta_done = 0;
        __threadfence();
      }
    }
    count = 0;
  };
  warp_acc_clear(&s_wacc);  // first use follows the loop's __syncthreads()
  for (int item = first;; ++item) {
    const int gi = item < stop ? cd.img0 + item / cpi : -1;
    const int t = item % cpi;
    if (gi != cur) {
      __syncthreads();
      if (count > 0) flush();
      if (item >= stop) break;
      cur = gi;
      slot = t;
      for (int q = threadIdx.x; q < KNODES / 2; q += blockDim.x)
        s_nodes[q] = __ldcg(reinterpret_cast<const float2*>(st[gi].node) + q);
      if (threadIdx.x == 0) s_mode = __ldcg(&st[gi].mode);
    }
    const ImgDesc& d = imgs[gi];
    ImgState* S = st + gi;
    const size_t off = (size_t)t * tile;
    float2* spec = d.S + off + b;
    if (t == 0) {  // the DC bin needs sum(u_E): total of the row pass's partials
      block_sum_columns(d.rowsum, row_items, 1, 1, red, s_tot);
      if (threadIdx.x == 0) S->sum_u = s_tot[0];
    }
    __syncthreads();  // the previous item's reads of the buffer are done
#pragma unroll
    for (int q = 0; q < E / r0; ++q) {
      const int beta = j + T * q;
      float2 x[r0];
#pragma unroll
      for (int i = 0; i < r0; ++i) x[i] = load_stream(spec + (beta + i * G::L1) * B);
      fft_first<FK_COL, M, false>(x, beta, buf, tw);
    }
    __syncthreads();
    if constexpr (G::S == 3) {
      fft_mid<FK_COL, M, false>(buf, j, tw);
      __syncthreads();
    }
    if (M < 4096) prefetch(item + 1);
    float2 x[E];  // U_E at rows j + T i
    fft_last<FK_COL, M, false>(x, j, buf);
    const bool mom = s_mode == MODE_MOM;
    const float c = s_nodes[0].x;
    const float2* Hc = d.H + off + b;
    const float2* Yc = d.Y + off + b;
    // residual terms |H U_E - Y|^2 and |H|^2 of one bin
    auto terms = [](float2 H, float2 Y, float2 U, float& r, float& a) {
      const float2 e = csub(cmul(H, U), Y);
      r = fmaf(e.x, e.x, e.y * e.y);
      a = fmaf(H.x, H.x, H.y * H.y);
    };
    bool pair0 = false;
    if (t == 0) {  // packed column 0: the rows k and M - k of the outputs meet in shared memory
      __syncthreads();
      pair0 = b == 0;
      if (pair0) {
#pragma unroll
        for (int i = 0; i < E; ++i) smem[j + T * i] = x[i];
      }
      __syncthreads();
    }
    if (!pair0) {
#pragma unroll
      for (int i = 0; i < E; ++i) spec[(j + T * i) * B] = x[i];
    }
    constexpr int G4 = E < 4 ? E : 4;  // bins whose loads are in flight together
    if (mom && !pair0) {
#pragma unroll
      for (int i0 = 0; i0 < E; i0 += G4) {
        float2 H[G4], Y[G4];
#pragma unroll
        for (int i = 0; i < G4; ++i) {
          H[i] = load_stream(Hc + (j + T * (i0 + i)) * B);
          Y[i] = load_stream(Yc + (j + T * (i0 + i)) * B);
        }
#pragma unroll
        for (int i = 0; i < G4; ++i) {
          float r, a;
          terms(H[i], Y[i], x[i0 + i], r, a);
          accum_bin_moments(2.0f * r, a, c, acc);  // bins l and N-l
        }
      }
    } else {
      // node sums (the first iterations) and column 0: a loop of G4 bins a
      // time, so that the code stays small in the instruction cache
      float2 nodes[KNODES / 2];
#pragma unroll
      for (int q = 0; q < KNODES / 2; ++q) nodes[q] = s_nodes[q];
#pragma unroll 1
      for (int i0 = 0; i0 < E; i0 += G4) {
        float r[2 * G4], a[2 * G4];  // terms of the bins, weights included
        if (!pair0) {
          float2 H[G4], Y[G4], U[G4];
#pragma unroll
          for (int i = 0; i < G4; ++i) {
            const int o = (j + T * (i0 + i)) * B;
            H[i] = load_stream(Hc + o);
            Y[i] = load_stream(Yc + o);
            U[i] = spec[o];
          }
#pragma unroll
          for (int i = 0; i < G4; ++i) {
            terms(H[i], Y[i], U[i], r[i], a[i]);
            r[i] *= 2.0f;  // bins l and N-l
          }
        } else {
          float2 HA[G4], HB[G4], YA[G4], YB[G4];
#pragma unroll
          for (int i = 0; i < G4; ++i) {
            const int k = j + T * (i0 + i);
            HA[i] = __ldcg(&d.H0[k]);
            HB[i] = __ldcg(&d.HN[k]);
            YA[i] = __ldcg(&d.Y0[k]);
            YB[i] = __ldcg(&d.YN[k]);
          }
#pragma unroll
          for (int i = 0; i < G4; ++i) {
            const int k = j + T * (i0 + i);
            float2 U = smem[k];
            const float2 Um = smem[(M - k) & (M - 1)];
            float2 UA, UB;
            unpack_pair(U, Um, UA, UB);
            terms(HA[i], YA[i], UA, r[i], a[i]);
            terms(HB[i], YB[i], UB, r[G4 + i], a[G4 + i]);
            if (k == 0) {
              // DC bin in FP64 from exact sums: d00 = sum(h) sum(u_E) - sum(y)
              const double su = s_tot[0];
              const double d00 = S->sum_h * su - S->sum_y;
              S->d00 = d00;
              r[i] = (float)(d00 * d00);
              U.x = (float)su;
            }
            spec[k * B] = U;
          }
        }
#pragma unroll
        for (int i = 0; i < 2 * G4; ++i) {
          if (i >= G4 && !pair0) break;
          if (mom)
            accum_bin_moments(r[i], a[i], c, acc);
          else
            accum_bin(r[i], a[i], nodes, acc);
        }
      }
    }
    warp_fold(acc, mom ? KMOM : KNODES, &s_wacc);
    ++count;
  }
}

// The node sums of Eq. 11 over `pairs` bin pairs (in tiled order) from pair p0
// on, by nt threads of which this is thread t, folded into wa.  Bins in pairs
// (b, b+1) of one tile row, read as 16-byte vectors; runs of 8 pairs per
// thread between folds (uniform control flow).
GFD_D void pass_bins(const ClassDesc& cd, const ImgDesc& d, const ImgState* S,
                     const float2 (&nodes)[KNODES / 2], int p0, int pairs, int t, int nt,
                     WarpAcc* wa) {
  const int TB = cd.TB, M = cd.M;
  const int lg_tile = __ffs(M * TB) - 1, lg_tb = __ffs(TB) - 1;  // powers of two
  const float4* S4 = reinterpret_cast<const float4*>(d.S);
  const float4* H4 = reinterpret_cast<const float4*>(d.H);
  const float4* Y4 = reinterpret_cast<const float4*>(d.Y);
  BinAcc acc;
  acc.clear();
  for (int base = 0; base < pairs; base += 8 * nt) {
#pragma unroll 4
    for (int q = 0; q < 8; ++q) {
      const int pi = base + q * nt + t;
      if (pi < pairs) {
        const int e = 2 * (p0 + pi);
        const int tl = e >> lg_tile, rem = e & ((1 << lg_tile) - 1);
        const int k = rem >> lg_tb, b = rem & (TB - 1);  // b even
        const float4 U2 = __ldcg(&S4[p0 + pi]);
        const float4 H2 = __ldcg(&H4[p0 + pi]), Y2 = __ldcg(&Y4[p0 + pi]);
        {  // bin b + 1 (never column 0)
          const float2 H = make_float2(H2.z, H2.w);
          const float2 r = csub(cmul(H, make_float2(U2.z, U2.w)), make_float2(Y2.z, Y2.w));
          accum_bin(2.0f * fmaf(r.x, r.x, r.y * r.y), fmaf(H.x, H.x, H.y * H.y), nodes, acc);
        }
        if (tl != 0 || b != 0) {
          const float2 H = make_float2(H2.x, H2.y);
          const float2 r = csub(cmul(H, make_float2(U2.x, U2.y)), make_float2(Y2.x, Y2.y));
          accum_bin(2.0f * fmaf(r.x, r.x, r.y * r.y), fmaf(H.x, H.x, H.y * H.y), nodes, acc);
        } else {  // packed column 0: bins (k, 0) and (k, N/2)
          const float2 U = make_float2(U2.x, U2.y);
          const float2 Um = __ldcg(&d.S[(size_t)((M - k) & (M - 1)) * TB]);
          float2 UA, UB;
          unpack_pair(U, Um, UA, UB);
          const float2 HA = d.H0[k], HB = d.HN[k], YA = d.Y0[k], YB = d.YN[k];
          float rA;
          if (k == 0) {
            const double d00 = __ldcg(&S->d00);
            rA = (float)(d00 * d00);
          } else {
            const float2 r = csub(cmul(HA, UA), YA);
            rA = fmaf(r.x, r.x, r.y * r.y);
          }
          const float2 rb = csub(cmul(HB, UB), YB);
          accum_bin(rA, fmaf(HA.x, HA.x, HA.y * HA.y), nodes, acc);
          accum_bin(fmaf(rb.x, rb.x, rb.y * rb.y), fmaf(HB.x, HB.x, HB.y * HB.y), nodes, acc);
        }
      }
    }
    warp_fold(acc, KNODES, wa);
  }
}

// Fallback evaluation of Eq. 11 over the stored spectrum U_E for images whose
// root is still open; a block covers `chunk` elements (in tiled order) of one
// image.
__global__ void __launch_bounds__(256)
k_lambda_pass(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st, int chunk, int iter,
              int last_chance) {
  __shared__ float s_nodes[KNODES];
  __shared__ double red[32 * (KNODES + 1)];
  __shared__ double s_tot[KNODES + 1];
  __shared__ int s_flag;
  __shared__ WarpAcc s_wacc;
  const int per_img = cd.M * (cd.N / 2);
  const int cpi = per_img / chunk;
  const int gi = cd.img0 + blockIdx.x / cpi;
  ImgState* S = st + gi;
  if (__ldcg(&S->need) == 0) return;
  const ImgDesc& d = imgs[gi];
  for (int q = threadIdx.x; q < KNODES; q += blockDim.x) s_nodes[q] = __ldcg(&S->node[q]);
  warp_acc_clear(&s_wacc);
  __syncthreads();
  float2 nodes[KNODES / 2];
#pragma unroll
  for (int q = 0; q < KNODES / 2; ++q) nodes[q] = make_float2(s_nodes[2 * q], s_nodes[2 * q + 1]);
  pass_bins(cd, d, S, nodes, (blockIdx.x % cpi) * (chunk / 2), chunk / 2, threadIdx.x, blockDim.x,
            &s_wacc);
  block_partials_folded(&s_wacc, d.part + (size_t)(blockIdx.x % cpi) * (KNODES + 1));
  if (last_item(&S->cta_done, cpi, &s_flag)) {
    block_sum_columns(d.part, cpi, KNODES + 1, KNODES + 1, red, s_tot);
    for (int q = threadIdx.x; q < cpi * (KNODES + 1); q += blockDim.x) d.part[q] = 0.0;
    if (threadIdx.x < 32)
      lambda_update_warp(S, s_tot, false, last_chance != 0, iter,
                         d.lam_out, d.res_out, threadIdx.x);
    if (threadIdx.x == 0) {
      S->cta_done = 0;
      __threadfence();
    }
  }
}


// All fallback passes of an iteration for small canvases: a cluster of
// LOOP_BLOCKS blocks per image repeats the pass until the image's root is
// resolved (npass at most), its blocks' sums meeting in the first block's
// shared memory.  One launch instead of npass, most of which find nothing to
// do and cost 2.5 to 4 us each on the chain of a small solve.
constexpr int LOOP_BLOCKS = 8, LOOP_THREADS = 512;

__global__ void __cluster_dims__(LOOP_BLOCKS, 1, 1) __launch_bounds__(LOOP_THREADS)
k_lambda_loop(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st, int iter, int npass) {
  namespace cg = cooperative_groups;
  __shared__ double s_part[LOOP_BLOCKS][KNODES + 1];  // of the cluster's first block
  __shared__ double s_tot[KNODES + 1];
  __shared__ WarpAcc s_wacc;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = blockIdx.x % LOOP_BLOCKS;
  const int gi = cd.img0 + blockIdx.x / LOOP_BLOCKS;
  ImgState* S = st + gi;
  // read by every block before the first cluster barrier, changed after it
  if (__ldcg(&S->need) == 0) return;
  // The first block's shared memory is written below: it has to have started.
  // (At the end no block touches another's memory after the last barrier.)
  cl.sync();
  const ImgDesc& d = imgs[gi];
  const int pairs = cd.M * (cd.N / 2) / 2;
  double* part = cl.map_shared_rank(&s_part[0][0], 0) + rank * (KNODES + 1);
  for (int p = 1; p <= npass; ++p) {
    float2 nodes[KNODES / 2];
#pragma unroll
    for (int q = 0; q < KNODES / 2; ++q)
      nodes[q] = __ldcg(reinterpret_cast<const float2*>(S->node) + q);
    warp_acc_clear(&s_wacc);
    __syncthreads();
    pass_bins(cd, d, S, nodes, 0, pairs, rank * LOOP_THREADS + threadIdx.x,
              LOOP_BLOCKS * LOOP_THREADS, &s_wacc);
    block_partials_folded(&s_wacc, part);
    cl.sync();
    if (rank == 0 && threadIdx.x < 32) {
      if (threadIdx.x <= KNODES) {
        double v[LOOP_BLOCKS];
#pragma unroll
        for (int r = 0; r < LOOP_BLOCKS; ++r) v[r] = s_part[r][threadIdx.x];
#pragma unroll
        for (int o = LOOP_BLOCKS / 2; o > 0; o /= 2)
#pragma unroll
          for (int r = 0; r < o; ++r) v[r] += v[r + o];
        s_tot[threadIdx.x] = v[0];
      }
      __syncwarp();
      lambda_update_warp(S, s_tot, false, p == npass, iter, d.lam_out, d.res_out, threadIdx.x);
      __threadfence();
    }
    cl.sync();
    if (__ldcg(&S->need) == 0) break;  // the same for the whole cluster
  }
}

// Eq. 8 and 9 at rows k of packed column 0, which holds the bins (k, 0) and
// (k, N/2): U_I and U_p of both, packed again.
__device__ __noinline__ float4 solve_col0(const ImgDesc& d, int M, int B, int k, float lam,
                                          float d2r) {
  const float2 U = __ldcg(&d.S[k * B]), Um = __ldcg(&d.S[((M - k) & (M - 1)) * B]);
  float2 UA, UB, IA, IB, PA, PB;
  unpack_pair(U, Um, UA, UB);
  solve_bin(UA, d.H0[k], d.Y0[k], lam, d2r, IA, PA);
  solve_bin(UB, d.HN[k], d.YN[k], lam, d2r + 4.0f, IB, PB);
  const float2 I = pack_pair(IA, IB), P = pack_pair(PA, PB);
  return make_float4(I.x, I.y, P.x, P.y);
}

// Spectral solves fused with the inverse column FFTs: the first stage's inputs
// are formed by Eq. 8 and 9 from U_E, H and Y as they are loaded (each bin once),
// U_I and U_p then go through one buffer each.  Batched solve of 256 images, 15
// iterations: 14.8 ms with staged tiles, 6.8 ms as it is; 4 images of 4096^2,
// 30 iterations: 22.6 -> 9.4 ms.  Three blocks per SM where the first radix is
// small enough for 80 registers (9.6 -> 8.6 ms); a first radix of 16 holds both
// planes' 16 inputs and keeps 128.
template <int M, int BT>
__global__ void __launch_bounds__(M >= 4096 ? 512 : 256,
                                  M >= 4096 ? 1 : (FftGeo<FK_COL, M>::RF <= 8 && M >= 512 ? 3 : 2))
k_col_solve_inv(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st,
                const float2* __restrict__ tw, const float* __restrict__ d2tab) {
  extern __shared__ __align__(16) float2 smem[];
  using G = FftGeo<FK_COL, M>;
  constexpr int T = G::T, r0 = G::RF, E = G::E;
  const int N = cd.N, Lc = N / 2, B = BT > 0 ? BT : cd.TB;
  const int cpi = Lc / B;
  const int n_items = cd.n_img * cpi;
  const int tile = M * B;
  const int b = threadIdx.x & (B - 1), j = threadIdx.x >> (__ffs(B) - 1);
  float2* bufI = smem + b * col_stride<M>(B);
  float2* bufP = bufI + B * col_stride<M>(B);
  const float* d2m = d2tab + tab_off(M);
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int gi = cd.img0 + item / cpi;
    const ImgDesc& d = imgs[gi];
    const int t = item % cpi;
    const int col = t * B + b;
    const size_t off = (size_t)t * tile + b;
    auto prefetch_next = [&]() {
      const int next = item + gridDim.x;
      if (next < n_items) {
        const ImgDesc& dn = imgs[cd.img0 + next / cpi];
        const size_t on = (size_t)(next % cpi) * tile;
        prefetch_l2(dn.S + on, (unsigned int)(tile * sizeof(float2)));
        prefetch_l2(dn.H + on, (unsigned int)(tile * sizeof(float2)));
        prefetch_l2(dn.Y + on, (unsigned int)(tile * sizeof(float2)));
      }
    };
    const double lamd = __ldcg(&st[gi].lam);
    const bool branch = !(lamd < 1e300);  // lambda = inf: u_I = u_p = u_E (Sec. 3.2)
    if (t == 0 && threadIdx.x == 0) {  // the inverse row pass re-forms them
      st[gi].absmax[0] = 0u;
      st[gi].absmax[1] = 0u;
    }
    const float lam = (float)lamd;
    const float d2c = __ldg(&d2tab[tab_off(N) + col]);
    const float2* Sc = d.S + off;
    const float2* Hc = d.H + off;
    const float2* Yc = d.Y + off;
    if (item != (int)blockIdx.x) __syncthreads();  // the previous item's reads are done
#pragma unroll
    for (int q = 0; q < E / r0; ++q) {
      const int beta = j + T * q;
      float2 xI[r0], xP[r0];
      if (branch) {
#pragma unroll
        for (int i = 0; i < r0; ++i) xI[i] = xP[i] = load_stream(Sc + (beta + i * G::L1) * B);
      } else if (col != 0) {
        constexpr int G4 = r0 < 4 ? r0 : 4;
#pragma unroll
        for (int i0 = 0; i0 < r0; i0 += G4) {
          float2 U[G4], H[G4], Y[G4];
#pragma unroll
          for (int i = 0; i < G4; ++i) {
            const int o = (beta + (i0 + i) * G::L1) * B;
            U[i] = load_stream(Sc + o);
            H[i] = load_stream(Hc + o);
            Y[i] = load_stream(Yc + o);
          }
#pragma unroll
          for (int i = 0; i < G4; ++i)
            solve_bin(U[i], H[i], Y[i], lam, __ldg(&d2m[beta + (i0 + i) * G::L1]) + d2c,
                      xI[i0 + i], xP[i0 + i]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < r0; ++i) {
          const int k = beta + i * G::L1;
          const float4 v = solve_col0(d, M, B, k, lam, __ldg(&d2m[k]));
          xI[i] = make_float2(v.x, v.y);
          xP[i] = make_float2(v.z, v.w);
        }
      }
      fft_first<FK_COL, M, true>(xI, beta, bufI, tw);
      fft_first<FK_COL, M, true>(xP, beta, bufP, tw);
    }
    __syncthreads();
    if constexpr (G::S == 3) {
      fft_mid<FK_COL, M, true>(bufI, j, tw);
      fft_mid<FK_COL, M, true>(bufP, j, tw);
      __syncthreads();
    }
    prefetch_next();
    float2 x[E];
    float2* qi = d.QI + off;
    fft_last<FK_COL, M, true>(x, j, bufI);
#pragma unroll
    for (int i = 0; i < E; ++i) qi[(j + T * i) * B] = x[i];
    float2* qp = d.Qp + off;
    fft_last<FK_COL, M, true>(x, j, bufP);
#pragma unroll
    for (int i = 0; i < E; ++i) qp[(j + T * i) * B] = x[i];
  }
}

// ---------------------------------------------------------------------------
// Column passes of small problems: one item per block, 4 rows per thread
// (short_fft), every global load requested before the transform.  Tiles of
// class_tile_width.  One 256 x 256 image: forward pass 25 us as the persistent
// radix-16 kernel (8 blocks of 256 threads), 15 us here, more than half of it
// the reductions and the root of lambda behind the transform; solve pass 11 ->
// 6 us.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512, 2)
k_col_fwd_lambda_short(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st,
                       const float2* __restrict__ tw, int lg, int iter) {
  extern __shared__ __align__(16) float2 smem[];
  __shared__ double s_tot[KNODES + 1];
  __shared__ int s_flag;
  __shared__ WarpAcc s_wacc;
  const int M = cd.M, B = cd.TB, Lc = cd.N / 2, cpi = Lc / B;
  const int b = threadIdx.x & (B - 1), j = threadIdx.x >> (__ffs(B) - 1);
  const int Q = M / 4;  // rows j + i Q
  const int cs = short_pos(M) + 1;
  double* red = reinterpret_cast<double*>(smem + ((B * cs + 1) & ~1));
  const int gi = cd.img0 + blockIdx.x / cpi, t = blockIdx.x % cpi;
  const ImgDesc& d = imgs[gi];
  ImgState* S = st + gi;
  const size_t off = (size_t)t * M * B + b;
  float2* spec = d.S + off;
  float2 x[1][4], H[4], Y[4];
  const bool pair0 = t == 0 && b == 0;  // packed column 0: bins (k, 0) and (k, N/2)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = j + i * Q;
    x[0][i] = load_stream(spec + k * B);
    H[i] = pair0 ? __ldcg(&d.H0[k]) : load_stream(d.H + off + k * B);
    Y[i] = pair0 ? __ldcg(&d.Y0[k]) : load_stream(d.Y + off + k * B);
  }
  __shared__ float2 s_nodes[KNODES / 2];
  for (int q = threadIdx.x; q < KNODES / 2; q += blockDim.x)
    s_nodes[q] = __ldcg(reinterpret_cast<const float2*>(S->node) + q);
  const bool mom = __ldcg(&S->mode) == MODE_MOM;
  warp_acc_clear(&s_wacc);  // first use follows the transform's barriers
  if (t == 0) {  // the DC bin needs sum(u_E): total of the row pass's sums
    block_sum_columns(d.rowsum, M, 1, 1, red, s_tot);
    if (threadIdx.x == 0) S->sum_u = s_tot[0];
  }
  float2* const bufs[1] = {smem + b * cs};
  short_fft<1, false>(x, bufs, lg, j, tw);
  if (t == 0) {  // rows k and M - k of column 0 meet in shared memory
    __syncthreads();
    if (pair0) {
#pragma unroll
      for (int i = 0; i < 4; ++i) smem[j + i * Q] = x[0][i];
    }
    __syncthreads();
  }
  BinAcc acc;
  acc.clear();
  auto bin = [&](float2 h, float2 y, float2 u, float w, bool dc) {
    const float2 e = csub(cmul(h, u), y);
    float r = w * fmaf(e.x, e.x, e.y * e.y);
    if (dc) {
      // DC bin in FP64 from exact sums: d00 = sum(h) sum(u_E) - sum(y)
      const double d00 = S->sum_h * s_tot[0] - S->sum_y;
      S->d00 = d00;
      r = (float)(d00 * d00);
    }
    const float a = fmaf(h.x, h.x, h.y * h.y);
    if (mom)
      accum_bin_moments(r, a, s_nodes[0].x, acc);
    else
      accum_bin(r, a, s_nodes, acc);
  };
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int k = j + i * Q;
    float2 U = x[0][i];
    if (pair0) {
      float2 UA, UB;
      unpack_pair(smem[k], smem[(M - k) & (M - 1)], UA, UB);
      bin(H[i], Y[i], UA, 1.0f, k == 0);
      bin(__ldcg(&d.HN[k]), __ldcg(&d.YN[k]), UB, 1.0f, false);
      if (k == 0) U.x = (float)s_tot[0];
    } else {
      bin(H[i], Y[i], U, 2.0f, false);  // bins l and N-l
    }
    spec[k * B] = U;
  }
  warp_fold(acc, mom ? KMOM : KNODES, &s_wacc);
  block_partials_folded(&s_wacc, d.part + (size_t)t * (KNODES + 1));
  if (last_item(&S->cta_done, cpi, &s_flag)) {
    block_sum_columns(d.part, cpi, KNODES + 1, KNODES + 1, red, s_tot);
    for (int q = threadIdx.x; q < cpi * (KNODES + 1); q += blockDim.x) d.part[q] = 0.0;
    if (threadIdx.x < 32)
      lambda_update_warp(S, s_tot, true, false, iter, d.lam_out, d.res_out,
                         threadIdx.x);
    if (threadIdx.x == 0) {
      S->cta_done = 0;
      __threadfence();
    }
  }
}

__global__ void __launch_bounds__(512)
k_col_solve_inv_short(ClassDesc cd, const ImgDesc* __restrict__ imgs, ImgState* st,
                      const float2* __restrict__ tw, const float* __restrict__ d2tab, int lg) {
  extern __shared__ __align__(16) float2 smem[];
  const int M = cd.M, B = cd.TB, Lc = cd.N / 2, cpi = Lc / B;
  const int b = threadIdx.x & (B - 1), j = threadIdx.x >> (__ffs(B) - 1);
  const int Q = M / 4, cs = short_pos(M) + 1;
  const int gi = cd.img0 + blockIdx.x / cpi, t = blockIdx.x % cpi;
  const ImgDesc& d = imgs[gi];
  const int col = t * B + b;
  const size_t off = (size_t)t * M * B + b;
  const double lamd = __ldcg(&st[gi].lam);
  const bool branch = !(lamd < 1e300);  // lambda = inf: u_I = u_p = u_E (Sec. 3.2)
  const float lam = (float)lamd;
  if (t == 0 && threadIdx.x == 0) {  // the inverse row pass re-forms them
    st[gi].absmax[0] = 0u;
    st[gi].absmax[1] = 0u;
  }
  const float d2c = __ldg(&d2tab[tab_off(cd.N) + col]);
  float2 x[2][4];
  if (branch) {
#pragma unroll
    for (int i = 0; i < 4; ++i) x[0][i] = x[1][i] = load_stream(d.S + off + (j + i * Q) * B);
  } else if (col != 0) {
    float2 U[4], H[4], Y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int o = (j + i * Q) * B;
      U[i] = load_stream(d.S + off + o);
      H[i] = load_stream(d.H + off + o);
      Y[i] = load_stream(d.Y + off + o);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      solve_bin(U[i], H[i], Y[i], lam, __ldg(&d2tab[tab_off(M) + j + i * Q]) + d2c, x[0][i],
                x[1][i]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = j + i * Q;
      const float4 v = solve_col0(d, M, B, k, lam, __ldg(&d2tab[tab_off(M) + k]));
      x[0][i] = make_float2(v.x, v.y);
      x[1][i] = make_float2(v.z, v.w);
    }
  }
  float2* const bufs[2] = {smem + b * cs, smem + (B + b) * cs};
  short_fft<2, true>(x, bufs, lg, j, tw);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    d.QI[off + (j + i * Q) * B] = x[0][i];
    d.Qp[off + (j + i * Q) * B] = x[1][i];
  }
}

// ---------------------------------------------------------------------------
// launch configuration and dispatch
// ---------------------------------------------------------------------------
static int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
  }
  return n;
}

// Persistent grid: as many blocks as fit on the device at once (never more
// than there are items).
template <class K>
static int persistent_grid(K kernel, int threads, size_t smem, int n_items, int div = 1) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) != cudaSuccess ||
      per_sm < 1)
    per_sm = 1;
  long long g = (long long)per_sm * sm_count();
  if (div > 1) g = (g + div - 1) / div;
  return (int)(g < n_items ? g : n_items);
}

// Largest power of two <= v (v >= 1): rows per item and tile widths are
// powers of two, so the tile copies index by shifts.
static int floor_pow2(int v) {
  int p = 1;
  while (2 * p <= v) p *= 2;
  return p;
}

// Threads of a row pass's team for rows of L packed values.
static int row_team(int L) { return L / fft_elems(FK_C2R, L); }

int rows_per_item(int L, int M, int row_threads) {
  int r = (row_threads > 0 ? row_threads : DEF_ROW_THREADS) / row_team(L);
  if (r < 1) r = 1;
  if (r > M) r = M;
  return floor_pow2(r);
}

// Tile width of a class's spectra = columns per column item: a block of about
// col_threads threads (512 for M = 4096), at least 2 columns (16-byte
// copies), at most N/2.
int class_tile_width(int M, int N, int col_threads, bool short_cols) {
  if (short_cols) {
    int B = M >= 1024 ? 2 : 4;  // M/4 threads per column: 512 per block at most
    while (B * M / 4 < 32 && B < N / 2) B *= 2;
    return B < N / 2 ? B : N / 2;
  }
  const int T = M / fft_elems(FK_COL, M);
  const int ct = col_threads > 0 ? (col_threads > 256 ? 256 : col_threads) : DEF_COL_THREADS;
  const int threads = M >= 4096 ? 512 : ct;
  int B = threads / T;
  if (B < 2) B = 2;
  if (B > N / 2) B = N / 2;
  return floor_pow2(B);
}

#define GFD_CASE_L(F, ...)             \
  case 4: F<4>(__VA_ARGS__); break;     \
  case 8: F<8>(__VA_ARGS__); break;     \
  case 16: F<16>(__VA_ARGS__); break;   \
  case 32: F<32>(__VA_ARGS__); break;   \
  case 64: F<64>(__VA_ARGS__); break;   \
  case 128: F<128>(__VA_ARGS__); break; \
  case 256: F<256>(__VA_ARGS__); break; \
  case 512: F<512>(__VA_ARGS__); break; \
  case 1024: F<1024>(__VA_ARGS__); break; \
  case 2048: F<2048>(__VA_ARGS__); break;

#define GFD_CASE_M(F, ...)               \
  case 8: F<8>(__VA_ARGS__); break;       \
  case 16: F<16>(__VA_ARGS__); break;     \
  case 32: F<32>(__VA_ARGS__); break;     \
  case 64: F<64>(__VA_ARGS__); break;     \
  case 128: F<128>(__VA_ARGS__); break;   \
  case 256: F<256>(__VA_ARGS__); break;   \
  case 512: F<512>(__VA_ARGS__); break;   \
  case 1024: F<1024>(__VA_ARGS__); break; \
  case 2048: F<2048>(__VA_ARGS__); break; \
  case 4096: F<4096>(__VA_ARGS__); break;

template <int L>
static void do_row_r2c(const ClassLaunch& c, const Tables& t, int src, int dst, int sum,
                       cudaStream_t s) {
  using G = FftGeo<FK_R2C, L>;
  const int rpc = rows_per_item(L, c.cd.M, c.row_threads);
  const int blocks = c.cd.n_img * c.cd.M / rpc;
  k_row_r2c<L><<<blocks, rpc * G::T, rpc * G::SIZE * sizeof(float2), s>>>(
      c.cd, c.imgs, one_desc(c), t.tw, rpc, src, dst, sum);
}

cudaError_t launch_row_r2c(const ClassLaunch& c, const Tables& t, int src, int dst,
                           bool do_sum, cudaStream_t s) {
  switch (c.cd.N / 2) {
    GFD_CASE_L(do_row_r2c, c, t, src, dst, do_sum ? 1 : 0, s)
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int L>
static void do_row_c2r(const ClassLaunch& c, const Tables& t, int sel0, int sel1, int dsel0,
                       int dsel1, float scale, cudaStream_t s) {
  using G = FftGeo<FK_C2R, L>;
  const int rpc = rows_per_item(L, c.cd.M, c.row_threads);
  int blocks = c.cd.n_img * c.cd.M / rpc;
  if (sel1 >= 0) blocks *= 2;
  k_row_c2r<L><<<blocks, rpc * G::T, rpc * G::SIZE * sizeof(float2), s>>>(
      c.cd, c.imgs, one_desc(c), t.tw, rpc, sel0, sel1, dsel0, dsel1, scale,
      dsel0 == SEL_UI ? c.st : nullptr);
}

cudaError_t launch_row_c2r(const ClassLaunch& c, const Tables& t, int sel0, int sel1, int dsel0,
                           int dsel1, float scale, cudaStream_t s) {
  switch (c.cd.N / 2) {
    GFD_CASE_L(do_row_c2r, c, t, sel0, sel1, dsel0, dsel1, scale, s)
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int M>
static void do_col_plain(const ClassLaunch& c, const Tables& t, int src, int dst, bool inv,
                         cudaStream_t s) {
  const int Lc = c.cd.N / 2;
  constexpr int T = FftGeo<FK_COL, M>::T;
  int B = 512 / T;
  if (B > Lc) B = Lc;
  if (B > c.cd.TB) B = c.cd.TB;  // a block stays inside one tile
  const size_t smem = (size_t)B * col_stride<M>(B) * sizeof(float2);
  const int nblk = c.cd.n_img * (Lc / B);
  if (inv)
    k_col_plain<M, true><<<nblk, B * T, smem, s>>>(c.cd, c.imgs, one_desc(c), t.tw, B, src, dst);
  else
    k_col_plain<M, false><<<nblk, B * T, smem, s>>>(c.cd, c.imgs, one_desc(c), t.tw, B, src, dst);
}

cudaError_t launch_col_plain(const ClassLaunch& c, const Tables& t, int src, int dst,
                             bool inverse, cudaStream_t s) {
  switch (c.cd.M) {
    GFD_CASE_M(do_col_plain, c, t, src, dst, inverse, s)
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Column kernels of the long transforms exist for every tile width that
// class_tile_width gives them, so that a thread's rows lie at constant offsets;
// shorter ones (BT = 0) take the width at run time.
#define GFD_COL_WIDTHS(F, M, B, ...)                                     \
  do {                                                                   \
    if constexpr ((M) >= 2048) {                                         \
      F<M, 2>(__VA_ARGS__);                                              \
    } else if constexpr ((M) == 1024) {                                  \
      if ((B) == 4) F<M, 4>(__VA_ARGS__); else F<M, 2>(__VA_ARGS__);     \
    } else if constexpr ((M) == 512) {                                   \
      if ((B) == 8) F<M, 8>(__VA_ARGS__);                                \
      else if ((B) == 4) F<M, 4>(__VA_ARGS__);                           \
      else F<M, 2>(__VA_ARGS__);                                         \
    } else if constexpr ((M) == 256) {                                   \
      if ((B) == 16) F<M, 16>(__VA_ARGS__);                              \
      else if ((B) == 8) F<M, 8>(__VA_ARGS__);                           \
      else if ((B) == 4) F<M, 4>(__VA_ARGS__);                           \
      else F<M, 2>(__VA_ARGS__);                                         \
    } else {                                                             \
      F<M, 0>(__VA_ARGS__);                                              \
    }                                                                    \
  } while (0)

template <int M, int BT>
static void do_col_fwd_lambda_w(const ClassLaunch& c, const Tables& t, int iter, cudaStream_t s) {
  const int Lc = c.cd.N / 2, B = c.cd.TB;
  const int nthr = B * FftGeo<FK_COL, M>::T;
  const size_t smem = (size_t)B * col_stride<M>(B) * sizeof(float2) + 16 * sizeof(double);
  const int n_items = c.cd.n_img * (Lc / B);
  const int grid = persistent_grid(k_col_fwd_lambda<M, BT>, nthr, smem, n_items, c.grid_div);
  k_col_fwd_lambda<M, BT><<<grid, nthr, smem, s>>>(c.cd, c.imgs, c.st, t.tw, iter, c.cd.M);
}

template <int M>
static void do_col_fwd_lambda(const ClassLaunch& c, const Tables& t, int iter, cudaStream_t s) {
  GFD_COL_WIDTHS(do_col_fwd_lambda_w, M, c.cd.TB, c, t, iter, s);
}

// Small problems (all images of a class together): the short column passes.
// Above SHORT_PIXELS the persistent ones, which pass fewer times through shared
// memory, take over.  Whole solves of 15 iterations, short against persistent
// passes: one 256^2 image 0.79 / 1.03 ms, one 512^2 1.00 / 1.06, one 1024^2 1.25 /
// 1.25 (the forward pass loses what the solve pass gains).
bool short_columns(int M, int N, int n_img) {
  // (a block holds at least the 16 threads that a lambda update needs)
  return M <= 1024 && M * N >= 128 && (long long)M * N * n_img <= SHORT_PIXELS;
}

static void do_col_fwd_lambda_short(const ClassLaunch& c, const Tables& t, int iter,
                                    cudaStream_t s) {
  const int M = c.cd.M, B = c.cd.TB, lg = __builtin_ctz(M);
  const size_t smem = (size_t)((B * (short_pos(M) + 1) + 1) & ~1) * sizeof(float2) +
                      16 * sizeof(double);
  k_col_fwd_lambda_short<<<c.cd.n_img * (c.cd.N / 2 / B), B * M / 4, smem, s>>>(c.cd, c.imgs, c.st,
                                                                               t.tw, lg, iter);
}

cudaError_t launch_col_fwd_lambda(const ClassLaunch& c, const Tables& t, int iter,
                                  cudaStream_t s) {
  if (c.short_cols) {
    do_col_fwd_lambda_short(c, t, iter, s);
    return cudaGetLastError();
  }
  switch (c.cd.M) {
    GFD_CASE_M(do_col_fwd_lambda, c, t, iter, s)
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_lambda_pass(const ClassLaunch& c, int iter, bool last_chance,
                               cudaStream_t s) {
  const int per_img = c.cd.M * (c.cd.N / 2);
  const int chunk = per_img < 16384 ? per_img : 16384;
  const int nblk = c.cd.n_img * (per_img / chunk);
  k_lambda_pass<<<nblk, 256, 0, s>>>(c.cd, c.imgs, c.st, chunk, iter, last_chance ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_lambda_loop(const ClassLaunch& c, int iter, int npass, cudaStream_t s) {
  k_lambda_loop<<<c.cd.n_img * LOOP_BLOCKS, LOOP_THREADS, 0, s>>>(c.cd, c.imgs, c.st, iter, npass);
  return cudaGetLastError();
}

template <int M, int BT>
static void do_col_solve_inv_w(const ClassLaunch& c, const Tables& t, cudaStream_t s) {
  const int Lc = c.cd.N / 2, B = c.cd.TB;
  const int nthr = B * FftGeo<FK_COL, M>::T;
  const size_t smem = (size_t)2 * B * col_stride<M>(B) * sizeof(float2);
  const int n_items = c.cd.n_img * (Lc / B);
  const int grid = persistent_grid(k_col_solve_inv<M, BT>, nthr, smem, n_items, c.grid_div);
  k_col_solve_inv<M, BT><<<grid, nthr, smem, s>>>(c.cd, c.imgs, c.st, t.tw, t.d2);
}

template <int M>
static void do_col_solve_inv(const ClassLaunch& c, const Tables& t, cudaStream_t s) {
  GFD_COL_WIDTHS(do_col_solve_inv_w, M, c.cd.TB, c, t, s);
}

cudaError_t launch_col_solve_inv(const ClassLaunch& c, const Tables& t, cudaStream_t s) {
  if (c.short_cols) {
    const int M = c.cd.M, B = c.cd.TB;
    k_col_solve_inv_short<<<c.cd.n_img * (c.cd.N / 2 / B), B * M / 4,
                            (size_t)2 * B * (short_pos(M) + 1) * sizeof(float2), s>>>(
        c.cd, c.imgs, c.st, t.tw, t.d2, __builtin_ctz(M));
    return cudaGetLastError();
  }
  switch (c.cd.M) {
    GFD_CASE_M(do_col_solve_inv, c, t, s)
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
static int smem_optin() {
  static int v = 0;
  if (v == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || v <= 0)
      v = 48 * 1024;
  }
  return v;
}

// Allow the kernel the device's opt-in shared memory minus its static part.
template <class K>
static cudaError_t allow_smem(K kernel) {
  cudaFuncAttributes a{};
  cudaError_t e = cudaFuncGetAttributes(&a, (const void*)kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              smem_optin() - (int)a.sharedSizeBytes);
}

template <int L>
static cudaError_t cfg_row() {
  cudaError_t e = allow_smem(k_row_r2c<L>);
  if (e != cudaSuccess) return e;
  return allow_smem(k_row_c2r<L>);
}
template <int M>
static cudaError_t cfg_col_fused();
template <int M>
static cudaError_t cfg_col() {
  cudaError_t e;
  if ((e = allow_smem(k_col_plain<M, false>)) != cudaSuccess) return e;
  if ((e = allow_smem(k_col_plain<M, true>)) != cudaSuccess) return e;
  return cfg_col_fused<M>();
}
template <int M, int BT>
static void cfg_col_width(cudaError_t& e) {
  if (e == cudaSuccess) e = allow_smem(k_col_fwd_lambda<M, BT>);
  if (e == cudaSuccess) e = allow_smem(k_col_solve_inv<M, BT>);
}
// Each width that GFD_COL_WIDTHS has for M once: 4096 / M (16 at most), halved down
// to 2; one kernel for all widths below 256 rows.
template <int M>
static cudaError_t cfg_col_fused() {
  cudaError_t e = cudaSuccess;
  constexpr int top = M >= 2048 || M < 256 ? 2 : 4096 / M;
  for (int B = 2; B <= top; B *= 2) GFD_COL_WIDTHS(cfg_col_width, M, B, e);
  return e;
}

cudaError_t configure_fft_kernels() {
  cudaError_t e;
#define GFD_CFG(x) if ((e = (x)) != cudaSuccess) return e;
  GFD_CFG(cfg_row<4>()) GFD_CFG(cfg_row<8>()) GFD_CFG(cfg_row<16>()) GFD_CFG(cfg_row<32>())
  GFD_CFG(cfg_row<64>()) GFD_CFG(cfg_row<128>()) GFD_CFG(cfg_row<256>()) GFD_CFG(cfg_row<512>())
  GFD_CFG(cfg_row<1024>()) GFD_CFG(cfg_row<2048>())
  GFD_CFG(cfg_col<8>()) GFD_CFG(cfg_col<16>()) GFD_CFG(cfg_col<32>()) GFD_CFG(cfg_col<64>())
  GFD_CFG(cfg_col<128>()) GFD_CFG(cfg_col<256>()) GFD_CFG(cfg_col<512>()) GFD_CFG(cfg_col<1024>())
  GFD_CFG(cfg_col<2048>()) GFD_CFG(cfg_col<4096>())
#undef GFD_CFG
  return cudaSuccess;
}

}  // namespace gfd
