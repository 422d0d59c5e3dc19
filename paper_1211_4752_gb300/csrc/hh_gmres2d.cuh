// Pieces shared by the 2-D GMRES step kernels of both precisions (method:
// hh_cheb.cuh; complex64: hh_gmres2d_32.cu, complex128: hh_gmres2d_64.cu).  A
// step is two kernels:
//
//   basis   w (the iterate, zero, or u + P e), q_0 = f - A w, the Chebyshev
//           vectors and the Gram matrix, per-block sums;
//   update  every block adds the partial Gram matrices, solves the m x m system
//           and forms u = w + s sum y_j q_j; on the way down also f - A u and its
//           full weighting.
//
// A block (or a warp) forms the vectors on its points and on a halo as wide as
// the number of products, so that no grid-wide step separates the products.
//
// Where a level's coefficients are uniform and real (outside the ECS layers)
// A u = (4 c_0 - beta k^2) u - c_0 (sum of the neighbours): with constant k, X u
// is then a multiple of that sum alone.
#pragma once
#include "hh_kernels.cuh"
#include "hh_launch.cuh"
#include "hh_tma.cuh"
#include "hh_gmres2d.h"

#include <algorithm>
#include <cstdlib>
#include <type_traits>

namespace hh {

namespace {

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

enum { GENERAL = 0, UNIFORM_K = 1, UNIFORM = 2 };   // UNIFORM_K: constant k as well

// the iterate a step starts from at (x, y) (zero outside the domain)
template <typename R, bool CORR>
__device__ __forceinline__ typename Cx<R>::T start_at(const LevelK<R> &L, const Gm2dIn<R> &in,
                                                      int b, bool zero, int x, int y) {
  using C = typename Cx<R>::T;
  const int N = L.N;
  C w = czero<C>();
  if ((unsigned)x >= (unsigned)N || (unsigned)y >= (unsigned)N) return w;
  if (!zero) w = in.u[(size_t)b * L.S + (size_t)y * L.P + x];
  if (CORR) w = cadd(w, prolong_at<R, 2>(in.e + (size_t)b * in.lc.S, in.lc, x, y, 0));
  return w;
}

// fc = c R r on a coarse point from the residual at its fine point (row pitch W)
template <typename R>
__device__ __forceinline__ typename Cx<R>::T weight_at(const typename Cx<R>::T *r, int W,
                                                       typename Cx<R>::T csc) {
  using C = typename Cx<R>::T;
  const C e = cadd(cadd(r[-1], r[1]), cadd(r[-W], r[W]));
  const C k = cadd(cadd(r[-W - 1], r[-W + 1]), cadd(r[W - 1], r[W + 1]));
  C a;
  a.x = fmaf_any(R(4), r[0].x, fmaf_any(R(2), e.x, k.x));
  a.y = fmaf_any(R(4), r[0].y, fmaf_any(R(2), e.y, k.y));
  return cmul(csc, a);
}

// Sum of the blocks' partial Gram matrices (fixed order), in every block of the
// update kernel: parts_sum leaves one sum per warp and quantity, solve_warp (one
// warp, after a barrier) adds those and solves.
template <typename R, int M>
__device__ __forceinline__ void parts_sum(const typename GramSum<R>::T *parts, int nparts,
                                          typename GramSum<R>::T *sums) {
  constexpr int NQP = Gram<M>::NQP;
  constexpr bool P = sizeof(R) == 4;
  const int q = threadIdx.x % NQP, g0 = threadIdx.x / NQP, ng = blockDim.x / NQP;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  GramAcc<R, P> t;
  t.zero();
  for (int i = g0; i < nparts; i += 4 * ng) {   // four loads in flight
    typename GramSum<R>::T v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (i + r * ng < nparts) v[r] = parts[(size_t)(i + r * ng) * NQP + q];
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (i + r * ng < nparts) gram_add(t, v[r]);
  }
#pragma unroll
  for (int o = NQP; o < 32; o <<= 1) t.add(t.shfl_xor(o));
  if (lane < NQP) sums[warp * NQP + lane] = gram_store(t);
}
template <typename R, int M>
__device__ __forceinline__ void solve_warp(typename GramSum<R>::T *sums, int nw, R s, double tol,
                                           StepCoef<R> *out) {
  constexpr int NQP = Gram<M>::NQP;
  const int lane = threadIdx.x & 31;
  GramAcc<R, sizeof(R) == 4> t;
  t.zero();
  for (int i = lane / NQP; i < nw; i += 32 / NQP) gram_add(t, sums[i * NQP + lane % NQP]);
#pragma unroll
  for (int o = NQP; o < 32; o <<= 1) t.add(t.shfl_xor(o));
  __syncwarp();
  if (lane < NQP) sums[lane] = gram_store(t);
  __syncwarp();
  gram_solve<R, M>(sums, s, tol, out);
}
template <typename R, int M>
__device__ __forceinline__ void step_coef(const typename GramSum<R>::T *parts, int nparts, R s,
                                          double tol, typename GramSum<R>::T *sums,
                                          StepCoef<R> *out) {
  parts_sum<R, M>(parts, nparts, sums);
  __syncthreads();
  if (threadIdx.x < 32) solve_warp<R, M>(sums, blockDim.x >> 5, s, tol, out);
  __syncthreads();
}

// complex128: the coefficients that k_gm2d_coef stored, with the correction from its nb
// blocks' sums.  By the whole block (sums: 8 slots per warp), ends with its barrier: one
// warp waits for ten rounds of loads at 152 blocks.
template <int M>
__device__ __forceinline__ void read_coef_block(const Gm2dWork<double> &wk, int b, int nb, double s,
                                                double *sums, StepCoef<double> *out) {
  const int tid = threadIdx.x, lane = tid & 31, nw = blockDim.x >> 5;
  static_assert(sizeof(StepCoef<double>) == kGm2dCoef * sizeof(double), "coefficients");
  if (tid < kGm2dCoef) reinterpret_cast<double *>(out)[tid] = wk.coef[(size_t)b * kGm2dCoef + tid];
  const double *p = wk.parts2 + (size_t)b * kGm2dCorr * 8 + (tid & 7);
  double d = 0.0;
#pragma unroll 4
  for (int i = tid >> 3; i < nb; i += 4 * nw) d += p[(size_t)i * 8];
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  d += __shfl_xor_sync(0xffffffffu, d, 16);
  if (lane < 8) sums[(tid >> 5) * 8 + lane] = d;
  __syncthreads();
  if (tid < 32) {
    d = 0.0;
    for (int w = lane >> 3; w < nw; w += 4) d += sums[w * 8 + (lane & 7)];
    d += __shfl_xor_sync(0xffffffffu, d, 8);
    d += __shfl_xor_sync(0xffffffffu, d, 16);
    __syncwarp();
    if (lane < 8) sums[lane] = d;
    __syncwarp();
    solve_correction<M>(sums, s, out);
  }
  __syncthreads();
}
// The same by one warp (the tiles, whose other warps form the basis meanwhile); sums: 8
// slots.
template <int M>
__device__ __forceinline__ void read_coef(const Gm2dWork<double> &wk, int b, int nb, double s,
                                          double *sums, StepCoef<double> *out) {
  const int lane = threadIdx.x & 31;
  if (lane < kGm2dCoef) reinterpret_cast<double *>(out)[lane] = wk.coef[(size_t)b * kGm2dCoef + lane];
  const double *p = wk.parts2 + (size_t)b * kGm2dCorr * 8 + (lane & 7);
  double t[4] = {0.0, 0.0, 0.0, 0.0};
  for (int i = lane >> 3; i < nb; i += 16)   // four loads in flight
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (i + 4 * r < nb) t[r] += p[(size_t)(i + 4 * r) * 8];
  double d = (t[0] + t[1]) + (t[2] + t[3]);
  d += __shfl_xor_sync(0xffffffffu, d, 8);
  d += __shfl_xor_sync(0xffffffffu, d, 16);
  if (lane < 8) sums[lane] = d;
  __syncwarp();
  solve_correction<M>(sums, s, out);
}

// ---------------------------------------------------------------------------
// Small levels: one thread per point of a T x T tile and its halo.  A march of
// a few rows is one warp's chain of dependent iterations; on levels of at most
// a few points per thread that chain, not the work, is the time (the paired sums
// alone are 320 instructions per point), so these kernels keep the q_j of the
// tile in shared memory, one barrier per product, and share each point's Gram
// products between two threads.
// ---------------------------------------------------------------------------
template <typename R> struct PointOp {
  using C = typename Cx<R>::T;
  C lox, upx, loy, upy, D;
  bool in;
  __device__ __forceinline__ void load(const LevelK<R> &L, int x, int y) {
    const int N = L.N;
    in = (unsigned)x < (unsigned)N && (unsigned)y < (unsigned)N;
    lox = upx = loy = upy = D = czero<C>();
    if (in) {
      lox = L.coef[x];
      upx = L.coef[2 * N + x];
      loy = L.coef[3 * N + y];
      upy = L.coef[5 * N + y];
      D = diag_at<R, 2>(L, x, y, 0);
    }
  }
  // the neighbours' part at q (pitch W); zero outside the domain
  __device__ __forceinline__ C nb(const C *q, int W) const {
    C n = cmul(lox, q[-1]);
    n = cfma(upx, q[1], n);
    n = cfma(loy, q[-W], n);
    return cfma(upy, q[W], n);
  }
  __device__ __forceinline__ C X(const C *q, int W, C sigma, R s) const {
    return in ? cscale(csub(cmul(csub(D, sigma), q[0]), nb(q, W)), s) : czero<C>();
  }
  __device__ __forceinline__ C resid(C f, const C *q, int W) const {
    return in ? cadd(csub(f, cmul(D, q[0])), nb(q, W)) : czero<C>();
  }
};

constexpr int round32(int v) { return (v + 31) / 32 * 32; }
constexpr int imax(int a, int b) { return a > b ? a : b; }

template <int M, int T> struct BasisTile {
  static constexpr int E = T + 2 * M, W = E + 2;       // q_0 region, iterate region
  static constexpr int NT = round32(imax(E * E, 2 * T * T));
};

// q_0 .. q_{M-1} (times g) of a tile's points in shared memory: q_j is valid j
// points inside the E x E region.  sw: the iterate on (E + 2)^2.  bar: barrier id of
// the `nt` threads that take part.
template <typename R, int M, int E>
__device__ __forceinline__ void tile_basis(const PointOp<R> &op, typename Cx<R>::T fv,
                                           const typename Cx<R>::T *sw,
                                           typename Cx<R>::T (*sq)[E * E],
                                           typename Cx<R>::T sigma, R s, R g, int tx, int ty, bool mine,
                                           int bar, int nt) {
  using C = typename Cx<R>::T;
  constexpr int W = E + 2;
  const int o = ty * E + tx;
  if (mine) sq[0][o] = cscale(op.resid(fv, sw + (ty + 1) * W + tx + 1, W), g);
#pragma unroll
  for (int j = 1; j < M; ++j) {
    bar_sync(bar, nt);
    const bool in = mine && tx >= j && tx < E - j && ty >= j && ty < E - j;
    if (in) {
      C v = op.X(sq[j - 1] + o, E, sigma, s);
      if (j >= 2) v = csub(cadd(v, v), sq[j - 2][o]);
      sq[j][o] = v;
    }
  }
  bar_sync(bar, nt);
}

template <typename R, int M, int T, bool CORR>
__global__ void __launch_bounds__(BasisTile<M, T>::NT)
k_gm2d_basis_tile(LevelK<R> L, typename Cx<R>::T sigma, R s, Gm2dIn<R> in, Gm2dWork<R> wk,
                  const SolveState *st, double *check) {
  using C = typename Cx<R>::T;
  using B = BasisTile<M, T>;
  using S = typename GramSum<R>::T;
  constexpr int E = B::E, W = B::W, NT = B::NT, NQP = Gram<M>::NQP, H = NQP / 2, NW = NT / 32;
  constexpr bool PAIR = sizeof(R) == 4, STORE = sizeof(R) == 8;
  using A = GramAcc<R, PAIR>;
  __shared__ C sw[W * W], sq[M][E * E];
  __shared__ S sums[NW * H];
  const int b = blockIdx.y, tid = threadIdx.x, N = L.N;
  const int nt = (N + T - 1) / T, x0 = (blockIdx.x % nt) * T, y0 = (blockIdx.x / nt) * T;
  const int tx = tid % E, ty = tid / E;
  const bool mine = tid < E * E;
  PointOp<R> op, gp;   // this thread's point, and the one whose products it sums
  op.load(L, mine ? x0 - M + tx : -1, y0 - M + ty);
  const int half = tid / (T * T), gi = tid % (T * T), ix = gi % T, iy = gi / T;
  gp.load(L, half < 2 ? x0 + ix : -1, y0 + iy);
  griddep_wait();
  griddep_launch_dependents();
  const R g = gram_scale_of<R>(wk.mag, b);   // (in flight early)
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  const bool zero = __syncthreads_or(in.zero_mode == ZERO_ALL ||
                                     (in.zero_mode == ZERO_FLAG && st && st[b].zero)) != 0;
  if (blockIdx.x == 0 && tid == 0) {
    wk.zflag[b] = zero;
    if (sizeof(R) == 4) wk.g[b] = (float)g;
  }
  const C fv = op.in ? in.f[(size_t)b * L.S + (size_t)(y0 - M + ty) * L.P + x0 - M + tx] : czero<C>();
  for (int i = tid; i < W * W; i += NT)
    sw[i] = start_at<R, CORR>(L, in, b, zero, x0 - M - 1 + i % W, y0 - M - 1 + i / W);
  __syncthreads();
  tile_basis<R, M, E>(op, fv, sw, sq, sigma, s, g, tx, ty, mine, 0, NT);
  A acc[NQP];
#pragma unroll
  for (int i = 0; i < NQP; ++i) acc[i].zero();
  if (half < 2) {
    const int o = (iy + M) * E + ix + M;
    const C t = cscale(sigma, s), xl = gp.X(sq[M - 1] + o, E, sigma, s);
    C v[M + 1];
    v[0] = sq[0][o];
    if (M >= 2) v[1] = cfma(t, v[0], sq[M >= 2 ? 1 : 0][o]);
    if (M == 3) v[2] = cfma(t, sq[M >= 2 ? 1 : 0][o], cscale(cadd(sq[M - 1][o], v[0]), R(0.5)));
    v[M] = cfma(t, sq[M - 1][o], xl);
    if (STORE && half == 0 && gp.in) {
      C *q = wk.q + (size_t)b * L.S + (size_t)(y0 + iy) * L.P + x0 + ix;
#pragma unroll
      for (int j = 0; j < M; ++j) q[j * wk.qs] = sq[j][o];
      q[M * wk.qs] = xl;
    }
    gram_point_half<R, M, PAIR>(acc, v, half);
  }
  // threads of the same half form whole warps (T^2 is a multiple of 32)
  static_assert((T * T) % 32 == 0, "whole warps per half");
  A h8[H];
#pragma unroll
  for (int i = 0; i < H; ++i) h8[i] = half == 0 ? acc[i] : acc[H + i];
  const A v = gram_warp_sum<A, H>(h8);
  constexpr int SH = H == 8 ? 2 : 4;
  const int lane = tid & 31, warp = tid >> 5;
  if ((lane & ((1 << SH) - 1)) == 0) sums[warp * H + (lane >> SH)] = gram_store(v);
  __syncthreads();
  if (tid < NQP) {
    constexpr int HW = T * T / 32;   // warps per half
    const int w0 = tid < H ? 0 : HW;
    A t;
    t.zero();
    for (int i = 0; i < HW; ++i) gram_add(t, sums[(w0 + i) * H + tid % H]);
    const S q = gram_store(t);
    wk.parts[((size_t)b * gridDim.x + blockIdx.x) * NQP + tid] = q;
    if (check && tid == 0) check[(size_t)b * gridDim.x + blockIdx.x] = gram_unscaled(q, (float)g);
  }
}

// Update of a tile (nparts: blocks of the basis kernel; complex128: of k_gm2d_coef):
// REST has T x T fine points (T even) and the residual on the
// (T + 1)^2 points its coarse points need, hence u on (T + 3)^2.
template <int M, int T, bool REST> struct UpdateTile {
  static constexpr int I = M - 1 + (REST ? 1 : 0);     // halo of q_0 below / left of the tile
  static constexpr int E = T + 2 * (M - 1) + (REST ? 3 : 0), W = E + 2;
  static constexpr int NC = round32(E * E);            // threads that own a point
  static constexpr int NT = NC + 32;                   // and the warp of the small solve
};

template <typename R, int M, int T, bool CORR, bool REST>
__global__ void __launch_bounds__(UpdateTile<M, T, REST>::NT)
k_gm2d_update_tile(LevelK<R> L, typename Cx<R>::T sigma, R s, Gm2dIn<R> in, Gm2dWork<R> wk,
                   int nparts, double tol, typename Cx<R>::T *u_out, typename Cx<R>::T *fc,
                   typename Cx<R>::T cs, Lay lc, const SolveState *st) {
  using C = typename Cx<R>::T;
  using B = UpdateTile<M, T, REST>;
  constexpr int E = B::E, W = B::W, NT = B::NT, I = B::I, NQP = Gram<M>::NQP, NC = B::NC;
  __shared__ C sw[W * W], sq[M][E * E];
  __shared__ typename GramSum<R>::T sums[NT / 32 * NQP];
  __shared__ StepCoef<R> sc;
  const int b = blockIdx.y, tid = threadIdx.x, N = L.N;
  const int nt = (N + T - 1) / T, x0 = (blockIdx.x % nt) * T, y0 = (blockIdx.x / nt) * T;
  const int tx = tid % E, ty = tid / E, x = x0 - I + tx, y = y0 - I + ty;
  const bool mine = tid < E * E;
  PointOp<R> op;
  op.load(L, mine ? x : -1, y);
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  const bool zero = wk.zflag[b] != 0;
  const C fv = op.in ? in.f[(size_t)b * L.S + (size_t)y * L.P + x] : czero<C>();
  for (int i = tid; i < W * W; i += NT)
    sw[i] = start_at<R, CORR>(L, in, b, zero, x0 - I - 1 + i % W, y0 - I - 1 + i / W);
  if constexpr (sizeof(R) == 4) parts_sum<R, M>(wk.parts + (size_t)b * nparts * NQP, nparts, sums);
  __syncthreads();
  // the last warp solves for the coefficients while the others form the basis
  if (tid >= NC) {
    if constexpr (sizeof(R) == 4) {
      solve_warp<R, M>(sums, NT / 32, s, tol, &sc);
      if (wk.track && blockIdx.x == 0 && tid == NC) gram_estimate(wk.mag, b, sums[0], wk.g[b]);
    }
    else read_coef<M>(wk, b, nparts, s, sums, &sc);
  }
  else tile_basis<R, M, E>(op, fv, sw, sq, sigma, s, R(1), tx, ty, mine, 1, NC);
  __syncthreads();
  const int o = ty * E + tx, ow = (ty + 1) * W + tx + 1;
  const bool have = mine && tx >= M - 1 && tx < E - (M - 1) && ty >= M - 1 && ty < E - (M - 1);
  C un = czero<C>();
  if (have) {   // (zero outside the domain, as w and the q_j are)
    un = sw[ow];
#pragma unroll
    for (int j = 0; j < M; ++j) un = cfma(sc.z[j], sq[j][o], un);
    if (op.in && x >= x0 && x < x0 + T && y >= y0 && y < y0 + T)
      u_out[(size_t)b * L.S + (size_t)y * L.P + x] = un;
  }
  if constexpr (REST) {
    __syncthreads();
    if (have) sw[ow] = un;
    __syncthreads();
    constexpr int J = M;   // the residual needs one point more
    if (mine && tx >= J && tx < E - J && ty >= J && ty < E - J) sq[0][o] = op.resid(fv, sw + ow, W);
    __syncthreads();
    constexpr int TC = T / 2;
    if (tid < TC * TC) {
      const int cx = tid % TC, cy = tid / TC, gx = x0 / 2 + cx, gy = y0 / 2 + cy;
      if (gx < lc.N && gy < lc.N) {
        const C *r = sq[0] + (2 * cy + 1 + I) * E + 2 * cx + 1 + I;   // centre
        fc[(size_t)b * lc.S + (size_t)gy * lc.P + gx] = weight_at<R>(r, E, cscale(cs, R(1.0 / 16.0)));
      }
    }
  }
}

inline int even_up(int v) { return (v + 1) & ~1; }

// calls fn with m as a compile-time constant
template <typename F> void with_m(int m, F fn) {
  if (m == 1) fn(std::integral_constant<int, 1>());
  else if (m == 2) fn(std::integral_constant<int, 2>());
  else fn(std::integral_constant<int, 3>());
}

template <typename R, int M, int T>
void basis_tile_launch(const LevelK<R> &L, typename Cx<R>::T sigma, R s, const Gm2dIn<R> &in,
                       const Gm2dWork<R> &w, int batch, const SolveState *st, double *check,
                       cudaStream_t stream) {
  const int nt = (L.N + T - 1) / T;
  auto go = [&](auto k) {
    launch_pdl(k, dim3(nt * nt, batch), dim3(BasisTile<M, T>::NT), 0, stream, L, sigma, s, in, w, st, check);
  };
  if (in.e) go(k_gm2d_basis_tile<R, M, T, true>);
  else go(k_gm2d_basis_tile<R, M, T, false>);
}
template <typename R, int M, int T, bool CORR, bool REST>
void update_tile_launch(const LevelK<R> &L, typename Cx<R>::T sigma, R s, const Gm2dIn<R> &in,
                        const Gm2dWork<R> &w, int nparts, double tol, typename Cx<R>::T *u_out,
                        typename Cx<R>::T *fc, typename Cx<R>::T cs, const Lay &lc, int batch,
                        const SolveState *st, cudaStream_t stream) {
  const int nt = (L.N + T - 1) / T;
  launch_pdl(k_gm2d_update_tile<R, M, T, CORR, REST>, dim3(nt * nt, batch),
             dim3(UpdateTile<M, T, REST>::NT), 0, stream, L, sigma, s, in, w, nparts, tol, u_out, fc,
             cs, lc, st);
}

}  // namespace

}  // namespace hh
