// GMRES(m) smoothing on 3-D levels, one reduction per step (method: hh_cheb.cuh):
// a kernel for each vector (q_0 = f - A w; q_1 = X q_0; q_2 = 2 X q_1 - q_0), one for
// the last product and the Gram matrix, and the update, every block of which adds
// the partial Gram matrices and solves the m x m system.  (A halo as wide as the
// products would cost five points per point in 3-D; two products per kernel on
// shared planes measured 119 us a step at 127^3 against 78 here, since the halo's
// arithmetic and two barriers a plane cost more than the reads they save.)
//
// A thread owns one (x, y) and walks along z: the values below, at and above are
// carried in registers, the four lateral ones come from L1, and the coefficients of
// x and y stay in registers.
//
// Measured (GB300, complex64, GMRES(3)): a step takes 76 us at 127^3 (151 with a
// reduction per Arnoldi step), 23 at 63^3 (49) and 10.4 at 31^3 (34); the 127^3 cycle
// 336 us (674).  complex128, 63^3: 154 us (154), the cycle 642 (734).
#pragma once
#include "hh_kernels.cuh"
#include "hh_launch.cuh"
#include "hh_gmres2d.cuh"
#include "hh_gmres3d.h"

namespace hh {

namespace {

constexpr int kBX = 32, kBY = 8, kT3 = kBX * kBY;    // columns of a block

// The block's planes [z0, z1) and the thread's column.
template <typename R> struct Walk3 {
  using C = typename Cx<R>::T;
  int x, y, z0, z1;
  bool in, w, e, n, t;     // inside the domain; neighbours inside
  size_t plane, kplane;
  int off;
  __device__ __forceinline__ Walk3(const LevelK<R> &L, int planes) {
    const int N = L.N, nx = (N + kBX - 1) / kBX, ny = (N + kBY - 1) / kBY;
    const int tile = blockIdx.x % (nx * ny), run = blockIdx.x / (nx * ny);
    x = (tile % nx) * kBX + threadIdx.x % kBX;
    y = (tile / nx) * kBY + threadIdx.x / kBX;
    z0 = run * planes;
    z1 = min(N, z0 + planes);
    in = x < N && y < N;
    w = x > 0;
    e = x < N - 1;
    n = y > 0;
    t = y < N - 1;
    plane = (size_t)N * L.P;
    kplane = (size_t)N * L.KP;
    off = in ? y * L.P + x : 0;
  }
};

// A of one column.
template <typename R> struct Column3 {
  using C = typename Cx<R>::T;
  C lx, ux, ly, uy, d;     // d: diagonal without its z part (less beta k^2 where k is constant)
  const C *cz;
  C beta;
  int N;
  bool kconst;
  const R *k2;
  __device__ __forceinline__ Column3(const LevelK<R> &L, int kc, const Walk3<R> &W)
      : cz(L.coef + 6 * L.N), beta(L.beta), N(L.N), kconst(kc != 0), k2(L.k2 + (size_t)W.y * L.KP + W.x) {
    lx = ux = ly = uy = d = czero<C>();
    if (W.in) {
      lx = L.coef[W.x];
      ux = L.coef[2 * N + W.x];
      ly = L.coef[3 * N + W.y];
      uy = L.coef[5 * N + W.y];
      d = cadd(L.coef[N + W.x], L.coef[4 * N + W.y]);
    }
    if (kconst) d = csub(d, cscale(beta, L.kc));
  }
  // the diagonal at plane z
  __device__ __forceinline__ C diag(int z, size_t kplane) const {
    C r = cadd(d, cz[N + z]);
    if (!kconst) r = csub(r, cscale(beta, k2[z * kplane]));
    return r;
  }
};

// fn(z, v, D, nb): v = a(z) at the thread's column, D the diagonal and nb the
// neighbours' part of A a there, for the block's planes.
template <typename R, typename F>
__device__ __forceinline__ void walk_z(const LevelK<R> &L, const Walk3<R> &W, const Column3<R> &K,
                                       const typename Cx<R>::T *a, F fn) {
  using C = typename Cx<R>::T;
  if (!W.in) return;
  const int N = L.N, P = L.P;
  const C *p = a + W.z0 * W.plane + W.off;
  C vm = W.z0 > 0 ? *(p - W.plane) : czero<C>(), v = *p;
#pragma unroll 2
  for (int z = W.z0; z < W.z1; ++z, p += W.plane) {
    const C vp = z + 1 < N ? p[W.plane] : czero<C>();
    const C vw = W.w ? p[-1] : czero<C>(), ve = W.e ? p[1] : czero<C>();
    const C vn = W.n ? *(p - P) : czero<C>(), vt = W.t ? p[P] : czero<C>();
    C nb = cmul(K.lx, vw);
    nb = cfma(K.ux, ve, nb);
    nb = cfma(K.ly, vn, nb);
    nb = cfma(K.uy, vt, nb);
    nb = cfma(K.cz[z], vm, nb);
    nb = cfma(K.cz[2 * N + z], vp, nb);
    fn(z, v, K.diag(z, W.kplane), nb);
    vm = v;
    v = vp;
  }
}

// Block sums of the Gram quantities into parts (and |q_0|^2, unscaled, into check).
template <typename R, int M, bool PAIR>
__device__ __forceinline__ void store_gram(GramAcc<R, PAIR> (&acc)[Gram<M>::NQP],
                                           const Gm2dWork<R> &wk, int b, double *check) {
  constexpr int NQP = Gram<M>::NQP, SH = NQP == 16 ? 1 : 3, NW = kT3 / 32;
  using S = typename GramSum<R>::T;
  __shared__ S sums[NW * NQP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const GramAcc<R, PAIR> v = gram_warp_sum<GramAcc<R, PAIR>, NQP>(acc);
  if ((lane & ((1 << SH) - 1)) == 0) sums[warp * NQP + (lane >> SH)] = gram_store(v);
  __syncthreads();
  if (threadIdx.x < NQP) {
    GramAcc<R, PAIR> t;
    t.zero();
    for (int i = 0; i < NW; ++i) gram_add(t, sums[i * NQP + threadIdx.x]);
    const S q = gram_store(t);
    wk.parts[((size_t)b * gridDim.x + blockIdx.x) * NQP + threadIdx.x] = q;
    if (check && threadIdx.x == 0)
      check[(size_t)b * gridDim.x + blockIdx.x] = gram_unscaled(q, sizeof(R) == 4 ? wk.g[b] : 1.f);
  }
}

// w = u + P e (trilinear) into out; a coarse plane is interpolated in x and y once
// for the two or three planes it serves.
template <typename R>
__global__ void __launch_bounds__(kT3)
k_gm3d_correct(LevelK<R> L, const typename Cx<R>::T *u, const typename Cx<R>::T *e, Lay lc,
               typename Cx<R>::T *out, int planes, const SolveState *st) {
  using C = typename Cx<R>::T;
  const int b = blockIdx.y;
  const Walk3<R> W(L, planes);
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  if (!W.in) return;
  u += (size_t)b * L.S;
  out += (size_t)b * L.S;
  e += (size_t)b * lc.S;
  const int Nc = lc.N, cx1 = W.x >> 1, cy1 = W.y >> 1;
  const int cx0 = (W.x & 1) ? cx1 : cx1 - 1, cy0 = (W.y & 1) ? cy1 : cy1 - 1;
  auto coarse = [&](int cz) {
    C v = czero<C>();
    if (cz < 0 || cz >= Nc) return v;
    const C *p = e + (size_t)cz * Nc * lc.P;
    auto g = [&](int cx, int cy) {
      return cx >= 0 && cx < Nc && cy >= 0 && cy < Nc ? p[(size_t)cy * lc.P + cx] : czero<C>();
    };
    v = cadd(cadd(g(cx0, cy0), g(cx1, cy0)), cadd(g(cx0, cy1), g(cx1, cy1)));
    return cscale(v, R(0.25));
  };
  C exB = coarse((W.z0 - 1) >> 1);
#pragma unroll 2
  for (int z = W.z0; z < W.z1; ++z) {
    C pe = exB;
    if (!(z & 1)) {   // between two coarse planes
      const C nx = coarse(z >> 1);
      pe = cscale(cadd(exB, nx), R(0.5));
      exB = nx;
    }
    const size_t o = z * W.plane + W.off;
    out[o] = cadd(u[o], pe);
  }
}

// J = 0: q_0 = g (f - A w) (g: hh_cheb.cuh; 1 in complex128); J = 1: q_1 = X q_0;
// J = 2: q_2 = 2 X q_1 - q_0.
template <typename R, int J>
__global__ void __launch_bounds__(kT3)
k_gm3d_vector(LevelK<R> L, typename Cx<R>::T sigma, R s, int kconst, Gm2dIn<R> in, Gm2dWork<R> wk,
              int planes, const SolveState *st) {
  using C = typename Cx<R>::T;
  const int b = blockIdx.y;
  const Walk3<R> W(L, planes);
  const Column3<R> K(L, kconst, W);
  griddep_wait();
  griddep_launch_dependents();
  const R g = J == 0 ? gram_scale_of<R>(wk.mag, b) : R(1);   // (in flight early)
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  C *q = wk.q + (size_t)b * L.S;
  if constexpr (J == 0) {
    const bool zero = __syncthreads_or(in.zero_mode == ZERO_ALL ||
                                       (in.zero_mode == ZERO_FLAG && st && st[b].zero)) != 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      wk.zflag[b] = zero;
      if (sizeof(R) == 4) wk.g[b] = (float)g;
    }
    const C *f = in.f + (size_t)b * L.S;
    if (zero) {
      if (W.in)
        for (int z = W.z0; z < W.z1; ++z) q[z * W.plane + W.off] = f[z * W.plane + W.off];
    } else {
      walk_z(L, W, K, in.u + (size_t)b * L.S, [&](int z, C v, C D, C nb) {
        const size_t o = z * W.plane + W.off;
        q[o] = cadd(csub(f[o], cmul(D, v)), nb);
      });
    }
    // (seldom: with the multiplication in the loop 127^3 took 42 us instead of 35)
    if (g != R(1) && W.in)
      for (int z = W.z0; z < W.z1; ++z) q[z * W.plane + W.off] = cscale(q[z * W.plane + W.off], g);
  } else {
    const C *a = q + (size_t)(J - 1) * wk.qs;
    C *out = q + (size_t)J * wk.qs;
    walk_z(L, W, K, a, [&](int z, C v, C D, C nb) {
      const size_t o = z * W.plane + W.off;
      C r = cscale(csub(cmul(csub(D, sigma), v), nb), s);
      if (J == 2) r = csub(cadd(r, r), q[o]);
      out[o] = r;
    });
  }
}

// The last product X q_{M-1} (stored in complex128) and the Gram matrix.
template <typename R, int M, bool PAIR>
__global__ void __launch_bounds__(kT3)
k_gm3d_gram(LevelK<R> L, typename Cx<R>::T sigma, R s, int kconst, Gm2dWork<R> wk, int planes,
            const SolveState *st, double *check) {
  using C = typename Cx<R>::T;
  const int b = blockIdx.y;
  const Walk3<R> W(L, planes);
  const Column3<R> K(L, kconst, W);
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  C *q = wk.q + (size_t)b * L.S;
  GramAcc<R, PAIR> acc[Gram<M>::NQP];
#pragma unroll
  for (int i = 0; i < Gram<M>::NQP; ++i) acc[i].zero();
  const C t = cscale(sigma, s);
  walk_z(L, W, K, q + (size_t)(M - 1) * wk.qs, [&](int z, C ql, C D, C nb) {
    const size_t o = z * W.plane + W.off;
    const C xl = cscale(csub(cmul(csub(D, sigma), ql), nb), s);
    if (sizeof(R) == 8) q[M * wk.qs + o] = xl;
    C v[M + 1];
    v[0] = M == 1 ? ql : q[o];
    const C q1 = M == 3 ? q[wk.qs + o] : ql;
    if (M >= 2) v[1] = cfma(t, v[0], q1);
    if (M == 3) v[M - 1] = cfma(t, q1, cscale(cadd(ql, v[0]), R(0.5)));
    v[M] = cfma(t, ql, xl);
    gram_point<R, M, PAIR>(acc, v);
    if (((z - W.z0) & 7) == 7) {
#pragma unroll
      for (int i = 0; i < Gram<M>::NQ; ++i) acc[i].fold();
    }
  });
#pragma unroll
  for (int i = 0; i < Gram<M>::NQP; ++i) acc[i].close();
  store_gram<R, M, PAIR>(acc, wk, b, check);
}

template <typename R, int M>
__global__ void __launch_bounds__(256)
k_gm3d_update(LevelK<R> L, R s, const typename Cx<R>::T *u_in, Gm2dWork<R> wk, int nparts, double tol,
              typename Cx<R>::T *u_out, const SolveState *st) {
  using C = typename Cx<R>::T;
  constexpr int NQP = Gram<M>::NQP;
  __shared__ typename GramSum<R>::T sums[8 * 16];
  __shared__ StepCoef<R> sc;
  const int b = blockIdx.y;
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  const bool zero = wk.zflag[b] != 0;
  if constexpr (sizeof(R) == 4) {   // (the stored q_j are g times the basis)
    const float g = wk.g[b];
    step_coef<R, M>(wk.parts + (size_t)b * nparts * NQP, nparts, s * gram_rcp(g), tol, sums, &sc);
    if (wk.track && blockIdx.x == 0 && threadIdx.x == 0) gram_estimate(wk.mag, b, sums[0], g);
  } else {
    read_coef_block<M>(wk, b, nparts, s, sums, &sc);
  }
  C z[M];
#pragma unroll
  for (int j = 0; j < M; ++j) z[j] = sc.z[j];
  const C *q = wk.q + (size_t)b * L.S;
  u_in += (size_t)b * L.S;
  u_out += (size_t)b * L.S;
  // every element of the right-hand side's rows: the padding column stays zero
  // (u and the q_j are zero there)
  const unsigned total = (unsigned)L.S;
#pragma unroll 2
  for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
    C v = zero ? czero<C>() : u_in[p];
#pragma unroll
    for (int j = 0; j < M; ++j) v = cfma(z[j], q[(size_t)j * wk.qs + p], v);
    u_out[p] = v;
  }
}

// complex64: paired sums up to 63 points per axis (2.5e5 points; see hh_cheb.cuh)
constexpr int kGramPairMaxN3 = 64;

template <typename R, typename F> void with_pair(int N, F fn) {
  if (sizeof(R) == 4 && N <= kGramPairMaxN3) fn(std::integral_constant<bool, sizeof(R) == 4>());
  else fn(std::false_type());
}

}  // namespace

template <typename R>
void launch_gm3d_basis(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int kconst, int m,
                       const Gm2dIn<R> &in_, const Gm2dWork<R> &w, const Gm3dPlan &p,
                       typename Cx<R>::T *u_out, int batch, const SolveState *st, double *check,
                       cudaStream_t stream) {
  const dim3 grid(p.vblocks, batch), blk(kT3);
  Gm2dIn<R> in = in_;
  if (in.e) {
    launch_pdl(k_gm3d_correct<R>, grid, blk, 0, stream, L, in.u, in.e, in.lc, u_out, p.vplanes, st);
    in.u = u_out;
  }
  auto vec = [&](auto k) {
    launch_pdl(k, grid, blk, 0, stream, L, sigma, s, kconst, in, w, p.vplanes, st);
  };
  vec(k_gm3d_vector<R, 0>);
  if (m >= 2) vec(k_gm3d_vector<R, 1>);
  if (m >= 3) vec(k_gm3d_vector<R, 2>);
  with_m(m, [&](auto mm) {
    with_pair<R>(L.N, [&](auto pr) {
      launch_pdl(k_gm3d_gram<R, decltype(mm)::value, decltype(pr)::value>, dim3(p.blocks, batch), blk, 0,
                 stream, L, sigma, s, kconst, w, p.planes, st, check);
    });
  });
}

template <typename R>
void launch_gm3d_update(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int m,
                        const Gm2dIn<R> &in, const Gm2dWork<R> &w, const Gm3dPlan &p,
                        typename Cx<R>::T *u_out, int batch, const SolveState *st,
                        cudaStream_t stream) {
  // (with a correction the corrected iterate is in u_out)
  const typename Cx<R>::T *from = in.e ? u_out : in.u;
  int nparts = p.blocks;
  if constexpr (sizeof(R) == 8) nparts = launch_gm_coef(L, L.N * L.N, sigma, s, m, w, p.blocks, batch, st, stream);
  const double tol = gram_tol<R>(L.N <= kGramPairMaxN3);
  with_m(m, [&](auto mm) {
    constexpr int M = decltype(mm)::value;
    launch_pdl(k_gm3d_update<R, M>, dim3(p.ublocks, batch), dim3(256), 0, stream, L, s, from, w, nparts, tol, u_out, st);
  });
}

#define HH_GM3D_INST(R)                                                                          \
  template void launch_gm3d_basis<R>(const LevelK<R> &, Cx<R>::T, R, int, int, const Gm2dIn<R> &, \
                                     const Gm2dWork<R> &, const Gm3dPlan &, Cx<R>::T *, int,     \
                                     const SolveState *, double *, cudaStream_t);                \
  template void launch_gm3d_update<R>(const LevelK<R> &, Cx<R>::T, R, int, const Gm2dIn<R> &,    \
                                      const Gm2dWork<R> &, const Gm3dPlan &, Cx<R>::T *, int,    \
                                      const SolveState *, cudaStream_t);

}  // namespace hh
