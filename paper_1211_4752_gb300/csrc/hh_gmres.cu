// GMRES(m) smoothing (Sec. 3.2, the smoother of the paper's experiments) on the
// small levels, 2-D and 3-D, complex64 and complex128: one block per right-hand
// side.  The larger levels: hh_gmres2d.h and hh_gmres3d.h; the step: hh_cheb.cuh.
#include "hh_kernels.cuh"
#include "hh_launch.cuh"
#include "hh_tma.cuh"
#include "hh_gmres.h"

namespace hh {

namespace {

// ---------------------------------------------------------------------------
// The GMRES-smoothed cycle of the small levels in one block per right-hand
// side, one reduction per step (hh_cheb.cuh).  Shared memory: per level its
// iterate U, right-hand side F, coefficient tables and k^2 (the level's LevelK
// is re-pointed at these copies, so the stencil arithmetic is that of the
// per-level kernels); the vectors q_0..q_2 are shared by the levels, since a
// coarser level runs only between a finer level's smoothing steps.  Rows have
// the pitch N + 1, a power of two, so that a thread gets its points'
// coordinates by shifts.
// ---------------------------------------------------------------------------
constexpr int TB = 512;

template <typename R, int DIM>
__device__ __forceinline__ LevelK<R> tail_level(const GmTailArgs<R> &A, typename Cx<R>::T *cm,
                                                R *km, int i) {
  LevelK<R> K = A.lv[i].K;
  const int N = K.N;
  K.coef = cm + A.lv[i].offT;
  K.k2 = km + A.lv[i].offK;
  K.KP = N + 1;
  K.P = N + 1;
  K.S = (long long)(N + 1) * (DIM == 2 ? N : N * N);
  return K;
}

// Calls fn(p, x, y, z) for the points of a level that this thread owns (p: the
// pitched position); the same points in every phase.
template <int DIM, typename F> __device__ __forceinline__ void tail_points(int N, F fn) {
  const int lg = 31 - __clz(N + 1);
  const int total = DIM == 2 ? N << lg : (N * N) << lg;
  for (int p = threadIdx.x; p < total; p += TB) {
    const int x = p & N, r = p >> lg;
    if (x == N) continue;
    if (DIM == 2) {
      fn(p, x, r, 0);
    } else {
      const int z = r / N;
      fn(p, x, r - z * N, z);
    }
  }
}

// One GMRES(M) step on level K (iterate U, right-hand side F; zero: U is taken
// as zero; g: scale of the vectors, hh_cheb.cuh).  res: Q0 holds f - A u of the new
// iterate afterwards.
template <typename R, int DIM, int M>
__device__ void tail_gm_step(const LevelK<R> &K, typename Cx<R>::T sigma, R s, R g,
                             typename Cx<R>::T *U, const typename Cx<R>::T *F,
                             typename Cx<R>::T *Q0, typename Cx<R>::T *Q1, typename Cx<R>::T *Q2,
                             typename Cx<R>::T *Q3, bool zero, bool res,
                             typename GramSum<R>::T *sums, StepCoef<R> *sc) {
  using C = typename Cx<R>::T;
  constexpr bool PAIR = sizeof(R) == 4;
  constexpr int NQP = Gram<M>::NQP;
  const int N = K.N, P = K.P;
  const C t = cscale(sigma, s);
  auto X = [&](const C *q, int x, int y, int z, C &qc) {
    auto get = [&](int xx, int yy, int zz) { return q[at<DIM>(xx, yy, zz, N, P)]; };
    C Aq, D;
    stencil<R, DIM>(K, x, y, z, get, Aq, D, qc);
    return cscale(csub(Aq, cmul(sigma, qc)), s);
  };
  {
    auto get = [&](int xx, int yy, int zz) { return U[at<DIM>(xx, yy, zz, N, P)]; };
    tail_points<DIM>(N, [&](int p, int x, int y, int z) {
      C r = F[p];
      if (!zero) {
        C Au, D, uc;
        stencil<R, DIM>(K, x, y, z, get, Au, D, uc);
        r = csub(r, Au);
      }
      Q0[p] = cscale(r, g);
    });
  }
  __syncthreads();
  if (M >= 2) {
    tail_points<DIM>(N, [&](int p, int x, int y, int z) {
      C qc;
      Q1[p] = X(Q0, x, y, z, qc);
    });
    __syncthreads();
  }
  if (M >= 3) {
    tail_points<DIM>(N, [&](int p, int x, int y, int z) {
      C qc;
      const C v = X(Q1, x, y, z, qc);
      Q2[p] = csub(cadd(v, v), Q0[p]);
    });
    __syncthreads();
  }
  GramAcc<R, PAIR> acc[NQP];
#pragma unroll
  for (int i = 0; i < NQP; ++i) acc[i].zero();
  tail_points<DIM>(N, [&](int p, int x, int y, int z) {
    C qc, v[M + 1];
    const C xl = X(M == 1 ? Q0 : (M == 2 ? Q1 : Q2), x, y, z, qc);
    v[0] = Q0[p];
    if (M >= 2) v[1] = cfma(t, v[0], Q1[p]);
    if (M == 3) v[M - 1] = cfma(t, Q1[p], cscale(cadd(qc, v[0]), R(0.5)));
    v[M] = cfma(t, qc, xl);
    if (sizeof(R) == 8) Q3[p] = xl;   // (read by this thread alone)
    gram_point<R, M, PAIR>(acc, v);
  });
  constexpr int SH = NQP == 16 ? 1 : 3;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  {
    const GramAcc<R, PAIR> v = gram_warp_sum<GramAcc<R, PAIR>, NQP>(acc);
    if ((lane & ((1 << SH) - 1)) == 0) sums[warp * NQP + (lane >> SH)] = gram_store(v);
  }
  __syncthreads();
  if (warp == 0) {
    // the warps that own points (the others' sums are zero)
    const int nw = min(TB / 32, ((int)K.S + 31) / 32);
    GramAcc<R, PAIR> v;
    v.zero();
    for (int i = lane / NQP; i < nw; i += 32 / NQP) gram_add(v, sums[i * NQP + lane % NQP]);
#pragma unroll
    for (int o = NQP; o < 32; o <<= 1) v.add(v.shfl_xor(o));
    __syncwarp();
    if (lane < NQP) sums[lane] = gram_store(v);
    __syncwarp();
    gram_solve<R, M>(sums, sizeof(R) == 4 ? s * (R)gram_rcp((float)g) : s, gram_tol<R>(PAIR), sc);
  }
  __syncthreads();
  if constexpr (sizeof(R) == 8) {   // the coefficients' correction (solve_correction)
    using A = GramAcc<double, false>;
    A cor[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) cor[i].zero();
    double2 yc[M];
#pragma unroll
    for (int j = 0; j < M; ++j) yc[j] = cscale(sc->z[j], 1.0 / s);
    tail_points<DIM>(N, [&](int p, int, int, int) {
      C a[M];
      const C qc = (M == 1 ? Q0 : (M == 2 ? Q1 : Q2))[p], xl = Q3[p];
      if (M >= 2) a[0] = cfma(t, Q0[p], Q1[p]);
      if (M == 3) a[1 % M] = cfma(t, Q1[p], cscale(cadd(qc, Q0[p]), 0.5));
      a[M - 1] = cfma(t, qc, xl);
      correction_point<M>(cor, a, yc, Q0[p]);
    });
    const A v = gram_warp_sum<A, 8>(cor);
    if ((lane & 3) == 0) sums[warp * 8 + (lane >> 2)] = v.h;
    __syncthreads();
    if (warp == 0) {
      const int nw = min(TB / 32, ((int)K.S + 31) / 32);   // (as above)
      double d = 0.0;
      for (int w = lane >> 3; w < nw; w += 4) d += sums[w * 8 + (lane & 7)];
      d += __shfl_xor_sync(0xffffffffu, d, 8);
      d += __shfl_xor_sync(0xffffffffu, d, 16);
      __syncwarp();
      if (lane < 8) sums[lane] = d;
      __syncwarp();
      solve_correction<M>(sums, s, sc);
    }
    __syncthreads();
  }
  tail_points<DIM>(N, [&](int p, int, int, int) {
    C v = zero ? czero<C>() : U[p];
    v = cfma(sc->z[0], Q0[p], v);
    if (M >= 2) v = cfma(sc->z[1], Q1[p], v);
    if (M >= 3) v = cfma(sc->z[2], Q2[p], v);
    U[p] = v;
  });
  __syncthreads();
  if (res) {
    auto get = [&](int xx, int yy, int zz) { return U[at<DIM>(xx, yy, zz, N, P)]; };
    tail_points<DIM>(N, [&](int p, int x, int y, int z) {
      C Au, D, uc;
      stencil<R, DIM>(K, x, y, z, get, Au, D, uc);
      Q0[p] = csub(F[p], Au);
    });
    __syncthreads();
  }
}

template <typename R, int DIM, int M>
__global__ void __launch_bounds__(TB) k_gm_tail(const __grid_constant__ GmTailArgs<R> A,
                                                const SolveState *st) {
  using C = typename Cx<R>::T;
  const int b = blockIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C *cm = reinterpret_cast<C *>(smem_raw);
  R *km = reinterpret_cast<R *>(smem_raw + A.kbase);
  double2 *sinv = reinterpret_cast<double2 *>(smem_raw + A.invbase);
  const int mm = A.mm;
  __shared__ typename GramSum<R>::T sums[(TB / 32) * 16];
  __shared__ StepCoef<R> sc;
  C *const Q0 = cm + A.offQ[0], *const Q1 = cm + A.offQ[1], *const Q2 = cm + A.offQ[2];
  C *const Q3 = cm + A.offQ[sizeof(R) == 8 ? 3 : 2];
  // every level's tables and k^2 and the coarsest inverse, which no kernel writes: staged
  // before the dependency wait
  for (int i = 0; i < A.nl; ++i) {
    const LevelK<R> &G = A.lv[i].K;
    const int N = G.N;
    C *tab = cm + A.lv[i].offT;
    for (int j = threadIdx.x; j < 3 * DIM * N; j += TB) tab[j] = G.coef[j];
    R *kk = km + A.lv[i].offK;
    tail_points<DIM>(N, [&](int p, int x, int y, int z) { kk[p] = G.k2[at<DIM>(x, y, z, N, G.KP)]; });
  }
  for (int j = threadIdx.x; j < mm * mm; j += TB) sinv[j] = A.inv[j];
  griddep_wait();
  griddep_launch_dependents();
  const R g = gram_scale_of<R>(A.mag, b);   // (in flight early)
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  {
    const int N = A.lv[0].K.N;
    const C *fb = A.f + (size_t)b * A.lay.S;
    C *F = cm + A.lv[0].offF;
    tail_points<DIM>(N, [&](int p, int x, int y, int z) { F[p] = fb[at<DIM>(x, y, z, N, A.lay.P)]; });
  }
  __syncthreads();
  // way down: smoothing from zero, full weighting of the last step's residual
  for (int i = 0; i + 1 < A.nl; ++i) {
    const LevelK<R> K = tail_level<R, DIM>(A, cm, km, i);
    const int N = K.N, P = K.P, Nc = A.lv[i + 1].K.N;
    C *U = cm + A.lv[i].offU;
    const C *F = cm + A.lv[i].offF;
    for (int s = 0; s < A.nu1; ++s)
      tail_gm_step<R, DIM, M>(K, A.lv[i].sigma, A.lv[i].s, g, U, F, Q0, Q1, Q2, Q3, s == 0,
                              s == A.nu1 - 1, sums, &sc);
    {
      const C *r = Q0;
      C *Fc = cm + A.lv[i + 1].offF;
      const int zlo = DIM == 3 ? -1 : 0, zhi = DIM == 3 ? 1 : 0;
      const R scale = DIM == 3 ? R(1.0 / 64.0) : R(1.0 / 16.0);
      const C cs = A.lv[i].c;
      tail_points<DIM>(Nc, [&](int, int cx, int cy, int cz) {
        C a = czero<C>();
        for (int dz = zlo; dz <= zhi; ++dz)
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
              const int x = 2 * cx + 1 + dx, y = 2 * cy + 1 + dy;
              const int z = DIM == 3 ? 2 * cz + 1 + dz : 0;
              const R w = R((2 - abs(dx)) * (2 - abs(dy)) * (DIM == 3 ? 2 - abs(dz) : 1));
              a = cadd(a, cscale(r[at<DIM>(x, y, z, N, P)], w));
            }
        Fc[at<DIM>(cx, cy, cz, Nc, Nc + 1)] = cmul(cs, cscale(a, scale));
      });
    }
    __syncthreads();
  }
  // coarsest level: u = A^{-1} f by the inverse that setup forms from the LU
  // factors (FP64).  Four threads per row, a quarter of the products each: a
  // warp's FP64 instruction takes 64 cycles, so that the 2 m dependent steps of the
  // substitutions took 3.5 us for m = 9 and 10 us for m = 27.
  {
    const int i = threadIdx.x >> 2, part = threadIdx.x & 3, N = A.lv[A.nl - 1].K.N;
    const C *fl = cm + A.lv[A.nl - 1].offF;
    C *ul = cm + A.lv[A.nl - 1].offU;
    if ((threadIdx.x & ~31) < 4 * mm) {   // whole warps
      double2 y = make_double2(0.0, 0.0);
      int x, yy, z;
      for (int j = part; i < mm && j < mm; j += 4) {
        coords<DIM>((size_t)j, N, x, yy, z);
        const C q = fl[at<DIM>(x, yy, z, N, N + 1)];
        y = cfma(sinv[i * mm + j], make_double2((double)q.x, (double)q.y), y);
      }
      for (int o = 1; o < 4; o <<= 1) {
        y.x += __shfl_xor_sync(0xffffffffu, y.x, o);
        y.y += __shfl_xor_sync(0xffffffffu, y.y, o);
      }
      if (i < mm && part == 0) {
        coords<DIM>((size_t)i, N, x, yy, z);
        ul[at<DIM>(x, yy, z, N, N + 1)] = cmk((R)y.x, (R)y.y);
      }
    }
  }
  __syncthreads();
  // way up: interpolated correction, smoothing
  for (int i = A.nl - 2; i >= 0; --i) {
    const LevelK<R> K = tail_level<R, DIM>(A, cm, km, i);
    const int N = K.N, Nc = A.lv[i + 1].K.N;
    C *U = cm + A.lv[i].offU;
    const C *F = cm + A.lv[i].offF;
    const C *E = cm + A.lv[i + 1].offU;
    const Lay lc{Nc, Nc + 1, 0};
    tail_points<DIM>(N, [&](int p, int x, int y, int z) {
      U[p] = cadd(U[p], prolong_at<R, DIM>(E, lc, x, y, z));
    });
    __syncthreads();
    for (int s = 0; s < A.nu2; ++s)
      tail_gm_step<R, DIM, M>(K, A.lv[i].sigma, A.lv[i].s, g, U, F, Q0, Q1, Q2, Q3, false, false,
                              sums, &sc);
  }
  {
    const int N = A.lv[0].K.N;
    C *ub = A.u + (size_t)b * A.lay.S;
    const C *U = cm + A.lv[0].offU;
    tail_points<DIM>(N, [&](int p, int x, int y, int z) { ub[at<DIM>(x, y, z, N, A.lay.P)] = U[p]; });
  }
}

}  // namespace

// Shared memory of the tail (layout of setup_gmres_tail): q_0..q_2 (complex128: and
// X q_{m-1}) of the first level, per level iterate, right-hand side, tables and k^2 (rows
// of pitch N + 1), the coarsest inverse.
static size_t tail_pts(int dim, int N) { return (size_t)(N + 1) * (dim == 2 ? N : N * N); }
template <typename R, int DIM> size_t gmres_tail_smem(const int *N, int nl, int m) {
  (void)m;
  using C = typename Cx<R>::T;
  size_t c = (sizeof(R) == 8 ? 4 : 3) * tail_pts(DIM, N[0]);
  size_t r = 0;
  for (int i = 0; i < nl; ++i) {
    c += 2 * tail_pts(DIM, N[i]) + 3 * DIM * (size_t)N[i];
    r += tail_pts(DIM, N[i]);
  }
  const size_t kb = (c * sizeof(C) + 15) / 16 * 16;
  const size_t lb = (kb + r * sizeof(R) + 15) / 16 * 16;
  const size_t mm = npts<DIM>(N[nl - 1]);
  return lb + mm * mm * sizeof(double2);
}

template <typename R, int DIM> cudaError_t init_gmres_tail() {
  cudaError_t e;
  auto set = [](auto k) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGmTailSmemMax);
  };
  if ((e = set(k_gm_tail<R, DIM, 1>)) != cudaSuccess) return e;
  if ((e = set(k_gm_tail<R, DIM, 2>)) != cudaSuccess) return e;
  return set(k_gm_tail<R, DIM, 3>);
}

template <typename R, int DIM>
void launch_gmres_tail(const GmTailArgs<R> &a, int batch, const SolveState *st, cudaStream_t s) {
  auto go = [&](auto k) { launch_pdl(k, dim3(batch), dim3(TB), a.smem_bytes, s, a, st); };
  if (a.m == 1) go(k_gm_tail<R, DIM, 1>);
  else if (a.m == 2) go(k_gm_tail<R, DIM, 2>);
  else go(k_gm_tail<R, DIM, 3>);
}

#define HH_GMTAIL_INST(R, DIM)                                                                 \
  template size_t gmres_tail_smem<R, DIM>(const int *, int, int);                              \
  template cudaError_t init_gmres_tail<R, DIM>();                                              \
  template void launch_gmres_tail<R, DIM>(const GmTailArgs<R> &, int, const SolveState *,      \
                                          cudaStream_t);
HH_GMTAIL_INST(float, 2)
HH_GMTAIL_INST(float, 3)
HH_GMTAIL_INST(double, 2)
HH_GMTAIL_INST(double, 3)

}  // namespace hh
