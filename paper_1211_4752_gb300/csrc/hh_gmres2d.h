// GMRES(m) smoothing steps on 2-D levels with one reduction per step
// (hh_gmres2d.cuh; the method is described in hh_cheb.cuh).
#pragma once
#include "hh_internal.h"
#include "hh_cheb.cuh"

namespace hh {

// Work split of one level: rows of a run or tile, warps per block (complex64) and
// blocks per right-hand side of the basis kernel (one partial Gram matrix per
// block) and of the update kernel.
struct Gm2dPlan {
  int rows, warps, blocks;
  int urows, uwarps, ublocks;
  int tile;                     // a thread per point of small tiles (small levels)
};

// Iterate a step starts from: u, or zero (ZERO_* mode), or u + P e.
template <typename R> struct Gm2dIn {
  const typename Cx<R>::T *u;
  const typename Cx<R>::T *f;
  const typename Cx<R>::T *e;   // coarse correction (layout lc), or null
  Lay lc;
  int zero_mode;
};

// Workspace: partial Gram matrices [b][block][NQP], whether the basis kernel
// took the iterate as zero ([b]), complex64: the scale of its sums ([b]), and
// (complex128) the stored basis.
template <typename R> struct Gm2dWork {
  typename GramSum<R>::T *parts;
  int *zflag;
  float *mag;                   // complex64: estimate of the level-0 residual's magnitude
  float *g;                     // and the scale that the step's basis kernel took from it
  int track;                    // the step is on level 0: its |r| is the next estimate
  typename Cx<R>::T *q;         // complex128: q_0 .. q_{m-1} and X q_{m-1}, stride qs,
  size_t qs;
  double *coef;                 // the solved coefficients ([b][kGm2dCoef]) and the
  double *parts2;               // sums of their correction ([b][block][8])
};
constexpr int kGm2dCoef = 24;   // StepCoef<double>: z_0..z_2, the inverse of N
constexpr int kGm2dCorr = 152;  // blocks of the correction's sums at most

template <typename R> cudaError_t init_gm2d();   // once per complex128 handle
template <typename R> Gm2dPlan gm2d_plan(int N, int m, int batch, int sms, bool restrict_);
int gm2d_max_parts(int batch, int sms);   // blocks per right-hand side at most

// Basis kernel: Gram matrix of the step from `in`.  check (level 0 of a solve):
// per-block |f - A w|^2 ([b][block]) for the stop test.
template <typename R>
void launch_gm2d_basis(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int kconst, int m,
                       const Gm2dIn<R> &in, const Gm2dWork<R> &w, const Gm2dPlan &p, int batch,
                       const SolveState *st, double *check, cudaStream_t stream);

// Update kernel: u_out = w + z; with fc: fc = c FW(f - A u_out) as well.  u_out
// must not be in.u.
template <typename R>
void launch_gm2d_update(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int kconst, int m,
                        const Gm2dIn<R> &in, const Gm2dWork<R> &w, const Gm2dPlan &p,
                        typename Cx<R>::T *u_out, typename Cx<R>::T *fc, typename Cx<R>::T cs,
                        const Lay &lc, int batch, const SolveState *st, cudaStream_t stream);

template <> Gm2dPlan gm2d_plan<float>(int, int, int, int, bool);
template <> Gm2dPlan gm2d_plan<double>(int, int, int, int, bool);
template <> cudaError_t init_gm2d<double>();
template <> void launch_gm2d_basis<float>(const LevelK<float> &, float2, float, int, int,
                                          const Gm2dIn<float> &, const Gm2dWork<float> &,
                                          const Gm2dPlan &, int, const SolveState *, double *,
                                          cudaStream_t);
template <> void launch_gm2d_basis<double>(const LevelK<double> &, double2, double, int, int,
                                           const Gm2dIn<double> &, const Gm2dWork<double> &,
                                           const Gm2dPlan &, int, const SolveState *, double *,
                                           cudaStream_t);
template <> void launch_gm2d_update<float>(const LevelK<float> &, float2, float, int, int,
                                           const Gm2dIn<float> &, const Gm2dWork<float> &,
                                           const Gm2dPlan &, float2 *, float2 *, float2, const Lay &,
                                           int, const SolveState *, cudaStream_t);
template <> void launch_gm2d_update<double>(const LevelK<double> &, double2, double, int, int,
                                            const Gm2dIn<double> &, const Gm2dWork<double> &,
                                            const Gm2dPlan &, double2 *, double2 *, double2,
                                            const Lay &, int, const SolveState *, cudaStream_t);

// (min, max) of the k^2 field of level 0 into out[0..1]; out: 2 + 2 kK2RangeBlocks.
constexpr int kK2RangeBlocks = 304;
void launch_k2_range(const double *k2, int N, int P, size_t rows, double *out, cudaStream_t s);

}  // namespace hh
