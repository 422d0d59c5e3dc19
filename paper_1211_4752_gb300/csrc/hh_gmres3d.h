// GMRES(m) smoothing steps on 3-D levels with one reduction per step
// (hh_gmres3d.cuh; the method is described in hh_cheb.cuh).
#pragma once
#include "hh_gmres2d.h"

namespace hh {

// Work split of one level: planes per run and blocks per right-hand side of the
// vector kernels, of the Gram kernel (one partial matrix per block) and blocks of
// the update kernel.
struct Gm3dPlan {
  int vplanes, vblocks;
  int planes, blocks;
  int ublocks;
};
Gm3dPlan gm3d_plan(int N, int batch, int sms, bool fp64);

// One step: basis kernels (q_0 .. q_{m-1} into w.q, the partial Gram matrices),
// check: per-block |f - A w|^2 for the stop test, or null), and the update
// u_out = w + z.  With in.e the corrected iterate u + P e is written to u_out first.
// u_out must not be in.u unless the step starts from zero.
template <typename R>
void launch_gm3d_basis(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int kconst, int m,
                       const Gm2dIn<R> &in, const Gm2dWork<R> &w, const Gm3dPlan &p,
                       typename Cx<R>::T *u_out, int batch, const SolveState *st, double *check,
                       cudaStream_t stream);
template <typename R>
void launch_gm3d_update(const LevelK<R> &L, typename Cx<R>::T sigma, R s, int m,
                        const Gm2dIn<R> &in, const Gm2dWork<R> &w, const Gm3dPlan &p,
                        typename Cx<R>::T *u_out, int batch, const SolveState *st,
                        cudaStream_t stream);

// complex128: the step's coefficients and their correction's sums for the update
// kernel; rows of N points per right-hand side.  Returns the blocks of the sums.
int launch_gm_coef(const LevelK<double> &L, int rows, double2 sigma, double s, int m,
                   const Gm2dWork<double> &w, int nparts, int batch, const SolveState *st,
                   cudaStream_t stream);

}  // namespace hh
