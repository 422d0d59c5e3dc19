// GMRES(m) smoothing on the small levels (hh_gmres.cu).
#pragma once
#include "hh_internal.h"
#include "hh_cheb.cuh"

namespace hh {

constexpr int kGmresMaxBatch = 64;   // right-hand sides per handle with GMRES smoothing

// The GMRES(m)-smoothed cycle on the small levels t0 .. coarsest in one
// block of 512 threads per right-hand side, every array in shared memory
// (hh_gmres.cu): from a zero initial guess, nu1 GMRES steps, residual and
// full weighting on the way down, the coarsest solve, and interpolated
// correction plus nu2 GMRES steps on the way up.  Only the right-hand side of
// level t0 is read from and its correction written to global memory.
constexpr int kGmTailMax = 8;
template <typename R> struct GmTailLevel {
  LevelK<R> K;                 // the level (tables and k^2 in global memory)
  typename Cx<R>::T c;         // scale of the residual restricted from it
  typename Cx<R>::T sigma;     // centre and inverse half width of its spectrum
  R s;                         // (hh_cheb.cuh)
  int offU, offF, offT;        // complex offsets in shared memory: iterate,
                               // right-hand side, coefficient tables (3 dim N)
  int offK;                    // real offset of k^2
};
template <typename R> struct GmTailArgs {
  int nl, m, nu1, nu2;
  GmTailLevel<R> lv[kGmTailMax];
  int offQ[4];                 // q_0..q_2, complex128: X q_{m-1} (sized for level t0)
  int kbase, invbase, smem_bytes;
  const typename Cx<R>::T *f;  // right-hand side of level t0 (library layout lay)
  typename Cx<R>::T *u;        // its correction
  Lay lay;
  const double2 *inv;          // inverse of the coarsest operator (FP64, mm x mm)
  const float *mag;            // complex64: Gm2dWork::mag
  int mm;
};
template <typename R, int DIM> size_t gmres_tail_smem(const int *N, int nl, int m);
template <typename R, int DIM> cudaError_t init_gmres_tail();
template <typename R, int DIM>
void launch_gmres_tail(const GmTailArgs<R> &a, int batch, const SolveState *st, cudaStream_t s);
constexpr size_t kGmTailSmemMax = 220 * 1024;   // of the 227 KB a block may use (2 KB static)

}  // namespace hh
