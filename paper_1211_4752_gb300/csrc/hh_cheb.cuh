// One GMRES(m) smoothing step from a single reduction (m <= 3).
//
// The Krylov space K_m(A, r) is the same for A and for the shifted, scaled
// operator X = s (A - sigma), with sigma the centre of the level's spectrum and
// 1/s its half width.  With the Chebyshev recurrence
//     q_0 = r,   q_1 = X q_0,   q_{j+1} = 2 X q_j - q_{j-1}
// the basis stays well conditioned without orthogonalisation (Joubert and
// Carey 1992; Hoemmen 2010, communication-avoiding GMRES), so all inner
// products of the step can be taken at once: with a_j = s A q_j =
// X q_j + s sigma q_j the minimiser of |r - sum y_j a_j| solves
//     N y = b,   N_ij = <a_i, a_j>,  b_i = <a_i, r>,
// whose entries, with |r|^2, are the Gram matrix of (r, a_0 .. a_{m-1}).  Then
//     z = s sum y_j q_j.
// complex64: the sums are those of g r and its basis, g a power of two that keeps the
// level-0 residual's norm within 2^-24 .. 2^25 (gram_scale): the products are squares,
// which leave FP32's range at 1e-19 and 1e19 (the pairs' second values at 1e-12).  y
// does not depend on g.
// (The new residual r - sum y_j a_j is not taken from the basis: in complex64 it
// would miss the rounding of u + z, which f - A (u + z) contains and the coarse
// levels correct; the cycles' error against FP64 was 2 to 4 times larger.)
// Against one reduction per Arnoldi step this leaves one per GMRES step.
//
// N's condition number is the square of the basis's (1e2 .. 1e5 on rough residuals, 1e6
// and more on smooth ones), so complex64 vectors' products are summed as unevaluated pairs
// of FP32 values (Dekker / Knuth: the product's and the sum's rounding errors are kept in a
// second FP32 value), which costs no FP64 arithmetic.  On levels of more than
// kGramPairMaxN points per axis a thread's own sums are plain FP32, folded into a second
// value every four rows (3-D: eight planes; above 1024 points per axis after each run of
// rows), and pairs from there on: relative errors of 2.7e-10 (511^2), 2.3e-10 (1023^2),
// 4.0e-10 (2047^2), 6.1e-10 (511^2, 16 right-hand sides) and 1.9e-10 (127^3; 3.6e-10 with
// 16); without the folds up to 1.3e-9 and 2.5e-9, with FP32 warp sums added in FP64 4.4e-10
// to 7.2e-10.  What the nearly parallel vectors of a smooth
// residual lose to their own rounding stays: a complex64 cycle from zero on smooth
// right-hand sides is 1 to 5 times as far from the exact one as with an orthogonalised
// basis (the step's residual is the same to 1e-7), on rough ones no further.
#pragma once
#include "hh_internal.h"
#include "hh_complex.cuh"

namespace hh {

constexpr int kGramPairMaxN = 256;   // complex64: paired sums up to this N (2-D)

// ---- accumulators ----------------------------------------------------------
template <typename R, bool PAIR> struct GramAcc;
template <> struct GramAcc<double, false> {
  double h;
  __device__ __forceinline__ void zero() { h = 0.0; }
  __device__ __forceinline__ void mac(double a, double b) { h = fma(a, b, h); }
  __device__ __forceinline__ void add(const GramAcc &o) { h += o.h; }
  __device__ __forceinline__ void fold() {}
  __device__ __forceinline__ void close() {}
  __device__ __forceinline__ GramAcc shfl_xor(int m) const {
    GramAcc r;
    r.h = __shfl_xor_sync(0xffffffffu, h, m);
    return r;
  }
};
// FP32 sums of FP32 products; the sums over threads carry their rounding
// errors in l (the same storage for the plain and the paired form).
template <bool PAIR> struct GramAcc<float, PAIR> {
  float h, l;
  __device__ __forceinline__ void zero() { h = l = 0.f; }
  __device__ __forceinline__ void two_sum(float p) {   // Knuth
    const float t = __fadd_rn(h, p), b = __fsub_rn(t, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(p, b)));
    h = t;
  }
  __device__ __forceinline__ void mac(float a, float b) {
    if (PAIR) {
      const float p = __fmul_rn(a, b);
      l = __fadd_rn(l, __fmaf_rn(a, b, -p));
      two_sum(p);
    } else {
      h = fmaf(a, b, h);
    }
  }
  // plain sums of a thread: h holds a few points', l those folded before (see above)
  __device__ __forceinline__ void fold() {
    if (PAIR) return;
    l = __fadd_rn(l, h);
    h = 0.f;
  }
  __device__ __forceinline__ void close() {   // (h, l) as a pair again
    if (PAIR) return;
    const float t = l;
    l = 0.f;
    two_sum(t);
  }
  __device__ __forceinline__ void add(const GramAcc &o) {
    l = __fadd_rn(l, o.l);
    two_sum(o.h);
  }
  __device__ __forceinline__ GramAcc shfl_xor(int m) const {
    GramAcc r;
    r.h = __shfl_xor_sync(0xffffffffu, h, m);
    r.l = __shfl_xor_sync(0xffffffffu, l, m);
    return r;
  }
};
// a sum as stored between threads and kernels: a double, or an FP32 pair
template <typename R> struct GramSum { using T = float2; };
template <> struct GramSum<double> { using T = double; };
template <bool P> __device__ __forceinline__ float2 gram_store(const GramAcc<float, P> &a) {
  return make_float2(a.h, a.l);
}
__device__ __forceinline__ double gram_store(const GramAcc<double, false> &a) { return a.h; }
template <bool P> __device__ __forceinline__ void gram_add(GramAcc<float, P> &a, float2 v) {
  a.l = __fadd_rn(a.l, v.y);
  a.two_sum(v.x);
}
__device__ __forceinline__ void gram_add(GramAcc<double, false> &a, double v) { a.h += v; }
__device__ __forceinline__ double gram_value(float2 v) { return (double)v.x + (double)v.y; }   // for the stop test
__device__ __forceinline__ double gram_value(double v) { return v; }

// g of a right-hand side from the estimate m[b] of its level-0 residual's magnitude:
// 1 for an m of 2^-24 .. 2^25 and where there is none (0, infinity, NaN), else the power
// of two that brings m to [1, 2).
__device__ __forceinline__ float gram_scale(const float *m, int b) {
  const float v = m[b];
  if (!(v > 0.f) || !(v < 3e38f)) return 1.f;
  const int e = min(80, max(-80, ((__float_as_int(v) >> 23) & 255) - 127));
  return e >= -24 && e <= 24 ? 1.f : __int_as_float((127 - e) << 23);
}
template <typename R> __device__ __forceinline__ R gram_scale_of(const float *m, int b) {
  if constexpr (sizeof(R) == 4) return gram_scale(m, b);
  else return R(1);
}
__device__ __forceinline__ float gram_rcp(float g) { return __int_as_float((254 << 23) - __float_as_int(g)); }   // 1 / g
// |r|^2 from the sum of |g r|^2
template <typename S> __device__ __forceinline__ double gram_unscaled(S sum, float g) {
  const double i = (double)gram_rcp(g);
  return gram_value(sum) * i * i;
}
// The next step's estimate from the sum of |g q_0|^2 of this one (left where that
// says nothing)
__device__ __forceinline__ void gram_estimate(float *m, int b, float2 sum, float g) {
  if (sum.x > 0.f && sum.x < 3e38f) m[b] = sqrtf(sum.x) * gram_rcp(g);
}

// Real numbers of the Gram matrix of m + 1 vectors, and that count rounded up
// to a power of two: entry i <= m is |v_i|^2; pair (i < j), counted in the order
// (0,1) (0,2) .. (0,m) (1,2) .., is at m + 1 + 2 pair (real and imaginary part
// of <v_i, v_j>).
template <int M> struct Gram {
  static constexpr int NV = M + 1, NQ = NV * NV, NQP = M == 1 ? 4 : 16;
  __host__ __device__ static constexpr int pair(int i, int j) {   // i < j
    return NV + 2 * (i * (2 * NV - i - 1) / 2 + (j - i - 1));
  }
};

template <typename R, int M, bool PAIR, typename C>
__device__ __forceinline__ void gram_point(GramAcc<R, PAIR> (&acc)[Gram<M>::NQP], const C (&v)[M + 1]) {
#pragma unroll
  for (int i = 0; i <= M; ++i) {
    acc[i].mac(v[i].x, v[i].x);
    acc[i].mac(v[i].y, v[i].y);
#pragma unroll
    for (int j = i + 1; j <= M; ++j) {
      const int p = Gram<M>::pair(i, j);
      acc[p].mac(v[i].x, v[j].x);
      acc[p].mac(v[i].y, v[j].y);
      acc[p + 1].mac(v[i].x, v[j].y);
      acc[p + 1].mac(-v[i].y, v[j].x);
    }
  }
}

// Half of a point's products: half 0 takes quantities 0 .. NQP/2 - 1, half 1 the
// others (the same number of products each for M = 3).
template <typename R, int M, bool PAIR, typename C>
__device__ __forceinline__ void gram_point_half(GramAcc<R, PAIR> (&acc)[Gram<M>::NQP],
                                                const C (&v)[M + 1], int half) {
  constexpr int H = Gram<M>::NQP / 2;
#pragma unroll
  for (int i = 0; i <= M; ++i) {
    if ((i >= H) == (half == 1)) {
      acc[i].mac(v[i].x, v[i].x);
      acc[i].mac(v[i].y, v[i].y);
    }
#pragma unroll
    for (int j = i + 1; j <= M; ++j) {
      const int p = Gram<M>::pair(i, j);
      if ((p >= H) == (half == 1)) {
        acc[p].mac(v[i].x, v[j].x);
        acc[p].mac(v[i].y, v[j].y);
      }
      if ((p + 1 >= H) == (half == 1)) {
        acc[p + 1].mac(v[i].x, v[j].y);
        acc[p + 1].mac(-v[i].y, v[j].x);
      }
    }
  }
}

// Sum of NQP quantities over a warp with NQP shuffles (instead of 5 NQP): at
// each step a lane keeps half of its quantities and hands the other half to
// its partner.  Lane l ends with the warp's sum of quantity l >> (5 - log2 NQP).
template <typename A, int NQP>
__device__ __forceinline__ A gram_warp_sum(A (&v)[NQP]) {
  const int lane = threadIdx.x & 31;
  int bit = 16;
#pragma unroll
  for (int n = NQP / 2; n >= 1; n >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int i = 0; i < NQP / 2; ++i) {
      if (i < n) {
        const A own = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
        v[i] = own;
        v[i].add(give.shfl_xor(bit));
      }
    }
    bit >>= 1;
  }
  for (; bit >= 1; bit >>= 1) v[0].add(v[0].shfl_xor(bit));
  return v[0];
}

// Arithmetic of the small solve: FP64 for complex128; for complex64 unevaluated
// pairs of FP32 values (Dekker 1971; about 46 bits).  An FP64 instruction takes a
// warp of this part 64 cycles, so that the solve took 2.6 us in FP64.
struct PairF {
  float h, l;
  __device__ __forceinline__ PairF() {}
  __device__ __forceinline__ PairF(float a, float b) : h(a), l(b) {}
  __device__ __forceinline__ explicit PairF(float2 v) {   // a stored sum, renormalised
    h = __fadd_rn(v.x, v.y);
    l = __fadd_rn(v.y, -__fsub_rn(h, v.x));
  }
  __device__ __forceinline__ static PairF zero() { return PairF(0.f, 0.f); }
  __device__ __forceinline__ PairF neg() const { return PairF(-h, -l); }
  __device__ __forceinline__ float lead() const { return h; }
  __device__ __forceinline__ PairF shfl(int src) const {
    return PairF(__shfl_sync(0xffffffffu, h, src), __shfl_sync(0xffffffffu, l, src));
  }
  __device__ __forceinline__ static PairF quick(float a, float b) {   // |a| >= |b|
    const float t = __fadd_rn(a, b);
    return PairF(t, __fsub_rn(b, __fsub_rn(t, a)));
  }
  __device__ __forceinline__ PairF mul(PairF o) const {
    const float p = __fmul_rn(h, o.h);
    return quick(p, __fmaf_rn(l, o.h, __fmaf_rn(h, o.l, __fmaf_rn(h, o.h, -p))));
  }
  __device__ __forceinline__ PairF add(PairF o) const {
    const float t = __fadd_rn(h, o.h), b = __fsub_rn(t, h);
    const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, b)), __fsub_rn(o.h, b));
    return quick(t, __fadd_rn(e, __fadd_rn(l, o.l)));
  }
  // 1 / this where the value exceeds tol * d (and FP32's smallest normal), else 0
  __device__ __forceinline__ PairF pivot_rcp(PairF d, double tol) const {
    if (!(h > (float)tol * d.h) || !(h > 2e-38f)) return zero();
    const float x = 1.0f / h;
    return quick(x, __fmul_rn(x, __fmaf_rn(-l, x, __fmaf_rn(-h, x, 1.0f))));
  }
};
struct Fp64 {
  double h;
  __device__ __forceinline__ Fp64() {}
  __device__ __forceinline__ explicit Fp64(double v) : h(v) {}
  __device__ __forceinline__ static Fp64 zero() { return Fp64(0.0); }
  __device__ __forceinline__ Fp64 neg() const { return Fp64(-h); }
  __device__ __forceinline__ double lead() const { return h; }
  __device__ __forceinline__ Fp64 shfl(int src) const { return Fp64(__shfl_sync(0xffffffffu, h, src)); }
  __device__ __forceinline__ Fp64 mul(Fp64 o) const { return Fp64(h * o.h); }
  __device__ __forceinline__ Fp64 add(Fp64 o) const { return Fp64(h + o.h); }
  __device__ __forceinline__ Fp64 pivot_rcp(Fp64 d, double tol) const {
    return h > tol * d.h ? Fp64(1.0 / h) : zero();
  }
};
template <typename R> struct SolveNum { using T = PairF; };
template <> struct SolveNum<double> { using T = Fp64; };

// Coefficients of one step's update, z_j = s y_j, in the vectors' precision;
// complex128: and the inverse of N, for the correction of y (solve_correction).
template <typename R> struct StepCoef {
  typename Cx<R>::T z[3];
};
template <> struct StepCoef<double> {
  double2 z[3];
  double2 inv[3][3];
};

// Solve N y = b from the Gram sums G (NQP entries, shared memory) by
// Gauss-Jordan elimination, one warp, lane 4 i + j holding entry (i, j) of
// [N | b], and store the step's coefficients (complex128: the inverse grows in N's place).  N is Hermitian and positive
// semidefinite; a pivot that is at most tol times its diagonal entry marks a
// vector in the span of the earlier ones: its coefficient is zero (the Krylov
// space has ended).  Called by the 32 lanes of one warp.
template <typename R, int M>
__device__ __forceinline__ void gram_solve(const typename GramSum<R>::T *G, R s, double tol,
                                           StepCoef<R> *out) {
  using T = typename SolveNum<R>::T;
  const int lane = threadIdx.x & 31;
  const int i = lane >> 2, j = lane & 3;
  T ax = T::zero(), ay = T::zero();
  if (i < M && (j < M || j == 3)) {
    const int p = i + 1, q = j == 3 ? 0 : j + 1;
    if (p == q) {
      ax = T(G[p]);
    } else {
      const int k = p < q ? Gram<M>::pair(p, q) : Gram<M>::pair(q, p);
      ax = T(G[k]);
      ay = T(G[k + 1]);
      if (p > q) ay = ay.neg();
    }
  }
  const T diag = ax;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const T pk = ax.shfl(5 * k), dk = diag.shfl(5 * k), rp = pk.pivot_rcp(dk, tol);
    // row k scaled, and this row's entry of column k
    T kx = ax.shfl(4 * k + j).mul(rp), ky = ay.shfl(4 * k + j).mul(rp);
    const T lx = ax.shfl(4 * i + k), ly = ay.shfl(4 * i + k);
    if (sizeof(R) == 8 && j == k) {   // the inverse's column, from the unit matrix
      kx = rp;
      ax = ay = ky = T::zero();
    }
    if (i == k) {
      ax = kx;
      ay = ky;
    } else {
      ax = ax.add(ly.mul(ky)).add(lx.mul(kx).neg());
      ay = ay.add(lx.mul(ky).add(ly.mul(kx)).neg());
    }
  }
  if (j == 3 && i < 3) {   // row i's solution
    out->z[i].x = R(ax.lead()) * s;
    out->z[i].y = R(ay.lead()) * s;
  }
  if constexpr (sizeof(R) == 8) {
    if (i < M && j < M) out->inv[i][j] = make_double2(ax.lead(), ay.lead());
  }
}

// complex128: y from the normal equations alone loses digits by N's condition (a cycle
// against quad precision 2e-15 to 7e-15 where an orthogonalised basis gave 0.8e-15, a step
// on smooth residuals 1e-13).  One correction restores them (corrected seminormal
// equations, Bjorck 1987): d_i = <a_i, r - sum y_j a_j> from the vectors, y += N^-1 d.
// Lanes 0 .. M - 1 of a warp; d: real and imaginary parts (shared memory).
template <int M>
__device__ __forceinline__ void solve_correction(const double *d, double s, StepCoef<double> *c) {
  const int i = threadIdx.x & 31;
  if (i >= M) return;
  double2 y = czero<double2>();
#pragma unroll
  for (int j = 0; j < M; ++j) y = cfma(c->inv[i][j], make_double2(d[2 * j], d[2 * j + 1]), y);
  c->z[i] = cadd(c->z[i], cscale(y, s));
}
// a point's part of d (acc[2 j], acc[2 j + 1]) from a_j and r
template <int M>
__device__ __forceinline__ void correction_point(GramAcc<double, false> (&acc)[8], const double2 (&a)[M],
                                                 const double2 (&y)[M], double2 r) {
#pragma unroll
  for (int j = 0; j < M; ++j) r = cfnma(y[j], a[j], r);
#pragma unroll
  for (int j = 0; j < M; ++j) {
    acc[2 * j].mac(a[j].x, r.x);
    acc[2 * j].mac(a[j].y, r.y);
    acc[2 * j + 1].mac(a[j].x, r.y);
    acc[2 * j + 1].mac(-a[j].y, r.x);
  }
}

// Pivot tolerance: above the rounding of the sums (1e-14 paired, 1e-9 plain
// FP32, 1e-16 FP64) and far below the pivots of a proper step.
template <typename R> __host__ __device__ constexpr double gram_tol(bool pair) {
  return sizeof(R) == 8 ? 1e-14 : (pair ? 1e-12 : 1e-8);
}

}  // namespace hh
