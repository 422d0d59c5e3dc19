// 2-D (5-point) kernels of the single steps: operator, weighted Jacobi sweep,
// residual + full weighting, correction + sweep.  They serve the step entry points,
// cycles with more than one sweep, and FGMRES's operator applications.
//
// A warp owns a strip of 32 adjacent columns, one per lane, and walks down a run of
// rows: the values above, at and below a point are in registers, the west and east
// ones come by shuffles (the strip's outer lanes are halo), so that every input is
// read about once and w = u + P e or the residual is formed once per point.  Where
// the strip and run lie outside the layers the coefficients are uniform and real:
// A u = D u - c_0 (sum of the neighbours), and on the finest level D is real too.
// In complex128, which these kernels are for, the FP64 pipe is the bound, so that
// is what counts: 10 to 12 FP64 instructions per point for the operator instead of
// 24, one division instead of three.
//
// Measured (GB300, complex128, 1023^2, variable k, three right-hand sides; before:
// a thread per point, five reads, the general coefficients everywhere): operator
// 143 -> 125 us, sweep 329 -> 246, residual + weighting 400 -> 225, correction +
// sweep 633 -> 305; 77 (operator) to 85 % of each is the FP64 pipe (a warp's instruction takes
// 64 cycles).  Runs of 32 rows, one warp each, took 161 / 327 / 258 / 348: blocks of
// general strips (layers) cost twice the others' work and set a single wave's time.
// A sequence of operator, adjoint operator, sweep, restriction, correction and coarse
// sweep on one right-hand side takes 1397 us at 2047^2 (2297), 420 at 1023^2 (605),
// 140 at 511^2 (181), 64 with four at 127^2 (78) and 70 with sixteen at 63^2 (78).
#include "hh_kernels.cuh"

#include <algorithm>

namespace hh {

namespace {

enum { APPLY = 0, SMOOTH = 1, CORRECT = 2, RESTRICT = 3 };

template <typename R> struct Walk2dArgs {
  using C = typename Cx<R>::T;
  LevelK<R> L;
  const C *u, *f, *e;
  C *out;                  // APPLY, SMOOTH, CORRECT: the level's array; RESTRICT: the coarse one
  Lay lc;
  C omega, cs;             // Jacobi weight; scale of the restricted residual
  int zero_mode, rows;
  const SolveState *st;
  double *partials;
};

template <typename C> __device__ __forceinline__ C lane_west(C v) {
  return cmk(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
template <typename C> __device__ __forceinline__ C lane_east(C v) {
  return cmk(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}

template <int KIND> constexpr int strip_cols() { return KIND == RESTRICT ? 28 : 30; }

template <typename R, int KIND, bool UNI>
__device__ __forceinline__ void walk_rows(const Walk2dArgs<R> &A, int b, bool zero, int x, int y0,
                                          int y1, bool own, double &acc) {
  using C = typename Cx<R>::T;
  const LevelK<R> &L = A.L;
  const int N = L.N, P = L.P;
  const bool inx = (unsigned)x < (unsigned)N;
  const C zc = czero<C>();
  const C *u = A.u + (size_t)b * L.S + x;
  const C *f = KIND == APPLY ? nullptr : A.f + (size_t)b * L.S + x;
  const R *kp = L.k2 + x;
  const C *cy = L.coef + 3 * N;
  const bool realD = UNI && L.beta.y == R(0);
  const bool realW = realD && A.omega.y == R(0);
  C lox = zc, upx = zc, dgx = zc;
  if (!UNI && inx) {
    lox = L.coef[x];
    dgx = L.coef[N + x];
    upx = L.coef[2 * N + x];
  }
  const R c0 = L.c0.x;
  C D = UNI ? L.dk : zc;   // for a constant k
  // CORRECT: the coarse row at or above the last fine row taken, interpolated in x
  const C *e = KIND == CORRECT ? A.e + (size_t)b * A.lc.S : nullptr;
  const bool el_in = inx && x >= 2 && !(x & 1), er_in = inx && (x >> 1) < A.lc.N;
  auto coarse = [&](int cr) {
    if (cr < 0 || cr >= A.lc.N) return zc;
    const C *p = e + (size_t)cr * A.lc.P + (x >> 1);
    const C r = er_in ? *p : zc;
    if (x & 1) return r;
    return cscale(cadd(el_in ? p[-1] : zc, r), R(0.5));
  };
  C ex = KIND == CORRECT ? coarse((y0 - 2) >> 1) : zc;
  auto load = [&](int y) {   // u (CORRECT: u + P e; rows in order) at row y
    const bool in = inx && (unsigned)y < (unsigned)N;
    C v = in && !zero ? u[(size_t)y * P] : zc;
    if (KIND == CORRECT) {
      C pe = ex;
      if (!(y & 1)) {
        const C nx = coarse(y >> 1);
        pe = cscale(cadd(ex, nx), R(0.5));
        ex = nx;
      }
      if (in) v = cadd(v, pe);
    }
    return v;
  };
  const int last = KIND == RESTRICT ? min(y1, N - 1) : y1 - 1;
  C vm = load(y0 - 1), v = load(y0), vp = load(y0 + 1);
  auto load_f = [&](int y) { return KIND != APPLY && inx && y <= last ? f[(size_t)y * P] : zc; };
  auto load_k = [&](int y) {
    return inx && y <= last && !(UNI && L.kconst) ? kp[(size_t)y * L.KP] : R(0);
  };
  C fv = load_f(y0);
  R kv = load_k(y0);
  C wacc = zc;
  C *out = KIND == RESTRICT ? A.out + (size_t)b * A.lc.S : A.out + (size_t)b * L.S + x;
  const C csc = cscale(A.cs, R(1.0 / 16.0));
  for (int y = y0; y <= last; ++y) {
    // the next row's inputs, in flight during this row's arithmetic
    const C vn = y < last ? load(y + 2) : zc, fn = load_f(y + 1);
    const R kn = load_k(y + 1);
    const C vw = lane_west(v), ve = lane_east(v);
    C r;                     // A v (APPLY), or f - A v
    if (UNI) {
      const C sn = cadd(cadd(vw, ve), cadd(vm, vp));
      if (!L.kconst) D = cmk(fmaf_any(-L.beta.x, kv, R(4) * c0), -L.beta.y * kv);
      if (KIND == APPLY) {
        r = cmk(fmaf_any(D.x, v.x, -c0 * sn.x), fmaf_any(D.x, v.y, -c0 * sn.y));
        if (!realD) r = cmk(fmaf_any(-D.y, v.y, r.x), fmaf_any(D.y, v.x, r.y));
      } else {
        r = cmk(fmaf_any(c0, sn.x, fmaf_any(-D.x, v.x, fv.x)),
                fmaf_any(c0, sn.y, fmaf_any(-D.x, v.y, fv.y)));
        if (!realD) r = cmk(fmaf_any(D.y, v.y, r.x), fmaf_any(-D.y, v.x, r.y));
      }
    } else {
      const C lo = cy[y], dg = cy[N + y], up = cy[2 * N + y];
      D = diag_less(cadd(dgx, dg), L.beta, kv);
      if (KIND == APPLY) {
        r = cmul(D, v);
        r = cfnma(lox, vw, r);
        r = cfnma(upx, ve, r);
        r = cfnma(lo, vm, r);
        r = cfnma(up, vp, r);
      } else {
        r = resid_row(fv, D, v, lox, vw, upx, ve, lo, vm, up, vp);
      }
    }
    if (KIND == APPLY) {
      if (own) out[(size_t)y * P] = r;
    } else if (KIND != RESTRICT) {
      C o;
      if (realW) {
        const R w = L.kconst ? L.wk.x : A.omega.x / D.x;
        o = cmk(fmaf_any(w, r.x, v.x), fmaf_any(w, r.y, v.y));
      } else {
        o = cfma(UNI && L.kconst ? L.wk : jacobi_weight(A.omega, D), r, v);
      }
      if (own) {
        out[(size_t)y * P] = o;
        if (KIND == SMOOTH && A.partials) acc += (double)r.x * r.x + (double)r.y * r.y;
      }
    } else {
      const C a = lane_west(r), c = lane_east(r);
      const C h = cmk(fmaf_any(R(2), r.x, a.x + c.x), fmaf_any(R(2), r.y, a.y + c.y));
      if (y & 1) {
        wacc = cmk(fmaf_any(R(2), h.x, wacc.x), fmaf_any(R(2), h.y, wacc.y));
      } else {
        if (y > y0 && own && (x & 1) && (x - 1) / 2 < A.lc.N)
          out[(size_t)(y / 2 - 1) * A.lc.P + (x - 1) / 2] = cmul(csc, cadd(wacc, h));
        wacc = h;
      }
    }
    vm = v;
    v = vp;
    vp = vn;
    fv = fn;
    kv = kn;
  }
}

template <typename R, int KIND>
__global__ void __launch_bounds__(256) k_walk2d(Walk2dArgs<R> A) {
  constexpr int OW = strip_cols<KIND>(), F = KIND == RESTRICT ? 2 : 1;
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (!__syncthreads_and(!(A.st && !A.st[b].active))) return;   // one decision per block
  const bool zero = A.zero_mode == ZERO_ALL || (A.zero_mode == ZERO_FLAG && A.st && A.st[b].zero);
  const LevelK<R> &L = A.L;
  const int N = L.N, strips = (N + OW - 1) / OW, runs = (N + A.rows - 1) / A.rows;
  double acc = 0.0;
  const int nw = blockDim.x >> 5;
  for (int i = blockIdx.x * nw + warp; i < strips * runs; i += gridDim.x * nw) {
    const int run = i / strips, xa = (i - run * strips) * OW - F, x = xa + lane;
    const int y0 = run * A.rows, y1 = min(N, y0 + A.rows);
    const bool own = lane >= F && lane < F + OW && x < N;
    const bool uni = xa >= L.ulo && xa + 31 <= L.uhi && y0 >= L.ulo && y1 <= L.uhi && L.c0.y == R(0);
    if (uni) walk_rows<R, KIND, true>(A, b, zero, x, y0, y1, own, acc);
    else walk_rows<R, KIND, false>(A, b, zero, x, y0, y1, own, acc);
  }
  if (KIND == SMOOTH && A.partials) {
    const double s = block_sum(acc);
    if (threadIdx.x == 0) A.partials[(size_t)b * gridDim.x + blockIdx.x] = s;
  }
}

// Rows per run, at most 32: short enough for about 64 warps per SM, several blocks
// each, which evens out the general strips' extra work (figures above); but up to 8
// as long as 16 warps per SM are left, since a run's first rows are loaded, and the
// restriction's residual is formed, twice.
template <typename R, int KIND>
void launch_walk2d(Walk2dArgs<R> a, int batch, int blocks, cudaStream_t s) {
  const int N = a.L.N, strips = (N + strip_cols<KIND>() - 1) / strip_cols<KIND>();
  const long long all = (long long)N * strips * batch, full = all / (64 * 152);
  const long long r = std::max(full, std::min<long long>(8, all / (16 * 152)));
  a.rows = (int)std::min<long long>(32, std::max<long long>(2, r)) & ~1;
  // two warps per block: with eight a few SMs got a block more than the others at
  // small sizes (four at 127^2: the sequence 83 us instead of 64).  With partial
  // sums the number of blocks is the caller's
  const int threads = blocks ? 256 : 64;
  if (!blocks) blocks = (strips * ((N + a.rows - 1) / a.rows) + 1) / 2;
  k_walk2d<R, KIND><<<dim3(blocks, batch), threads, 0, s>>>(a);
}

template <typename R> void smooth2d(const LevelK<R> &L, const typename Cx<R>::T *u_in, int zero_mode,
                                    const typename Cx<R>::T *f, typename Cx<R>::T *u_out,
                                    typename Cx<R>::T omega, int batch, const SolveState *st,
                                    double *partials, int nparts, cudaStream_t s) {
  Walk2dArgs<R> a{L, u_in, f, nullptr, u_out, Lay{0, 0, 0}, omega, czero<typename Cx<R>::T>(),
                  zero_mode, 0, st, partials};
  launch_walk2d<R, SMOOTH>(a, batch, partials ? nparts : 0, s);
}
template <typename R> void restrict2d(const LevelK<R> &L, const typename Cx<R>::T *u,
                                      const typename Cx<R>::T *f, typename Cx<R>::T *fc, const Lay &lc,
                                      typename Cx<R>::T cs, int batch, const SolveState *st,
                                      cudaStream_t s) {
  Walk2dArgs<R> a{L, u, f, nullptr, fc, lc, czero<typename Cx<R>::T>(), cs, ZERO_NONE, 0, st, nullptr};
  launch_walk2d<R, RESTRICT>(a, batch, 0, s);
}
template <typename R> void correct2d(const LevelK<R> &L, const typename Cx<R>::T *u_in,
                                     const typename Cx<R>::T *e, const Lay &lc,
                                     const typename Cx<R>::T *f, typename Cx<R>::T *u_out,
                                     typename Cx<R>::T omega, int batch, const SolveState *st,
                                     cudaStream_t s) {
  Walk2dArgs<R> a{L, u_in, f, e, u_out, lc, omega, czero<typename Cx<R>::T>(), ZERO_NONE, 0, st, nullptr};
  launch_walk2d<R, CORRECT>(a, batch, 0, s);
}
template <typename R> void apply2d(const LevelK<R> &L, const typename Cx<R>::T *x,
                                   typename Cx<R>::T *y, int batch, cudaStream_t s) {
  const auto z = czero<typename Cx<R>::T>();
  Walk2dArgs<R> a{L, x, nullptr, nullptr, y, Lay{0, 0, 0}, z, z, ZERO_NONE, 0, nullptr, nullptr};
  launch_walk2d<R, APPLY>(a, batch, 0, s);
}

}  // namespace

#define HH_STEPS2D(R)                                                                          \
  template <>                                                                                  \
  void launch_smooth<R, 2>(const LevelK<R> &L, const Cx<R>::T *u_in, int zero_mode,            \
                           const Cx<R>::T *f, Cx<R>::T *u_out, Cx<R>::T omega, int batch,      \
                           const SolveState *st, double *partials, int nparts, cudaStream_t s) { \
    smooth2d<R>(L, u_in, zero_mode, f, u_out, omega, batch, st, partials, nparts, s);          \
  }                                                                                            \
  template <>                                                                                  \
  void launch_resid_restrict<R, 2>(const LevelK<R> &L, const Cx<R>::T *u, const Cx<R>::T *f,   \
                                   Cx<R>::T *fc, const Lay &lc, Cx<R>::T cs, int batch,        \
                                   const SolveState *st, cudaStream_t s) {                     \
    restrict2d<R>(L, u, f, fc, lc, cs, batch, st, s);                                          \
  }                                                                                            \
  template <>                                                                                  \
  void launch_correct_smooth<R, 2>(const LevelK<R> &L, const Cx<R>::T *u_in, const Cx<R>::T *e, \
                                   const Lay &lc, const Cx<R>::T *f, Cx<R>::T *u_out,          \
                                   Cx<R>::T omega, int batch, const SolveState *st,            \
                                   cudaStream_t s) {                                           \
    correct2d<R>(L, u_in, e, lc, f, u_out, omega, batch, st, s);                               \
  }                                                                                            \
  template <>                                                                                  \
  void launch_apply<R, 2>(const LevelK<R> &L, const Cx<R>::T *x, Cx<R>::T *y, int batch,       \
                          cudaStream_t s) {                                                    \
    apply2d<R>(L, x, y, batch, s);                                                             \
  }
HH_STEPS2D(float)
HH_STEPS2D(double)

HH_INSTANTIATE_DIM(2)

}  // namespace hh
