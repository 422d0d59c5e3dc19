// complex128 kernels of the 2-D GMRES steps (hh_gmres2d.cuh), and the helpers
// that do not depend on the precision.  These kernels are bound by the FP64 pipe
// (a warp's FP64 instruction takes 64 cycles), so the basis is stored for the
// update instead of formed twice, and the halo, which costs arithmetic, is kept
// small: a block works on tiles of 56 columns and up to 32 rows in shared memory,
// a thread per column and run of rows, the values above and below carried in
// registers.  Small levels: a thread per point of 8 x 8 tiles (hh_gmres2d.cuh).
// Measured (GB300, constant k with layers; in brackets a kernel and a reduction per Arnoldi
// step): a GMRES(3) step takes 479 us at 1023^2 (394), 165 at 511^2 (140), 90 at 255^2 (76),
// 38 at 127^2 (51) and 24 at 63^2 (51), and of four right-hand sides at 1023^2 1460 (1424);
// the cycle of one at 1023^2 1.98 ms (1.99), of four there 5.40 (5.49) and at 255^2 0.82
// (1.05).  A fifth of a step is the correction of its coefficients (k_gm2d_coef), without
// which these kernels lose digits.  The FP64 pipe is 86 % busy in the basis kernel at 1023^2,
// 89 % in k_gm2d_coef and 71 to 76 % in the update.
#include "hh_gmres2d.cuh"
#include "hh_gmres3d.h"

namespace hh {

namespace {

// Operator of one column of a tile.  GENERAL: the column's coefficients and a
// row's (lo, dg, up) are zero outside the domain; with every vector zero there
// too, X and resid are zero outside the domain without a test.
template <typename R, int MODE> struct ColumnOp {
  using C = typename Cx<R>::T;
  C c0, D0, sb, sd;        // uniform: c_0, 4 c_0, s beta, s (4 c_0 - sigma)
  C lo, up, dg, dgs, sigma, beta;   // dgs = dg - sigma
  R cf, s, kc;
  bool realb;              // beta is real (a comparison per point is an FP64 instruction)
  __device__ __forceinline__ ColumnOp(const LevelK<R> &L, C sigma_, R s_)
      : sigma(sigma_), beta(L.beta), s(s_), kc(L.kc), realb(L.beta.y == R(0)) {
    if (MODE != GENERAL) {
      c0 = L.c0;
      D0 = cscale(c0, R(4));
      cf = s * c0.x;
      sb = cscale(L.beta, s);
      sd = cscale(csub(D0, sigma), s);
    }
  }
  __device__ __forceinline__ void column(const LevelK<R> &L, int x) {
    if (MODE != GENERAL) return;
    const bool in = (unsigned)x < (unsigned)L.N;
    lo = in ? L.coef[x] : czero<C>();
    dg = in ? L.coef[L.N + x] : czero<C>();
    dgs = csub(dg, sigma);
    up = in ? L.coef[2 * L.N + x] : czero<C>();
  }
  __device__ __forceinline__ C neighbours(const C *rc, C vw, C ve, C vn, C vs) const {
    C nb = cmul(lo, vw);
    nb = cfma(up, ve, nb);
    nb = cfma(rc[0], vn, nb);
    return cfma(rc[2], vs, nb);
  }
  // X v = s (A - sigma) v; rc: the row's coefficients, kv: k^2 of the point
  __device__ __forceinline__ C X(C v, C vw, C ve, C vn, C vs, const C *rc, R kv) const {
    if (MODE == GENERAL) {
      const C d = diag_less(cadd(dgs, rc[1]), beta, kv);
      return cscale(csub(cmul(d, v), neighbours(rc, vw, ve, vn, vs)), s);
    }
    const C sn = cadd(cadd(vw, ve), cadd(vn, vs));
    C r = cmk(-cf * sn.x, -cf * sn.y);
    if (MODE == UNIFORM) {
      // (beta and sigma are real on the finest level: uniform branches leave out
      // the products with zero here and below)
      const R dx = fmaf_any(-sb.x, kv, sd.x);
      r = cmk(fmaf_any(dx, v.x, r.x), fmaf_any(dx, v.y, r.y));
      if (!realb) {
        const R dy = fmaf_any(-sb.y, kv, sd.y);
        r = cmk(fmaf_any(-dy, v.y, r.x), fmaf_any(dy, v.x, r.y));
      }
    }
    return r;
  }
  __device__ __forceinline__ C resid(C f, C v, C vw, C ve, C vn, C vs, const C *rc, R kv) const {
    if (MODE == GENERAL) {
      const C d = diag_less(cadd(dg, rc[1]), beta, kv);
      return resid_row(f, d, v, lo, vw, up, ve, rc[0], vn, rc[2], vs);
    }
    const C sn = cadd(cadd(vw, ve), cadd(vn, vs));
    const R kk = MODE == UNIFORM_K ? kc : kv;
    const R dx = fmaf_any(-beta.x, kk, D0.x);
    C r;
    r.x = fmaf_any(c0.x, sn.x, fmaf_any(-dx, v.x, f.x));
    r.y = fmaf_any(c0.x, sn.y, fmaf_any(-dx, v.y, f.y));
    if (!realb) {
      const R dy = beta.y * kk;
      r = cmk(fmaf_any(-dy, v.y, r.x), fmaf_any(dy, v.x, r.y));
    }
    return r;
  }
};

constexpr int kTX = 56, kTP = 64;      // tile columns; row pitch of its buffers
constexpr int kTileThreads = 512;
// Buffers hold the tile and m + 1 points around it (the iterate around m products).

// Calls fn(column, first row, end row) for the thread's run of rows of a region
// of W columns and H rows (compile-time W: the threads' columns are fixed).
template <int W, typename F> __device__ __forceinline__ void column_runs(int H, F fn) {
  constexpr int NS = kTileThreads / W;
  const int tx = threadIdx.x % W, sg = threadIdx.x / W;
  const int rs = (H + NS - 1) / NS, r0 = sg * rs, r1 = min(H, r0 + rs);
  if (sg < NS && r0 < r1) fn(tx, r0, r1);
}

// The tile in flight.  Buffer coordinates: (x - bx, y - by).
template <typename R, int MODE> struct TileCtx {
  using C = typename Cx<R>::T;
  const LevelK<R> &L;
  int bx, by;              // the point at buffer position (0, 0)
  const C *rows;           // shared row coefficients: lo, dg, up of buffer row r at 3 r
  __device__ __forceinline__ R k2(int x, int y) const {
    if (MODE == UNIFORM_K) return R(0);
    if (MODE == GENERAL && ((unsigned)x >= (unsigned)L.N || (unsigned)y >= (unsigned)L.N)) return R(0);
    return L.k2[(size_t)y * L.KP + x];
  }
  // Walks the W x H region whose first point is buffer (o, o): put(position, x, y,
  // X v or f - A v) from the vector in buffer src; f: its values (null: X).
  template <int W, bool RES, typename F, typename P>
  __device__ __forceinline__ void walk(ColumnOp<R, MODE> &op, const C *src, int o, int H, F fval, P put) const {
    column_runs<W>(H, [&](int tx, int r0, int r1) {
      op.column(L, bx + o + tx);
      const C *p = src + (r0 + o) * kTP + tx + o;
      C vn = p[-kTP], v = p[0];
      for (int r = r0; r < r1; ++r, p += kTP) {
        const C vs = p[kTP], vw = p[-1], ve = p[1];
        const int pos = (r + o) * kTP + tx + o, x = bx + o + tx, y = by + o + r;
        const R kv = k2(x, y);
        const C *rc = rows + 3 * (r + o);
        put(pos, x, y, RES ? op.resid(fval(pos, x, y), v, vw, ve, vn, vs, rc, kv)
                           : op.X(v, vw, ve, vn, vs, rc, kv));
        vn = v;
        v = vs;
      }
    });
  }
};

// Stages the iterate and the right-hand side of a tile (h buffer rows) and, off
// the uniform region, the row coefficients.  u, f: arrays of one right-hand side.
template <typename R, bool CORR>
__device__ __forceinline__ void stage_tile(const LevelK<R> &L, const Gm2dIn<R> &in, int b, bool zero,
                                           bool rows, int bx, int by, int h, typename Cx<R>::T *A,
                                           typename Cx<R>::T *F, typename Cx<R>::T *sr) {
  using C = typename Cx<R>::T;
  const int N = L.N;
  const int tx = threadIdx.x % kTP, x = bx + tx;
  const C *f = in.f + (size_t)b * L.S;
  const bool inx = (unsigned)x < (unsigned)N;
#pragma unroll 4
  for (int r = threadIdx.x / kTP; r < h; r += kTileThreads / kTP) {
    const int y = by + r;
    A[r * kTP + tx] = start_at<R, CORR>(L, in, b, zero, x, y);
    F[r * kTP + tx] = inx && (unsigned)y < (unsigned)N ? f[(size_t)y * L.P + x] : czero<C>();
  }
  if (rows) {
    for (int i = threadIdx.x; i < 3 * h; i += kTileThreads) {
      const int y = by + i / 3;
      sr[i] = (unsigned)y < (unsigned)N ? L.coef[(3 + i % 3) * N + y] : czero<C>();
    }
  }
}

// Body of a tile: x in [xlo, xhi], y in [ylo, yhi] are the points whose
// coefficients it uses.
template <typename R>
__device__ __forceinline__ int tile_mode(const LevelK<R> &L, int kconst, int xlo, int xhi, int ylo, int yhi) {
  const bool uni = xlo >= L.ulo && xhi <= L.uhi && ylo >= L.ulo && yhi <= L.uhi && L.c0.y == R(0);
  return !uni ? GENERAL : (kconst ? UNIFORM_K : UNIFORM);
}

// Dynamic shared memory of the tile kernels: three buffers of `ty` + 2 (m + 1) + 1
// rows and the row coefficients.
__host__ __device__ constexpr int tile_rows(int m, int ty) { return ty + 2 * m + 3; }
size_t tile_smem(int m, int ty) {
  return (size_t)tile_rows(m, ty) * (3 * kTP + 3) * sizeof(double2);
}

// Basis of a tile whose iterate is in A and right-hand side in F: q_0 -> B,
// q_1 -> A, q_2 -> F (M - 1 products), each with the block's barrier after it.
// The region of q_j is the tile and M - j points around it.
template <typename R, int M, int MODE, int TX, int XH>
__device__ __forceinline__ void tile_vectors(const TileCtx<R, MODE> &t, ColumnOp<R, MODE> &op, int H,
                                             typename Cx<R>::T *A, typename Cx<R>::T *B,
                                             typename Cx<R>::T *F) {
  using C = typename Cx<R>::T;
  // q_0 on buffer [1, TX + XH - 1) x [1, H - 1)
  t.template walk<TX + XH - 2, true>(op, A, 1, H - 2, [&](int p, int, int) { return F[p]; },
                                     [&](int p, int, int, C r) { B[p] = r; });
  __syncthreads();
  if (M >= 2) {
    t.template walk<TX + XH - 4, false>(op, B, 2, H - 4, [](int, int, int) { return C(); },
                                        [&](int p, int, int, C r) { A[p] = r; });
    __syncthreads();
  }
  if (M >= 3) {
    t.template walk<TX + XH - 6, false>(op, A, 3, H - 6, [](int, int, int) { return C(); },
                                        [&](int p, int, int, C r) { F[p] = cmk(fmaf_any(R(2), r.x, -B[p].x), fmaf_any(R(2), r.y, -B[p].y)); });
    __syncthreads();
  }
}

template <typename R, int M, int MODE, bool CORR>
__device__ __forceinline__ void basis_body(const LevelK<R> &L, const Gm2dWork<R> &wk,
                                           typename Cx<R>::T sigma, R s, int b, int bx, int by,
                                           int ty, typename Cx<R>::T *A, typename Cx<R>::T *B,
                                           typename Cx<R>::T *F, const typename Cx<R>::T *sr,
                                           GramAcc<R, false> (&acc)[Gram<M>::NQP]) {
  using C = typename Cx<R>::T;
  constexpr int XH = 2 * (M + 1);
  const TileCtx<R, MODE> t{L, bx, by, sr};
  ColumnOp<R, MODE> op(L, sigma, s);
  tile_vectors<R, M, MODE, kTX, XH>(t, op, ty + XH, A, B, F);
  const C sg = cscale(sigma, s);
  const bool reals = sg.y == R(0);
  const C *src = M == 1 ? B : (M == 2 ? A : F);
  t.template walk<kTX, false>(op, src, M + 1, ty, [](int, int, int) { return C(); },
                              [&](int p, int x, int y, C xl) {
    C v[M + 1];   // (zero outside the domain)
    v[0] = B[p];
    auto shifted = [&](C q, C xq) {   // X q + s sigma q
      C r = cmk(fmaf_any(sg.x, q.x, xq.x), fmaf_any(sg.x, q.y, xq.y));
      if (!reals) r = cmk(fmaf_any(-sg.y, q.y, r.x), fmaf_any(sg.y, q.x, r.y));
      return r;
    };
    if (M == 1) v[1] = shifted(v[0], xl);
    if (M >= 2) v[1] = shifted(v[0], A[p]);
    if (M == 2) v[2] = shifted(A[p], xl);
    if (M == 3) {
      v[M - 1] = shifted(A[p], cscale(cadd(F[p], v[0]), R(0.5)));
      v[M] = shifted(F[p], xl);
    }
    gram_point<R, M, false>(acc, v);
    if (x < L.N && y < L.N) {
      C *q = wk.q + (size_t)b * L.S + (size_t)y * L.P + x;
      q[0] = v[0];
      if (M >= 2) q[wk.qs] = A[p];
      if (M >= 3) q[2 * wk.qs] = F[p];
      q[M * wk.qs] = xl;
    }
  });
}

// ty: rows of a tile.
template <int M, bool CORR>
__global__ void __launch_bounds__(kTileThreads)
k_gm2d_basis(LevelK<double> L, double2 sigma, double s, int kconst, Gm2dIn<double> in, Gm2dWork<double> wk,
             int ty, const SolveState *st, double *check) {
  using R = double;
  using C = double2;
  constexpr int NQP = Gram<M>::NQP, NW = kTileThreads / 32;
  using S = typename GramSum<R>::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ S sums[NW * NQP];
  const int hb = tile_rows(M, ty);
  C *A = reinterpret_cast<C *>(smem_raw), *B = A + hb * kTP, *F = B + hb * kTP, *sr = F + hb * kTP;
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  const bool zero = __syncthreads_or(in.zero_mode == ZERO_ALL ||
                                     (in.zero_mode == ZERO_FLAG && st && st[b].zero)) != 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) wk.zflag[b] = zero;
  using Acc = GramAcc<R, false>;
  Acc acc[NQP];
#pragma unroll
  for (int i = 0; i < NQP; ++i) acc[i].zero();
  const int N = L.N, nx = (N + kTX - 1) / kTX, ntiles = nx * ((N + ty - 1) / ty);
  for (int i = blockIdx.x; i < ntiles; i += gridDim.x) {
    const int x0 = (i % nx) * kTX, y0 = (i / nx) * ty, bx = x0 - M - 1, by = y0 - M - 1;
    const int mode = tile_mode(L, kconst, x0 - M, x0 + kTX + M - 1, y0 - M, y0 + ty + M - 1);
    if (i != (int)blockIdx.x) __syncthreads();   // the previous tile's last reads
    stage_tile<R, CORR>(L, in, b, zero, mode == GENERAL, bx, by, ty + 2 * (M + 1), A, F, sr);
    __syncthreads();
    if (mode == UNIFORM_K) basis_body<R, M, UNIFORM_K, CORR>(L, wk, sigma, s, b, bx, by, ty, A, B, F, sr, acc);
    else if (mode == UNIFORM) basis_body<R, M, UNIFORM, CORR>(L, wk, sigma, s, b, bx, by, ty, A, B, F, sr, acc);
    else basis_body<R, M, GENERAL, CORR>(L, wk, sigma, s, b, bx, by, ty, A, B, F, sr, acc);
  }
  // block sums, in a fixed order
  constexpr int SH = NQP == 16 ? 1 : 3;   // lane l holds quantity l >> SH
  const Acc v = gram_warp_sum<Acc, NQP>(acc);
  if ((lane & ((1 << SH) - 1)) == 0) sums[warp * NQP + (lane >> SH)] = gram_store(v);
  __syncthreads();
  if (threadIdx.x < NQP) {
    Acc t;
    t.zero();
    for (int i = 0; i < NW; ++i) gram_add(t, sums[i * NQP + threadIdx.x]);
    const S g = gram_store(t);
    wk.parts[((size_t)b * gridDim.x + blockIdx.x) * NQP + threadIdx.x] = g;
    if (check && threadIdx.x == 0) check[(size_t)b * gridDim.x + blockIdx.x] = gram_value(g);
  }
}

// Residual of the new iterate in buffer U on the tile and the point after it, and
// its weighting (T: scratch).  o: buffer position of the tile's first point.
template <typename R, int MODE, int TX>
__device__ __forceinline__ void restrict_body(const TileCtx<R, MODE> &t, ColumnOp<R, MODE> &op,
                                              const typename Cx<R>::T *f, const typename Cx<R>::T *U,
                                              typename Cx<R>::T *T, int o, int ty, int x0, int y0,
                                              typename Cx<R>::T *fc, typename Cx<R>::T csc,
                                              const Lay &lc) {
  using C = typename Cx<R>::T;
  const int N = t.L.N, P = t.L.P;
  t.template walk<TX + 1, true>(op, U, o, ty + 1,
                                [&](int, int x, int y) {
                                  return x < N && y < N ? f[(size_t)y * P + x] : czero<C>();
                                },
                                [&](int p, int, int, C r) { T[p] = r; });
  __syncthreads();
  constexpr int TC = TX / 2;
  for (int i = threadIdx.x; i < TC * (ty / 2); i += kTileThreads) {
    const int cx = i % TC, cy = i / TC, gx = x0 / 2 + cx, gy = y0 / 2 + cy;
    if (gx < lc.N && gy < lc.N)
      fc[(size_t)gy * lc.P + gx] =
          weight_at<R>(T + (2 * cy + 1 + o) * kTP + 2 * cx + 1 + o, kTP, csc);
  }
}

// The step's coefficients from the partial Gram matrices, for the update kernel
// (every block of this kernel adds and solves; block 0 stores), and per block the sums of
// their correction (solve_correction) from the stored vectors.  Bound by the FP64 pipe
// (89 % busy, 32 instructions per point on the finest level, 38 below): 77 us at 1023^2, 40
// at 511^2, 11 on small levels.
template <int M>
__global__ void __launch_bounds__(1024)
k_gm2d_coef(LevelK<double> L, int rows, double2 sigma, double s, Gm2dWork<double> wk, int nparts,
            double tol, const SolveState *st) {
  constexpr int NQP = Gram<M>::NQP;
  using A = GramAcc<double, false>;
  __shared__ double sums[32 * 16];
  __shared__ StepCoef<double> sc;
  const int b = blockIdx.y;
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  step_coef<double, M>(wk.parts + (size_t)b * nparts * NQP, nparts, s, tol, sums, &sc);
  if (blockIdx.x == 0 && threadIdx.x < kGm2dCoef)
    wk.coef[(size_t)b * kGm2dCoef + threadIdx.x] = reinterpret_cast<const double *>(&sc)[threadIdx.x];
  A acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i].zero();
  double2 y[M];
#pragma unroll
  for (int j = 0; j < M; ++j) y[j] = cscale(sc.z[j], (M == 3 && j == 1 ? 0.5 : 1.0) / s);
  const double2 t = cscale(sigma, s), t2 = cadd(t, t);
  const double2 *q = wk.q + (size_t)b * L.S;
  const int N = L.N;
  // (real t, the finest level's: two loops; with a condition in one both sides' products
  // were formed, 89 us)
  auto walk = [&](auto real) {
    auto shifted = [](double2 c, double2 q, double2 xq) {   // xq + c q
      double2 r = make_double2(fma(c.x, q.x, xq.x), fma(c.x, q.y, xq.y));
      if (!decltype(real)::value) r = make_double2(fma(-c.y, q.y, r.x), fma(c.y, q.x, r.y));
      return r;
    };
    for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < (unsigned)rows * (unsigned)N; p += gridDim.x * blockDim.x) {
      const unsigned yy = p / (unsigned)N, o = yy * (unsigned)L.P + (p - yy * (unsigned)N);
      double2 v[M + 1], a[M];
#pragma unroll
      for (int j = 0; j <= M; ++j) v[j] = q[(size_t)j * wk.qs + o];   // v[M] = X q_{M-1}
      a[0] = shifted(t, v[0], v[1]);
      if (M == 2) a[M - 1] = shifted(t, v[1], v[M]);
      if (M == 3) {   // (twice a_1, with half of y_1 and of d_1)
        a[1 % M] = shifted(t2, v[1], cadd(v[2 % (M + 1)], v[0]));
        a[M - 1] = shifted(t, v[M - 1], v[M]);
      }
      correction_point<M>(acc, a, y, v[0]);
    }
  };
  if (t.y == 0.0) walk(std::true_type());
  else walk(std::false_type());
  const A v = gram_warp_sum<A, 8>(acc);
  __syncthreads();   // (block 0 has read the coefficients; the Gram sums are used up)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((lane & 3) == 0) sums[warp * 8 + (lane >> 2)] = v.h;
  __syncthreads();
  if (threadIdx.x < 8) {
    double r = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sums[w * 8 + threadIdx.x];
    if (M == 3 && threadIdx.x >> 1 == 1) r *= 0.5;
    wk.parts2[((size_t)b * kGm2dCorr + blockIdx.x) * 8 + threadIdx.x] = r;
  }
}

// complex128: from the stored basis.  With REST the new iterate of the tile and
// two points around it (three at the high ends) in a shared buffer, then as above.
template <int M, bool CORR, bool REST>
__global__ void __launch_bounds__(kTileThreads)
k_gm2d_update(LevelK<double> L, double2 sigma, double s, int kconst, Gm2dIn<double> in,
                     Gm2dWork<double> wk, int nparts, int ty, double2 *u_out,
                     double2 *fc, double2 cs, Lay lc, const SolveState *st) {
  constexpr int TX = kTX, O = REST ? 1 : 0, XH = REST ? 3 : 0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sums[kTileThreads / 4];
  __shared__ StepCoef<double> sc;
  const int hb = tile_rows(M, ty);
  double2 *A = reinterpret_cast<double2 *>(smem_raw), *B = A + hb * kTP, *sr = B + 2 * hb * kTP;
  const int b = blockIdx.y, N = L.N, P = L.P;
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  const bool zero = wk.zflag[b] != 0;
  read_coef_block<M>(wk, b, nparts, s, sums, &sc);
  const double2 *q = wk.q + (size_t)b * L.S;
  u_out += (size_t)b * L.S;
  if (REST) fc += (size_t)b * lc.S;
  const int nx = (N + TX - 1) / TX, ntiles = nx * ((N + ty - 1) / ty);
  for (int i = blockIdx.x; i < ntiles; i += gridDim.x) {
    const int x0 = (i % nx) * TX, y0 = (i / nx) * ty, bx = x0 - O, by = y0 - O;
    if (i != (int)blockIdx.x) __syncthreads();
    const int tx = threadIdx.x % kTP, x = bx + tx;
#pragma unroll 2
    for (int r = threadIdx.x / kTP; r < ty + XH; r += kTileThreads / kTP) {
      const int y = by + r;
      double2 w = start_at<double, CORR>(L, in, b, zero, x, y);
      if (tx < TX + XH && (unsigned)x < (unsigned)N && (unsigned)y < (unsigned)N) {
        const size_t o = (size_t)y * P + x;
#pragma unroll
        for (int j = 0; j < M; ++j) w = cfma(sc.z[j], q[(size_t)j * wk.qs + o], w);
        if (x >= x0 && x < x0 + TX && y >= y0 && y < y0 + ty) u_out[o] = w;
      }
      if (REST) A[r * kTP + tx] = w;
    }
    if constexpr (REST) {
      const int mode = tile_mode(L, kconst, x0, x0 + TX, y0, y0 + ty);
      if (mode == GENERAL)
        for (int j = threadIdx.x; j < 3 * (ty + XH); j += kTileThreads) {
          const int y = by + j / 3;
          sr[j] = (unsigned)y < (unsigned)N ? L.coef[(3 + j % 3) * N + y] : czero<double2>();
        }
      __syncthreads();
      const double2 *f = in.f + (size_t)b * L.S;
      const double2 csc = cscale(cs, 1.0 / 16.0);
      auto go = [&](auto m) {
        constexpr int MODE = decltype(m)::value;
        const TileCtx<double, MODE> t{L, bx, by, sr};
        ColumnOp<double, MODE> op(L, sigma, s);
        restrict_body<double, MODE, TX>(t, op, f, A, B, O, ty, x0, y0, fc, csc, lc);
      };
      if (mode == UNIFORM_K) go(std::integral_constant<int, UNIFORM_K>());
      else if (mode == UNIFORM) go(std::integral_constant<int, UNIFORM>());
      else go(std::integral_constant<int, GENERAL>());
    }
  }
}

// Tiles of 8 x 8 points on small levels: the FP64 pipe binds these too, and small
// tiles spread over more SMs.
constexpr int kSmallTile = 8;
bool use_tiles(int N, int batch) {
  const int nt = (N + kSmallTile - 1) / kSmallTile;
  return nt * nt * batch <= 256;
}
constexpr int kMaxRows = 32;   // rows of a large tile

// (min, max) over the rows a block takes, into part[2 blockIdx.x ..].
__global__ void __launch_bounds__(256) k_k2_range(const double *k2, int N, int P, size_t rows, double *part) {
  __shared__ double lo[8], hi[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double a = k2[0], c = k2[0];
  for (size_t r = (size_t)blockIdx.x * 8 + warp; r < rows; r += (size_t)gridDim.x * 8)
    for (int x = lane; x < N; x += 32) {
      const double v = k2[r * P + x];
      a = fmin(a, v);
      c = fmax(c, v);
    }
  for (int o = 16; o > 0; o >>= 1) {
    a = fmin(a, __shfl_xor_sync(0xffffffffu, a, o));
    c = fmax(c, __shfl_xor_sync(0xffffffffu, c, o));
  }
  if (lane == 0) {
    lo[warp] = a;
    hi[warp] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) {
      lo[0] = fmin(lo[0], lo[i]);
      hi[0] = fmax(hi[0], hi[i]);
    }
    part[2 * blockIdx.x] = lo[0];
    part[2 * blockIdx.x + 1] = hi[0];
  }
}

}  // namespace

// Partial Gram matrices per right-hand side at most: about two blocks per SM
// over the batch (every block of the update kernel adds them all).
int gm2d_max_parts(int batch, int sms) { return std::max(256, 2 * sms / std::max(1, batch)); }

// Blocks of eight rows, and one over their results: min(all) and max(all) of the pairs.
// (One block for the whole field took 10 ms at 4095^2.)
void launch_k2_range(const double *k2, int N, int P, size_t rows, double *out, cudaStream_t s) {
  const int blocks = (int)std::min<size_t>(kK2RangeBlocks, (rows + 7) / 8);
  k_k2_range<<<blocks, 256, 0, s>>>(k2, N, P, rows, out + 2);
  k_k2_range<<<1, 256, 0, s>>>(out + 2, 2 * blocks, 2 * blocks, 1, out);
}

// Rows of a tile: as many as leave about two tiles per SM over the batch (tall
// tiles waste fewer halo rows), at most what shared memory holds.
template <> Gm2dPlan gm2d_plan<double>(int N, int m, int batch, int sms, bool) {
  const int nx = (N + kTX - 1) / kTX;
  const int ny = std::max(1, 2 * sms / (nx * batch));   // tile rows wanted
  Gm2dPlan p{};
  p.tile = use_tiles(N, batch);
  p.rows = p.urows = std::min(kMaxRows, std::max(4, even_up((N + ny - 1) / ny)));
  const int tiles = nx * ((N + p.rows - 1) / p.rows);
  p.blocks = std::min(tiles, gm2d_max_parts(batch, sms));
  p.ublocks = std::min(tiles, std::max(1, 2 * sms / batch));
  if (p.tile) {
    const int nt = (N + kSmallTile - 1) / kSmallTile;
    p.blocks = nt * nt;
  }
  (void)m;
  return p;
}

template <> cudaError_t init_gm2d<double>() {
  cudaError_t e = cudaSuccess;
  for (int m = 1; m <= 3; ++m)
    with_m(m, [&](auto mm) {
      constexpr int M = decltype(mm)::value;
      auto set = [&](auto k) {
        if (e == cudaSuccess)
          e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tile_smem(M, kMaxRows));
      };
      set(k_gm2d_basis<M, true>);
      set(k_gm2d_basis<M, false>);
      set(k_gm2d_update<M, true, false>);
      set(k_gm2d_update<M, false, true>);
      set(k_gm2d_update<M, false, false>);
    });
  return e;
}

template <>
void launch_gm2d_basis<double>(const LevelK<double> &L, double2 sigma, double s, int kconst, int m,
                               const Gm2dIn<double> &in, const Gm2dWork<double> &w, const Gm2dPlan &p,
                               int batch, const SolveState *st, double *check, cudaStream_t stream) {
  with_m(m, [&](auto mm) {
    constexpr int M = decltype(mm)::value;
    if (p.tile) {
      basis_tile_launch<double, M, kSmallTile>(L, sigma, s, in, w, batch, st, check, stream);
      return;
    }
    auto go = [&](auto k) {
      launch_pdl(k, dim3(p.blocks, batch), dim3(kTileThreads), tile_smem(M, p.rows), stream, L, sigma, s,
                 kconst, in, w, p.rows, st, check);
    };
    if (in.e) go(k_gm2d_basis<M, true>);
    else go(k_gm2d_basis<M, false>);
  });
}

int launch_gm_coef(const LevelK<double> &L, int rows, double2 sigma, double s, int m,
                   const Gm2dWork<double> &w, int nparts, int batch, const SolveState *st,
                   cudaStream_t stream) {
  // Small levels: a point per thread.  Large ones: 32 warps per SM (with 8 of them 1023^2
  // took 320 us), blocks on every SM for two right-hand sides or more (the others of a
  // batch may have stopped; every block adds and solves before its points)
  const long long pts = (long long)rows * L.N;
  const int threads = pts < 65536 ? 256 : 1024;
  const int nb = (int)std::min<long long>((pts + threads - 1) / threads, batch == 1 || threads == 256 ? kGm2dCorr : kGm2dCorr / 2);
  const double tol = gram_tol<double>(false);
  with_m(m, [&](auto mm) {
    launch_pdl(k_gm2d_coef<decltype(mm)::value>, dim3(nb, batch), dim3(threads), 0, stream, L, rows, sigma, s,
               w, nparts, tol, st);
  });
  return nb;
}

template <>
void launch_gm2d_update<double>(const LevelK<double> &L, double2 sigma, double s, int kconst, int m,
                                const Gm2dIn<double> &in, const Gm2dWork<double> &w, const Gm2dPlan &p,
                                double2 *u_out, double2 *fc, double2 cs, const Lay &lc, int batch,
                                const SolveState *st, cudaStream_t stream) {
  const double tol = gram_tol<double>(false);
  with_m(m, [&](auto mm) {
    constexpr int M = decltype(mm)::value;
    const int nb = launch_gm_coef(L, L.N, sigma, s, M, w, p.blocks, batch, st, stream);
    // (a corrected iterate is never restricted: it belongs to the way up)
    auto go = [&](auto corr, auto rest) {
      constexpr bool CORR = decltype(corr)::value, REST = decltype(rest)::value;
      if (p.tile)
        update_tile_launch<double, M, kSmallTile, CORR, REST>(L, sigma, s, in, w, nb, tol, u_out,
                                                              fc, cs, lc, batch, st, stream);
      else
        launch_pdl(k_gm2d_update<M, CORR, REST>, dim3(p.ublocks, batch), dim3(kTileThreads),
                   tile_smem(M, p.urows), stream, L, sigma, s, kconst, in, w, nb, p.urows,
                   u_out, fc, cs, lc, st);
    };
    if (in.e) go(std::true_type(), std::false_type());
    else if (fc) go(std::false_type(), std::true_type());
    else go(std::false_type(), std::false_type());
  });
}

}  // namespace hh
