// complex64 kernels of the 2-D GMRES steps (hh_gmres2d.cuh).  Nothing is kept
// between a step's two kernels: the update forms the basis again from u and f
// (16 B read per point instead of 24 B written and read).
//
// Large levels march: a warp owns a strip of 32 adjacent columns, one per lane,
// and walks down a run of rows.  q_0 of row y, X q_0 of row y-1, X q_1 of row y-2
// and X q_2 of row y-3 are formed in the same iteration, so that every vector
// lives in a register window of four rows; west and east neighbours come by
// shuffles.  The strip's outer lanes are halo (one more on each side per product),
// as are the rows above and below a run: no shared memory, no block barrier and
// no vector in memory.
//
// Small levels (at most 255 points per axis and few right-hand sides): a block
// per tile, a thread per point (hh_gmres2d.cuh), because there one warp's chain
// of march iterations is the time.
//
// Measured (GB300, one right-hand side, constant k with layers; in brackets a kernel and a
// reduction per Arnoldi step): a GMRES(3) step takes 32.1 us at 1023^2 (67.2), 18.6 at 511^2
// (41.6), 10.9 at 255^2 (36.4), 6.8 at 127^2 (30.3) and 6.3 at 63^2 (29.5; 20.6 with
// marches); the 1023^2 cycle 207 us (539).  At 1023^2 the basis kernel uses 45 % and the
// update 41 % of the issue slots with 12 and 15 warps per SM: chains of dependent rows; at
// 2047^2 59 and 46 %.  Two columns per lane, or the tiles of hh_gmres2d_64.cu, were slower
// (44 and 54 us a step).
#include "hh_gmres2d.cuh"

namespace hh {

namespace {

template <typename C> __device__ __forceinline__ C shfl_left(C v) {    // the lane to the west
  C r;
  r.x = __shfl_up_sync(0xffffffffu, v.x, 1);
  r.y = __shfl_up_sync(0xffffffffu, v.y, 1);
  return r;
}
template <typename C> __device__ __forceinline__ C shfl_right(C v) {
  C r;
  r.x = __shfl_down_sync(0xffffffffu, v.x, 1);
  r.y = __shfl_down_sync(0xffffffffu, v.y, 1);
  return r;
}

// Strip of a march with NX products: the first lane whose X q_{NX-1} (with REST:
// whose new residual's weighting) is complete, and the columns owned (with REST
// an even number, which keeps the coarse columns on fixed lanes).
template <int NX, bool REST = false> struct Strip {
  static constexpr int F = REST ? NX + 2 : NX + 1;
  static constexpr int OW = REST ? (31 - 2 * F) / 2 * 2 : 32 - 2 * F;
};

// The march of one warp.  NX products X q_j are formed (q_1 = X q_0,
// q_{j+1} = 2 X q_j - q_{j-1}); M vectors q_j are kept.  Rows [y0, y1) are emitted
// (y0 even where CORR).  hook<j>(slot, q_j) is called when q_j of a row is formed,
// row y - j, whose window slot is given; emit(slot, row, X q_{NX-1}) when row `row`
// is done.  w0(slot, w) receives the iterate with q_0.  FROWS keeps the
// right-hand side of the window's rows.
template <typename R, int M, int NX, int MODE, bool CORR, bool FROWS = false> struct March {
  using C = typename Cx<R>::T;
  struct Raw { C u, el, er; };
  const LevelK<R> &L;
  const Gm2dIn<R> &in;
  C sigma;
  R s, g;                  // g: factor of q_0
  int x, wmax, fmax;
  bool zero, inx;          // inx: the lane's column is inside the domain
  const C *u, *f, *e;
  const R *kp;
  const C *cy;             // row tables lo, dg, up
  int N, P;
  C lox, upx, dxs, dxu;    // GENERAL: the columns' coefficients (dxu = dg_x, dxs = dg_x - sigma)
  C c0, D0, sb;
  R cf;
  bool el_in, er_in;
  C w[4], q0[4], q1[4], q2[4];
  C fr[4];
  R k[4];
  Raw pw[2];
  C pf[2];
  R pk[2];
  C exB;

  __device__ __forceinline__ March(const LevelK<R> &L_, const Gm2dIn<R> &in_, C sigma_, R s_,
                                   R g_, int b, bool zero_, int x_)
      : L(L_), in(in_), sigma(sigma_), s(s_), g(g_), x(x_), zero(zero_) {
    N = L.N;
    P = L.P;
    inx = MODE != GENERAL || (unsigned)x < (unsigned)N;
    u = in.u + (size_t)b * L.S + x;
    f = in.f + (size_t)b * L.S + x;
    kp = L.k2 + x;
    cy = L.coef + 3 * N;
    if (CORR) {
      e = in.e + (size_t)b * in.lc.S;
      // coarse columns around x: x/2 - 1 and x/2, or (x - 1)/2 for an odd x
      el_in = inx && x >= 2 && !(x & 1);
      er_in = inx && (x >> 1) < in.lc.N;
    }
    const C zc = czero<C>();
    if (MODE == GENERAL) {
      lox = inx ? L.coef[x] : zc;
      upx = inx ? L.coef[2 * N + x] : zc;
      dxu = inx ? L.coef[N + x] : zc;
      dxs = csub(dxu, sigma);
    } else {
      c0 = L.c0;
      D0 = cscale(c0, R(4));
      cf = s * c0.x;
      sb = cscale(L.beta, s);
    }
  }

  __device__ __forceinline__ C fetch(const C *p, int yy) const { return p[(size_t)(unsigned)yy * P]; }
  __device__ __forceinline__ bool row_in(int yy, int last) const {
    return MODE != GENERAL ? yy <= last : (inx && yy <= last && (unsigned)yy < (unsigned)N);
  }
  __device__ __forceinline__ C coarse(int cyr, bool ok, int cx) const {
    return ok && cyr >= 0 && cyr < in.lc.N ? e[(size_t)cyr * in.lc.P + cx] : czero<C>();
  }
  __device__ __forceinline__ Raw load_w(int yy, bool even) const {
    Raw r;
    r.u = czero<C>();
    if (CORR) r.el = r.er = czero<C>();
    if (!zero && row_in(yy, wmax)) r.u = fetch(u, yy);
    if (CORR && even && yy <= wmax) {   // a new coarse row yy / 2
      r.el = coarse(yy >> 1, el_in, (x >> 1) - 1);
      r.er = coarse(yy >> 1, er_in, x >> 1);
    }
    return r;
  }
  // the coarse row interpolated to the lane's column
  __device__ __forceinline__ C spread(C el, C er) const {
    return (x & 1) ? er : cscale(cadd(el, er), R(0.5));
  }
  __device__ __forceinline__ C fin_w(const Raw &r, int, bool even) {
    if (!CORR) return r.u;
    C pe = exB;
    if (even) {
      const C nx = spread(r.el, r.er);
      pe = cscale(cadd(exB, nx), R(0.5));
      exB = nx;
    }
    return cadd(r.u, pe);   // (the coarse values outside the domain are zero)
  }
  __device__ __forceinline__ C load_f(int yy) const {
    return row_in(yy, fmax) ? fetch(f, yy) : czero<C>();
  }
  __device__ __forceinline__ R load_k(int yy) const {
    return MODE != UNIFORM_K && row_in(yy, fmax) ? kp[(size_t)(unsigned)yy * L.KP] : R(0);
  }
  // Row coefficients of the general body: zero outside the domain.  With the
  // columns' lox = upx = 0 there and every vector zero outside the domain, X and
  // resid are zero outside it without a test.
  struct RowCoef { C lo, dg, up; };
  __device__ __forceinline__ RowCoef row_coef(int yy) const {
    RowCoef r;
    r.lo = r.dg = r.up = czero<C>();
    if (MODE == GENERAL && (unsigned)yy < (unsigned)N) {
      r.lo = cy[yy];
      r.dg = cy[N + yy];
      r.up = cy[2 * N + yy];
    }
    return r;
  }
  __device__ __forceinline__ C neighbours(const RowCoef &rc, C vw, C ve, C vn, C vs) const {
    C nb = cmul(lox, vw);
    nb = cfma(upx, ve, nb);
    nb = cfma(rc.lo, vn, nb);
    return cfma(rc.up, vs, nb);
  }
  // X v at row yy (v, its rows above and below, k^2 of the point)
  __device__ __forceinline__ C X(C vn, C v, C vs, int yy, R kv) const {
    const C vw = shfl_left(v), ve = shfl_right(v);
    if (MODE == GENERAL) {
      const RowCoef rc = row_coef(yy);
      const C d = csub(cadd(dxs, rc.dg), cscale(L.beta, kv));
      return cscale(csub(cmul(d, v), neighbours(rc, vw, ve, vn, vs)), s);
    }
    const C sn = cadd(cadd(vw, ve), cadd(vn, vs));
    C r = cmk(-cf * sn.x, -cf * sn.y);
    if (MODE == UNIFORM) {   // s (4 c_0 - beta k^2 - sigma) v
      C d;
      d.x = fmaf_any(-sb.x, kv, s * (D0.x - sigma.x));
      d.y = fmaf_any(-sb.y, kv, -s * sigma.y);
      r = cfma(d, v, r);
    }
    return r;
  }
  // f - A w at row yy
  __device__ __forceinline__ C resid(C fv, C vn, C v, C vs, int yy, R kv) const {
    const C vw = shfl_left(v), ve = shfl_right(v);
    if (MODE == GENERAL) {
      const RowCoef rc = row_coef(yy);
      const C d = csub(cadd(dxu, rc.dg), cscale(L.beta, kv));
      return cadd(csub(fv, cmul(d, v)), neighbours(rc, vw, ve, vn, vs));
    }
    const C sn = cadd(cadd(vw, ve), cadd(vn, vs));
    const R kk = MODE == UNIFORM_K ? L.kc : kv;
    C d, r;
    d.x = fmaf_any(-L.beta.x, kk, D0.x);
    d.y = -L.beta.y * kk;
    r.x = fmaf_any(c0.x, sn.x, fmaf_any(-d.x, v.x, fmaf_any(d.y, v.y, fv.x)));
    r.y = fmaf_any(c0.x, sn.y, fmaf_any(-d.x, v.y, fmaf_any(-d.y, v.x, fv.y)));
    return r;
  }

  template <int S, typename W0, typename H, typename E>
  __device__ __forceinline__ void step(int y, W0 &w0, H &hook, E &emit) {
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    constexpr int S1 = (S + 1) & 3, S2 = (S + 2) & 3, S3 = (S + 3) & 3, O = S & 1;
    // with CORR the run's first row y0 is even: y = y0 - NX + t has a static parity
    constexpr bool even1 = ((NX + S + 1) & 1) == 0;
    w[S1] = fin_w(pw[O ^ 1], y + 1, even1);
    pw[O ^ 1] = load_w(y + 3, even1);
    const C fv = pf[O];
    pf[O] = load_f(y + 2);
    if (MODE != UNIFORM_K) {
      k[S] = pk[O];
      pk[O] = load_k(y + 2);
    }
    if (FROWS) fr[S] = fv;
    q0[S] = cscale(zero ? fv : resid(fv, w[S3], w[S], w[S1], y, k[S]), g);
    w0(S, w[S]);
    hook(I0(), S, q0[S]);
    C xl = czero<C>();
    if (NX >= 1) {
      xl = X(q0[S2], q0[S3], q0[S], y - 1, k[S3]);
      if (M >= 2) {
        q1[S3] = xl;
        hook(I1(), S3, q1[S3]);
      }
    }
    if (NX >= 2) {
      xl = X(q1[S1], q1[S2], q1[S3], y - 2, k[S2]);
      if (M >= 3) {
        q2[S2] = csub(cadd(xl, xl), q0[S2]);
        hook(I2(), S2, q2[S2]);
      }
    }
    if (NX >= 3) xl = X(q2[S], q2[S1], q2[S2], y - 3, k[S1]);
    emit((S + 4 - NX) & 3, y - NX, xl);
  }

  // rows [y0, y1); rows outside the domain are zero
  // (fold: called every four rows)
  template <typename W0, typename H, typename E, typename D>
  __device__ __forceinline__ void run(int y0, int y1, W0 w0, H hook, E emit, D fold) {
    const int ys = y0 - NX, T = y1 - y0 + 2 * NX;
    wmax = y1 + NX;
    fmax = y1 - 1 + NX;
    const C zv = czero<C>();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      w[i] = q0[i] = q1[i] = q2[i] = zv;
      if (FROWS) fr[i] = zv;
      k[i] = R(0);
    }
    // row r of the iterate has the parity of NX + (r - ys)
    constexpr bool ev_m1 = ((NX + 1) & 1) == 0, ev_0 = (NX & 1) == 0;
    if (CORR) {
      const int c = (ys - 2) >> 1;   // the coarse row at or above row ys - 1
      exB = spread(coarse(c, el_in, (x >> 1) - 1), coarse(c, er_in, x >> 1));
    }
    const Raw a = load_w(ys - 1, ev_m1), b0 = load_w(ys, ev_0);
    pw[1] = load_w(ys + 1, ev_m1);
    pw[0] = load_w(ys + 2, ev_0);
    pf[0] = load_f(ys);
    pf[1] = load_f(ys + 1);
    pk[0] = load_k(ys);
    pk[1] = load_k(ys + 1);
    w[3] = fin_w(a, ys - 1, ev_m1);
    w[0] = fin_w(b0, ys, ev_0);
#pragma unroll 1
    for (int t = 0; t < T; t += 4) {
      step<0>(ys + t, w0, hook, emit);
      if (t + 1 < T) step<1>(ys + t + 1, w0, hook, emit);
      if (t + 2 < T) step<2>(ys + t + 2, w0, hook, emit);
      if (t + 3 < T) step<3>(ys + t + 3, w0, hook, emit);
      fold();
    }
  }
};

// Work of a march kernel: strips x runs of `rows` rows.  Strips and runs that
// touch the region of non-uniform coefficients (the layers, the domain's edge)
// take the general body, about twice the instructions; so that they do not
// set the kernel's time, such a run is halved between two warps: the first
// strips * runs items are runs (general ones: their first half), the items after
// them the second halves of the general ones.
struct MarchWork {
  int strips, runs, rows, F, OW;
  int su0, su1, ru0, ru1;   // strips and runs of the uniform body: [su0, su1), [ru0, ru1)
  int nsec;                 // second halves
  template <typename R>
  __device__ __forceinline__ MarchWork(const LevelK<R> &L, int rows_, int F_, int OW_, int hy)
      : rows(rows_), F(F_), OW(OW_) {
    strips = (L.N + OW - 1) / OW;
    runs = (L.N + rows - 1) / rows;
    su0 = ru0 = su1 = ru1 = 0;
    // (the uniform body reads the rows next to the run's unchecked: inside the domain)
    const int ulo = max(L.ulo, 1), uhi = min(L.uhi, L.N - 2);
    if (L.c0.y == R(0) && ulo <= uhi) {
      su0 = (ulo + F + OW - 1) / OW;                    // strip OW - F >= ulo
      su1 = uhi + F - 31 < 0 ? 0 : (uhi + F - 31) / OW + 1;   // strip OW - F + 31 <= uhi
      ru0 = (ulo + hy + rows - 1) / rows;               // run rows - hy >= ulo
      ru1 = (uhi - hy + 1) / rows;                      // (run + 1) rows - 1 + hy <= uhi
      su1 = max(su0, min(su1, strips));
      ru1 = max(ru0, min(ru1, runs));
    }
    nsec = strips * runs - (su1 - su0) * (ru1 - ru0);
  }
  __device__ __forceinline__ int items() const { return strips * runs + nsec; }
  // strip, rows [y0, y1) and body of item i
  __device__ __forceinline__ bool item(int i, int N, int &strip, int &y0, int &y1) const {
    int run;
    const bool second = i >= strips * runs;
    if (!second) {
      run = i / strips;
      strip = i - run * strips;
    } else {
      i -= strips * runs;
      const int nr = runs - (ru1 - ru0), ns = strips - (su1 - su0);
      if (i < nr * strips) {            // runs outside [ru0, ru1)
        run = i / strips;
        strip = i - run * strips;
        if (run >= ru0) run += ru1 - ru0;
      } else {                          // strips outside [su0, su1) of the others
        i -= nr * strips;
        run = i / ns;
        strip = i - run * ns;
        run += ru0;
        if (strip >= su0) strip += su1 - su0;
      }
    }
    const bool uni = strip >= su0 && strip < su1 && run >= ru0 && run < ru1;
    y0 = run * rows;
    y1 = min(N, y0 + rows);
    if (!uni) {
      const int mid = min(y1, y0 + ((rows / 2 + 1) & ~1));   // even: see March
      if (second) y0 = mid;
      else y1 = mid;
    }
    return uni;
  }
};

constexpr int kMaxWarps = 16;   // per block: 128 registers per thread
// Plain sums, folded every four rows, need more.  Twelve warps with 168 registers where
// these hold all items at once (four right-hand sides at 511^2 38 us a step, 46 unfolded with
// 128 registers; one at 1023^2 32.2 and 31.9), else 16 that spill a little (four at 1023^2 120
// us and 126 with twelve, 113 unfolded).
constexpr int kPlainWarps = 12;
// Larger levels have so many runs that a warp's sums of whole ones are near enough (4.0e-10
// at 2047^2, 5.2e-10 with FP32 warp sums added in FP64): added up as pairs after each item,
// 2047^2 112 us a step, 4095^2 441 (folded every four rows 119 and 458, not at all 110 and 436).
constexpr int kFoldRowsMaxN = 1024;
enum { PAIRED, FOLD_ROWS, FOLD_ITEM };

template <typename R, int M, bool PAIR, int SUMS, int MODE, bool CORR>
__device__ __forceinline__ void basis_run(const LevelK<R> &L, const Gm2dIn<R> &in,
                                          typename Cx<R>::T sigma, R s, R g, int b, bool zero, int x,
                                          int y0, int y1, bool own,
                                          GramAcc<R, PAIR> (&acc)[Gram<M>::NQP]) {
  using C = typename Cx<R>::T;
  March<R, M, M, MODE, CORR> m(L, in, sigma, s, g, b, zero, x);
  const C t = cscale(sigma, s);
  auto none0 = [](int, C) {};
  auto none = [](auto, int, C) {};
  auto emit = [&](int sl, int row, C xl) {
    if (row < y0 || !own) return;
    C v[M + 1];   // (zero outside the domain)
    v[0] = m.q0[sl];
    if (M == 1) v[1] = cfma(t, v[0], xl);
    if (M >= 2) v[1] = cfma(t, v[0], m.q1[sl]);
    if (M == 2) v[2] = cfma(t, m.q1[sl], xl);
    if (M == 3) {
      v[M - 1] = cfma(t, m.q1[sl], cscale(cadd(m.q2[sl], v[0]), R(0.5)));
      v[M] = cfma(t, m.q2[sl], xl);
    }
    gram_point<R, M, PAIR>(acc, v);
  };
  m.run(y0, y1, none0, none, emit, [&] {
    if (SUMS != FOLD_ROWS) return;
#pragma unroll
    for (int i = 0; i < Gram<M>::NQ; ++i) acc[i].fold();
  });
}

template <typename R, int M, bool PAIR, bool CORR, int WARPS, int SUMS>
__global__ void __launch_bounds__(32 * WARPS)
k_gm2d_basis(LevelK<R> L, typename Cx<R>::T sigma, R s, int kconst, Gm2dIn<R> in, Gm2dWork<R> wk,
             int rows, const SolveState *st, double *check) {
  constexpr int NQP = Gram<M>::NQP;
  using G = Strip<M>;
  using S = typename GramSum<R>::T;
  __shared__ S sums[WARPS * NQP];
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const MarchWork work(L, rows, G::F, G::OW, M);
  griddep_wait();
  griddep_launch_dependents();
  const R g = gram_scale_of<R>(wk.mag, b);   // (in flight early)
  if (!__syncthreads_and(!(st && !st[b].active))) return;   // one decision per block
  const bool zero = __syncthreads_or(in.zero_mode == ZERO_ALL ||
                                     (in.zero_mode == ZERO_FLAG && st && st[b].zero)) != 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    wk.zflag[b] = zero;
    wk.g[b] = g;
  }
  constexpr int SH = NQP == 16 ? 1 : 3;   // lane l holds quantity l >> SH of a warp's sums
  const bool holds = (lane & ((1 << SH) - 1)) == 0;
  S *mine = sums + warp * NQP + (lane >> SH);
  GramAcc<R, PAIR> acc[NQP];
  auto clear = [&] {
#pragma unroll
    for (int i = 0; i < NQP; ++i) acc[i].zero();
  };
  clear();
  if (SUMS == FOLD_ITEM && holds) *mine = make_float2(0.f, 0.f);
  const bool own = lane >= G::F && lane < G::F + G::OW;
  for (int wi = blockIdx.x * nw + warp; wi < work.items(); wi += gridDim.x * nw) {
    int strip, y0, y1;
    const bool uni = work.item(wi, L.N, strip, y0, y1);
    const int x = strip * G::OW - G::F + lane;
    if (y0 >= y1) continue;
    if (!uni) basis_run<R, M, PAIR, SUMS, GENERAL, CORR>(L, in, sigma, s, g, b, zero, x, y0, y1, own, acc);
    else if (kconst) basis_run<R, M, PAIR, SUMS, UNIFORM_K, CORR>(L, in, sigma, s, g, b, zero, x, y0, y1, own, acc);
    else basis_run<R, M, PAIR, SUMS, UNIFORM, CORR>(L, in, sigma, s, g, b, zero, x, y0, y1, own, acc);
    if (SUMS == FOLD_ITEM) {
      GramAcc<R, PAIR> v = gram_warp_sum<GramAcc<R, PAIR>, NQP>(acc);
      if (holds) {
        gram_add(v, *mine);
        *mine = gram_store(v);
      }
      clear();
    }
  }
  // block sums, in a fixed order
  if (SUMS != FOLD_ITEM) {
    if (SUMS == FOLD_ROWS) {
#pragma unroll
      for (int i = 0; i < NQP; ++i) acc[i].close();
    }
    const GramAcc<R, PAIR> v = gram_warp_sum<GramAcc<R, PAIR>, NQP>(acc);
    if (holds) *mine = gram_store(v);
  }
  __syncthreads();
  if (threadIdx.x < NQP) {
    GramAcc<R, PAIR> t;
    t.zero();
    for (int i = 0; i < nw; ++i) gram_add(t, sums[i * NQP + threadIdx.x]);
    const S q = gram_store(t);
    wk.parts[((size_t)b * gridDim.x + blockIdx.x) * NQP + threadIdx.x] = q;
    if (check && threadIdx.x == 0) check[(size_t)b * gridDim.x + blockIdx.x] = gram_unscaled(q, g);
  }
}

// Full weighting of consecutive rows from y0 (even) that a warp holds one after
// the other, a column per lane; acc collects 1-2-1 over three rows.
template <typename R> struct WeightRows {
  using C = typename Cx<R>::T;
  C acc;
  __device__ __forceinline__ void row(C r, int row, int y0, bool write, int x, C csc, C *fc, int Pc) {
    const C a = shfl_left(r), c = shfl_right(r);
    C h;
    h.x = fmaf_any(R(2), r.x, a.x + c.x);
    h.y = fmaf_any(R(2), r.y, a.y + c.y);
    if (row & 1) {
      acc.x = fmaf_any(R(2), h.x, acc.x);
      acc.y = fmaf_any(R(2), h.y, acc.y);
    } else {
      if (row > y0 && write) fc[(size_t)(row / 2 - 1) * Pc + (x - 1) / 2] = cmul(csc, cadd(acc, h));
      acc = h;
    }
  }
};

// complex64: the basis again from u and f.  REST: f - A u of the new iterate one
// row behind it, and its full weighting.
template <typename R, int M, int MODE, bool CORR, bool REST>
__device__ __forceinline__ void update_run(const LevelK<R> &L, const Gm2dIn<R> &in,
                                           typename Cx<R>::T sigma, R s, const StepCoef<R> &sc,
                                           int b, bool zero, int x, int y0, int y1, bool own,
                                           typename Cx<R>::T *u_out, typename Cx<R>::T *fc,
                                           typename Cx<R>::T csc, const Lay &lc) {
  using C = typename Cx<R>::T;
  constexpr int NX = M - 1;
  March<R, M, NX, MODE, CORR, REST> m(L, in, sigma, s, R(1), b, zero, x);
  const int N = L.N;
  const bool cown = REST && own && (x & 1) && (x - 1) / 2 < lc.N;
  C o[4], un[4];
  WeightRows<R> fw;
  fw.acc = czero<C>();
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = un[i] = czero<C>();
  C *up = u_out + x;
  auto w0 = [&](int sl, C w) { o[sl] = w; };
  auto hook = [&](auto J, int sl, C q) {
    constexpr int j = decltype(J)::value;
    if (j < M) o[sl] = cfma(sc.z[j < M ? j : 0], q, o[sl]);
  };
  auto emit = [&](int sl, int row, C) {
    if (row < (REST ? y0 - 1 : y0)) return;
    if (own && m.inx && row >= y0 && row < y1) up[(size_t)(unsigned)row * L.P] = o[sl];
    if (REST) {
      un[sl] = o[sl];
      if (row > y0) {   // the residual of row - 1
        const int p = (sl + 3) & 3;
        C r = m.resid(m.fr[p], un[(sl + 2) & 3], un[p], un[sl], row - 1, m.k[p]);
        fw.row(r, row - 1, y0, cown, x, csc, fc, lc.P);
      }
    }
  };
  auto nofold = [] {};
  if (REST) m.run(y0 - 1, y1 + 2, w0, hook, emit, nofold);
  else m.run(y0, y1, w0, hook, emit, nofold);
}

template <typename R, int M, bool CORR, bool REST>
__global__ void __launch_bounds__(32 * kMaxWarps)
k_gm2d_update(LevelK<R> L, typename Cx<R>::T sigma, R s, int kconst, Gm2dIn<R> in, Gm2dWork<R> wk,
              int nparts, double tol, int rows, typename Cx<R>::T *u_out, typename Cx<R>::T *fc,
              typename Cx<R>::T cs, Lay lc, const SolveState *st) {
  using C = typename Cx<R>::T;
  constexpr int NQP = Gram<M>::NQP, NX = M - 1;
  using G = Strip<NX, REST>;
  __shared__ typename GramSum<R>::T sums[kMaxWarps * NQP];
  __shared__ StepCoef<R> sc;
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const MarchWork work(L, rows, G::F, G::OW, NX + (REST ? 2 : 0));
  griddep_wait();
  griddep_launch_dependents();
  if (!__syncthreads_and(!(st && !st[b].active))) return;
  const bool zero = wk.zflag[b] != 0;
  step_coef<R, M>(wk.parts + (size_t)b * nparts * NQP, nparts, s, tol, sums, &sc);
  if (wk.track && blockIdx.x == 0 && threadIdx.x == 0) gram_estimate(wk.mag, b, sums[0], wk.g[b]);
  const C csc = cscale(cs, R(1.0 / 16.0));
  u_out += (size_t)b * L.S;
  if (REST) fc += (size_t)b * lc.S;
  const bool own = lane >= G::F && lane < G::F + G::OW;
  for (int wi = blockIdx.x * nw + warp; wi < work.items(); wi += gridDim.x * nw) {
    int strip, y0, y1;
    const bool uni = work.item(wi, L.N, strip, y0, y1);
    const int x = strip * G::OW - G::F + lane;
    if (y0 >= y1) continue;
    if (!uni) update_run<R, M, GENERAL, CORR, REST>(L, in, sigma, s, sc, b, zero, x, y0, y1, own, u_out, fc, csc, lc);
    else if (kconst) update_run<R, M, UNIFORM_K, CORR, REST>(L, in, sigma, s, sc, b, zero, x, y0, y1, own, u_out, fc, csc, lc);
    else update_run<R, M, UNIFORM, CORR, REST>(L, in, sigma, s, sc, b, zero, x, y0, y1, own, u_out, fc, csc, lc);
  }
}

// Tiles of 16 x 16 points (484 threads), the restricting update 14 x 14 (441).
constexpr int kBasisTile = 16;
template <bool REST> constexpr int update_tile() { return REST ? 14 : 16; }
bool use_tiles(int N, int batch) {
  const int nt = (N + kBasisTile - 1) / kBasisTile;
  return nt * nt <= 256 && nt * nt * batch <= 1024;
}

}  // namespace

// Rows per run: long runs waste fewer halo rows, short ones give more warps:
// about 12 warps per SM over the batch.  Blocks: about one per SM, so that few
// partial sums reach the update kernel.
template <> Gm2dPlan gm2d_plan<float>(int N, int m, int batch, int sms, bool restrict_) {
  auto split = [&](int width, int cap, int wmax, int *rows, int *warps, int *blocks) {
    const int strips = (N + width - 1) / width;
    const long long want = 12LL * sms;
    long long r = ((long long)N * strips * batch + want - 1) / want;
    r = std::min<long long>(std::max<long long>(r, 4), 32);
    int most;
    // (longer where the items would not fit one block of wmax warps per SM: with a second
    // wave of the 168-register blocks a 1023^2 step took 41 us)
    for (*rows = even_up((int)r);; *rows += 2) {
      const int total = strips * ((N + *rows - 1) / *rows);
      most = total + total / 4;   // general runs are halved (MarchWork)
      if (*rows >= 32 || (long long)most * batch <= (long long)wmax * sms) break;
    }
    const int per = (int)std::min<long long>(wmax, std::max<long long>(1, ((long long)most * batch + sms - 1) / sms));
    *warps = per;
    *blocks = (most + per - 1) / per;
    if (cap > 0) *blocks = std::min(*blocks, cap);
  };
  Gm2dPlan p;
  p.tile = use_tiles(N, batch);
  const int cap = gm2d_max_parts(batch, sms);
  split(30 - 2 * m, cap, N > kGramPairMaxN ? kPlainWarps : kMaxWarps, &p.rows, &p.warps, &p.blocks);
  if (N > kGramPairMaxN && p.blocks * batch > sms) split(30 - 2 * m, cap, kMaxWarps, &p.rows, &p.warps, &p.blocks);
  split(restrict_ ? 28 - 2 * m : 32 - 2 * m, 0, kMaxWarps, &p.urows, &p.uwarps, &p.ublocks);
  if (p.tile) {
    const int nt = (N + kBasisTile - 1) / kBasisTile;
    p.blocks = nt * nt;
  }
  return p;
}

template <>
void launch_gm2d_basis<float>(const LevelK<float> &L, float2 sigma, float s, int kconst, int m,
                              const Gm2dIn<float> &in, const Gm2dWork<float> &w, const Gm2dPlan &p,
                              int batch, const SolveState *st, double *check, cudaStream_t stream) {
  with_m(m, [&](auto mm) {
    constexpr int M = decltype(mm)::value;
    if (p.tile) {
      basis_tile_launch<float, M, kBasisTile>(L, sigma, s, in, w, batch, st, check, stream);
      return;
    }
    auto go = [&](auto k) {
      launch_pdl(k, dim3(p.blocks, batch), dim3(32 * p.warps), 0, stream, L, sigma, s, kconst, in, w,
                 p.rows, st, check);
    };
    auto corr = [&](auto c) {
      constexpr bool CORR = decltype(c)::value;
      if (L.N <= kGramPairMaxN) go(k_gm2d_basis<float, M, true, CORR, kMaxWarps, PAIRED>);
      else if (p.warps <= kPlainWarps) go(k_gm2d_basis<float, M, false, CORR, kPlainWarps, FOLD_ROWS>);
      else if (L.N <= kFoldRowsMaxN) go(k_gm2d_basis<float, M, false, CORR, kMaxWarps, FOLD_ROWS>);
      else go(k_gm2d_basis<float, M, false, CORR, kMaxWarps, FOLD_ITEM>);
    };
    if (in.e) corr(std::true_type());
    else corr(std::false_type());
  });
}

template <>
void launch_gm2d_update<float>(const LevelK<float> &L, float2 sigma, float s, int kconst, int m,
                               const Gm2dIn<float> &in, const Gm2dWork<float> &w, const Gm2dPlan &p,
                               float2 *u_out, float2 *fc, float2 cs, const Lay &lc, int batch,
                               const SolveState *st, cudaStream_t stream) {
  const double tol = gram_tol<float>(L.N <= kGramPairMaxN);
  with_m(m, [&](auto mm) {
    constexpr int M = decltype(mm)::value;
    // (a corrected iterate is never restricted: it belongs to the way up)
    auto go = [&](auto corr, auto rest) {
      constexpr bool CORR = decltype(corr)::value, REST = decltype(rest)::value;
      if (p.tile)
        update_tile_launch<float, M, update_tile<REST>(), CORR, REST>(L, sigma, s, in, w, p.blocks,
                                                                      tol, u_out, fc, cs, lc, batch, st, stream);
      else
        launch_pdl(k_gm2d_update<float, M, CORR, REST>, dim3(p.ublocks, batch), dim3(32 * p.uwarps), 0,
                   stream, L, sigma, s, kconst, in, w, p.blocks, tol, p.urows, u_out, fc, cs, lc, st);
    };
    if (in.e) go(std::true_type(), std::false_type());
    else if (fc) go(std::false_type(), std::true_type());
    else go(std::false_type(), std::false_type());
  });
}

}  // namespace hh
