// Jerk-controlled Dubins car with Gaussian obstacle bumps (Sec. V-A's second
// system, with the time state dropped).  x = [px, py, theta, v, a],
// u = [omega, jerk], explicit Euler:
//   px+ = px + dt v cos(theta),  py+ = py + dt v sin(theta),
//   theta+ = theta + dt omega,   v+ = v + dt a,   a+ = a + dt jerk.
// Running cost w_u |u|^2 + bumps(p); terminal w_pT |p|^2 + w_vT v^2 + w_aT a^2.
#pragma once
#include "common.cuh"

namespace to {

template <class R>
struct DubinsParams {
  R dt, wu, bamp, bsig, wpT, wvT, waT;
  int nb;
  R bc[8][2];
  R is2, inv, inv2;   // 1 / sigma^2, half of it, 1 / (2 sigma^2)
  // the quotients a rollout step would divide out again, rounded as there
  void derive() {
    is2 = R(1) / (bsig * bsig);
    inv = R(0.5) * is2;
    inv2 = R(1) / (R(2) * bsig * bsig);
  }
};

template <class D, class S>
inline void cast_params(const DubinsParams<S>& s, DubinsParams<D>& d) {
  d.dt = (D)s.dt; d.wu = (D)s.wu; d.bamp = (D)s.bamp; d.bsig = (D)s.bsig;
  d.wpT = (D)s.wpT; d.wvT = (D)s.wvT; d.waT = (D)s.waT;
  d.nb = s.nb;
  for (int b = 0; b < 8; ++b) { d.bc[b][0] = (D)s.bc[b][0]; d.bc[b][1] = (D)s.bc[b][1]; }
  d.derive();
}

struct SysDubins {
  static constexpr int n = 5, m = 2;
  static constexpr bool kActor = false;
  template <class R> using ParamsT = DubinsParams<R>;
  template <class R> struct Scratch { static constexpr int elems = 1; };
  template <int G> static constexpr bool kGroupStep = false;
  static constexpr bool kKnotParallel = false;
  static constexpr bool kStoredDerivs = false;


  template <class R>
  TO_DEV static R bumps(const ParamsT<R>& P, R px, R py) {
    R s = 0;
    each_bump(P.bc, P.nb, px, py, P.inv2, [&](R, R, R e) { s += P.bamp * e; });
    return s;
  }

  template <class R>
  TO_DEV static R running_cost(const ParamsT<R>& P, const R* x, const R* u) {
    return P.wu * (u[0] * u[0] + u[1] * u[1]) + bumps(P, x[0], x[1]);
  }

  // the same step on a state carried as (hi, lo) pairs, in place
  template <class R>
  TO_DEV static R cost_step2(const ParamsT<R>& P, R* xh, R* xl, const R* u) {
    const R l = running_cost(P, xh, u);
    step2(P, xh, xl, u);
    return l;
  }
  // the next state alone: the running cost (three exponentials) is off the
  // rollout's chain
  static constexpr bool kDeferCost = true;
  template <class R>
  TO_DEV static void step2(const ParamsT<R>& P, R* xh, R* xl, const R* u) {
    R s, c;
    sincos(xh[2], &s, &c);
    const R v = xh[3] + xl[3];
    const R dpx = P.dt * (v * c), dpy = P.dt * (v * s), dv = P.dt * xh[4] + P.dt * xl[4];
    acc2(xh[0], xl[0], dpx);
    acc2(xh[1], xl[1], dpy);
    acc2(xh[2], xl[2], P.dt * u[0]);
    acc2(xh[3], xl[3], dv);
    acc2(xh[4], xl[4], P.dt * u[1]);
  }

  template <class R>
  TO_DEV static R terminal_cost(const ParamsT<R>& P, const R* x) {
    return P.wpT * (x[0] * x[0] + x[1] * x[1]) + P.wvT * x[3] * x[3] + P.waT * x[4] * x[4];
  }

  // What a knot's derivatives hold besides constants, computed for every knot
  // before the backward pass, one knot per lane, and kept in the knot's gain
  // record (free until that knot's gains are written):
  //   [0..3] A(0, 2), A(0, 3), A(1, 2), A(1, 3)  [4..6] the clipped position
  //   block of l_xx (xx, xy, yy)  [7..8] l_x  [9..10] l_u  [11] padding
  // The bumps act on the position block only, so the clipped 5x5 state Hessian
  // is the clipped 2x2 position block with the clip of 0 on the other diagonal
  // entries.
  static constexpr bool kGainDerivs = true;
  static constexpr int kBlock = 11, kBlockPad = 12;
  template <class R>
  TO_DEV static void block(const ParamsT<R>& P, const R* x, const R* u, R eps, R* d) {
    R gx = 0, gy = 0, hxx = 0, hxy = 0, hyy = 0;
    const R is2 = P.is2;
    each_bump(P.bc, P.nb, x[0], x[1], P.inv, [&](R dx, R dy, R e) {
      const R es = P.bamp * e * is2;
      gx -= es * dx;
      gy -= es * dy;
      hxx += es * (dx * dx * is2 - R(1));
      hyy += es * (dy * dy * is2 - R(1));
      hxy += es * dx * dy * is2;
    });
    eigclip_2x2(hxx, hxy, hyy, eps);
    R s, c;
    sincos(x[2], &s, &c);
    const R w2 = R(2) * P.wu;
    d[0] = -P.dt * x[3] * s;
    d[1] = P.dt * c;
    d[2] = P.dt * x[3] * c;
    d[3] = P.dt * s;
    d[4] = hxx; d[5] = hxy; d[6] = hyy;
    d[7] = gx; d[8] = gy;
    d[9] = w2 * u[0]; d[10] = w2 * u[1];
    d[11] = R(0);
  }
  // Sparsity of A and B.  Column j of A has its nonzeros in rows a_row(j, q), q <
  // kA, in ascending order (filled up with rows whose entry is 0); column c of
  // B has one, in row b_row(c).
  static constexpr int kA = 3;
  static constexpr TO_HD int a_row(int j, int q) {
    return q == 0 ? 0 : q == 1 ? (j == 4 ? 3 : 1) : (j == 3 ? 3 : j == 4 ? 4 : 2);
  }
  static constexpr TO_HD bool a_nz(int r, int j) { return r == j || (r < 2 && (j == 2 || j == 3)) || (r == 3 && j == 4); }
  static constexpr TO_HD int b_row(int c) { return 2 + 2 * c; }
  // the constant entries: A, B, and l_xx, l_x, l_uu outside the block (lane
  // of a group of G)
  template <class R>
  TO_DEV static void block_consts(const ParamsT<R>& P, int lane, int G, R eps, R* A, R* B, R* lxx, R* lx, R* luu) {
    const R w2 = R(2) * P.wu;
    for (int e = lane; e < n * n; e += G) {
      const int i = e / n, j = e % n;
      A[e] = (i == j) ? R(1) : ((i == 3 && j == 4) ? P.dt : R(0));
      lxx[e] = (i == j && i >= 2) ? clip0(eps) : R(0);
    }
    for (int e = lane; e < n * m; e += G) B[e] = (e == 2 * m || e == 4 * m + 1) ? P.dt : R(0);
    for (int e = lane; e < n; e += G) lx[e] = R(0);
    for (int e = lane; e < m * m; e += G) luu[e] = (e / m == e % m) ? (w2 > eps ? w2 : eps) : R(0);
  }
  // where entry e of the block goes; the mirrored entry of a symmetric pair
  // (second), else the same place
  template <class R>
  TO_DEV static R* block_dst(int e, bool second, R* A, R* lxx, R* lx, R* lu) {
    return e < 4 ? A + (e >> 1) * n + 2 + (e & 1)
                 : e == 4 ? lxx : e == 5 ? lxx + (second ? n : 1) : e == 6 ? lxx + n + 1 : e < 9 ? lx + (e - 7) : lu + (e - 9);
  }

  // the whole derivatives on one lane (single-lane groups)
  template <class R>
  TO_DEV static void derivs_lane(const ParamsT<R>& P, const R* x, const R* u, R eps, R* A, R* B, R* lxx, R* lx,
                                 R* luu, R* lu) {
    R d[kBlockPad];
    block(P, x, u, eps, d);
#pragma unroll
    for (int i = 0; i < n; ++i)
#pragma unroll
      for (int j = 0; j < n; ++j) A[i * n + j] = (i == j) ? R(1) : R(0);
    A[0 * n + 2] = d[0];
    A[0 * n + 3] = d[1];
    A[1 * n + 2] = d[2];
    A[1 * n + 3] = d[3];
    A[3 * n + 4] = P.dt;
#pragma unroll
    for (int i = 0; i < n * m; ++i) B[i] = R(0);
    B[2 * m + 0] = P.dt;
    B[4 * m + 1] = P.dt;
#pragma unroll
    for (int i = 0; i < n * n; ++i) lxx[i] = 0;
    lxx[0] = d[4]; lxx[1] = d[5]; lxx[n] = d[5]; lxx[n + 1] = d[6];
    lxx[2 * n + 2] = clip0(eps); lxx[3 * n + 3] = clip0(eps); lxx[4 * n + 4] = clip0(eps);
    lx[0] = d[7]; lx[1] = d[8]; lx[2] = 0; lx[3] = 0; lx[4] = 0;
    const R w2 = R(2) * P.wu;
    const R q = w2 > eps ? w2 : eps;
    luu[0] = q; luu[1] = 0; luu[2] = 0; luu[3] = q;
    lu[0] = d[9]; lu[1] = d[10];
  }

  template <class R>
  TO_DEV static void terminal_derivs(const ParamsT<R>& P, const R* x, R eps, R* lxx, R* lx) {
    const R a = R(2) * P.wpT, b = R(2) * P.wvT, c = R(2) * P.waT;
#pragma unroll
    for (int i = 0; i < n * n; ++i) lxx[i] = 0;
    lxx[0] = a > eps ? a : eps; lxx[n + 1] = lxx[0];
    lxx[2 * n + 2] = clip0(eps);
    lxx[3 * n + 3] = b > eps ? b : eps;
    lxx[4 * n + 4] = c > eps ? c : eps;
    lx[0] = a * x[0]; lx[1] = a * x[1]; lx[2] = 0; lx[3] = b * x[3]; lx[4] = c * x[4];
  }
};

}  // namespace to
