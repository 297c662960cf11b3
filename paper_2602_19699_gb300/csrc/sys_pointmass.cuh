// Point-mass double integrator with Gaussian obstacle bumps (Sec. V-A systems;
// the synthetic workload's cost).  x = [px, py, vx, vy], u = [ax, ay],
// explicit Euler: p+ = p + dt v, v+ = v + dt u.
#pragma once
#include "common.cuh"

namespace to {

template <class R>
struct PointMassParams {
  R dt, wu, bamp, bsig, wpT, wvT;
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
inline void cast_params(const PointMassParams<S>& s, PointMassParams<D>& d) {
  d.dt = (D)s.dt; d.wu = (D)s.wu; d.bamp = (D)s.bamp; d.bsig = (D)s.bsig; d.wpT = (D)s.wpT; d.wvT = (D)s.wvT;
  d.nb = s.nb;
  for (int b = 0; b < 8; ++b) { d.bc[b][0] = (D)s.bc[b][0]; d.bc[b][1] = (D)s.bc[b][1]; }
  d.derive();
}

struct SysPointMass {
  static constexpr int n = 4, m = 2;
  static constexpr bool kActor = false;
  template <class R> using ParamsT = PointMassParams<R>;
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
    const R dpx = P.dt * xh[2] + P.dt * xl[2], dpy = P.dt * xh[3] + P.dt * xl[3];
    acc2(xh[0], xl[0], dpx);
    acc2(xh[1], xl[1], dpy);
    acc2(xh[2], xl[2], P.dt * u[0]);
    acc2(xh[3], xl[3], P.dt * u[1]);
  }

  template <class R>
  TO_DEV static R terminal_cost(const ParamsT<R>& P, const R* x) {
    return P.wpT * (x[0] * x[0] + x[1] * x[1]) + P.wvT * (x[2] * x[2] + x[3] * x[3]);
  }

  // What a knot's derivatives hold besides constants, computed for every knot
  // before the backward pass, one knot per lane, and kept in the knot's gain
  // record (free until that knot's gains are written):
  //   [0..2] the clipped position block of l_xx (xx, xy, yy)  [3..4] l_x
  //   [5..6] l_u  [7] padding
  // The bumps act on the position block only, so the clip of the full 4x4
  // state Hessian is the clip of the 2x2 position block with eps on the
  // velocity diagonal (the remaining eigenpairs are (0, e_i)).
  static constexpr bool kGainDerivs = true;
  static constexpr int kBlock = 7, kBlockPad = 8;
  template <class R>
  TO_DEV static void block(const ParamsT<R>& P, const R* x, const R* u, R eps, R* d) {
    R gx = 0, gy = 0, hxx = 0, hxy = 0, hyy = 0;
    const R is2 = P.is2;
    each_bump(P.bc, P.nb, x[0], x[1], P.inv, [&](R dx, R dy, R ex) {
      const R e = P.bamp * ex;
      // d/dp e = -e d / s2 ;  d2/dp2 e = e (d d^T / s2^2 - I / s2)
      const R es = e * is2;
      gx -= es * dx;
      gy -= es * dy;
      hxx += es * (dx * dx * is2 - R(1));
      hyy += es * (dy * dy * is2 - R(1));
      hxy += es * dx * dy * is2;
    });
    eigclip_2x2(hxx, hxy, hyy, eps);
    const R w2 = R(2) * P.wu;
    d[0] = hxx; d[1] = hxy; d[2] = hyy;
    d[3] = gx; d[4] = gy;
    d[5] = w2 * u[0]; d[6] = w2 * u[1];
    d[7] = R(0);
  }
  // Sparsity of A and B.  Column j of A has its nonzeros in rows a_row(j, q), q <
  // kA, in ascending order (filled up with rows whose entry is 0); column c of
  // B has one, in row b_row(c).
  static constexpr int kA = 2;
  static constexpr TO_HD int a_row(int j, int q) { return q == 0 ? (j >= 2 ? j - 2 : j) : (j >= 2 ? j : j + 2); }
  static constexpr TO_HD bool a_nz(int r, int j) { return r == j || r + 2 == j; }
  static constexpr TO_HD int b_row(int c) { return c + 2; }
  // the constant entries: A, B, and l_xx, l_x, l_uu outside the block (lane
  // of a group of G)
  template <class R>
  TO_DEV static void block_consts(const ParamsT<R>& P, int lane, int G, R eps, R* A, R* B, R* lxx, R* lx, R* luu) {
    const R w2 = R(2) * P.wu;
    for (int e = lane; e < n * n; e += G) {
      const int i = e / n, j = e % n;
      A[e] = (i == j) ? R(1) : ((j == i + 2) ? P.dt : R(0));
      lxx[e] = (i == j && i >= 2) ? clip0(eps) : R(0);
    }
    for (int e = lane; e < n * m; e += G) B[e] = (e / m == e % m + 2) ? P.dt : R(0);
    for (int e = lane; e < n; e += G) lx[e] = R(0);
    for (int e = lane; e < m * m; e += G) luu[e] = (e / m == e % m) ? (w2 > eps ? w2 : eps) : R(0);
  }
  // where entry e of the block goes; the mirrored entry of a symmetric pair
  // (second), else the same place
  template <class R>
  TO_DEV static R* block_dst(int e, bool second, R*, R* lxx, R* lx, R* lu) {
    return e == 0 ? lxx : e == 1 ? lxx + (second ? n : 1) : e == 2 ? lxx + n + 1 : e < 5 ? lx + (e - 3) : lu + (e - 5);
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
      for (int j = 0; j < n; ++j) A[i * n + j] = (i == j) ? R(1) : ((j == i + 2) ? P.dt : R(0));
#pragma unroll
    for (int i = 0; i < n; ++i)
#pragma unroll
      for (int j = 0; j < m; ++j) B[i * m + j] = (i == j + 2) ? P.dt : R(0);
#pragma unroll
    for (int i = 0; i < n * n; ++i) lxx[i] = 0;
    lxx[0] = d[0]; lxx[1] = d[1]; lxx[n] = d[1]; lxx[n + 1] = d[2];
    lxx[2 * n + 2] = clip0(eps); lxx[3 * n + 3] = clip0(eps);
    lx[0] = d[3]; lx[1] = d[4]; lx[2] = 0; lx[3] = 0;
    const R w2 = R(2) * P.wu;
    const R q = w2 > eps ? w2 : eps;
    luu[0] = q; luu[1] = 0; luu[2] = 0; luu[3] = q;
    lu[0] = d[5]; lu[1] = d[6];
  }

  template <class R>
  TO_DEV static void terminal_derivs(const ParamsT<R>& P, const R* x, R eps, R* lxx, R* lx) {
    const R a = R(2) * P.wpT, b = R(2) * P.wvT;
#pragma unroll
    for (int i = 0; i < n * n; ++i) lxx[i] = 0;
    lxx[0] = a > eps ? a : eps; lxx[5] = lxx[0];
    lxx[10] = b > eps ? b : eps; lxx[15] = lxx[10];
    lx[0] = a * x[0]; lx[1] = a * x[1]; lx[2] = b * x[2]; lx[3] = b * x[3];
  }
};

}  // namespace to
