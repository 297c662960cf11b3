// Rigid-body trees for the 7-DoF arm and the quadruped-shaped floating base
// (Sec. V-A's manipulators, Sec. V-D's quadruped; the synthetic workloads'
// parameters).  x = [q; qd], u = torques of joints a0..N-1.
//
// Dynamics: M(q) qdd + h(q, qd) = [0; u] (+ soft ground contact at the feet
// for the quadruped), n_sub semi-implicit Euler substeps of h = dt / n_sub:
//   qd+ = qd + h qdd,  q+ = q + h qd+.
// * h(q, qd): body-frame spatial Newton-Euler (Featherstone 2008, ch. 5) with
//   gravity as a base acceleration and the contact forces as external forces;
// * M(q): composite-rigid-body algorithm (Featherstone 2008, Sec. 6.2),
//   Cholesky-factored.
// Derivatives: each lane propagates one tangent direction (a state
// coordinate, or a control) through the substeps:
//   dqdd = M^{-1} (dtau - d ID(q, qd, qdd) / d(q, qd) . (dq, dqd)),
// with the directional derivative of the inverse dynamics (qdd held fixed)
// from a hand-written tangent pass over per-body primal quantities (the
// product rule of the Newton-Euler recursion).  The primal quantities of
// every knot's substeps are computed before the backward pass, one knot per
// lane, and stored; the tangent lanes stage them into shared memory.  A
// dual-number pass of the same recursion serves the arm's nested terminal
// Hessian.
#pragma once
#include "common.cuh"

namespace to {

// ---------------------------------------------------------------------------
// a dual number: value and one directional derivative
// ---------------------------------------------------------------------------
template <class R>
struct Dl {
  R v, d;
  TO_DEV Dl() {}
  TO_DEV Dl(R a) : v(a), d(0) {}
  TO_DEV Dl(R a, R b) : v(a), d(b) {}
};
template <class R> TO_DEV Dl<R> operator+(Dl<R> a, Dl<R> b) { return Dl<R>(a.v + b.v, a.d + b.d); }
template <class R> TO_DEV Dl<R> operator-(Dl<R> a, Dl<R> b) { return Dl<R>(a.v - b.v, a.d - b.d); }
template <class R> TO_DEV Dl<R> operator-(Dl<R> a) { return Dl<R>(-a.v, -a.d); }
template <class R> TO_DEV Dl<R> operator*(Dl<R> a, Dl<R> b) { return Dl<R>(a.v * b.v, a.v * b.d + a.d * b.v); }
template <class R> TO_DEV Dl<R> operator*(R a, Dl<R> b) { return Dl<R>(a * b.v, a * b.d); }
template <class R> TO_DEV Dl<R> operator/(Dl<R> a, Dl<R> b) {
  const R iv = R(1) / b.v;
  return Dl<R>(a.v * iv, (a.d - a.v * iv * b.d) * iv);
}
template <class R> TO_DEV Dl<R>& operator+=(Dl<R>& a, Dl<R> b) { a = a + b; return a; }
template <class R> TO_DEV Dl<R>& operator-=(Dl<R>& a, Dl<R> b) { a = a - b; return a; }
TO_DEV float dexp(float a) { return expf(a); }
TO_DEV double dexp(double a) { return exp(a); }
TO_DEV float dlog1p(float a) { return log1pf(a); }
TO_DEV double dlog1p(double a) { return log1p(a); }
TO_DEV void dsincos(float a, float* s, float* c) { sincosf(a, s, c); }
TO_DEV void dsincos(double a, double* s, double* c) { sincos(a, s, c); }
TO_DEV float value_of(float a) { return a; }
TO_DEV double value_of(double a) { return a; }
template <class R> TO_DEV auto value_of(Dl<R> a) { return value_of(a.v); }
template <class R> TO_DEV Dl<R> dexp(Dl<R> a) { const R e = dexp(a.v); return Dl<R>(e, e * a.d); }
template <class R> TO_DEV Dl<R> dlog1p(Dl<R> a) { return Dl<R>(dlog1p(a.v), a.d / (R(1) + a.v)); }
template <class R> TO_DEV void dsincos(Dl<R> a, Dl<R>* s, Dl<R>* c) {
  R sv, cv;
  dsincos(a.v, &sv, &cv);
  *s = Dl<R>(sv, cv * a.d);
  *c = Dl<R>(cv, -(sv * a.d));
}

// ---------------------------------------------------------------------------
// parameters
// ---------------------------------------------------------------------------
enum { RK_ARM7 = 3, RK_QUAD = 4 };

template <class R, int N>
struct RigidParams {
  R dt, g[3];
  int n_sub, a0;
  int parent[N], jtype[N];
  R off[N][3], mass[N], com[N][3], inertia[N][3];
  // arm reaching cost
  R wtau, wv, tgt[3], wee, wvT, ee_pt[3];
  int ee_body;
  // quadruped cost and contact
  R znom, wz, wrpy, wvx, vxt, tscale, kc, dc, beta;
  int nfeet, foot_body[4];
  R foot_pt[4][3];
  int free_base;   // quadruped: bodies 0..4 massless, the base's joints all at one point
};

template <class D, class S, int N>
inline void cast_params(const RigidParams<S, N>& s, RigidParams<D, N>& d) {
  d.dt = (D)s.dt;
  for (int k = 0; k < 3; ++k) { d.g[k] = (D)s.g[k]; d.tgt[k] = (D)s.tgt[k]; d.ee_pt[k] = (D)s.ee_pt[k]; }
  d.n_sub = s.n_sub; d.a0 = s.a0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    d.parent[i] = s.parent[i]; d.jtype[i] = s.jtype[i]; d.mass[i] = (D)s.mass[i];
    for (int k = 0; k < 3; ++k) { d.off[i][k] = (D)s.off[i][k]; d.com[i][k] = (D)s.com[i][k]; d.inertia[i][k] = (D)s.inertia[i][k]; }
  }
  d.wtau = (D)s.wtau; d.wv = (D)s.wv; d.wee = (D)s.wee; d.wvT = (D)s.wvT; d.ee_body = s.ee_body;
  d.znom = (D)s.znom; d.wz = (D)s.wz; d.wrpy = (D)s.wrpy; d.wvx = (D)s.wvx; d.vxt = (D)s.vxt;
  d.free_base = s.free_base;
  d.tscale = (D)s.tscale; d.kc = (D)s.kc; d.dc = (D)s.dc; d.beta = (D)s.beta; d.nfeet = s.nfeet;
  for (int f = 0; f < 4; ++f) {
    d.foot_body[f] = s.foot_body[f];
    for (int k = 0; k < 3; ++k) d.foot_pt[f][k] = (D)s.foot_pt[f][k];
  }
}

// ---------------------------------------------------------------------------
// Joint trees, fixed at compile time: every loop over the bodies and over an
// ancestor chain has a compile-time trip count and unrolls, so the per-body
// arrays of the recursions are registers (or fixed stack slots) rather than
// dynamically indexed local memory.  parent(i) < i (parents first); depth(i)
// counts the ancestors of body i and anc(i, d) is its d-th ancestor
// (anc(i, 0) = i).  Joint types: 0..2 revolute about x, y, z; 3..5 prismatic
// along x, y, z.  The host parser accepts exactly these trees.
// ---------------------------------------------------------------------------
template <int KIND>
struct RigidTopo;

// 7-DoF arm: a chain of revolute joints about z, y, z, y, z, y, z; the end
// effector on the last body
template <>
struct RigidTopo<RK_ARM7> {
  static constexpr int kBodies = 7, kDepthMax = 6, kFeet = 0, kEeBody = 6;
  static constexpr int parent(int i) { return i - 1; }
  static constexpr int jtype(int i) { return (i & 1) ? 1 : 2; }
  static constexpr int depth(int i) { return i; }
  static constexpr int anc(int i, int d) { return i - d; }
  static constexpr int foot_body(int) { return -1; }
};

// quadruped: the floating base as the chain Px, Py, Pz, Rz, Ry, Rx (bodies
// 0..5, the base's mass on body 5), then four legs of hip (x), thigh (y) and
// calf (y) joints hanging from body 5; the feet on the calves
template <>
struct RigidTopo<RK_QUAD> {
  static constexpr int kBodies = 18, kDepthMax = 8, kFeet = 4, kEeBody = -1;
  static constexpr int parent(int i) { return i < 6 ? i - 1 : ((i - 6) % 3 == 0 ? 5 : i - 1); }
  static constexpr int jtype(int i) { return i < 3 ? 3 + i : (i < 6 ? 5 - i : ((i - 6) % 3 == 0 ? 0 : 1)); }
  static constexpr int depth(int i) { return i < 6 ? i : 6 + (i - 6) % 3; }
  static constexpr int anc(int i, int d) { return (i < 6 || d <= (i - 6) % 3) ? i - d : 6 + (i - 6) % 3 - d; }
  static constexpr int foot_body(int f) { return 8 + 3 * f; }
};

// ---------------------------------------------------------------------------
// the model
// ---------------------------------------------------------------------------
template <int N_, int A0, int KIND>
struct SysRigid {
  static constexpr int N = N_;
  static constexpr int n = 2 * N, m = N - A0;
  static constexpr bool kActor = (KIND == RK_QUAD);   // 36 -> 256 -> 256 -> 12 actor warm start
  template <class R> using ParamsT = RigidParams<R, N>;
  typedef RigidTopo<KIND> Topo;
  static_assert(Topo::kBodies == N, "joint tree size");
  static constexpr int kDepthMax = Topo::kDepthMax, kFeet = Topo::kFeet, kEeBody = Topo::kEeBody;
  static constexpr int parent(int i) { return Topo::parent(i); }
  static constexpr int jtype(int i) { return Topo::jtype(i); }
  static constexpr int depth(int i) { return Topo::depth(i); }
  static constexpr int anc(int i, int d) { return Topo::anc(i, d); }
  static constexpr int foot_body(int f) { return Topo::foot_body(f); }

  // The arm's float32 solves are chaotic: after any change of rounding they can
  // be compared with what they replace only by their distribution against the
  // oracle.  The cheaper forms whose rounding differs (shared joint transforms,
  // the sparse products of the mass matrix) are therefore not used there; that is
  // a way of comparing, not a limit (13.7 ms against 16.4 for B = 2048, T = 50 to
  // 200 with shared transforms, on the device).
  template <class R> static constexpr bool kKeepBits = KIND == RK_ARM7 && sizeof(R) == 4;

  // a body without mass needs no force of its own (the joints that place the
  // quadruped's base: 5 of 18 bodies; uniform over the grid)
  template <class R> TO_DEV static bool massless(const ParamsT<R>& P, int i) {
    if constexpr (KIND == RK_QUAD) return P.free_base && i < 5;
    else return false;
  }

  // 3-vectors
  template <class S> TO_DEV static void cross(const S* a, const S* b, S* c) {
    const S c0 = a[1] * b[2] - a[2] * b[1], c1 = a[2] * b[0] - a[0] * b[2], c2 = a[0] * b[1] - a[1] * b[0];
    c[0] = c0; c[1] = c1; c[2] = c2;
  }
  // y += a x b and y -= a x b.  In float64 fused: 6 operations, each of which
  // holds the scheduler's FP64 pipe for 64 cycles, where the compiler makes 9.
  // In float32 as the compiler fuses them: the arms are chaotic there, and
  // their bits are kept.
  template <class S> TO_DEV static void cross_acc(const S* a, const S* b, S* y) {
    if constexpr (sizeof(S) == 8) {
      y[0] = fma_rn(a[1], b[2], fma_rn(-a[2], b[1], y[0]));
      y[1] = fma_rn(a[2], b[0], fma_rn(-a[0], b[2], y[1]));
      y[2] = fma_rn(a[0], b[1], fma_rn(-a[1], b[0], y[2]));
    } else {
      y[0] += a[1] * b[2] - a[2] * b[1];
      y[1] += a[2] * b[0] - a[0] * b[2];
      y[2] += a[0] * b[1] - a[1] * b[0];
    }
  }
  template <class S> TO_DEV static void cross_sub(const S* a, const S* b, S* y) {
    if constexpr (sizeof(S) == 8) {
      cross_acc(b, a, y);
    } else {
      S c[3];
      cross(a, b, c);
#pragma unroll
      for (int k = 0; k < 3; ++k) y[k] -= c[k];
    }
  }
  // y += a x (s e_ax): a joint's own motion is along one axis, so 4 of the 6
  // products of cross_acc would multiply by zero (which the compiler may not
  // drop: 0 x is not 0 for every x)
  template <class S> TO_DEV static S axpy(S a, S b, S y) {
    if constexpr (sizeof(S) == 8) return fma_rn(a, b, y);
    else return y + mul_rn(a, b);
  }
  template <class S> TO_DEV static void axis_acc(const S* a, int ax, S s, S* y) {
    if (ax == 0) { y[1] = axpy(a[2], s, y[1]); y[2] = axpy(-a[1], s, y[2]); }
    else if (ax == 1) { y[0] = axpy(-a[2], s, y[0]); y[2] = axpy(a[0], s, y[2]); }
    else { y[0] = axpy(a[1], s, y[0]); y[1] = axpy(-a[0], s, y[1]); }
  }
  // y = E x and y = E^T x for a row-major 3x3 E
  template <class S> TO_DEV static void mv(const S* E, const S* x, S* y) {
    const S y0 = E[0] * x[0] + E[1] * x[1] + E[2] * x[2];
    const S y1 = E[3] * x[0] + E[4] * x[1] + E[5] * x[2];
    const S y2 = E[6] * x[0] + E[7] * x[1] + E[8] * x[2];
    y[0] = y0; y[1] = y1; y[2] = y2;
  }
  template <class S> TO_DEV static void mtv(const S* E, const S* x, S* y) {
    const S y0 = E[0] * x[0] + E[3] * x[1] + E[6] * x[2];
    const S y1 = E[1] * x[0] + E[4] * x[1] + E[7] * x[2];
    const S y2 = E[2] * x[0] + E[5] * x[1] + E[8] * x[2];
    y[0] = y0; y[1] = y1; y[2] = y2;
  }

  // y = E x and y = E^T x for a joint transform: a rotation about the joint's
  // coordinate axis (4 nonzeros besides the unit entry) or the identity
  // (prismatic).  The joint type is a compile-time constant at every call
  // (the body loops unroll), so the switch folds away.
  template <class S> TO_DEV static void jmv(int jt, const S* E, const S* x, S* y) {
    const S x0 = x[0], x1 = x[1], x2 = x[2];
    switch (jt) {
      case 0: { const S c = E[4], s = E[5]; y[0] = x0; y[1] = c * x1 + s * x2; y[2] = c * x2 - s * x1; break; }
      case 1: { const S c = E[0], s = E[6]; y[0] = c * x0 - s * x2; y[1] = x1; y[2] = c * x2 + s * x0; break; }
      case 2: { const S c = E[0], s = E[1]; y[0] = c * x0 + s * x1; y[1] = c * x1 - s * x0; y[2] = x2; break; }
      default: y[0] = x0; y[1] = x1; y[2] = x2;
    }
  }
  template <class S> TO_DEV static void jmtv(int jt, const S* E, const S* x, S* y) {
    const S x0 = x[0], x1 = x[1], x2 = x[2];
    switch (jt) {
      case 0: { const S c = E[4], s = E[5]; y[0] = x0; y[1] = c * x1 - s * x2; y[2] = c * x2 + s * x1; break; }
      case 1: { const S c = E[0], s = E[6]; y[0] = c * x0 + s * x2; y[1] = x1; y[2] = c * x2 - s * x0; break; }
      case 2: { const S c = E[0], s = E[1]; y[0] = c * x0 - s * x1; y[1] = c * x1 + s * x0; y[2] = x2; break; }
      default: y[0] = x0; y[1] = x1; y[2] = x2;
    }
  }

  // Entry (r, k) of E M, of M E and of E^T M for a joint transform E (M
  // row-major 3x3): a rotation about a coordinate axis leaves one row or column
  // alone and mixes the other two (the identity, prismatic, none), so a product
  // takes 12 multiply-adds where the full 3x3 one takes 27.
  template <class R> TO_DEV static R e_row(int jt, const R* E, const R* M, int r, int k) {
    if (jt > 2 || r == jt) return M[r * 3 + k];
    const int i = (jt + 1) % 3, j = (jt + 2) % 3;
    return E[r * 3 + i] * M[i * 3 + k] + E[r * 3 + j] * M[j * 3 + k];
  }
  template <class R> TO_DEV static R e_col(int jt, const R* M, const R* E, int r, int k) {
    if (jt > 2 || k == jt) return M[r * 3 + k];
    const int i = (jt + 1) % 3, j = (jt + 2) % 3;
    return M[r * 3 + i] * E[i * 3 + k] + M[r * 3 + j] * E[j * 3 + k];
  }
  template <class R> TO_DEV static R et_row(int jt, const R* E, const R* M, int r, int k) {
    if (jt > 2 || r == jt) return M[r * 3 + k];
    const int i = (jt + 1) % 3, j = (jt + 2) % 3;
    return E[i * 3 + r] * M[i * 3 + k] + E[j * 3 + r] * M[j * 3 + k];
  }

  // Plucker transform of joint i: E maps parent coordinates to body
  // coordinates (a rotation by q about the joint axis, or identity), r is the
  // body origin in parent coordinates
  template <class R, class S>
  TO_DEV static void joint_transform(const ParamsT<R>& P, int i, S q, S* E, S* r) {
    const int jt = jtype(i);
#pragma unroll
    for (int k = 0; k < 3; ++k) r[k] = S(P.off[i][k]);
#pragma unroll
    for (int k = 0; k < 9; ++k) E[k] = S(R(0));
    if (jt <= 2) {
      S s, c;
      dsincos(q, &s, &c);
      const int a = jt, b = (jt + 1) % 3, cc = (jt + 2) % 3;
      E[a * 3 + a] = S(R(1));
      E[b * 3 + b] = c; E[b * 3 + cc] = s;
      E[cc * 3 + b] = -s; E[cc * 3 + cc] = c;
    } else {
      E[0] = S(R(1)); E[4] = S(R(1)); E[8] = S(R(1));
      r[jt - 3] = r[jt - 3] + q;
    }
  }

  // world pose: E0 maps world to body coordinates, p0 is the body origin
  template <class R, class S>
  TO_DEV static void world_pose(const ParamsT<R>& P, const S* q, S (*E0)[9], S (*p0)[3]) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      S E[9], r[3];
      joint_transform(P, i, q[i], E, r);
      const int pa = parent(i);
      if (pa < 0) {
#pragma unroll
        for (int k = 0; k < 9; ++k) E0[i][k] = E[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) p0[i][k] = r[k];
      } else {
        // E0_i = E E0_p ;  p0_i = p0_p + E0_p^T r
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
          for (int b = 0; b < 3; ++b)
            E0[i][a * 3 + b] = E[a * 3 + 0] * E0[pa][0 * 3 + b] + E[a * 3 + 1] * E0[pa][1 * 3 + b] + E[a * 3 + 2] * E0[pa][2 * 3 + b];
        S wr[3];
        mtv(E0[pa], r, wr);
#pragma unroll
        for (int k = 0; k < 3; ++k) p0[i][k] = p0[pa][k] + wr[k];
      }
    }
  }

  // spatial inertia times a motion vector (w, v): momentum about the body
  // origin, (I_c w + c x p, p) with p = m (v + w x c)
  template <class R, class S>
  TO_DEV static void inertia_mul(const ParamsT<R>& P, int i, const S* w, const S* v, S* n, S* f) {
    S c[3] = {S(P.com[i][0]), S(P.com[i][1]), S(P.com[i][2])};
    S p[3];
    if constexpr (sizeof(S) == 8) {
#pragma unroll
      for (int k = 0; k < 3; ++k) p[k] = v[k];
      cross_acc(w, c, p);
#pragma unroll
      for (int k = 0; k < 3; ++k) { p[k] *= P.mass[i]; n[k] = P.inertia[i][k] * w[k]; f[k] = p[k]; }
      cross_acc(c, p, n);
    } else {
      S wc[3];
      cross(w, c, wc);
#pragma unroll
      for (int k = 0; k < 3; ++k) p[k] = P.mass[i] * (v[k] + wc[k]);
      S cp[3];
      cross(c, p, cp);
#pragma unroll
      for (int k = 0; k < 3; ++k) { n[k] = P.inertia[i][k] * w[k] + cp[k]; f[k] = p[k]; }
    }
  }

  // With the axis products and the sparse joint products (e_row), 7-DoF arm
  // B=304 float64 17.2 -> 15.3 ms (V_x, 2 iterations), B=2048 float32 29.5 ->
  // 27.5 ms (the same bits), quadruped B=512 float32 10.7 -> 9.5 ms.
  // One body's velocity and its acceleration at qdd = 0, from its parent's
  // (pa < 0: the fixed base, whose acceleration is -g): v and a transformed,
  // the joint's own motion S qd, the velocity product v x (S qd); then the body
  // force I a + v x* (I v).  Ept (nullable): the parent's linear velocity in
  // body axes; Epw the angular one.
  template <class R>
  TO_DEV static void body_bias(const ParamsT<R>& P, int i, const R* E, const R* r, R qd, const R* pw, const R* pv,
                               const R* paw, const R* pav, R* Epw, R* Ept, R* vw, R* vv, R* aw, R* av, R* hn, R* hf,
                               R* fn, R* ff) {
    const int pa = parent(i), jt = jtype(i), ax = jt <= 2 ? jt : jt - 3;
    R t[3];
    if (pa < 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) { Epw[k] = R(0); Ept[k] = R(0); aw[k] = R(0); t[k] = -P.g[k]; }
      // (no force depends on where a sliding root stands: a non-finite position
      // still ends in a non-finite cost)
      if (jt > 2) t[ax] += R(0) * r[ax];
    } else {
      // X m = (E w, E (v - r x w))
#pragma unroll
      for (int k = 0; k < 3; ++k) t[k] = pv[k];
      cross_sub(r, pw, t);
      jmv(jt, E, pw, Epw);
      jmv(jt, E, t, Ept);
#pragma unroll
      for (int k = 0; k < 3; ++k) t[k] = pav[k];
      cross_sub(r, paw, t);
      jmv(jt, E, paw, aw);
    }
    jmv(jt, E, t, av);
#pragma unroll
    for (int k = 0; k < 3; ++k) { vw[k] = Epw[k]; vv[k] = Ept[k]; }
    if (jt <= 2) vw[ax] += qd; else vv[ax] += qd;
    if (pa >= 0) {
      if (jt <= 2) {
        axis_acc(vw, ax, qd, aw);
        axis_acc(vv, ax, qd, av);
      } else {
        axis_acc(vw, ax, qd, av);
      }
    }
    if (massless(P, i)) {
#pragma unroll
      for (int k = 0; k < 3; ++k) { hn[k] = R(0); hf[k] = R(0); fn[k] = R(0); ff[k] = R(0); }
      return;
    }
    inertia_mul(P, i, aw, av, fn, ff);
    inertia_mul(P, i, vw, vv, hn, hf);
    cross_acc(vw, hn, fn);
    cross_acc(vv, hf, fn);
    cross_acc(vw, hf, ff);
  }

  // the bias torques: inverse dynamics at qdd = 0 with gravity and contact; the
  // joint transforms are left in E and r
  template <class R, class S>
  TO_DEV static void rnea(const ParamsT<R>& P, const S* q, const S* qd, S* tau, S (*E)[9], S (*r)[3]) {
    constexpr bool contact = KIND == RK_QUAD;
    S vw[N][3], vv[N][3], fn[N][3], ff[N][3];
    S E0[KIND == RK_QUAD ? N : 1][9], p0[KIND == RK_QUAD ? N : 1][3];
    S awb[N][3], avb[N][3];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      joint_transform(P, i, q[i], E[i], r[i]);
      const int pa = parent(i), jt = jtype(i), pb = pa < 0 ? 0 : pa;
      S Epw[3], Ept[3], hn[3], hf[3];
      body_bias(P, i, E[i], r[i], qd[i], vw[pb], vv[pb], awb[pb], avb[pb], Epw, Ept, vw[i], vv[i], awb[i], avb[i], hn,
                hf, fn[i], ff[i]);
      if (KIND == RK_QUAD) {
        if (pa < 0) {
#pragma unroll
          for (int k = 0; k < 9; ++k) E0[i][k] = E[i][k];
#pragma unroll
          for (int k = 0; k < 3; ++k) p0[i][k] = r[i][k];
        } else {
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) E0[i][a * 3 + b] = e_row(jt, E[i], E0[pa], a, b);
          S wr[3];
          mtv(E0[pa], r[i], wr);
#pragma unroll
          for (int k = 0; k < 3; ++k) p0[i][k] = p0[pa][k] + wr[k];
        }
      }
      (void)jt;
    }
    if (contact) {
#pragma unroll
      for (int ft = 0; ft < kFeet; ++ft) {
        const int bi = foot_body(ft);
        S pt[3] = {S(P.foot_pt[ft][0]), S(P.foot_pt[ft][1]), S(P.foot_pt[ft][2])};
        S wpt[3], Pw[3], wxp[3], vb[3], vwld[3];
        mtv(E0[bi], pt, wpt);
#pragma unroll
        for (int k = 0; k < 3; ++k) Pw[k] = p0[bi][k] + wpt[k];
        cross(vw[bi], pt, wxp);
#pragma unroll
        for (int k = 0; k < 3; ++k) vb[k] = vv[bi][k] + wxp[k];
        mtv(E0[bi], vb, vwld);
        // normal: k softplus_beta(-z) - d sigmoid(-beta z) zdot; tangential damper
        // softplus_beta(-z) = log(1 + exp(-beta z)) / beta and sigmoid(-beta z),
        // evaluated with exp of a non-positive argument only (no overflow)
        const S bz = P.beta * Pw[2];
        S sp, gate;
        if (value_of(bz) >= R(0)) {
          const S e = dexp(-bz);
          sp = (R(1) / P.beta) * dlog1p(e);
          gate = e / (S(R(1)) + e);
        } else {
          const S e = dexp(bz);
          sp = (R(1) / P.beta) * (dlog1p(e) - bz);
          gate = S(R(1)) / (S(R(1)) + e);
        }
        S F[3];
        F[0] = -(P.dc * (gate * vwld[0]));
        F[1] = -(P.dc * (gate * vwld[1]));
        F[2] = P.kc * sp - P.dc * (gate * vwld[2]);
        S mw[3], mb[3], fb[3];
        cross(wpt, F, mw);
        mv(E0[bi], mw, mb);
        mv(E0[bi], F, fb);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[bi][k] = fn[bi][k] - mb[k]; ff[bi][k] = ff[bi][k] - fb[k]; }
      }
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int jt = jtype(i);
      tau[i] = jt <= 2 ? fn[i][jt] : ff[i][jt - 3];
      const int pa = parent(i);
      if (pa >= 0) {
        // X^T f = (E^T n + r x E^T f, E^T f)
        S en[3], ef[3], rf[3];
        jmtv(jt, E[i], fn[i], en);
        jmtv(jt, E[i], ff[i], ef);
        cross(r[i], ef, rf);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[pa][k] = fn[pa][k] + en[k] + rf[k]; ff[pa][k] = ff[pa][k] + ef[k]; }
      }
    }
  }

  // Joint-space mass matrix by the composite-rigid-body algorithm
  // (Featherstone 2008, Sec. 6.2), written into the lower triangle of L and
  // factored in place as M = L^T L along the tree (reciprocal pivots).  A subtree's composite
  // inertia is kept about its root body's origin, in that body's coordinates,
  // as (mass, first moment h = mass * com, rotational inertia about the
  // origin); moving it to the parent frame rotates it and applies the
  // parallel-axis shift.  Bodies are ordered parents first.
  // Eb, rb (nullable): the joint transforms of q from its bias pass, which save a
  // second evaluation of each sine and cosine, 25 FP64 instructions a joint
  // (float64 arm, B = 304, T = 10 to 20: 8.93 -> 8.54 ms with the fused position
  // update; quadruped, B = 512, T = 4 to 8: 6.79 -> 6.60 ms).  The float32 arm
  // evaluates them twice (kKeepBits: the compiler fuses other multiply-adds with
  // shared ones).
  template <class R>
  TO_DEV static void mass_chol(const ParamsT<R>& P, const R* q, R* L, const R (*Eb)[9] = nullptr,
                               const R (*rb)[3] = nullptr) {
    constexpr bool kFull = kKeepBits<R>;   // the full products of a joint transform
    R E[N][9], r[N][3];
    R cm[N], ch[N][3], cI[N][6];   // cI: xx, yy, zz, xy, xz, yz
#pragma unroll
    for (int i = 0; i < N; ++i) {
      if (!Eb) {
        joint_transform(P, i, q[i], E[i], r[i]);
      } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) E[i][k] = Eb[i][k];
#pragma unroll
        for (int k = 0; k < 3; ++k) r[i][k] = rb[i][k];
      }
      const R mi = P.mass[i], c0 = P.com[i][0], c1 = P.com[i][1], c2 = P.com[i][2];
      cm[i] = mi;
      ch[i][0] = mi * c0; ch[i][1] = mi * c1; ch[i][2] = mi * c2;
      // I_origin = I_com + m (|c|^2 1 - c c^T)
      cI[i][0] = P.inertia[i][0] + mi * (c1 * c1 + c2 * c2);
      cI[i][1] = P.inertia[i][1] + mi * (c0 * c0 + c2 * c2);
      cI[i][2] = P.inertia[i][2] + mi * (c0 * c0 + c1 * c1);
      cI[i][3] = -mi * c0 * c1; cI[i][4] = -mi * c0 * c2; cI[i][5] = -mi * c1 * c2;
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int pa = parent(i);
      if (pa < 0) continue;
      const R* e = E[i];
      const R* rr = r[i];
      const R mi = cm[i];
      // h_A = E^T h (parent coordinates, about the child origin)
      R hA[3];
      jmtv(jtype(i), e, ch[i], hA);
      // I_A = E^T I E
      const R I3[9] = {cI[i][0], cI[i][3], cI[i][4], cI[i][3], cI[i][1], cI[i][5], cI[i][4], cI[i][5], cI[i][2]};
      R T[9];   // I E
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
          T[a * 3 + b] = kFull ? I3[a * 3 + 0] * e[0 * 3 + b] + I3[a * 3 + 1] * e[1 * 3 + b] + I3[a * 3 + 2] * e[2 * 3 + b]
                               : e_col(jtype(i), I3, e, a, b);
      R IA[6];
      const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
#pragma unroll
      for (int k = 0; k < 6; ++k)
        IA[k] = kFull ? e[0 * 3 + ia[k]] * T[0 * 3 + ib[k]] + e[1 * 3 + ia[k]] * T[1 * 3 + ib[k]] + e[2 * 3 + ia[k]] * T[2 * 3 + ib[k]]
                      : et_row(jtype(i), e, T, ia[k], ib[k]);
      // shift to the parent origin (child origin at r):
      // I_O = I_A + m (|r|^2 1 - r r^T) + 2 (r.h_A) 1 - (h_A r^T + r h_A^T)
      const R r2 = rr[0] * rr[0] + rr[1] * rr[1] + rr[2] * rr[2];
      const R rh = rr[0] * hA[0] + rr[1] * hA[1] + rr[2] * hA[2];
#pragma unroll
      for (int k = 0; k < 3; ++k) cI[pa][k] += IA[k] + mi * (r2 - rr[k] * rr[k]) + R(2) * (rh - hA[k] * rr[k]);
#pragma unroll
      for (int k = 3; k < 6; ++k) cI[pa][k] += IA[k] - mi * rr[ia[k]] * rr[ib[k]] - (hA[ia[k]] * rr[ib[k]] + rr[ia[k]] * hA[ib[k]]);
#pragma unroll
      for (int k = 0; k < 3; ++k) ch[pa][k] += hA[k] + mi * rr[k];
      cm[pa] += mi;
    }
    // only (body, ancestor) entries are formed and read: the others are zero
#pragma unroll
    for (int i = 0; i < N; ++i) {
      // F = Ic_i S_i: revolute about axis a: (I e_a, e_a x h); prismatic along a: (h x e_a, m e_a)
      R fn[3], ff[3];
      const int jt = jtype(i);
      const R* c6 = cI[i];
      if (jt <= 2) {
        const int a = jt;
        const int col[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
        fn[0] = c6[col[0][a]]; fn[1] = c6[col[1][a]]; fn[2] = c6[col[2][a]];
        R ea[3] = {R(0), R(0), R(0)};
        ea[a] = R(1);
        cross(ea, ch[i], ff);
      } else {
        const int a = jt - 3;
        R ea[3] = {R(0), R(0), R(0)};
        ea[a] = R(1);
        cross(ch[i], ea, fn);
        ff[0] = R(0); ff[1] = R(0); ff[2] = R(0);
        ff[a] = cm[i];
      }
      L[i * N + i] = jt <= 2 ? fn[jt] : ff[jt - 3];
#pragma unroll
      for (int d = 0; d < kDepthMax; ++d) {
        if (d >= depth(i)) continue;
        // force across joint j into its parent's frame: f_p = E^T f, n_p = E^T n + r x f_p
        const int j = anc(i, d), jp = anc(i, d + 1);
        R en[3], ef[3], rf[3];
        jmtv(jtype(j), E[j], fn, en);
        jmtv(jtype(j), E[j], ff, ef);
        cross(r[j], ef, rf);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[k] = en[k] + rf[k]; ff[k] = ef[k]; }
        const int jj = jtype(jp);
        L[i * N + jp] = jj <= 2 ? fn[jj] : ff[jj - 3];
      }
    }
    // M = L^T L with L lower triangular and the tree's sparsity (Featherstone
    // 2008, Sec. 6.5): eliminating from the last body up touches only
    // (body, ancestor) pairs, so nothing fills in; 1 / L_kk on the diagonal
#pragma unroll
    for (int k = N - 1; k >= 0; --k) {
      const R rk = rsqrt_(L[k * N + k]);
      L[k * N + k] = rk;
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d)
        if (d <= depth(k)) L[k * N + anc(k, d)] *= rk;
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d) {
        if (d > depth(k)) continue;
        const int i = anc(k, d);
        const R lki = L[k * N + i];
#pragma unroll
        for (int e = 0; e <= kDepthMax; ++e)
          if (e <= depth(i)) L[i * N + anc(i, e)] -= lki * L[k * N + anc(i, e)];
      }
    }
  }
  // mass_chol of q held in (shared) memory into (shared) memory: q read once,
  // the factor formed in registers, then only its tree-sparse entries (the
  // diagonal and the (body, ancestor) pairs, all that chol_solve reads) stored
  template <class R>
  TO_DEV static void mass_chol_mem(const ParamsT<R>& P, const R* qm, R* Lm) {
    R q[N], L[N * N];
#pragma unroll
    for (int i = 0; i < N; ++i) q[i] = qm[i];
    mass_chol(P, q, L);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      Lm[k * N + k] = L[k * N + k];
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d)
        if (d <= depth(k)) Lm[k * N + anc(k, d)] = L[k * N + anc(k, d)];
    }
  }

  // x = M^{-1} b with M = L^T L from mass_chol: L^T y = b from the leaves up,
  // then L x = y from the root down, each along the ancestor chains
  template <class R>
  TO_DEV static void chol_solve(const ParamsT<R>& P, const R* L, const R* b, R* x) {
    R y[N];
#pragma unroll
    for (int i = 0; i < N; ++i) y[i] = b[i];
#pragma unroll
    for (int k = N - 1; k >= 0; --k) {
      y[k] *= L[k * N + k];
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d)
        if (d <= depth(k)) y[anc(k, d)] -= L[k * N + anc(k, d)] * y[k];
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
      R t = y[k];
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d)
        if (d <= depth(k)) t -= L[k * N + anc(k, d)] * x[anc(k, d)];
      x[k] = t * L[k * N + k];
    }
  }

  // one substep's acceleration: qdd = M^{-1} (tau - h); also returns L
  template <class R>
  TO_DEV static void accel(const ParamsT<R>& P, const R* q, const R* qd, const R* tau, R* qdd, R* L) {
    R h[N], rhs[N], E[N][9], r[N][3];
    rnea<R, R>(P, q, qd, h, E, r);
    if constexpr (kKeepBits<R>) mass_chol(P, q, L);
    else mass_chol(P, q, L, E, r);
#pragma unroll
    for (int i = 0; i < N; ++i) rhs[i] = tau[i] - h[i];
    chol_solve(P, L, rhs, qdd);
  }


  // ---- costs ----
  template <class R, class S>
  TO_DEV static void ee_world(const ParamsT<R>& P, const S* q, S* ee) {
    S E0[N][9], p0[N][3];
    world_pose(P, q, E0, p0);
    const int b = kEeBody < 0 ? 0 : kEeBody;   // the arm's end-effector body (unused for the quadruped)
    S pt[3] = {S(P.ee_pt[0]), S(P.ee_pt[1]), S(P.ee_pt[2])}, w[3];
    mtv(E0[b], pt, w);
#pragma unroll
    for (int k = 0; k < 3; ++k) ee[k] = p0[b][k] + w[k];
  }

  template <class R>
  TO_DEV static R running_cost(const ParamsT<R>& P, const R* x, const R* u) {
    R l = 0;
    for (int j = 0; j < m; ++j) l += P.wtau * u[j] * u[j];
    if (KIND == RK_ARM7) {
#pragma unroll
      for (int j = 0; j < N; ++j) l += P.wv * x[N + j] * x[N + j];
    } else {
      const R dz = x[2] - P.znom, dv = x[N] - P.vxt;
      l += P.wz * dz * dz + P.wrpy * (x[3] * x[3] + x[4] * x[4] + x[5] * x[5]) + P.wvx * dv * dv;
    }
    return l;
  }
  // the same step on a state carried as (hi, lo) pairs, in place
  template <class R>
  TO_DEV static R cost_step2(const ParamsT<R>& P, R* xh, R* xl, const R* u) {
    const R l = running_cost(P, xh, u);
    R tau[N], qdd[N], L[N * N];
#pragma unroll
    for (int i = 0; i < N; ++i) tau[i] = i < A0 ? R(0) : u[i - A0];
    const R h = P.dt / (R)P.n_sub;
    for (int s = 0; s < P.n_sub; ++s) {
      accel(P, xh, xh + N, tau, qdd, L);
      semi_implicit2<R, N>(xh, xl, xh + N, xl + N, qdd, h);
    }
    return l;
  }
  // -------------------------------------------------------------------------
  // The quadruped's step by teams.  G / 16 lanes take a candidate, one or two
  // legs each: the same code for every leg (the body index is data), the base
  // on every lane, and only sums over the legs cross the lanes.  The base is a
  // free body (P.free_base: its six joints only place it), so the step is solved
  // in its spatial acceleration a_b instead of its joints':
  //   [ I_c  F ] [ a_b  ]   [ -(bias wrench) ]     F: the legs' joint columns
  //   [ F^T  H ] [ qdd  ] = [ tau - bias     ]     H: 3 x 3 per leg
  // each lane eliminates its legs, the 6 x 6 Schur complement is summed and
  // solved on every lane, and the joints' accelerations follow from the axes.
  // A substep is ~1.5 k instructions on all lanes; by partner lanes it is ~4.4 k on
  // a candidate's lane beside ~4 k on its partner's, half of the lanes, in four
  // times the code.
  // Quadruped B=512 float32, T 4..8, 1 iteration, V_x: 9.7 -> 7.8 ms.
  // -------------------------------------------------------------------------
  static constexpr int kTeamSlot = 4 * N + m;      // x hi, x lo, joint torques of a candidate
  // the joint rotations of a leg: c = cos q, s = sin q, axis JT (0: x, 1: y)
  template <int JT, class R> TO_DEV static void rot(R c, R s, const R* x, R* y) {
    const R x0 = x[0], x1 = x[1], x2 = x[2];
    if (JT == 0) { y[0] = x0; y[1] = c * x1 + s * x2; y[2] = c * x2 - s * x1; }
    else { y[0] = c * x0 - s * x2; y[1] = x1; y[2] = c * x2 + s * x0; }
  }
  template <int JT, class R> TO_DEV static void rot_t(R c, R s, const R* x, R* y) { rot<JT>(c, -s, x, y); }
  // a spatial force (n, f) in body axes to the parent's: (E^T n + r x E^T f, E^T f)
  template <int JT, class R> TO_DEV static void force_up(R c, R s, const R* r, const R* n_, const R* f_, R* n2, R* f2) {
    rot_t<JT>(c, s, f_, f2);
    rot_t<JT>(c, s, n_, n2);
    cross_acc(r, f2, n2);
  }
  // composite inertia (mass, first moment, rotational inertia xx yy zz xy xz yz
  // about the origin) of a child added to its parent's
  template <int JT, class R>
  TO_DEV static void inertia_up(R c, R s, const R* r, R mi, const R* hc, const R* I, R& mp, R* hp, R* Ip) {
    R hA[3];
    rot_t<JT>(c, s, hc, hA);
    // E^T I E for a rotation in the plane (j, k): the 2 x 2 block turned twice
    R A[6];
    if (JT == 0) {
      const R ty = c * I[1] - s * I[5], tz = c * I[5] - s * I[2], uy = s * I[1] + c * I[5], uz = s * I[5] + c * I[2];
      A[0] = I[0]; A[1] = c * ty - s * tz; A[5] = s * ty + c * tz; A[2] = s * uy + c * uz;
      A[3] = c * I[3] - s * I[4]; A[4] = s * I[3] + c * I[4];
    } else {
      const R tz = c * I[2] - s * I[4], tx = c * I[4] - s * I[0], uz = s * I[2] + c * I[4], ux = s * I[4] + c * I[0];
      A[1] = I[1]; A[2] = c * tz - s * tx; A[4] = s * tz + c * tx; A[0] = s * uz + c * ux;
      A[5] = c * I[5] - s * I[3]; A[3] = s * I[5] + c * I[3];
    }
    const R r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2], rh = r[0] * hA[0] + r[1] * hA[1] + r[2] * hA[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) Ip[k] += A[k] + mi * (r2 - r[k] * r[k]) + R(2) * (rh - hA[k] * r[k]);
    Ip[3] += A[3] - mi * r[0] * r[1] - (hA[0] * r[1] + r[0] * hA[1]);
    Ip[4] += A[4] - mi * r[0] * r[2] - (hA[0] * r[2] + r[0] * hA[2]);
    Ip[5] += A[5] - mi * r[1] * r[2] - (hA[1] * r[2] + r[1] * hA[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) hp[k] += hA[k] + mi * r[k];
    mp += mi;
  }
  template <class R> TO_DEV static void body_inertia(const ParamsT<R>& P, int i, R& mi, R* h, R* I) {
    const R c0 = P.com[i][0], c1 = P.com[i][1], c2 = P.com[i][2];
    mi = P.mass[i];
    h[0] = mi * c0; h[1] = mi * c1; h[2] = mi * c2;
    I[0] = P.inertia[i][0] + (h[1] * c1 + h[2] * c2);
    I[1] = P.inertia[i][1] + (h[0] * c0 + h[2] * c2);
    I[2] = P.inertia[i][2] + (h[0] * c0 + h[1] * c1);
    I[3] = -h[0] * c1; I[4] = -h[0] * c2; I[5] = -h[1] * c2;
  }
  // a leg body's velocity and acceleration at qdd = 0 and the force they need
  template <int JT, class R>
  TO_DEV static void leg_body(const ParamsT<R>& P, int i, R c, R s, const R* r, R qd, const R* pw, const R* pv, const R* paw,
                              const R* pav, R* vw, R* vv, R* aw, R* av, R* fn, R* ff) {
    R t[3], hn[3], hf[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = pv[k];
    cross_sub(r, pw, t);
    rot<JT>(c, s, pw, vw);
    rot<JT>(c, s, t, vv);
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k] = pav[k];
    cross_sub(r, paw, t);
    rot<JT>(c, s, paw, aw);
    rot<JT>(c, s, t, av);
    vw[JT] += qd;
    axis_acc(vw, JT, qd, aw);
    axis_acc(vv, JT, qd, av);
    inertia_mul(P, i, aw, av, fn, ff);
    inertia_mul(P, i, vw, vv, hn, hf);
    cross_acc(vw, hn, fn);
    cross_acc(vv, hf, fn);
    cross_acc(vw, hf, ff);
  }

  // a knot's substeps by its team, from the state and the joint torques in its
  // slot, where the new state is left; prims (nullable): the state and the
  // accelerations of every substep are put into the knot's stored Prims
  template <class R, int G>
  TO_DEV static void team_steps(const ParamsT<R>& P, bool on, R* slot, int sub, R* prims) {
    constexpr int TL = G / kStepSlots, LP = 4 / TL;
    R bq[6], bql[6], bv[6], bvl[6], lq[LP][3], lql[LP][3], lv[LP][3], lvl[LP][3], tau[LP][3];
#pragma unroll
    for (int i = 0; i < 6; ++i) { bq[i] = slot[i]; bql[i] = slot[n + i]; bv[i] = slot[N + i]; bvl[i] = slot[n + N + i]; }
#pragma unroll
    for (int p = 0; p < LP; ++p)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int j = 3 * (sub * LP + p) + k;
        lq[p][k] = slot[6 + j]; lql[p][k] = slot[n + 6 + j];
        lv[p][k] = slot[N + 6 + j]; lvl[p][k] = slot[n + N + 6 + j];
        tau[p][k] = slot[2 * n + j];
      }
    const R h = P.dt / (R)P.n_sub, ib = R(1) / P.beta;
    for (int st = 0; st < P.n_sub; ++st) {
      if (prims && on) {
        Prim<R>& pr = *reinterpret_cast<Prim<R>*>(prims + (size_t)st * kPrimStride<R>);
        if (sub == 0)
#pragma unroll
          for (int i = 0; i < 6; ++i) { pr.q[i] = bq[i]; pr.qd[i] = bv[i]; }
#pragma unroll
        for (int p = 0; p < LP; ++p)
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int j = 6 + 3 * (sub * LP + p) + k;
            pr.q[j] = lq[p][k]; pr.qd[j] = lv[p][k]; pr.tin[j] = tau[p][k];
          }
      }
      // the base: E0 maps world to body axes
      R sz, cz, sy, cy, sx, cx;
      dsincos(bq[3], &sz, &cz);
      dsincos(bq[4], &sy, &cy);
      dsincos(bq[5], &sx, &cx);
      const R E0[9] = {cy * cz,                cy * sz,                -sy,
                       sx * sy * cz - cx * sz, sx * sy * sz + cx * cz, sx * cy,
                       cx * sy * cz + sx * sz, cx * sy * sz - sx * cz, cx * cy};
      R w[3], v[3], aw[3], av[3], fb[3], nb[3];
      const R dz = bv[3], dy = bv[4], dx = bv[5], zy = dz * dy;
      w[0] = dx - sy * dz; w[1] = cx * dy + sx * cy * dz; w[2] = cx * cy * dz - sx * dy;
      aw[0] = -cy * zy; aw[1] = w[2] * dx - sx * sy * zy; aw[2] = -(w[1] * dx) - cx * sy * zy;
      mv(E0, bv, v);
      mv(E0, P.g, av);
#pragma unroll
      for (int k = 0; k < 3; ++k) av[k] = -av[k];
      // (no force depends on where the base stands in the plane: a non-finite
      // position still ends in a non-finite cost)
      av[0] += R(0) * bq[0] + R(0) * bq[1];
      cross_acc(v, w, av);
      // sums over the legs: the 6 x 6 matrix (lower, rows n then f) and the right-hand side
      R S[21], y[6];
      {
        R hn[3], hf[3];
        inertia_mul(P, 5, aw, av, nb, fb);
        inertia_mul(P, 5, w, v, hn, hf);
        cross_acc(w, hn, nb);
        cross_acc(v, hf, nb);
        cross_acc(w, hf, fb);
      }
#pragma unroll
      for (int i = 0; i < 21; ++i) S[i] = R(0);
#pragma unroll
      for (int i = 0; i < 6; ++i) y[i] = R(0);
      R mc = R(0), hc[3] = {R(0), R(0), R(0)}, Ic[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
      R F[LP][3][6], yr[LP][3], l00[LP], l10[LP], l20[LP], l11[LP], l21[LP], l22[LP];
#pragma unroll
      for (int p = 0; p < LP; ++p) {
        const int leg = sub * LP + p, bi = 6 + 3 * leg;
        R s0, c0, s1, c1, s2, c2;
        dsincos(lq[p][0], &s0, &c0);
        dsincos(lq[p][1], &s1, &c1);
        dsincos(lq[p][2], &s2, &c2);
        const R* r0 = P.off[bi];
        const R* r1 = P.off[bi + 1];
        const R* r2 = P.off[bi + 2];
        R w0[3], v0[3], a0[3], b0[3], n0[3], f0[3], w1[3], v1[3], a1[3], b1[3], n1[3], f1[3], w2[3], v2[3], a2[3], b2[3],
            n2[3], f2[3];
        leg_body<0>(P, bi, c0, s0, r0, lv[p][0], w, v, aw, av, w0, v0, a0, b0, n0, f0);
        leg_body<1>(P, bi + 1, c1, s1, r1, lv[p][1], w0, v0, a0, b0, w1, v1, a1, b1, n1, f1);
        leg_body<1>(P, bi + 2, c2, s2, r2, lv[p][2], w1, v1, a1, b1, w2, v2, a2, b2, n2, f2);
        {  // contact at the foot: height and velocity in world axes, the force back in the calf's
          const R pt[3] = {P.foot_pt[leg][0], P.foot_pt[leg][1], P.foot_pt[leg][2]};
          R t[3], q[3], vel[3], Fw[3];
          rot_t<1>(c2, s2, pt, t);
#pragma unroll
          for (int k = 0; k < 3; ++k) t[k] += r2[k];
          rot_t<1>(c1, s1, t, q);
#pragma unroll
          for (int k = 0; k < 3; ++k) q[k] += r1[k];
          rot_t<0>(c0, s0, q, t);
#pragma unroll
          for (int k = 0; k < 3; ++k) t[k] += r0[k];
          const R bz = P.beta * (bq[2] + (E0[2] * t[0] + E0[5] * t[1] + E0[8] * t[2]));
#pragma unroll
          for (int k = 0; k < 3; ++k) t[k] = v2[k];
          cross_acc(w2, pt, t);
          rot_t<1>(c2, s2, t, q);
          rot_t<1>(c1, s1, q, t);
          rot_t<0>(c0, s0, t, q);
          mtv(E0, q, vel);
          R sp, gate;
          if (bz >= R(0)) {
            const R e = dexp(-bz);
            sp = ib * dlog1p(e);
            gate = e / (R(1) + e);
          } else {
            const R e = dexp(bz);
            sp = ib * (dlog1p(e) - bz);
            gate = R(1) / (R(1) + e);
          }
          const R dg = P.dc * gate;
          Fw[0] = -(dg * vel[0]);
          Fw[1] = -(dg * vel[1]);
          Fw[2] = P.kc * sp - dg * vel[2];
          mv(E0, Fw, q);
          rot<0>(c0, s0, q, t);
          rot<1>(c1, s1, t, q);
          rot<1>(c2, s2, q, t);
#pragma unroll
          for (int k = 0; k < 3; ++k) f2[k] -= t[k];
          cross_sub(pt, t, n2);
        }
        // bias torques, and the leg's wrench on the base
        R rhs[3], nu[3], fu[3];
        rhs[2] = tau[p][2] - n2[1];
        force_up<1>(c2, s2, r2, n2, f2, nu, fu);
#pragma unroll
        for (int k = 0; k < 3; ++k) { n1[k] += nu[k]; f1[k] += fu[k]; }
        rhs[1] = tau[p][1] - n1[1];
        force_up<1>(c1, s1, r1, n1, f1, nu, fu);
#pragma unroll
        for (int k = 0; k < 3; ++k) { n0[k] += nu[k]; f0[k] += fu[k]; }
        rhs[0] = tau[p][0] - n0[0];
        force_up<0>(c0, s0, r0, n0, f0, nu, fu);
#pragma unroll
        for (int k = 0; k < 3; ++k) { y[k] -= nu[k]; y[3 + k] -= fu[k]; }
        // composite inertias and joint columns (I e, e x h), carried to the base
        R H00, H10, H20, H11, H21, H22;
        {
          R m2, h2[3], I2[6], m1, h1[3], I1[6], m0, h0[3], I0[6], n_[3], f_[3];
          body_inertia(P, bi + 2, m2, h2, I2);
          body_inertia(P, bi + 1, m1, h1, I1);
          body_inertia(P, bi, m0, h0, I0);
          inertia_up<1>(c2, s2, r2, m2, h2, I2, m1, h1, I1);
          inertia_up<1>(c1, s1, r1, m1, h1, I1, m0, h0, I0);
          inertia_up<0>(c0, s0, r0, m0, h0, I0, mc, hc, Ic);
          const R cn[3] = {I2[3], I2[1], I2[5]}, cf[3] = {h2[2], R(0), -h2[0]};
          H22 = I2[1];
          force_up<1>(c2, s2, r2, cn, cf, n_, f_);
          H21 = n_[1];
          force_up<1>(c1, s1, r1, n_, f_, nu, fu);
          H20 = nu[0];
          force_up<0>(c0, s0, r0, nu, fu, &F[p][2][0], &F[p][2][3]);
          const R tn[3] = {I1[3], I1[1], I1[5]}, tf[3] = {h1[2], R(0), -h1[0]};
          H11 = I1[1];
          force_up<1>(c1, s1, r1, tn, tf, nu, fu);
          H10 = nu[0];
          force_up<0>(c0, s0, r0, nu, fu, &F[p][1][0], &F[p][1][3]);
          const R xn[3] = {I0[0], I0[3], I0[4]}, xf[3] = {R(0), -h0[2], h0[1]};
          H00 = I0[0];
          force_up<0>(c0, s0, r0, xn, xf, &F[p][0][0], &F[p][0][3]);
        }
        // H = L L^T (reciprocal diagonal); F <- L^-1 F^T, yr = L^-1 rhs
        l00[p] = rsqrt_(H00);
        l10[p] = H10 * l00[p];
        l20[p] = H20 * l00[p];
        l11[p] = rsqrt_(H11 - l10[p] * l10[p]);
        l21[p] = (H21 - l20[p] * l10[p]) * l11[p];
        l22[p] = rsqrt_(H22 - l20[p] * l20[p] - l21[p] * l21[p]);
        yr[p][0] = rhs[0] * l00[p];
        yr[p][1] = (rhs[1] - l10[p] * yr[p][0]) * l11[p];
        yr[p][2] = (rhs[2] - l20[p] * yr[p][0] - l21[p] * yr[p][1]) * l22[p];
#pragma unroll
        for (int j = 0; j < 6; ++j) {
          F[p][0][j] *= l00[p];
          F[p][1][j] = (F[p][1][j] - l10[p] * F[p][0][j]) * l11[p];
          F[p][2][j] = (F[p][2][j] - l20[p] * F[p][0][j] - l21[p] * F[p][1][j]) * l22[p];
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) {
#pragma unroll
          for (int j = 0; j <= i; ++j)
            S[i * (i + 1) / 2 + j] -= F[p][0][i] * F[p][0][j] + F[p][1][i] * F[p][1][j] + F[p][2][i] * F[p][2][j];
          y[i] -= F[p][0][i] * yr[p][0] + F[p][1][i] * yr[p][1] + F[p][2][i] * yr[p][2];
        }
      }
      // the legs' composite inertia in spatial form: n = I a + h x b, f = m b - h x a
      S[0] += Ic[0]; S[2] += Ic[1]; S[5] += Ic[2]; S[1] += Ic[3]; S[3] += Ic[4]; S[4] += Ic[5];
      S[9] += mc; S[14] += mc; S[20] += mc;
      S[7] += hc[2]; S[8] -= hc[1]; S[10] -= hc[2]; S[12] += hc[0]; S[15] += hc[1]; S[16] -= hc[0];
#pragma unroll
      for (int o = 1; o < TL; o <<= 1) {
#pragma unroll
        for (int i = 0; i < 21; ++i) S[i] += __shfl_xor_sync(0xffffffffu, S[i], o);
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] += __shfl_xor_sync(0xffffffffu, y[i], o);
      }
      {  // the base body itself
        R m5, h5[3], I5[6];
        body_inertia(P, 5, m5, h5, I5);
        S[0] += I5[0]; S[2] += I5[1]; S[5] += I5[2]; S[1] += I5[3]; S[3] += I5[4]; S[4] += I5[5];
        S[9] += m5; S[14] += m5; S[20] += m5;
        S[7] += h5[2]; S[8] -= h5[1]; S[10] -= h5[2]; S[12] += h5[0]; S[15] += h5[1]; S[16] -= h5[0];
#pragma unroll
        for (int k = 0; k < 3; ++k) { y[k] -= nb[k]; y[3 + k] -= fb[k]; }
      }
      // a_b: Cholesky of the 6 x 6 (reciprocal diagonal), two triangular solves
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        R d = S[j * (j + 1) / 2 + j];
#pragma unroll
        for (int k = 0; k < j; ++k) d -= S[j * (j + 1) / 2 + k] * S[j * (j + 1) / 2 + k];
        const R rd = rsqrt_(d);
        S[j * (j + 1) / 2 + j] = rd;
#pragma unroll
        for (int i = j + 1; i < 6; ++i) {
          R t = S[i * (i + 1) / 2 + j];
#pragma unroll
          for (int k = 0; k < j; ++k) t -= S[i * (i + 1) / 2 + k] * S[j * (j + 1) / 2 + k];
          S[i * (i + 1) / 2 + j] = t * rd;
        }
      }
#pragma unroll
      for (int i = 0; i < 6; ++i) {
#pragma unroll
        for (int k = 0; k < i; ++k) y[i] -= S[i * (i + 1) / 2 + k] * y[k];
        y[i] *= S[i * (i + 1) / 2 + i];
      }
#pragma unroll
      for (int i = 5; i >= 0; --i) {
#pragma unroll
        for (int k = i + 1; k < 6; ++k) y[i] -= S[k * (k + 1) / 2 + i] * y[k];
        y[i] *= S[i * (i + 1) / 2 + i];
      }
      // joint accelerations: the legs' by back substitution, the base's from its axes
#pragma unroll
      for (int p = 0; p < LP; ++p) {
        R z[3], a[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          z[k] = yr[p][k];
#pragma unroll
          for (int j = 0; j < 6; ++j) z[k] -= F[p][k][j] * y[j];
        }
        a[2] = z[2] * l22[p];
        a[1] = (z[1] - l21[p] * a[2]) * l11[p];
        a[0] = (z[0] - l10[p] * a[1] - l20[p] * a[2]) * l00[p];
        semi_implicit2<R, 3>(lq[p], lql[p], lv[p], lvl[p], a, h);
        if (prims && on) {
          Prim<R>& pr = *reinterpret_cast<Prim<R>*>(prims + (size_t)st * kPrimStride<R>);
#pragma unroll
          for (int k = 0; k < 3; ++k) pr.qdd[6 + 3 * (sub * LP + p) + k] = a[k];
        }
      }
      R ba[6];
      mtv(E0, y + 3, ba);
      ba[3] = (sx * y[1] + cx * y[2]) / cy;
      ba[4] = cx * y[1] - sx * y[2];
      ba[5] = y[0] + sy * ba[3];
      semi_implicit2<R, 6>(bq, bql, bv, bvl, ba, h);
      if (prims && on && sub == 0) {
        Prim<R>& pr = *reinterpret_cast<Prim<R>*>(prims + (size_t)st * kPrimStride<R>);
#pragma unroll
        for (int i = 0; i < 6; ++i) { pr.qdd[i] = ba[i]; pr.tin[i] = R(0); }
      }
    }
    if (on) {
      if (sub == 0)
#pragma unroll
        for (int i = 0; i < 6; ++i) { slot[i] = bq[i]; slot[n + i] = bql[i]; slot[N + i] = bv[i]; slot[n + N + i] = bvl[i]; }
#pragma unroll
      for (int p = 0; p < LP; ++p)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const int j = 3 * (sub * LP + p) + k;
          slot[6 + j] = lq[p][k]; slot[n + 6 + j] = lql[p][k];
          slot[N + 6 + j] = lv[p][k]; slot[n + N + 6 + j] = lvl[p][k];
        }
    }
  }

  template <class R, int G>
  TO_DEV static R cost_step_team(const ParamsT<R>& P, const Group<G>& g, bool mine, R* xh, R* xl, const R* u, R* scratch) {
    static_assert(kGroupStep<G> && (G == 32 || G == 64), "16 teams of 2 or 4 lanes");
    constexpr int TL = G / kStepSlots;
    R* flag = scratch + kStepSlots * kTeamSlot;
    R l = R(0);
    if (mine) {
      R* s = scratch + g.lane * kTeamSlot;
      l = running_cost(P, xh, u);
#pragma unroll
      for (int i = 0; i < n; ++i) { s[i] = xh[i]; s[n + i] = xl[i]; }
#pragma unroll
      for (int i = 0; i < m; ++i) s[2 * n + i] = u[i];
    }
    if (g.lane < kStepSlots) flag[g.lane] = mine ? R(1) : R(0);
    g.sync();
    const int cand = g.lane / TL, sub = g.lane % TL;
    const bool on = flag[cand] != R(0);
    R* slot = scratch + cand * kTeamSlot;
    // a warp's teams run together (their sums are shuffles)
    if (__any_sync(0xffffffffu, on)) team_steps<R, G>(P, on, slot, sub, nullptr);
    g.sync();
    if (mine) {
      const R* s = scratch + g.lane * kTeamSlot;
#pragma unroll
      for (int i = 0; i < n; ++i) { xh[i] = s[i]; xl[i] = s[n + i]; }
    }
    return l;
  }

  // cost_step2 shared by a candidate lane and its partner (kGroupStep): every
  // lane of the group calls it, mine on the candidate lanes (all < kStepSlots);
  // returns the running cost on those.  Two group barriers per substep.  A base
  // that is a free body goes to the teams; this path serves the others.
  template <class R, int G>
  TO_DEV static R cost_step_group(const ParamsT<R>& P, const Group<G>& g, bool mine, R* xh, R* xl, const R* u,
                                  R* scratch) {
    if (P.free_base) return cost_step_team(P, g, mine, xh, xl, u, scratch);   // uniform over the grid
    static_assert(kGroupStep<G>, "a partner lane in the group's other half");
    constexpr int H = G / 2;                  // candidate c's partner is lane c + H
    static_assert(H >= kStepSlots, "a partner for every candidate slot");
    const int c = g.lane;
    const int slot = c < H ? c : c - H;
    R* sq = scratch + slot * kStepSlot;       // q of the candidate's substep
    R* sL = sq + N;                           // the factor of M(q)
    R* flag = scratch + kStepSlots * kStepSlot;
    R l = R(0), tau[N];
    if (mine) {
      l = running_cost(P, xh, u);
#pragma unroll
      for (int i = 0; i < N; ++i) tau[i] = i < A0 ? R(0) : u[i - A0];
    }
    if (c < kStepSlots) flag[c] = mine ? R(1) : R(0);
    const R h = P.dt / (R)P.n_sub;
    for (int s = 0; s < P.n_sub; ++s) {
      if (mine)
#pragma unroll
        for (int i = 0; i < N; ++i) sq[i] = xh[i];
      g.sync();
      R hb[N];
      if (mine) {
        R E[N][9], r[N][3];
        rnea<R, R>(P, xh, xh + N, hb, E, r);
      } else if (c >= H && slot < kStepSlots && flag[slot] != R(0)) {
        mass_chol_mem(P, sq, sL);
      }
      g.sync();
      if (mine) {
        R rhs[N], qdd[N];
#pragma unroll
        for (int i = 0; i < N; ++i) rhs[i] = tau[i] - hb[i];
        chol_solve(P, sL, rhs, qdd);
        semi_implicit2<R, N>(xh, xl, xh + N, xl + N, qdd, h);
      }
    }
    return l;
  }

  template <class R>
  TO_DEV static R terminal_cost(const ParamsT<R>& P, const R* x) {
    R l = 0;
    if (KIND == RK_ARM7) {
      R ee[3];
      ee_world(P, x, ee);
      for (int k = 0; k < 3; ++k) { const R d = ee[k] - P.tgt[k]; l += P.wee * d * d; }
#pragma unroll
      for (int j = 0; j < N; ++j) l += P.wvT * x[N + j] * x[N + j];
    } else {
      const R dz = x[2] - P.znom, dv = x[N] - P.vxt;
      l = P.tscale * (P.wz * dz * dz + P.wrpy * (x[3] * x[3] + x[4] * x[4] + x[5] * x[5]) + P.wvx * dv * dv);
    }
    return l;
  }

  // Separable running costs: the clipped Hessians are diagonal, max(d, eps), and
  // the same at every knot, so they are set once a pass; a knot's gradients are
  // linear in x and u.  By the lanes of the group.
  template <class R>
  TO_DEV static void running_consts(const ParamsT<R>& P, int lane, int G, R eps, R* lxx, R* lx, R* luu) {
    const R w2 = R(2) * P.wtau;
    for (int e = lane; e < n * n; e += G) {
      const int i = e / n;
      R d = R(0);
      bool cost = false;
      if (KIND == RK_ARM7) {
        cost = i >= N;
        d = R(2) * P.wv;
      } else {
        cost = i == 2 || (i >= 3 && i < 6) || i == N;
        d = R(2) * (i == 2 ? P.wz : i == N ? P.wvx : P.wrpy);
      }
      lxx[e] = i != e % n ? R(0) : cost ? (d > eps ? d : eps) : clip0(eps);
    }
    for (int e = lane; e < m * m; e += G) luu[e] = e / m != e % m ? R(0) : (w2 > eps ? w2 : eps);
    for (int e = lane; e < n; e += G) lx[e] = R(0);
  }
  template <class R, int G>
  TO_DEV static void running_grads(const ParamsT<R>& P, int lane, const R* x, const R* u, R* lx, R* lu) {
    for (int i = lane; i < m; i += G) lu[i] = (R(2) * P.wtau) * u[i];
    if (KIND == RK_ARM7) {
      for (int i = lane; i < N; i += G) lx[N + i] = (R(2) * P.wv) * x[N + i];
    } else {
      if (lane == 2) lx[2] = (R(2) * P.wz) * (x[2] - P.znom);
      else if (lane >= 3 && lane < 6) lx[lane] = (R(2) * P.wrpy) * x[lane];
      else if (lane == 6) lx[N] = (R(2) * P.wvx) * (x[N] - P.vxt);
    }
  }

  // Terminal-cost derivatives (V and v in shared memory), by a group of whole
  // warps; on is uniform over it.  The arm's end-effector term goes through
  // forward kinematics: gradient and exact Hessian by nested dual numbers, one
  // pair of joints per lane, then the q-block is eigen-clipped by the lanes
  // together (scratch: 2 N^2 elements).  On one lane the 28 pairs and the Jacobi
  // sweeps are a third of a solve: 7-DoF arm B=304 float64, T 10..20, 2 iterations,
  // V_x 15.3 ms there, 9.0 here; B=2048 float32, T 50..200, 2 iterations 27.5 and
  // 17.2 ms (the same bits; 582 and 343 KB of code).
  template <class R, int G>
  TO_DEV static void terminal_group(const ParamsT<R>& P, const Group<G>& g, bool on, const R* x, R eps, R* lxx, R* lx,
                                    R* scratch) {
    if (on) {
      for (int e = g.lane; e < n * n; e += G) lxx[e] = R(0);
      for (int e = g.lane; e < n; e += G) lx[e] = R(0);
    }
    g.sync();
    if constexpr (KIND == RK_ARM7) {
      static_assert(G == 32 && N * (N + 1) / 2 <= G, "a lane per pair of joints");
      R* A = scratch;
      if (on && g.lane < N * (N + 1) / 2) {
        typedef Dl<Dl<R>> H;
        int a = 0, b = g.lane;                        // pair (a, b), a <= b
        while (b >= N - a) { b -= N - a; ++a; }
        b += a;
        H q[N];
#pragma unroll
        for (int k = 0; k < N; ++k) q[k] = H(Dl<R>(x[k], k == a ? R(1) : R(0)), Dl<R>(k == b ? R(1) : R(0), R(0)));
        H ee[3];
        ee_world(P, q, ee);
        H l(Dl<R>(R(0)));
        const H wee(Dl<R>(P.wee));
        for (int k = 0; k < 3; ++k) {
          const H d = ee[k] - H(Dl<R>(P.tgt[k]));
          l = l + wee * (d * d);
        }
        A[a * N + b] = l.d.d;
        A[b * N + a] = l.d.d;
        if (a == b) lx[a] = l.v.d;
      }
      g.sync();
      eigclip_warp<R, N>(A, A + N * N, eps, g.lane, on);
      if (on) {
        for (int e = g.lane; e < N * N; e += G) lxx[(e / N) * n + e % N] = A[e];
        const R v2 = R(2) * P.wvT;
        if (g.lane < N) {
          lx[N + g.lane] = v2 * x[N + g.lane];
          lxx[(N + g.lane) * n + N + g.lane] = v2 > eps ? v2 : eps;
        }
      }
    } else if (on) {
      const R s = P.tscale;
      const R z2 = R(2) * P.wz * s, r2 = R(2) * P.wrpy * s, x2 = R(2) * P.wvx * s;
      for (int i = g.lane; i < n; i += G) {
        const R d = i == 2 ? z2 : i >= 3 && i < 6 ? r2 : i == N ? x2 : R(0);
        lxx[i * n + i] = i == 2 || (i >= 3 && i < 6) || i == N ? (d > eps ? d : eps) : clip0(eps);
        if (i == 2) lx[i] = z2 * (x[2] - P.znom);
        else if (i >= 3 && i < 6) lx[i] = r2 * x[i];
        else if (i == N) lx[i] = x2 * (x[N] - P.vxt);
      }
    }
  }

  // ---- group-shared primal of one substep and the per-lane tangent pass ----
  static constexpr int NF = (KIND == RK_QUAD) ? 4 : 1;
  // Per-body quantities of the Newton-Euler pass at (q, qd, qdd), the mass
  // matrix factor and the contact terms: computed once per substep by one
  // lane into shared memory, read by every tangent lane.
  template <class R>
  struct Prim {
    R q[N], qd[N], qdd[N], tau[N], tin[N];
    R L[N * N];
    R E[N][9], r[N][3];
    R vw[N][3], vv[N][3];       // body velocity
    R Epw[N][3], Ept[N][3];     // E pw and E (pv - r x pw): the parent's velocity in body coordinates
    R Epa[N][3], Epb[N][3];     // E paw and E (pav - r x paw): the same for the acceleration
    R aw[N][3];                 // body angular acceleration
    R hn[N][3], hf[N][3];       // I v
    R fn[N][3], ff[N][3];       // body force as sent to the parent (children and contact included)
    R E0[KIND == RK_QUAD ? N : 1][9], p0[KIND == RK_QUAD ? N : 1][3];
    R wpt[NF][3], F[NF][3], vb[NF][3], vwld[NF][3], gate[NF];
  };
  // Knot-parallel derivatives (both trees): before each backward pass every
  // lane runs the substep primal chains of its own knots (primal_knot; a
  // free quadruped's group shares them, primals_group) and stores each
  // substep's Prim in a per-knot global scratch; inside the
  // backward pass the group stages those Prims into shared memory
  // (cp.async, one substep ahead) and every direction lane runs its tangent
  // pass at once (derivs_staged).  No lane waits for a primal.
  static constexpr bool kKnotParallel = true;
  static constexpr bool kStoredDerivs = false;
  static constexpr bool kGainDerivs = false;
  static constexpr bool kDeferCost = false;
  // elements per stored substep primal (a whole number of 16-byte chunks)
  template <class R> static constexpr int kPrimStride = (int)(((sizeof(Prim<R>) + 15) / 16 * 16) / sizeof(R));

  // Line search of the quadruped's groups: every workload's base is a free body,
  // whose candidates step by teams of lanes (cost_step_team).  For any other base,
  // candidate lane c < kStepSlots steps its rollout with lane c + G/2 as its
  // partner (the other warp of a 64-lane group, the other half-warp of a 32-lane
  // one), which forms and factors the mass matrix while lane c runs the bias
  // Newton-Euler pass; per candidate the scratch holds its substep's q and the
  // factor (a team's slot is smaller).  The 7-DoF arm's candidates step alone: its
  // 7-body mass matrix is cheap, and the partner split measured 2 % slower there in
  // mixed mode.
  template <int G> static constexpr bool kGroupStep = (KIND == RK_QUAD) && G >= 32;
  static constexpr int kStepSlots = 16, kStepSlot = N + N * N;
  // the group's shared-memory scratch (the solver reserves it in its work
  // area): the derivative primal, or the line search's per-candidate slots
  template <class R>
  struct Scratch {
    static constexpr int prim = 2 * kPrimStride<R>;   // the staged substep primals, double-buffered
    static constexpr int step = KIND == RK_QUAD ? kStepSlots * kStepSlot + kStepSlots : 0;
    static_assert(KIND != RK_QUAD || kTeamSlot <= kStepSlot, "the teams' slots fit the partners'");
    static constexpr int elems = prim > step ? prim : step;
  };

  // y -= s (e_ax x z): the change of E x under dq about joint axis ax
  template <class S> TO_DEV static void rot_tangent(int ax, S s, const S* z, S* y) {
    if (ax == 0) { y[1] += s * z[2]; y[2] -= s * z[1]; }
    else if (ax == 1) { y[0] -= s * z[2]; y[2] += s * z[0]; }
    else { y[0] += s * z[1]; y[1] -= s * z[0]; }
  }
  // A substep's primal for the derivative lanes comes in two halves around
  // the solve for qdd, so that the joint transforms, the velocities, the
  // world poses and the contact forces are evaluated once (the tangent pass
  // reads them all from pr):
  // bias_store (one lane): those quantities, I v, and the inverse dynamics at
  // qdd = 0 (gravity, velocity products, contact), i.e. the bias torques h.
  // The joint transforms are also left in Ej and rj.
  template <class R>
  TO_DEV static void bias_store(const ParamsT<R>& P, Prim<R>& pr, const R* q, const R* qd, R* h, R (*Ej)[9],
                                R (*rj)[3]) {
    R aw[N][3], av[N][3], fn[N][3], ff[N][3];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int pa = parent(i), jt = jtype(i);
      R* E = Ej[i];
      R* r = rj[i];
      joint_transform(P, i, q[i], E, r);
#pragma unroll
      for (int k = 0; k < 9; ++k) pr.E[i][k] = E[k];
#pragma unroll
      for (int k = 0; k < 3; ++k) pr.r[i][k] = r[k];
      const int pb = pa < 0 ? 0 : pa;
      R Epw[3], Ept[3], vw[3], vv[3], hn[3], hf[3], pw[3], pv[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) { pw[k] = pr.vw[pb][k]; pv[k] = pr.vv[pb][k]; }
      body_bias(P, i, E, r, qd[i], pw, pv, aw[pb], av[pb], Epw, Ept, vw, vv, aw[i], av[i], hn, hf, fn[i], ff[i]);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        pr.Epw[i][k] = Epw[k]; pr.Ept[i][k] = Ept[k];
        pr.vw[i][k] = vw[k]; pr.vv[i][k] = vv[k];
        pr.hn[i][k] = hn[k]; pr.hf[i][k] = hf[k];
      }
      if (KIND == RK_QUAD) {
        if (pa < 0) {
#pragma unroll
          for (int k = 0; k < 9; ++k) pr.E0[i][k] = E[k];
#pragma unroll
          for (int k = 0; k < 3; ++k) pr.p0[i][k] = r[k];
        } else {
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) pr.E0[i][a * 3 + b] = e_row(jt, E, pr.E0[pa], a, b);
          R wr[3];
          mtv(pr.E0[pa], r, wr);
#pragma unroll
          for (int k = 0; k < 3; ++k) pr.p0[i][k] = pr.p0[pa][k] + wr[k];
        }
      }
    }
    if (KIND == RK_QUAD) {
#pragma unroll
      for (int ft = 0; ft < kFeet; ++ft) {
        const int bi = foot_body(ft);
        const R pt[3] = {P.foot_pt[ft][0], P.foot_pt[ft][1], P.foot_pt[ft][2]};
        R wpt[3], vb[3], vwld[3], wxp[3];
        mtv(pr.E0[bi], pt, wpt);
        cross(pr.vw[bi], pt, wxp);
#pragma unroll
        for (int k = 0; k < 3; ++k) vb[k] = pr.vv[bi][k] + wxp[k];
        mtv(pr.E0[bi], vb, vwld);
        const R bz = P.beta * (pr.p0[bi][2] + wpt[2]);
        R sp, gate;
        if (bz >= R(0)) {
          const R e = dexp(-bz);
          sp = (R(1) / P.beta) * dlog1p(e);
          gate = e / (R(1) + e);
        } else {
          const R e = dexp(bz);
          sp = (R(1) / P.beta) * (dlog1p(e) - bz);
          gate = R(1) / (R(1) + e);
        }
        R F[3];
        F[0] = -(P.dc * (gate * vwld[0]));
        F[1] = -(P.dc * (gate * vwld[1]));
        F[2] = P.kc * sp - P.dc * (gate * vwld[2]);
        pr.gate[ft] = gate;
#pragma unroll
        for (int k = 0; k < 3; ++k) { pr.wpt[ft][k] = wpt[k]; pr.vb[ft][k] = vb[k]; pr.vwld[ft][k] = vwld[k]; pr.F[ft][k] = F[k]; }
        R mw[3], mb[3], fb[3];
        cross(wpt, F, mw);
        mv(pr.E0[bi], mw, mb);
        mv(pr.E0[bi], F, fb);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[bi][k] -= mb[k]; ff[bi][k] -= fb[k]; }
      }
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int jt = jtype(i);
      h[i] = jt <= 2 ? fn[i][jt] : ff[i][jt - 3];
      const int pa = parent(i);
      if (pa >= 0) {
        R en[3], ef[3], rf[3];
        jmtv(jt, pr.E[i], fn[i], en);
        jmtv(jt, pr.E[i], ff[i], ef);
        cross(pr.r[i], ef, rf);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[pa][k] += en[k] + rf[k]; ff[pa][k] += ef[k]; }
      }
    }
  }

  // accel_store (one lane, after the solve put qdd in pr): the accelerations
  // with qdd, the parents' acceleration transforms, and the body forces as
  // sent to the parent (children and contact included), from the stored
  // transforms, velocities, I v and contact forces.
  template <class R>
  TO_DEV static void accel_store(const ParamsT<R>& P, Prim<R>& pr) {
    R av[N][3], fn[N][3], ff[N][3];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int pa = parent(i), jt = jtype(i);
      const R* E = pr.E[i];
      const int ax = jt <= 2 ? jt : jt - 3;
      R t[3], Epa[3], Epb[3], vw[3], vv[3], hn[3], hf[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) { vw[k] = pr.vw[i][k]; vv[k] = pr.vv[i][k]; hn[k] = pr.hn[i][k]; hf[k] = pr.hf[i][k]; }
      if (pa < 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { Epa[k] = R(0); t[k] = -P.g[k]; }
      } else {
        R paw[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) { paw[k] = pr.aw[pa][k]; t[k] = av[pa][k]; }
        cross_sub(pr.r[i], paw, t);
        jmv(jt, E, paw, Epa);
      }
      jmv(jt, E, t, Epb);
      R aw[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) { pr.Epa[i][k] = Epa[k]; pr.Epb[i][k] = Epb[k]; aw[k] = Epa[k]; av[i][k] = Epb[k]; }
      if (pa >= 0) {
        if (jt <= 2) {
          axis_acc(vw, ax, pr.qd[i], aw);
          axis_acc(vv, ax, pr.qd[i], av[i]);
        } else {
          axis_acc(vw, ax, pr.qd[i], av[i]);
        }
      }
      if (jt <= 2) aw[jt] += pr.qdd[i]; else av[i][jt - 3] += pr.qdd[i];
#pragma unroll
      for (int k = 0; k < 3; ++k) pr.aw[i][k] = aw[k];
      if (massless(P, i)) {
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[i][k] = R(0); ff[i][k] = R(0); }
        continue;
      }
      R In[3], If[3];
      inertia_mul(P, i, aw, av[i], In, If);
#pragma unroll
      for (int k = 0; k < 3; ++k) { fn[i][k] = In[k]; ff[i][k] = If[k]; }
      cross_acc(vw, hn, fn[i]);
      cross_acc(vv, hf, fn[i]);
      cross_acc(vw, hf, ff[i]);
    }
    if (KIND == RK_QUAD) {
#pragma unroll
      for (int ft = 0; ft < kFeet; ++ft) {
        const int bi = foot_body(ft);
        R mw[3], mb[3], fb[3];
        cross(pr.wpt[ft], pr.F[ft], mw);
        mv(pr.E0[bi], mw, mb);
        mv(pr.E0[bi], pr.F[ft], fb);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[bi][k] -= mb[k]; ff[bi][k] -= fb[k]; }
      }
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      const int jt = jtype(i);
      pr.tau[i] = jt <= 2 ? fn[i][jt] : ff[i][jt - 3];
#pragma unroll
      for (int k = 0; k < 3; ++k) { pr.fn[i][k] = fn[i][k]; pr.ff[i][k] = ff[i][k]; }
      const int pa = parent(i);
      if (pa >= 0) {
        R en[3], ef[3], rf[3];
        jmtv(jt, pr.E[i], fn[i], en);
        jmtv(jt, pr.E[i], ff[i], ef);
        cross(pr.r[i], ef, rf);
#pragma unroll
        for (int k = 0; k < 3; ++k) { fn[pa][k] += en[k] + rf[k]; ff[pa][k] += ef[k]; }
      }
    }
  }

  // Directional derivative of the inverse dynamics along (dq, dqd) at the
  // stored substep (qdd held fixed): the product rule through the forward
  // recursion (velocities, accelerations, body forces, world poses and
  // contact) and the backward force recursion.  Only the tangents live in
  // the lane's own arrays.
  // One body of the forward recursion: its tangents and its force's from its
  // parent's (pa < 0: none).
  template <class R>
  TO_DEV static void tan_body(const ParamsT<R>& P, const Prim<R>& pr, int jt, int i, int pa, R dq, R dqd, const R* pdvw,
                              const R* pdvv, const R* pdaw, const R* pdav, R* dvw, R* dvv, R* daw, R* dav, R* dfn, R* dff) {
    const bool rev = jt <= 2;
    const int ax = rev ? jt : jt - 3;
    const R* E = pr.E[i];
    const R* r = pr.r[i];
    R t[3];
    if (pa < 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) { dvw[k] = R(0); dvv[k] = R(0); daw[k] = R(0); dav[k] = R(0); }
    } else {
      R pw[3], paw[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) { pw[k] = pr.vw[pa][k]; paw[k] = pr.aw[pa][k]; }
      // velocity
      jmv(jt, E, pdvw, dvw);
      if (rev) rot_tangent(ax, dq, pr.Epw[i], dvw);
#pragma unroll
      for (int k = 0; k < 3; ++k) t[k] = pdvv[k];
      cross_sub(r, pdvw, t);
      if (!rev) axis_acc(pw, ax, dq, t);
      jmv(jt, E, t, dvv);
      if (rev) rot_tangent(ax, dq, pr.Ept[i], dvv);
      // acceleration (qdd fixed)
      jmv(jt, E, pdaw, daw);
      if (rev) rot_tangent(ax, dq, pr.Epa[i], daw);
#pragma unroll
      for (int k = 0; k < 3; ++k) t[k] = pdav[k];
      cross_sub(r, pdaw, t);
      if (!rev) axis_acc(paw, ax, dq, t);
      jmv(jt, E, t, dav);
    }
    if (rev) rot_tangent(ax, dq, pr.Epb[i], dav);
    if (rev) dvw[ax] += dqd; else dvv[ax] += dqd;
    if (pa >= 0) {
      if (rev) {
        axis_acc(dvw, ax, pr.qd[i], daw);
        axis_acc(pr.vw[i], ax, dqd, daw);
        axis_acc(dvv, ax, pr.qd[i], dav);
        axis_acc(pr.vv[i], ax, dqd, dav);
      } else {
        axis_acc(dvw, ax, pr.qd[i], dav);
        axis_acc(pr.vw[i], ax, dqd, dav);
      }
    }
    // body force
    if (massless(P, i)) {
#pragma unroll
      for (int k = 0; k < 3; ++k) { dfn[k] = R(0); dff[k] = R(0); }
      return;
    }
    R dhn[3], dhf[3];
    inertia_mul(P, i, daw, dav, dfn, dff);
    inertia_mul(P, i, dvw, dvv, dhn, dhf);
    cross_acc(dvw, pr.hn[i], dfn);
    cross_acc(pr.vw[i], dhn, dfn);
    cross_acc(dvv, pr.hf[i], dfn);
    cross_acc(pr.vv[i], dhf, dfn);
    cross_acc(dvw, pr.hf[i], dff);
    cross_acc(pr.vw[i], dhf, dff);
  }
  // its world pose's: dE0_i = dE_i E0_p + E_i dE0_p, dp0_i = dp0_p + dE0_p^T r + E0_p^T dr
  template <class R>
  TO_DEV static void tan_pose(const Prim<R>& pr, int jt, int i, int pa, R dq, const R* pdE0, const R* pdp0, R* dE0, R* dp0) {
    const bool rev = jt <= 2;
    const int ax = rev ? jt : jt - 3;
    if (pa < 0) {
#pragma unroll
      for (int k = 0; k < 9; ++k) dE0[k] = R(0);
#pragma unroll
      for (int k = 0; k < 3; ++k) dp0[k] = !rev && k == ax ? dq : R(0);
    } else {
      const R* E = pr.E[i];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) dE0[a * 3 + b] = e_row(jt, E, pdE0, a, b);
      R w1[3];
      mtv(pdE0, pr.r[i], w1);
#pragma unroll
      for (int k = 0; k < 3; ++k) dp0[k] = pdp0[k] + w1[k];
      if (!rev)
#pragma unroll
        for (int k = 0; k < 3; ++k) dp0[k] += pr.E0[pa][ax * 3 + k] * dq;
    }
    if (rev) {
      // column b of E0_i turns with the joint: -dq (e_ax x column)
      const R* E0 = pr.E0[i];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const R col[3] = {E0[0 * 3 + b], E0[1 * 3 + b], E0[2 * 3 + b]};
        R y[3] = {dE0[0 * 3 + b], dE0[1 * 3 + b], dE0[2 * 3 + b]};
        rot_tangent(ax, dq, col, y);
#pragma unroll
        for (int a = 0; a < 3; ++a) dE0[a * 3 + b] = y[a];
      }
    }
  }
  // the contact force of foot ft on body bi
  template <class R>
  TO_DEV static void tan_contact(const ParamsT<R>& P, const Prim<R>& pr, int ft, int bi, const R* dE0, const R* dp0,
                                 const R* dvw, const R* dvv, R* dfn, R* dff) {
    const R pt[3] = {P.foot_pt[ft][0], P.foot_pt[ft][1], P.foot_pt[ft][2]};
    const R* E0 = pr.E0[bi];
    R dwpt[3], dvb[3], dvwld[3], w1[3];
    mtv(dE0, pt, dwpt);
    const R dz = dp0[2] + dwpt[2];
    cross(dvw, pt, w1);
#pragma unroll
    for (int k = 0; k < 3; ++k) dvb[k] = dvv[k] + w1[k];
    mtv(dE0, pr.vb[ft], dvwld);
    mtv(E0, dvb, w1);
#pragma unroll
    for (int k = 0; k < 3; ++k) dvwld[k] += w1[k];
    const R gate = pr.gate[ft];
    const R dgate = -P.beta * gate * (R(1) - gate) * dz;
    const R dsp = -gate * dz;
    R dF[3];
    dF[0] = -P.dc * (dgate * pr.vwld[ft][0] + gate * dvwld[0]);
    dF[1] = -P.dc * (dgate * pr.vwld[ft][1] + gate * dvwld[1]);
    dF[2] = P.kc * dsp - P.dc * (dgate * pr.vwld[ft][2] + gate * dvwld[2]);
    R mw[3], dmw[3] = {R(0), R(0), R(0)}, dmb[3], dfb[3];
    cross(pr.wpt[ft], pr.F[ft], mw);
    cross_acc(dwpt, pr.F[ft], dmw);
    cross_acc(pr.wpt[ft], dF, dmw);
    mv(dE0, mw, dmb);
    mv(E0, dmw, w1);
#pragma unroll
    for (int k = 0; k < 3; ++k) dmb[k] += w1[k];
    mv(dE0, pr.F[ft], dfb);
    mv(E0, dF, w1);
#pragma unroll
    for (int k = 0; k < 3; ++k) { dfn[k] -= dmb[k]; dff[k] -= dfb[k] + w1[k]; }
  }
  // a body's force tangent added to its parent's:
  // d(E^T y) = E^T dy + dq E^T (e_ax x y) for a revolute joint
  template <class R>
  TO_DEV static void tan_up(const Prim<R>& pr, int jt, int i, R dq, const R* dfn, const R* dff, R* pfn, R* pff) {
    const bool rev = jt <= 2;
    const int ax = rev ? jt : jt - 3;
    const R* E = pr.E[i];
    R yn[3], yf[3], den[3], def[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) { yn[k] = dfn[k]; yf[k] = dff[k]; }
    if (rev) {
      rot_tangent(ax, -dq, pr.fn[i], yn);
      rot_tangent(ax, -dq, pr.ff[i], yf);
    }
    jmtv(jt, E, yn, den);
    jmtv(jt, E, yf, def);
    if (!rev) {
      R ef[3];
      jmtv(jt, E, pr.ff[i], ef);
      axis_acc(ef, ax, -dq, den);
    }
    cross_acc(pr.r[i], def, den);
#pragma unroll
    for (int k = 0; k < 3; ++k) { pfn[k] += den[k]; pff[k] += def[k]; }
  }

  template <class R>
  TO_DEV static void rnea_tangent(const ParamsT<R>& P, const Prim<R>& pr, const R* dq, const R* dqd, R* dtau) {
    constexpr int NB = KIND == RK_QUAD ? 6 : N;     // bodies of the chain that the pass unrolls
    R dvw[NB][3], dvv[NB][3], daw[NB][3], dav[NB][3], dfn[NB][3], dff[NB][3];
    R dE0[KIND == RK_QUAD ? NB : 1][9], dp0[KIND == RK_QUAD ? NB : 1][3];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int pa = parent(i), pb = pa < 0 ? 0 : pa;
      tan_body(P, pr, jtype(i), i, pa, dq[i], dqd[i], dvw[pb], dvv[pb], daw[pb], dav[pb], dvw[i], dvv[i], daw[i], dav[i],
               dfn[i], dff[i]);
      if constexpr (KIND == RK_QUAD) tan_pose(pr, jtype(i), i, pa, dq[i], dE0[pb], dp0[pb], dE0[i], dp0[i]);
    }
    if constexpr (KIND == RK_QUAD) {
      // The legs one after another in a loop: the body index is data, so their
      // code is there once, and only one leg's tangents are live.  Unrolled, the
      // 18 bodies' arrays did not fit the registers and the warps waited for
      // their spills and for instructions: B=512 float32, T 4..8, 1 iteration, V_x
      // 7.8 -> 6.8 ms.
#pragma unroll 1
      for (int leg = 3; leg >= 0; --leg) {
        const int b = 6 + 3 * leg;
        auto pick = [&](const R* d, int k) { return leg == 0 ? d[6 + k] : leg == 1 ? d[9 + k] : leg == 2 ? d[12 + k] : d[15 + k]; };
        R lw[3][3], lv[3][3], la[3][3], lb[3][3], ln[3][3], lf[3][3], lE[9], lp[3], mE[9], mp[3], lq[3], lqd[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) { lq[k] = pick(dq, k); lqd[k] = pick(dqd, k); }
        tan_body(P, pr, 0, b, 5, lq[0], lqd[0], dvw[5], dvv[5], daw[5], dav[5], lw[0], lv[0], la[0], lb[0], ln[0], lf[0]);
        tan_pose(pr, 0, b, 5, lq[0], dE0[5], dp0[5], lE, lp);
        tan_body(P, pr, 1, b + 1, b, lq[1], lqd[1], lw[0], lv[0], la[0], lb[0], lw[1], lv[1], la[1], lb[1], ln[1], lf[1]);
        tan_pose(pr, 1, b + 1, b, lq[1], lE, lp, mE, mp);
        tan_body(P, pr, 1, b + 2, b + 1, lq[2], lqd[2], lw[1], lv[1], la[1], lb[1], lw[2], lv[2], la[2], lb[2], ln[2], lf[2]);
        tan_pose(pr, 1, b + 2, b + 1, lq[2], mE, mp, lE, lp);
        tan_contact(P, pr, leg, b + 2, lE, lp, lw[2], lv[2], ln[2], lf[2]);
        R t[3];
        t[2] = ln[2][1];
        tan_up(pr, 1, b + 2, lq[2], ln[2], lf[2], ln[1], lf[1]);
        t[1] = ln[1][1];
        tan_up(pr, 1, b + 1, lq[1], ln[1], lf[1], ln[0], lf[0]);
        t[0] = ln[0][0];
        tan_up(pr, 0, b, lq[0], ln[0], lf[0], dfn[5], dff[5]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int k = 0; k < 3; ++k) dtau[6 + 3 * j + k] = j == leg ? t[k] : dtau[6 + 3 * j + k];
      }
    }
#pragma unroll
    for (int i = NB - 1; i >= 0; --i) {
      const int jt = jtype(i), pa = parent(i);
      dtau[i] = jt <= 2 ? dfn[i][jt <= 2 ? jt : 0] : dff[i][jt <= 2 ? 0 : jt - 3];
      if (pa >= 0) tan_up(pr, jt, i, dq[i], dfn[i], dff[i], dfn[pa], dff[pa]);
    }
  }

  template <class R> TO_DEV static void store_factor(Prim<R>& pr, const R* L) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      pr.L[k * N + k] = L[k * N + k];
#pragma unroll
      for (int d = 1; d <= kDepthMax; ++d)
        if (d <= depth(k)) pr.L[k * N + anc(k, d)] = L[k * N + anc(k, d)];
    }
  }

  // The stored primals of knots 0..T-1 by the whole group (a quadruped whose
  // base is a free body): the substeps' states and accelerations by teams, 16
  // knots at a time, then every substep's Prim by a lane of its own.  On one
  // lane a knot's 10 substeps follow each other through 10 k instructions of
  // straight-line code, and a short horizon fills a few lanes: a third of a
  // solve.  B = 512 float32, 1 iteration with V_x: T = 4 to 8 6.60 -> 5.38 ms,
  // T = 1 (device) 1.45 -> 0.75, T = 17 7.55 -> 7.28, T = 40 to 50 the same
  // (21.8: the lanes were full).
  template <class R, int G, class Rec, class Out>
  TO_DEV static void primals_group(const ParamsT<R>& P, const Group<G>& g, int T, Rec rec, Out out, R* scratch) {
    const int cand = g.lane / (G / kStepSlots), sub = g.lane % (G / kStepSlots);
    for (int k0 = 0; k0 < T; k0 += kStepSlots) {
      if (g.lane < kStepSlots && k0 + g.lane < T) {
        const R* r = rec(k0 + g.lane);
        R* s = scratch + g.lane * kTeamSlot;
#pragma unroll
        for (int i = 0; i < n; ++i) { s[i] = r[i]; s[n + i] = R(0); }
#pragma unroll
        for (int i = 0; i < m; ++i) s[2 * n + i] = r[n + i];
      }
      g.sync();
      const bool on = k0 + cand < T;
      if (__any_sync(0xffffffffu, on))
        team_steps<R, G>(P, on, scratch + cand * kTeamSlot, sub, out(on ? k0 + cand : 0));
      g.sync();
    }
    for (int e = g.lane; e < T * P.n_sub; e += G) {
      Prim<R>& pr = *reinterpret_cast<Prim<R>*>(out(e / P.n_sub) + (size_t)(e % P.n_sub) * kPrimStride<R>);
      R q[N], qd[N], hb[N], L[N * N], E[N][9], r[N][3];
#pragma unroll
      for (int i = 0; i < N; ++i) { q[i] = pr.q[i]; qd[i] = pr.qd[i]; }
      bias_store(P, pr, q, qd, hb, E, r);
      mass_chol(P, q, L, E, r);
      store_factor(pr, L);
      accel_store(P, pr);
    }
  }

  // The substep primal chain of one knot on one lane, every substep's Prim
  // stored at out + s kPrimStride (global memory), the mass matrix formed and
  // factored on this lane: the 7-DoF arm's knots, and those of a quadruped whose
  // base is not a free body.
  template <class R>
  TO_DEV static void primal_knot(const ParamsT<R>& P, const R* x, const R* u, R* out) {
    R q[N], qd[N], tin[N];
#pragma unroll
    for (int i = 0; i < N; ++i) { q[i] = x[i]; qd[i] = x[N + i]; tin[i] = i < A0 ? R(0) : u[i - A0]; }
    const R h = P.dt / (R)P.n_sub;
    for (int s = 0; s < P.n_sub; ++s) {
      Prim<R>& pr = *reinterpret_cast<Prim<R>*>(out + (size_t)s * kPrimStride<R>);
      R hb[N], L[N * N], rhs[N], qdd[N], E[N][9], r[N][3];
      bias_store(P, pr, q, qd, hb, E, r);
      if constexpr (kKeepBits<R>) mass_chol(P, q, L);
      else mass_chol(P, q, L, E, r);
      store_factor(pr, L);
#pragma unroll
      for (int i = 0; i < N; ++i) rhs[i] = tin[i] - hb[i];
      chol_solve(P, L, rhs, qdd);
#pragma unroll
      for (int i = 0; i < N; ++i) { pr.q[i] = q[i]; pr.qd[i] = qd[i]; pr.tin[i] = tin[i]; pr.qdd[i] = qdd[i]; }
      accel_store(P, pr);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        qd[i] = qd[i] + h * qdd[i];
        q[i] = q[i] + h * qd[i];
      }
    }
  }

  // group copy of one stored Prim into shared memory, 16 bytes per cp.async
  template <class R, int G>
  TO_DEV static void stage_prim(const Group<G>& g, const R* src, R* dst) {
    constexpr int chunks = kPrimStride<R> * (int)sizeof(R) / 16;
    const char* s = reinterpret_cast<const char*>(src);
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    for (int c = g.lane; c < chunks; c += G)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d + 16u * c), "l"(s + 16 * c) : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }

  // Columns of [A | B] from the knot's stored substep primals (prims, global):
  // each substep's Prim is staged into shared memory one substep ahead while
  // the direction lanes run the tangent pass of the current one.  A group
  // narrower than the n + m directions takes them in passes of G (the
  // substeps are staged again for each pass).
  template <class R, int G>
  TO_DEV static void derivs_staged(const ParamsT<R>& P, const Group<G>& g, const R* x, const R* u, R* A, R* B, R* lx,
                                   R* lu, R* scratch, const R* prims) {
    for (int pass = 0; pass < (n + m + G - 1) / G; ++pass) {
    if (pass > 0) g.sync();   // every lane done with the staging buffers of the previous pass
    const int c = pass * G + g.lane;
    const bool dir = c < n + m;
    R dq[N], dqd[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      dq[i] = (c == i) ? R(1) : R(0);
      dqd[i] = (c == N + i) ? R(1) : R(0);
    }
    const R h = P.dt / (R)P.n_sub;
    stage_prim<R, G>(g, prims, scratch);
    for (int s = 0; s < P.n_sub; ++s) {
      asm volatile("cp.async.wait_all;\n" ::: "memory");
      g.sync();   // substep s staged by every lane; every lane done with the other buffer
      if (s + 1 < P.n_sub)
        stage_prim<R, G>(g, prims + (size_t)(s + 1) * kPrimStride<R>, scratch + ((s + 1) & 1) * kPrimStride<R>);
      const Prim<R>& pr = *reinterpret_cast<const Prim<R>*>(scratch + (s & 1) * kPrimStride<R>);
      if (dir) {
        R dtau[N], rhs[N], dqdd[N];
        rnea_tangent(P, pr, dq, dqd, dtau);
#pragma unroll
        for (int i = 0; i < N; ++i) rhs[i] = ((c >= n && i == A0 + (c - n)) ? R(1) : R(0)) - dtau[i];
        chol_solve(P, pr.L, rhs, dqdd);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          dqd[i] = dqd[i] + h * dqdd[i];
          dq[i] = dq[i] + h * dqd[i];
        }
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    if (dir) {
      if (c < n) {
#pragma unroll
        for (int i = 0; i < N; ++i) { A[i * n + c] = dq[i]; A[(N + i) * n + c] = dqd[i]; }
      } else {
#pragma unroll
        for (int i = 0; i < N; ++i) { B[i * m + (c - n)] = dq[i]; B[(N + i) * m + (c - n)] = dqd[i]; }
      }
    }
    }
    running_grads<R, G>(P, g.lane, x, u, lx, lu);
  }

};

typedef SysRigid<7, 0, RK_ARM7> SysArm7;
typedef SysRigid<18, 6, RK_QUAD> SysQuad;

}  // namespace to

namespace to {
template <class R> using RigidArm7P = RigidParams<R, 7>;
template <class R> using RigidQuadP = RigidParams<R, 18>;
}  // namespace to
