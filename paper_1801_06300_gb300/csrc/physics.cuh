// Euler physics for the DG kernels (Sec. 4.1, 4.4 of the paper), written once
// over the dimension D (2 or 3; D + 2 conservative variables) and over a scalar
// type S that is a real type (the residual), Tangent<T> (value + directional
// derivative: J v; through the reverse sweeps, second order) or Jet<T, N> (point Jacobians).
//
// Riemann flux: Roe's solver with square-root-density averages and no entropy
// fix, F~ = 1/2 (F_n(U_L) + F_n(U_R)) - 1/2 sum_k |lambda_k| alpha_k r_k.
// Ghost states: slip wall mirrors the normal velocity; the far field uses the
// one-dimensional Riemann invariants R+- = q_n +- 2 c / (gamma - 1), with R+
// from the interior unless its normal Mach number is <= -1, R- from the free
// stream unless it is >= 1, entropy and tangential velocity from the interior
// when the boundary normal velocity is >= 0, else from the free stream.
#pragma once
#include <cuda_runtime.h>

#define PCEXP_DEV __device__ __forceinline__

namespace pcexp {

// ---------------------------------------------------------------- tangent scalar
template <class T>
struct Tangent {
  T v, d;  // value and derivative along the direction
};

template <class T> PCEXP_DEV T val(T x) { return x; }
template <class T> PCEXP_DEV T val(Tangent<T> x) { return x.v; }

template <class T> PCEXP_DEV Tangent<T> operator+(Tangent<T> a, Tangent<T> b) { return {a.v + b.v, a.d + b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator-(Tangent<T> a, Tangent<T> b) { return {a.v - b.v, a.d - b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator-(Tangent<T> a) { return {-a.v, -a.d}; }
template <class T> PCEXP_DEV Tangent<T> operator*(Tangent<T> a, Tangent<T> b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator/(Tangent<T> a, Tangent<T> b) {
  T q = a.v / b.v;
  return {q, (a.d - q * b.d) / b.v};
}
template <class T> PCEXP_DEV Tangent<T> operator+(Tangent<T> a, T b) { return {a.v + b, a.d}; }
template <class T> PCEXP_DEV Tangent<T> operator+(T a, Tangent<T> b) { return {a + b.v, b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator-(Tangent<T> a, T b) { return {a.v - b, a.d}; }
template <class T> PCEXP_DEV Tangent<T> operator-(T a, Tangent<T> b) { return {a - b.v, -b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator*(Tangent<T> a, T b) { return {a.v * b, a.d * b}; }
template <class T> PCEXP_DEV Tangent<T> operator*(T a, Tangent<T> b) { return {a * b.v, a * b.d}; }
template <class T> PCEXP_DEV Tangent<T> operator/(Tangent<T> a, T b) { return {a.v / b, a.d / b}; }
template <class T> PCEXP_DEV Tangent<T> operator/(T a, Tangent<T> b) {
  T q = a / b.v;
  return {q, -q * b.d / b.v};
}

PCEXP_DEV double sqrt_s(double x) { return sqrt(x); }
PCEXP_DEV float sqrt_s(float x) { return sqrtf(x); }
template <class T> PCEXP_DEV Tangent<T> sqrt_s(Tangent<T> x) {
  T s = sqrt_s(x.v);
  return {s, x.d / (T(2) * s)};
}
// |x| with derivative sign(x) * dx, sign(0) = 0
PCEXP_DEV double abs_s(double x) { return fabs(x); }
PCEXP_DEV float abs_s(float x) { return fabsf(x); }
template <class T> PCEXP_DEV Tangent<T> abs_s(Tangent<T> x) {
  T sg = x.v > T(0) ? T(1) : (x.v < T(0) ? T(-1) : T(0));
  return {sg * x.v, sg * x.d};
}
PCEXP_DEV double pow_s(double x, double e) { return pow(x, e); }
PCEXP_DEV float pow_s(float x, float e) { return powf(x, e); }
template <class T> PCEXP_DEV Tangent<T> pow_s(Tangent<T> x, T e) {
  T pv = pow_s(x.v, e);
  return {pv, e * pv / x.v * x.d};
}
template <class S> PCEXP_DEV S select_s(bool c, S a, S b) { return c ? a : b; }


// ------------------------------------------------- multi-direction tangent (Jacobians)
// Jet<T, N>: value and its derivatives along N directions; evaluating a flux on
// Jets seeded with unit directions gives N columns of its exact Jacobian.
template <class T, int N>
struct Jet {
  T v;
  T d[N];
};
template <class T, int N> PCEXP_DEV T val(const Jet<T, N>& x) { return x.v; }
#define PCEXP_JET_BIN(OP, DEXPR)                                                        \
  template <class T, int N>                                                             \
  PCEXP_DEV Jet<T, N> operator OP(const Jet<T, N>& a, const Jet<T, N>& b) {             \
    Jet<T, N> r;                                                                        \
    r.v = a.v OP b.v;                                                                   \
    _Pragma("unroll") for (int k = 0; k < N; ++k) r.d[k] = DEXPR;                       \
    return r;                                                                           \
  }
PCEXP_JET_BIN(+, a.d[k] + b.d[k])
PCEXP_JET_BIN(-, a.d[k] - b.d[k])
PCEXP_JET_BIN(*, a.d[k] * b.v + a.v * b.d[k])
#undef PCEXP_JET_BIN
template <class T, int N> PCEXP_DEV Jet<T, N> operator/(const Jet<T, N>& a, const Jet<T, N>& b) {
  Jet<T, N> r;
  r.v = a.v / b.v;
  const T ib = T(1) / b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = (a.d[k] - r.v * b.d[k]) * ib;
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> operator-(const Jet<T, N>& a) {
  Jet<T, N> r;
  r.v = -a.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = -a.d[k];
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> operator+(const Jet<T, N>& a, T b) { Jet<T, N> r = a; r.v += b; return r; }
template <class T, int N> PCEXP_DEV Jet<T, N> operator+(T a, const Jet<T, N>& b) { Jet<T, N> r = b; r.v += a; return r; }
template <class T, int N> PCEXP_DEV Jet<T, N> operator-(const Jet<T, N>& a, T b) { Jet<T, N> r = a; r.v -= b; return r; }
template <class T, int N> PCEXP_DEV Jet<T, N> operator-(T a, const Jet<T, N>& b) {
  Jet<T, N> r;
  r.v = a - b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = -b.d[k];
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> operator*(const Jet<T, N>& a, T b) {
  Jet<T, N> r;
  r.v = a.v * b;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = a.d[k] * b;
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> operator*(T a, const Jet<T, N>& b) { return b * a; }
template <class T, int N> PCEXP_DEV Jet<T, N> operator/(const Jet<T, N>& a, T b) { return a * (T(1) / b); }
template <class T, int N> PCEXP_DEV Jet<T, N> operator/(T a, const Jet<T, N>& b) {
  Jet<T, N> r;
  r.v = a / b.v;
  const T f = -r.v / b.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = f * b.d[k];
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> sqrt_s(const Jet<T, N>& x) {
  Jet<T, N> r;
  r.v = sqrt_s(x.v);
  const T f = T(0.5) / r.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = f * x.d[k];
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> abs_s(const Jet<T, N>& x) {
  const T sg = x.v > T(0) ? T(1) : (x.v < T(0) ? T(-1) : T(0));
  Jet<T, N> r;
  r.v = sg * x.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = sg * x.d[k];
  return r;
}
template <class T, int N> PCEXP_DEV Jet<T, N> pow_s(const Jet<T, N>& x, T e) {
  Jet<T, N> r;
  r.v = pow_s(x.v, e);
  const T f = e * r.v / x.v;
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = f * x.d[k];
  return r;
}
PCEXP_DEV double exp_s(double x) { return exp(x); }
template <class T, int N> PCEXP_DEV Jet<T, N> exp_s(const Jet<T, N>& x) {
  Jet<T, N> r;
  r.v = exp(x.v);
#pragma unroll
  for (int k = 0; k < N; ++k) r.d[k] = r.v * x.d[k];
  return r;
}
template <class S, class T> struct Lift {
  PCEXP_DEV static S of(T x) { return S(x); }
};
template <class T> struct Lift<Tangent<T>, T> {
  PCEXP_DEV static Tangent<T> of(T x) { return {x, T(0)}; }
};
template <class T, int N> struct Lift<Jet<T, N>, T> {
  PCEXP_DEV static Jet<T, N> of(T x) {
    Jet<T, N> r;
    r.v = x;
#pragma unroll
    for (int k = 0; k < N; ++k) r.d[k] = T(0);
    return r;
  }
};

// ---------------------------------------------------------------- free stream
// vel holds the free-stream velocity in x, y (and z in 3D; zero in the x-y-plane cases)
template <class T>
struct Free {
  T gamma, rho, p;
  T vel[3];
};

// ------------------------------------------------------ fluxes (D dimensions, D+2 variables)
// Physical fluxes F[d] along the Cartesian axes of U = (rho, rho v_1..rho v_D, rho E).
template <int D, class S, class T>
PCEXP_DEV void euler_flux(const S (&U)[D + 2], T g, S (&F)[D][D + 2]) {
  constexpr int NV = D + 2;
  const S ir = T(1) / U[0];
  S vel[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vel[d] = U[1 + d] * ir;
  S ke = U[1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = ke + U[1 + d] * vel[d];
  const S p = (g - T(1)) * (U[NV - 1] - T(0.5) * ke);
  const S e = U[NV - 1] + p;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    F[d][0] = U[1 + d];
#pragma unroll
    for (int k = 0; k < D; ++k) F[d][1 + k] = (k == d) ? U[1 + k] * vel[d] + p : U[1 + k] * vel[d];
    F[d][NV - 1] = e * vel[d];
  }
}

template <int D, class S, class T>
PCEXP_DEV S dot_n(const S (&a)[D], const T (&n)[D]) {
  S r = a[0] * n[0];
#pragma unroll
  for (int d = 1; d < D; ++d) r = r + a[d] * n[d];
  return r;
}

// Roe flux F~(U_L, U_R) . n.  vrn = v_r . n, the normal velocity of a rotating frame at the
// face point (Sec. 4.1): F . n = F_abs . n - vrn U and the waves' speeds are shifted by -vrn
// (vrn = 0: the fixed frame, the same operations as without it).
template <int D, class S, class T>
PCEXP_DEV void roe_flux(const S (&L)[D + 2], const S (&R)[D + 2], const T (&n)[D], T g, S (&F)[D + 2],
                        T vrn = T(0)) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  S rL = L[0], irL = T(1) / rL, rR = R[0], irR = T(1) / rR;
  S vL[D], vR[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vL[d] = L[1 + d] * irL;
    vR[d] = R[1 + d] * irR;
  }
  S keL = L[1] * vL[0], keR = R[1] * vR[0];
#pragma unroll
  for (int d = 1; d < D; ++d) {
    keL = keL + L[1 + d] * vL[d];
    keR = keR + R[1 + d] * vR[d];
  }
  S pL = gm * (L[NV - 1] - T(0.5) * keL);
  S pR = gm * (R[NV - 1] - T(0.5) * keR);
  S qL = dot_n<D>(vL, n), qR = dot_n<D>(vR, n);
  S HL = (L[NV - 1] + pL) * irL, HR = (R[NV - 1] + pR) * irR;
  // central part
  S c[NV];
  c[0] = rL * qL + rR * qR;
#pragma unroll
  for (int d = 0; d < D; ++d) c[1 + d] = L[1 + d] * qL + R[1 + d] * qR + (pL + pR) * n[d];
  c[NV - 1] = (L[NV - 1] + pL) * qL + (R[NV - 1] + pR) * qR;
  // Roe averages
  S sL = sqrt_s(rL), sR = sqrt_s(rR), is = T(1) / (sL + sR);
  S rh = sL * sR;
  S vh[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vh[d] = (sL * vL[d] + sR * vR[d]) * is;
  S Hh = (sL * HL + sR * HR) * is;
  S q2 = vh[0] * vh[0];
#pragma unroll
  for (int d = 1; d < D; ++d) q2 = q2 + vh[d] * vh[d];
  S cc = gm * (Hh - T(0.5) * q2);
  S cs = sqrt_s(cc);
  S qh = dot_n<D>(vh, n);
  // jumps and wave strengths
  S dp = pR - pL, dr = rR - rL;
  S dv[D];
#pragma unroll
  for (int d = 0; d < D; ++d) dv[d] = vR[d] - vL[d];
  S dq = dot_n<D>(dv, n);
  const S qs = vrn != T(0) ? qh - vrn : qh;  // wave speeds relative to the frame
  S l1 = abs_s(qs - cs), l2 = abs_s(qs), l4 = abs_s(qs + cs);
  S i2c = T(0.5) / cc;
  S a1 = (dp - rh * cs * dq) * i2c;
  S a4 = (dp + rh * cs * dq) * i2c;
  S a2 = dr - dp / cc;
  S t1 = l1 * a1, t4 = l4 * a4, t2 = l2 * a2, ts = l2 * rh;
  S dd[NV];
  dd[0] = t1 + t2 + t4;
  S vdv = vh[0] * dv[0];
#pragma unroll
  for (int d = 1; d < D; ++d) vdv = vdv + vh[d] * dv[d];
#pragma unroll
  for (int d = 0; d < D; ++d)
    dd[1 + d] = t1 * (vh[d] - cs * n[d]) + t2 * vh[d] + ts * (dv[d] - dq * n[d]) + t4 * (vh[d] + cs * n[d]);
  dd[NV - 1] = t1 * (Hh - cs * qh) + t2 * (T(0.5) * q2) + ts * (vdv - qh * dq) + t4 * (Hh + cs * qh);
  if (vrn != T(0)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) c[v] = c[v] - vrn * (L[v] + R[v]);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) F[v] = T(0.5) * (c[v] - dd[v]);
}

// Slip wall and symmetry plane: the velocity relative to the wall (which moves with a
// rotating frame: vrn = v_r . n) has its normal component mirrored; density and pressure are
// kept.  v_g = v - 2 q n with q = v . n - vrn, so |v_g|^2 = |v|^2 - 4 q vrn and the ghost's
// total energy is rho E - 2 rho q vrn (unchanged in a fixed frame).
template <int D, class S, class T>
PCEXP_DEV void ghost_slip_wall(const S (&U)[D + 2], const T (&n)[D], S (&G)[D + 2], T vrn = T(0)) {
  constexpr int NV = D + 2;
  const S ir = T(1) / U[0];
  S m[D];
#pragma unroll
  for (int d = 0; d < D; ++d) m[d] = U[1 + d];
  S qn = dot_n<D>(m, n) * ir;  // normal velocity
  if (vrn != T(0)) qn = qn - vrn;
  G[0] = U[0];
#pragma unroll
  for (int d = 0; d < D; ++d) G[1 + d] = U[1 + d] - T(2) * U[0] * qn * n[d];
  G[NV - 1] = U[NV - 1];
  if (vrn != T(0)) G[NV - 1] = G[NV - 1] - T(2) * vrn * (U[0] * qn);
}

template <int D, class S, class T>
PCEXP_DEV void ghost_farfield(const S (&U)[D + 2], const T (&n)[D], const Free<T>& fs, S (&G)[D + 2]) {
  constexpr int NV = D + 2;
  const T g = fs.gamma, gm = g - T(1);
  const S ir = T(1) / U[0];
  S vel[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vel[d] = U[1 + d] * ir;
  S ke = U[1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = ke + U[1 + d] * vel[d];
  const S p = gm * (U[NV - 1] - T(0.5) * ke);
  const S c = sqrt_s(g * p * ir);
  const S qn = dot_n<D>(vel, n);
  const T cinf = sqrt_s(g * fs.p / fs.rho);
  T qinf = fs.vel[0] * n[0];
#pragma unroll
  for (int d = 1; d < D; ++d) qinf += fs.vel[d] * n[d];
  const T mn = val(qn) / val(c);
  const S rp = select_s(mn > T(-1), qn + T(2) * c / gm, Lift<S, T>::of(qinf + T(2) * cinf / gm));
  const S rm = select_s(mn < T(1), Lift<S, T>::of(qinf - T(2) * cinf / gm), qn - T(2) * c / gm);
  const S qb = T(0.5) * (rp + rm);
  const S cb = T(0.25) * gm * (rp - rm);
  const bool out = val(qb) >= T(0);
  const S s_in = p / pow_s(U[0], g);
  const T s_inf = fs.p / pow_s(fs.rho, g);
  const S sb = select_s(out, s_in, Lift<S, T>::of(s_inf));
  const S rb = pow_s(cb * cb / (g * sb), T(1) / gm);
  const S pb = rb * cb * cb / g;
  S kb = Lift<S, T>::of(T(0));
  G[0] = rb;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const S vt = select_s(out, vel[d] - qn * n[d], Lift<S, T>::of(fs.vel[d] - qinf * n[d]));
    const S vb = vt + qb * n[d];
    G[1 + d] = rb * vb;
    kb = kb + vb * vb;
  }
  G[NV - 1] = pb / gm + T(0.5) * rb * kb;
}

// The far-field ghost state of ghost_farfield with the free-stream velocity as a scalar of
// type S, for derivatives with respect to the free stream (the Mach number and the flow
// angle enter the scheme only through this velocity).  Same arithmetic, operation by
// operation, as ghost_farfield.
template <int D, class S, class T>
PCEXP_DEV void ghost_farfield_v(const S (&U)[D + 2], const T (&n)[D], T g, T rho_inf, T p_inf, const S (&vinf)[3],
                                S (&G)[D + 2]) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  const S ir = T(1) / U[0];
  S vel[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vel[d] = U[1 + d] * ir;
  S ke = U[1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = ke + U[1 + d] * vel[d];
  const S p = gm * (U[NV - 1] - T(0.5) * ke);
  const S c = sqrt_s(g * p * ir);
  const S qn = dot_n<D>(vel, n);
  const T cinf = sqrt_s(g * p_inf / rho_inf);
  S qinf = vinf[0] * n[0];
#pragma unroll
  for (int d = 1; d < D; ++d) qinf = qinf + vinf[d] * n[d];
  const T mn = val(qn) / val(c);
  const S rp = select_s(mn > T(-1), qn + T(2) * c / gm, qinf + T(2) * cinf / gm);
  const S rm = select_s(mn < T(1), qinf - T(2) * cinf / gm, qn - T(2) * c / gm);
  const S qb = T(0.5) * (rp + rm);
  const S cb = T(0.25) * gm * (rp - rm);
  const bool out = val(qb) >= T(0);
  const S s_in = p / pow_s(U[0], g);
  const T s_inf = p_inf / pow_s(rho_inf, g);
  const S sb = select_s(out, s_in, Lift<S, T>::of(s_inf));
  const S rb = pow_s(cb * cb / (g * sb), T(1) / gm);
  const S pb = rb * cb * cb / g;
  S kb = Lift<S, T>::of(T(0));
  G[0] = rb;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const S vt = select_s(out, vel[d] - qn * n[d], vinf[d] - qinf * n[d]);
    const S vb = vt + qb * n[d];
    G[1 + d] = rb * vb;
    kb = kb + vb * vb;
  }
  G[NV - 1] = pb / gm + T(0.5) * rb * kb;
}

// ------------------------------------------------------------ reverse mode of the fluxes
// Each *_vjp takes the adjoint of an output and adds the adjoints of the inputs, the exact
// transpose of the forward function (sign(0) = 0 for |x|).  One evaluation costs two to three
// forward ones, whatever the number of inputs.  On S = Tangent<T> with the inputs' tangents t, the
// derivative parts of the results are d/dU [ybar^T F'(U) t]: the second-order term of the reverse
// step, without seeding a direction per input (hyper-dual numbers carry 2 (D + 2) + 2 components
// through every operation and need a pass per side).
template <class T> PCEXP_DEV T sign_of(T x) { return x > T(0) ? T(1) : (x < T(0) ? T(-1) : T(0)); }

// Fb[d][v]: adjoint of the flux along axis d (no state in it); Ub += dF^T Fb
template <int D, class S, class T>
PCEXP_DEV void euler_flux_vjp(const S (&U)[D + 2], T g, const T (&Fb)[D][D + 2], S (&Ub)[D + 2]) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  const S ir = T(1) / U[0];
  S vel[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vel[d] = U[1 + d] * ir;
  S ke = U[1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = ke + U[1 + d] * vel[d];
  const S e = U[NV - 1] + gm * (U[NV - 1] - T(0.5) * ke);
  T trace = Fb[0][1];
#pragma unroll
  for (int d = 1; d < D; ++d) trace += Fb[d][1 + d];
  S eb = Fb[0][NV - 1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) eb = eb + Fb[d][NV - 1] * vel[d];
  const S pb = eb + trace;
  const S keb = (T(-0.5) * gm) * pb;
  S irb = Lift<S, T>::of(T(0));
#pragma unroll
  for (int d = 0; d < D; ++d) {
    S vb = keb * U[1 + d] + Fb[d][NV - 1] * e;
    S mb = keb * vel[d] + Fb[d][0];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      vb = vb + Fb[d][1 + k] * U[1 + k];
      mb = mb + Fb[k][1 + d] * vel[k];
    }
    Ub[1 + d] = Ub[1 + d] + mb + vb * ir;
    irb = irb + vb * U[1 + d];
  }
  Ub[NV - 1] = Ub[NV - 1] + eb + gm * pb;
  Ub[0] = Ub[0] - ir * ir * irb;
}

// adjoints of one side's state from those of its Roe-flux intermediates: rho, velocity, pressure,
// total enthalpy H, energy E (mass row and momenta already in Ub)
template <int D, class S, class T>
PCEXP_DEV void primitives_vjp(const S (&U)[D + 2], const S& ir, const S (&v)[D], const S& p, T gm, const S (&vb)[D],
                              S pb, const S& Hb, S (&Ub)[D + 2]) {
  constexpr int NV = D + 2;
  const S Hi = Hb * ir;  // H = (E + p) / rho
  pb = pb + Hi;
  const S keb = (T(-0.5) * gm) * pb;
  S irb = Hb * (U[NV - 1] + p);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const S w = vb[d] + keb * U[1 + d];
    Ub[1 + d] = Ub[1 + d] + keb * v[d] + w * ir;
    irb = irb + w * U[1 + d];
  }
  Ub[NV - 1] = Ub[NV - 1] + Hi + gm * pb;
  Ub[0] = Ub[0] - ir * ir * irb;
}

// Lb, Rb += (dF~/dL)^T Fb, (dF~/dR)^T Fb for the Roe flux of roe_flux (same intermediates)
template <int D, class S, class T>
PCEXP_DEV void roe_flux_vjp(const S (&L)[D + 2], const S (&R)[D + 2], const T (&n)[D], T g, const T (&Fb)[D + 2],
                            S (&Lb)[D + 2], S (&Rb)[D + 2], T vrn = T(0)) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  const S rL = L[0], irL = T(1) / rL, rR = R[0], irR = T(1) / rR;
  S vL[D], vR[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vL[d] = L[1 + d] * irL;
    vR[d] = R[1 + d] * irR;
  }
  S keL = L[1] * vL[0], keR = R[1] * vR[0];
#pragma unroll
  for (int d = 1; d < D; ++d) {
    keL = keL + L[1 + d] * vL[d];
    keR = keR + R[1 + d] * vR[d];
  }
  const S pL = gm * (L[NV - 1] - T(0.5) * keL), pR = gm * (R[NV - 1] - T(0.5) * keR);
  const S qL = dot_n<D>(vL, n), qR = dot_n<D>(vR, n);
  const S hL = L[NV - 1] + pL, hR = R[NV - 1] + pR;
  const S HL = hL * irL, HR = hR * irR;
  const S sL = sqrt_s(rL), sR = sqrt_s(rR), is = T(1) / (sL + sR);
  const S wL = sL * is, wR = sR * is, rh = sL * sR;
  S vh[D], dv[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vh[d] = wL * vL[d] + wR * vR[d];
    dv[d] = vR[d] - vL[d];
  }
  const S Hh = wL * HL + wR * HR;
  S q2 = vh[0] * vh[0], vdv = vh[0] * dv[0];
#pragma unroll
  for (int d = 1; d < D; ++d) {
    q2 = q2 + vh[d] * vh[d];
    vdv = vdv + vh[d] * dv[d];
  }
  const S cc = gm * (Hh - T(0.5) * q2), cs = sqrt_s(cc), i2c = T(0.5) / cc;
  const S qh = dot_n<D>(vh, n), dq = dot_n<D>(dv, n), dp = pR - pL, dr = rR - rL;
  const S qs = vrn != T(0) ? qh - vrn : qh;
  const T s1 = sign_of(val(qs) - val(cs)), s2 = sign_of(val(qs)), s4 = sign_of(val(qs) + val(cs));
  const S l1 = s1 * (qs - cs), l2 = s2 * qs, l4 = s4 * (qs + cs);
  const S w = rh * cs * dq;
  const S a1 = (dp - w) * i2c, a4 = (dp + w) * i2c, a2 = dr - T(2) * dp * i2c;
  const S t1 = l1 * a1, t4 = l4 * a4, t2 = l2 * a2, ts = l2 * rh;
  // F~ = (c - dd) / 2: the dissipation's adjoint is -Fb / 2
  const T d0 = T(-0.5) * Fb[0], dE = T(-0.5) * Fb[NV - 1];
  T dm[D], dmn = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    dm[d] = T(-0.5) * Fb[1 + d];
    dmn += dm[d] * n[d];
  }
  // dd_0 = t1 + t2 + t4, dd_m = (t1 + t2 + t4) vh + (t4 - t1) cs n + ts (dv - dq n),
  // dd_E = (t1 + t4) Hh + (t4 - t1) cs qh + t2 q2 / 2 + ts (vdv - qh dq)
  S dmvh = dm[0] * vh[0], dmdv = dm[0] * dv[0];
#pragma unroll
  for (int d = 1; d < D; ++d) {
    dmvh = dmvh + dm[d] * vh[d];
    dmdv = dmdv + dm[d] * dv[d];
  }
  const S mc = t4 - t1;
  const S base = dmvh + d0, sb = base + dE * Hh, t2b = base + (T(0.5) * dE) * q2;
  const S mcb = dE * qh + dmn, mb = mcb * cs;
  const S tsb = dmdv - dmn * dq + dE * (vdv - qh * dq);
  S csb = mcb * mc;
  S qhb = dE * (mc * cs - ts * dq);
  S dqb = -(ts * mcb);
  S q2b = (T(0.5) * dE) * t2;
  const S sum = t1 + t2 + t4;
  S Hhb = dE * (t1 + t4);
  const S t1b = sb - mb, t4b = sb + mb;
  const S l1b = s1 * (t1b * a1), l4b = s4 * (t4b * a4), l2b = s2 * (t2b * a2 + tsb * rh);
  qhb = qhb + l1b + l2b + l4b;
  csb = csb - l1b + l4b;
  const S a1b = t1b * l1, a4b = t4b * l4, a2b = t2b * l2;
  S rhb = tsb * l2;
  const S ab = a1b + a4b, wb = (a4b - a1b) * i2c;
  const S dpb = (ab - T(2) * a2b) * i2c;
  const S i2cb = (ab - T(2) * a2b) * dp + (a4b - a1b) * w;
  const S wrc = wb * rh, wcd = wb * dq;
  rhb = rhb + wcd * cs;
  csb = csb + wcd * rh;
  dqb = dqb + wrc * cs;
  const S ccb = csb * cs * i2c - T(2) * (i2c * i2c) * i2cb;  // cs = sqrt(cc), i2c = 1 / (2 cc)
  Hhb = Hhb + gm * ccb;
  q2b = q2b - (T(0.5) * gm) * ccb;
  // central part: c_0 = rL qL + rR qR, c_m = m qL + m' qR + (pL + pR) n, c_E = hL qL + hR qR
  const T c0 = -d0, cE = -dE, cmn = -dmn;
  S qLb = c0 * rL + cE * hL, qRb = c0 * rR + cE * hR;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    qLb = qLb - dm[d] * L[1 + d];
    qRb = qRb - dm[d] * R[1 + d];
  }
  const S eL = cE * qL, eR = cE * qR;  // adjoint of h = E + p of each side
  S vLb[D], vRb[D], wd = Hhb * (HL - HR);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const S vhb = dm[d] * sum + (dE * ts) * dv[d] + qhb * n[d] + T(2) * q2b * vh[d];
    const S dvb = dm[d] * ts + (dE * ts) * vh[d] + dqb * n[d];
    vLb[d] = wL * vhb - dvb + qLb * n[d];
    vRb[d] = wR * vhb + dvb + qRb * n[d];
    wd = wd - vhb * dv[d];
    Lb[1 + d] = Lb[1 + d] - dm[d] * qL;
    Rb[1 + d] = Rb[1 + d] - dm[d] * qR;
  }
  // wL = sL / (sL + sR), wR = 1 - wL; rh = sL sR; s = sqrt(r)
  const S wi = wd * is;
  const S sLb = wi * wR + rhb * sR, sRb = rhb * sL - wi * wL;
  Lb[0] = Lb[0] + c0 * qL - a2b + T(0.5) * sLb / sL;
  Rb[0] = Rb[0] + c0 * qR + a2b + T(0.5) * sRb / sR;
  Lb[NV - 1] = Lb[NV - 1] + eL;
  Rb[NV - 1] = Rb[NV - 1] + eR;
  primitives_vjp<D, S, T>(L, irL, vL, pL, gm, vLb, eL - dpb + cmn, wL * Hhb, Lb);
  primitives_vjp<D, S, T>(R, irR, vR, pR, gm, vRb, eR + dpb + cmn, wR * Hhb, Rb);
  if (vrn != T(0)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Lb[v] = Lb[v] - (T(0.5) * vrn) * Fb[v];
      Rb[v] = Rb[v] - (T(0.5) * vrn) * Fb[v];
    }
  }
}

// Ub += (dG/dU)^T Gb for ghost_slip_wall (linear in U)
template <int D, class S, class T>
PCEXP_DEV void ghost_slip_wall_vjp(const T (&n)[D], const S (&Gb)[D + 2], S (&Ub)[D + 2], T vrn = T(0)) {
  constexpr int NV = D + 2;
  S a = Gb[1] * n[0];
#pragma unroll
  for (int d = 1; d < D; ++d) a = a + Gb[1 + d] * n[d];
  S b = T(2) * a;
  Ub[0] = Ub[0] + Gb[0];
  if (vrn != T(0)) {
    b = b + (T(2) * vrn) * Gb[NV - 1];
    Ub[0] = Ub[0] + vrn * b;
  }
#pragma unroll
  for (int d = 0; d < D; ++d) Ub[1 + d] = Ub[1 + d] + Gb[1 + d] - b * n[d];
  Ub[NV - 1] = Ub[NV - 1] + Gb[NV - 1];
}

// Ub += (dG/dU)^T Gb and vib += (dG/dv_inf)^T Gb for ghost_farfield (same intermediates)
template <int D, class S, class T>
PCEXP_DEV void ghost_farfield_vjp(const S (&U)[D + 2], const T (&n)[D], const Free<T>& fs, const S (&Gb)[D + 2],
                                  S (&Ub)[D + 2], S (&vib)[D]) {
  constexpr int NV = D + 2;
  const T g = fs.gamma, gm = g - T(1);
  const S ir = T(1) / U[0];
  S vel[D];
#pragma unroll
  for (int d = 0; d < D; ++d) vel[d] = U[1 + d] * ir;
  S ke = U[1] * vel[0];
#pragma unroll
  for (int d = 1; d < D; ++d) ke = ke + U[1 + d] * vel[d];
  const S p = gm * (U[NV - 1] - T(0.5) * ke);
  const S c = sqrt_s(g * p * ir);
  const S qn = dot_n<D>(vel, n);
  const T cinf = sqrt_s(g * fs.p / fs.rho);
  T qinf = fs.vel[0] * n[0];
#pragma unroll
  for (int d = 1; d < D; ++d) qinf += fs.vel[d] * n[d];
  const T mn = val(qn) / val(c);
  const bool in_p = mn > T(-1), in_m = !(mn < T(1));  // invariants taken from the interior
  const S rp = select_s(in_p, qn + T(2) * c / gm, Lift<S, T>::of(qinf + T(2) * cinf / gm));
  const S rm = select_s(!in_m, Lift<S, T>::of(qinf - T(2) * cinf / gm), qn - T(2) * c / gm);
  const S qb = T(0.5) * (rp + rm);
  const S cb = T(0.25) * gm * (rp - rm);
  const bool out = val(qb) >= T(0);
  const S s_in = p / pow_s(U[0], g);
  const T s_inf = fs.p / pow_s(fs.rho, g);
  const S sb = select_s(out, s_in, Lift<S, T>::of(s_inf));
  const S rb = pow_s(cb * cb / (g * sb), T(1) / gm);
  S vb[D], kb = Lift<S, T>::of(T(0)), rbb = Gb[0], qbb = Lift<S, T>::of(T(0)), vbb[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const S vt = select_s(out, vel[d] - qn * n[d], Lift<S, T>::of(fs.vel[d] - qinf * n[d]));
    vb[d] = vt + qb * n[d];
    kb = kb + vb[d] * vb[d];
    rbb = rbb + Gb[1 + d] * vb[d];
  }
  rbb = rbb + T(0.5) * Gb[NV - 1] * kb;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    vbb[d] = rb * (Gb[1 + d] + Gb[NV - 1] * vb[d]);
    qbb = qbb + vbb[d] * n[d];
  }
  const S pbb = Gb[NV - 1] / gm;  // G_E = p_b / gm + rho_b |v_b|^2 / 2, p_b = rho_b c_b^2 / g
  rbb = rbb + pbb * cb * cb / g;
  S cbb = T(2) / g * pbb * rb * cb;
  const S lr = rbb * rb / gm;  // rho_b = (c_b^2 / (g s_b))^(1 / gm)
  cbb = cbb + T(2) * lr / cb;
  S qnb = Lift<S, T>::of(T(0)), qib = qnb, cib = qnb, pb = qnb;
  const S rpb = T(0.5) * qbb + (T(0.25) * gm) * cbb, rmb = T(0.5) * qbb - (T(0.25) * gm) * cbb;
  if (in_p) {
    qnb = qnb + rpb;
    cib = cib + rpb;
  } else {
    qib = qib + rpb;
  }
  if (in_m) {
    qnb = qnb + rmb;
    cib = cib - rmb;
  } else {
    qib = qib + rmb;
  }
  if (out) {
    qnb = qnb - qbb;
    pb = pb - lr / p;         // s_in = p rho^-g
    Ub[0] = Ub[0] + g * lr * ir;
  } else {
    qib = qib - qbb;
  }
  const S ch = (T(1) / gm) * cib * c;  // (2 / gm) cib * dc, dc = c / 2 (dp / p - drho / rho)
  pb = pb + ch / p;
  Ub[0] = Ub[0] - ch * ir;
  const S keb = (T(-0.5) * gm) * pb;
  S irb = Lift<S, T>::of(T(0));
#pragma unroll
  for (int d = 0; d < D; ++d) {
    S w = keb * U[1 + d] + qnb * n[d];
    if (out) w = w + vbb[d];
    else vib[d] = vib[d] + vbb[d];
    vib[d] = vib[d] + qib * n[d];
    Ub[1 + d] = Ub[1 + d] + keb * vel[d] + w * ir;
    irb = irb + w * U[1 + d];
  }
  Ub[NV - 1] = Ub[NV - 1] + gm * pb;
  Ub[0] = Ub[0] - ir * ir * irb;
}

// ------------------------------------------------- Roe-flux derivative from a stored record
// What the Roe flux's linearisation at (L, R) needs besides the normal; 16 values (D = 2: 14) that
// replace its 2 (D + 2)^2 Jacobian entries.  H total enthalpy, w = sqrt(rho_L) / (sqrt(rho_L) +
// sqrt(rho_R)), c Roe's sound speed, i2c = 1 / (2 c^2), dp = p_R - p_L.
template <class T, int D>
struct RoeRecord {
  T vL[D], HL, rL, irL, vR[D], HR, rR, irR, w, c, i2c, dp;
};

template <int D, class T>
PCEXP_DEV RoeRecord<T, D> roe_record(const T (&L)[D + 2], const T (&R)[D + 2], T g) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  RoeRecord<T, D> r;
  r.rL = L[0];
  r.rR = R[0];
  r.irL = T(1) / L[0];
  r.irR = T(1) / R[0];
  T kL = T(0), kR = T(0), q2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    r.vL[d] = L[1 + d] * r.irL;
    r.vR[d] = R[1 + d] * r.irR;
    kL += L[1 + d] * r.vL[d];
    kR += R[1 + d] * r.vR[d];
  }
  const T pL = gm * (L[NV - 1] - T(0.5) * kL), pR = gm * (R[NV - 1] - T(0.5) * kR);
  r.HL = (L[NV - 1] + pL) * r.irL;
  r.HR = (R[NV - 1] + pR) * r.irR;
  const T sL = sqrt_s(L[0]), sR = sqrt_s(R[0]), is = T(1) / (sL + sR);
  r.w = sL * is;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const T vh = (sL * r.vL[d] + sR * r.vR[d]) * is;
    q2 += vh * vh;
  }
  const T cc = gm * ((sL * r.HL + sR * r.HR) * is - T(0.5) * q2);
  r.c = sqrt_s(cc);
  r.i2c = T(0.5) / cc;
  r.dp = pR - pL;
  return r;
}

// One side's primitive derivatives along a (its conservative direction), and its share of the
// central flux's derivative added to C.
template <class T, int D>
struct SideDerivative {
  T lr, v[D], p, q, H;  // d ln rho, dv, dp, d(v . n), dH
};
template <int D, class T>
PCEXP_DEV SideDerivative<T, D> side_derivative(const T (&v)[D], T H, T ir, T qn, const T (&n)[D], T gm,
                                               const T (&a)[D + 2], T (&C)[D + 2]) {
  constexpr int NV = D + 2;
  SideDerivative<T, D> s;
  T k2 = T(0), e = a[NV - 1], mn = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    k2 = fma(T(0.5) * v[d], v[d], k2);
    e = fma(-v[d], a[1 + d], e);
    mn = fma(a[1 + d], n[d], mn);
    s.v[d] = fma(-v[d], a[0], a[1 + d]) * ir;
  }
  s.p = gm * fma(k2, a[0], e);
  const T h = a[NV - 1] + s.p, w = fma(-qn, a[0], mn);  // d(E + p), rho dq
  s.lr = a[0] * ir;
  s.q = w * ir;
  s.H = fma(-H, a[0], h) * ir;
  C[0] += mn;
#pragma unroll
  for (int d = 0; d < D; ++d) C[1 + d] = fma(qn, a[1 + d], fma(v[d], w, fma(s.p, n[d], C[1 + d])));
  C[NV - 1] = fma(qn, h, fma(H, w, C[NV - 1]));
  return s;
}

// dF = dF~/dU_L a + dF~/dU_R b (the derivative of roe_flux, sign(0) = 0 for |x|).
template <int D, class T>
PCEXP_DEV void roe_derivative(const RoeRecord<T, D>& r, const T (&n)[D], T g, T vrn, const T (&a)[D + 2],
                              const T (&b)[D + 2], T (&dF)[D + 2]) {
  constexpr int NV = D + 2;
  const T gm = g - T(1);
  T qL = T(0), qR = T(0), C[NV];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    qL = fma(r.vL[d], n[d], qL);
    qR = fma(r.vR[d], n[d], qR);
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) C[v] = T(0);
  const SideDerivative<T, D> dL = side_derivative<D, T>(r.vL, r.HL, r.irL, qL, n, gm, a, C);
  const SideDerivative<T, D> dR = side_derivative<D, T>(r.vR, r.HR, r.irR, qR, n, gm, b, C);
  const T wL = r.w, wR = T(1) - r.w, t = T(0.5) * wL * wR * (dL.lr - dR.lr);  // t = dw_L
  const T dH = r.HR - r.HL, dq = qR - qL, ddq = dR.q - dL.q;
  const T Hh = fma(wR, dH, r.HL), qh = fma(wR, dq, qL), rh = fma(r.rL, wR, r.rR * wL);
  const T dHh = fma(wL, dL.H, fma(wR, dR.H, -t * dH)), drh = T(0.5) * rh * (dL.lr + dR.lr);
  T vh[D], dvh[D], dv[D], ddv[D], vhd = T(0), dqh = T(0), vdv = T(0), dvdv = T(0), k2 = T(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    dv[d] = r.vR[d] - r.vL[d];
    ddv[d] = dR.v[d] - dL.v[d];
    vh[d] = fma(wR, dv[d], r.vL[d]);
    dvh[d] = fma(wL, dL.v[d], fma(wR, dR.v[d], -t * dv[d]));
    vhd = fma(vh[d], dvh[d], vhd);
    dqh = fma(dvh[d], n[d], dqh);
    vdv = fma(vh[d], dv[d], vdv);
    dvdv = fma(dvh[d], dv[d], fma(vh[d], ddv[d], dvdv));
    k2 = fma(T(0.5) * vh[d], vh[d], k2);
  }
  const T dcc = gm * (dHh - vhd), c = r.c, dc = dcc * r.i2c * c;  // c = sqrt(cc), i2c = 1 / (2 cc)
  const T qs = qh - vrn;
  const T s1 = sign_of(qs - c), s2 = sign_of(qs), s4 = sign_of(qs + c);
  const T l1 = s1 * (qs - c), l2 = s2 * qs, l4 = s4 * (qs + c);
  const T dl1 = s1 * (dqh - dc), dl2 = s2 * dqh, dl4 = s4 * (dqh + dc);
  const T w0 = rh * c * dq, dw0 = fma(drh * c, dq, rh * fma(dc, dq, c * ddq));
  const T ddp = dR.p - dL.p, ri = T(-2) * r.i2c * dcc;  // di2c = i2c ri
  const T a1 = (r.dp - w0) * r.i2c, a4 = (r.dp + w0) * r.i2c, a2 = fma(T(-2) * r.dp, r.i2c, r.rR - r.rL);
  const T da1 = fma(ddp - dw0, r.i2c, a1 * ri), da4 = fma(ddp + dw0, r.i2c, a4 * ri);
  const T da2 = fma(T(-2) * r.i2c, fma(r.dp, ri, ddp), b[0] - a[0]);
  const T t1 = l1 * a1, t4 = l4 * a4, t2 = l2 * a2, ts = l2 * rh;
  const T dt1 = fma(dl1, a1, l1 * da1), dt4 = fma(dl4, a4, l4 * da4), dt2 = fma(dl2, a2, l2 * da2);
  const T dts = fma(dl2, rh, l2 * drh);
  const T e = t1 + t4, de = dt1 + dt4, S = e + t2, dS = de + dt2;
  const T m = t4 - t1, mc = m * c, dmc = fma(dt4 - dt1, c, m * dc);
  const T cn = dmc - fma(dts, dq, ts * ddq);
  dF[0] = T(0.5) * (C[0] - dS);
#pragma unroll
  for (int d = 0; d < D; ++d)
    dF[1 + d] = T(0.5) * (C[1 + d] - fma(dS, vh[d], fma(S, dvh[d], fma(cn, n[d], fma(dts, dv[d], ts * ddv[d])))));
  const T dE = fma(de, Hh, fma(e, dHh, fma(dmc, qh, fma(mc, dqh, fma(dt2, k2, t2 * vhd))))) +
               fma(dts, fma(-qh, dq, vdv), ts * (dvdv - fma(dqh, dq, qh * ddq)));
  dF[NV - 1] = T(0.5) * (C[NV - 1] - dE);
  if (vrn != T(0)) {
#pragma unroll
    for (int v = 0; v < NV; ++v) dF[v] = fma(T(-0.5) * vrn, a[v] + b[v], dF[v]);
  }
}

}  // namespace pcexp
