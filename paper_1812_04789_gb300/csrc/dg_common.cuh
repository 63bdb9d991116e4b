// Shared device definitions: forward-mode dual numbers, pointwise compressible
// Navier-Stokes physics (Sec. 2 closure, Sec. 3.1 fluxes), device mesh view.
//
// Every pointwise routine is templated on the scalar S (T = float/double for a
// residual, Dual<T> for a Jacobian-vector product: value + directional
// derivative, so the JVP is the exact linearisation of the discrete residual)
// and on the dimension D (2 or 3); m = D + 2 conservative variables
// (rho, rho v_1..rho v_D, rho e0).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace dgk {

// 8 consecutive BF16 values (16 bytes, read-only, not kept in L1) widened to
// FP32: a BF16 value is the upper half of the FP32 with the same bits.
__device__ __forceinline__ void ld_bf16x8(const unsigned short* p, float* v) {
  unsigned a, b, c, d;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
               : "l"(p));
  v[0] = __uint_as_float(a << 16);
  v[1] = __uint_as_float(a & 0xffff0000u);
  v[2] = __uint_as_float(b << 16);
  v[3] = __uint_as_float(b & 0xffff0000u);
  v[4] = __uint_as_float(c << 16);
  v[5] = __uint_as_float(c & 0xffff0000u);
  v[6] = __uint_as_float(d << 16);
  v[7] = __uint_as_float(d & 0xffff0000u);
}

// ----------------------------------------------------------------- duals
template <class T>
struct Dual {
  T v, d;
  __host__ __device__ Dual() {}
  __host__ __device__ Dual(T a) : v(a), d(T(0)) {}
  __host__ __device__ Dual(T a, T b) : v(a), d(b) {}
};
template <class T> __host__ __device__ __forceinline__ Dual<T> operator+(Dual<T> a, Dual<T> b) { return Dual<T>(a.v + b.v, a.d + b.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator-(Dual<T> a, Dual<T> b) { return Dual<T>(a.v - b.v, a.d - b.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator-(Dual<T> a) { return Dual<T>(-a.v, -a.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator*(Dual<T> a, Dual<T> b) { return Dual<T>(a.v * b.v, a.d * b.v + a.v * b.d); }
// one division per quotient: the tangent reuses the reciprocal of the value
template <class T> __host__ __device__ __forceinline__ Dual<T> operator/(Dual<T> a, Dual<T> b) {
  const T r = T(1) / b.v;
  const T q = a.v * r;
  return Dual<T>(q, (a.d - q * b.d) * r);
}
template <class T> __host__ __device__ __forceinline__ Dual<T> operator+(Dual<T> a, T b) { return Dual<T>(a.v + b, a.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator+(T a, Dual<T> b) { return Dual<T>(a + b.v, b.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator-(Dual<T> a, T b) { return Dual<T>(a.v - b, a.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator-(T a, Dual<T> b) { return Dual<T>(a - b.v, -b.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator*(Dual<T> a, T b) { return Dual<T>(a.v * b, a.d * b); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator*(T a, Dual<T> b) { return Dual<T>(a * b.v, a * b.d); }
template <class T> __host__ __device__ __forceinline__ Dual<T> operator/(Dual<T> a, T b) {
  const T r = T(1) / b;
  return Dual<T>(a.v * r, a.d * r);
}
template <class T> __host__ __device__ __forceinline__ Dual<T> operator/(T a, Dual<T> b) {
  const T r = T(1) / b.v;
  const T q = a * r;
  return Dual<T>(q, -q * b.d * r);
}
template <class T> __host__ __device__ __forceinline__ Dual<T> dsqrt(Dual<T> a) {
  const T s = sqrt(a.v);
  return Dual<T>(s, a.d * (T(0.5) / s));
}
__host__ __device__ __forceinline__ double dsqrt(double a) { return sqrt(a); }
__host__ __device__ __forceinline__ float dsqrt(float a) { return sqrtf(a); }

template <class T> __host__ __device__ __forceinline__ T val(Dual<T> a) { return a.v; }
__host__ __device__ __forceinline__ double val(double a) { return a; }
__host__ __device__ __forceinline__ float val(float a) { return a; }
template <class T> __host__ __device__ __forceinline__ T tan_part(Dual<T> a) { return a.d; }
__host__ __device__ __forceinline__ double tan_part(double a) { return a; }
__host__ __device__ __forceinline__ float tan_part(float a) { return a; }

// |x| continued so that the derivative at x = 0 is +1 (x >= 0 is "positive")
template <class S> __host__ __device__ __forceinline__ S sabs(S x) { return val(x) >= 0 ? x : -x; }

// c + a b and c - a b (a, b, c numbers or duals), written so that every product
// of a dual's tangent fuses with an addition: three multiply-adds, where the
// separate product and sum take five operations
__host__ __device__ __forceinline__ double madd(double a, double b, double c) { return a * b + c; }
__host__ __device__ __forceinline__ float madd(float a, float b, float c) { return a * b + c; }
__host__ __device__ __forceinline__ double msub(double a, double b, double c) { return c - a * b; }
__host__ __device__ __forceinline__ float msub(float a, float b, float c) { return c - a * b; }
template <class T> __host__ __device__ __forceinline__ Dual<T> madd(Dual<T> a, Dual<T> b, Dual<T> c) {
  return Dual<T>(a.v * b.v + c.v, a.d * b.v + (a.v * b.d + c.d));
}
template <class T> __host__ __device__ __forceinline__ Dual<T> msub(Dual<T> a, Dual<T> b, Dual<T> c) {
  return Dual<T>(c.v - a.v * b.v, (c.d - a.v * b.d) - a.d * b.v);
}
template <class T> __host__ __device__ __forceinline__ Dual<T> madd(T a, Dual<T> b, Dual<T> c) {
  return Dual<T>(a * b.v + c.v, a * b.d + c.d);
}
template <class T> __host__ __device__ __forceinline__ Dual<T> msub(T a, Dual<T> b, Dual<T> c) {
  return Dual<T>(c.v - a * b.v, c.d - a * b.d);
}
// sqrt(a) where ia = 1/a is at hand: the tangent a' / (2 sqrt(a)) = a' sqrt(a) ia / 2
// needs no division
template <class T> __host__ __device__ __forceinline__ Dual<T> dsqrt(Dual<T> a, Dual<T> ia) {
  const T r = sqrt(a.v);
  return Dual<T>(r, a.d * (T(0.5) * r * ia.v));
}
__host__ __device__ __forceinline__ double dsqrt(double a, double) { return sqrt(a); }
__host__ __device__ __forceinline__ float dsqrt(float a, float) { return sqrtf(a); }

// ----------------------------------------------------------------- physics
// The FP64 kernels are bound by the number of FP64 operations (two lanes per
// clock and SM), so the pointwise physics spends as few as it can: primitives
// once per trace, four divisions and three square roots per face point, the
// symmetric parts of the stress and of rho v v once, the viscosity multiplied
// into the stress only, structural zeros never touched.  A face point of the
// JVP takes about 700 FP64 operations (2,050 when every routine formed its
// own primitives and full tensors), a volume point 250.
template <class T>
struct Phys {
  T gamma, gm1, Pr, mu, Rgas, eta, roe_delta, kappa;  // kappa = mu c_p / Pr
  T kq = T(0);    // kappa (gamma - 1) / R; 0 = form it here
  T hrd = T(0);   // 1 / (2 roe_delta); 0 = form it here
  __host__ __device__ __forceinline__ T heat() const { return kq != T(0) ? kq : kappa * (gm1 / Rgas); }
  __host__ __device__ __forceinline__ T half_inv_delta() const { return hrd != T(0) ? hrd : T(0.5) / roe_delta; }
};

// 1/rho, velocity, specific total energy, pressure, total enthalpy
template <int D, class S>
struct Prim {
  S ir, vel[D], e0, p, h0;
};
template <int D, class S, class T>
__host__ __device__ __forceinline__ void primitives(const S* u, const Phys<T>& ph, Prim<D, S>& P) {
  constexpr int M = D + 2;
  P.ir = T(1) / u[0];
#pragma unroll
  for (int j = 0; j < D; ++j) P.vel[j] = u[1 + j] * P.ir;
  S mv = u[1] * P.vel[0];
#pragma unroll
  for (int j = 1; j < D; ++j) mv = madd(u[1 + j], P.vel[j], mv);
  P.p = ph.gm1 * msub(T(0.5), mv, u[M - 1]);
  P.e0 = u[M - 1] * P.ir;
  P.h0 = madd(P.p, P.ir, P.e0);
}

// Inviscid flux column k: (rho v_k, rho v_j v_k + p delta_jk, rho v_k h0)
// Full tensor F_c + F_v at a point: F[v][k].
template <int D, class S, class T>
__host__ __device__ __forceinline__ void flux_total(const S* u, const S (*g)[D], S (*F)[D],
                                           const Phys<T>& ph) {
  constexpr int M = D + 2;
  Prim<D, S> P;
  primitives<D, S, T>(u, ph, P);
  // rho grad v_j = grad(rho v_j) - v_j grad rho, and rho (grad e0 - v . grad v)
  S a[D][D], b[D];
#pragma unroll
  for (int k = 0; k < D; ++k) {
    b[k] = msub(P.e0, g[0][k], g[M - 1][k]);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      a[j][k] = msub(P.vel[j], g[0][k], g[1 + j][k]);
      b[k] = msub(P.vel[j], a[j][k], b[k]);
    }
  }
  S div = a[0][0];
#pragma unroll
  for (int j = 1; j < D; ++j) div = div + a[j][j];
  const S mi = ph.mu * P.ir, ki = ph.heat() * P.ir;
  S tau[D][D];
#pragma unroll
  for (int k = 0; k < D; ++k)
#pragma unroll
    for (int j = 0; j <= k; ++j) {
      const S t = mi * (j == k ? msub(T(2) / T(3), div, T(2) * a[k][k]) : a[j][k] + a[k][j]);
      tau[j][k] = t;
      tau[k][j] = t;
    }
#pragma unroll
  for (int k = 0; k < D; ++k) {
    F[0][k] = u[1 + k];
#pragma unroll
    for (int j = 0; j <= k; ++j) {
      S f = madd(u[1 + j], P.vel[k], -tau[j][k]);
      if (j == k) f = f + P.p;
      F[1 + j][k] = f;
      F[1 + k][j] = f;
    }
    S q = ki * b[k];
#pragma unroll
    for (int j = 0; j < D; ++j) q = madd(P.vel[j], tau[j][k], q);
    F[M - 1][k] = madd(u[1 + k], P.h0, -q);
  }
}

// Fk += c F_v column k (F_v = -(0, tau, v.tau - q)), given the primitives.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void add_visc_col(const Prim<D, S>& P, const S (*g)[D], T c, S* Fk,
                                                      const Phys<T>& ph) {
  constexpr int M = D + 2;
  S an[D], b = msub(P.e0, g[0][k], g[M - 1][k]), dt = T(0);   // rho d_k v_j; the other directions' divergence
#pragma unroll
  for (int j = 0; j < D; ++j) {
    an[j] = msub(P.vel[j], g[0][k], g[1 + j][k]);
    b = msub(P.vel[j], an[j], b);
  }
  const S mi = (c * ph.mu) * P.ir;
  S q = (c * ph.heat()) * P.ir * b;
  bool first = true;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    if (j == k) continue;
    const S ajj = msub(P.vel[j], g[0][j], g[1 + j][j]);
    dt = first ? ajj : dt + ajj;
    first = false;
    const S akj = msub(P.vel[k], g[0][j], g[1 + k][j]);      // rho d_j v_k
    const S t = mi * (an[j] + akj);
    Fk[1 + j] = Fk[1 + j] - t;
    q = madd(P.vel[j], t, q);
  }
  const S t = mi * msub(T(2) / T(3), dt, (T(4) / T(3)) * an[k]);
  Fk[1 + k] = Fk[1 + k] - t;
  q = madd(P.vel[k], t, q);
  Fk[M - 1] = Fk[M - 1] - q;
}

// Viscous flux only (F_v = -(0, tau, v.tau - q)), column k, for face averages.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void flux_visc_col(const S* u, const S (*g)[D], S* Fk,
                                              const Phys<T>& ph) {
  Prim<D, S> P;
  primitives<D, S, T>(u, ph, P);
#pragma unroll
  for (int v = 0; v < D + 2; ++v) Fk[v] = T(0);
  add_visc_col<D, k, S, T>(P, g, T(1), Fk, ph);
}

// c K(u)(a (x) e_k) = -c F_v(u, a (x) e_k), the viscous operator applied to the
// rank-one gradient a e_k^T (the BR2 lifting of eq. re and the dual-consistency
// term of eq. dg_ns), by its independent entries: with m_j = c mu (d v_j along
// e_k) the tensor G[v][kk] is
//   G[0][.] = 0,  G[1+j][k] = m_j (j != k), 4/3 m_k (j = k),
//   kk != k: G[1+k][kk] = m_kk, G[1+kk][kk] = -2/3 m_k, else 0,  G[M-1][kk] = e_kk.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void visc_rank1(const Prim<D, S>& P, const S* a, T c, S* m, S* e,
                                                    const Phys<T>& ph) {
  constexpr int M = D + 2;
  S b = msub(P.e0, a[0], a[M - 1]), av[D];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    av[j] = msub(P.vel[j], a[0], a[1 + j]);
    b = msub(P.vel[j], av[j], b);
  }
  const S mi = (c * ph.mu) * P.ir;
#pragma unroll
  for (int j = 0; j < D; ++j) m[j] = mi * av[j];
  S en = madd((T(4) / T(3)) * P.vel[k], m[k], (c * ph.heat()) * P.ir * b);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    if (j == k) continue;
    en = madd(P.vel[j], m[j], en);
    e[j] = msub((T(2) / T(3)) * P.vel[j], m[k], P.vel[k] * m[j]);
  }
  e[k] = en;
}
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void rank1_tensor(const S* m, const S* e, S (*G)[D]) {
#pragma unroll
  for (int kk = 0; kk < D; ++kk) {
    G[0][kk] = T(0);
#pragma unroll
    for (int j = 0; j < D; ++j)
      G[1 + j][kk] = kk == k ? (j == k ? (T(4) / T(3)) * m[k] : m[j])
                             : j == k ? m[kk] : j == kk ? (T(-2) / T(3)) * m[k] : S(T(0));
    G[D + 1][kk] = e[kk];
  }
}
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void visc_K_rank1(const S* u, const S* a, S (*G)[D],
                                             const Phys<T>& ph) {
  Prim<D, S> P;
  primitives<D, S, T>(u, ph, P);
  S m[D], e[D];
  visc_rank1<D, k, S, T>(P, a, T(1), m, e, ph);
  rank1_tensor<D, k, S, T>(m, e, G);
}

// |lam| smoothed to (lam^2 + delta^2) / (2 delta) below delta; ihd = 1 / (2 delta)
template <class S, class T>
__host__ __device__ __forceinline__ S entropy_fixed_abs(S lam, S delta, S ihd) {
  const S a = sabs(lam);
  if (val(delta) > T(0) && val(a) < val(delta)) return madd(lam, lam, delta * delta) * ihd;
  return a;
}

// Roe flux with normal +e_k: 1/2 (F_c(uL) + F_c(uR)).e_k - 1/2 |A_Roe| (uR - uL),
// the primitives of both sides given.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void roe_flux(const S* uL, const S* uR, const Prim<D, S>& L, const Prim<D, S>& R,
                                                  S* Fh, const Phys<T>& ph) {
  constexpr int M = D + 2;
  const S sL = dsqrt(uL[0], L.ir), sR = dsqrt(uR[0], R.ir);
  const S wL = sL * (T(1) / (sL + sR));          // Roe weight of L; R has 1 - wL
  const S rho = sL * sR;
  S vel[D], dv[D], q2 = T(0), vt = T(0);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    dv[j] = R.vel[j] - L.vel[j];
    vel[j] = msub(wL, dv[j], R.vel[j]);
    q2 = j == 0 ? vel[0] * vel[0] : madd(vel[j], vel[j], q2);
  }
  const S h0 = msub(wL, R.h0 - L.h0, R.h0);
  const S c2 = ph.gm1 * msub(T(0.5), q2, h0), ic2 = T(1) / c2;
  const S c = dsqrt(c2, ic2);
  const S vn = vel[k], dp = R.p - L.p;
  const S pa = dp * (T(0.5) * ic2), pb = (rho * dv[k]) * (T(0.5) * c * ic2);   // wave strengths pa -+ pb
  const S delta = ph.roe_delta * c;
  const S ihd = ph.roe_delta > T(0) ? (ph.half_inv_delta() * c) * ic2 : S(T(0));
  const S l1 = entropy_fixed_abs<S, T>(vn - c, delta, ihd) * (pa - pb);
  const S l2 = entropy_fixed_abs<S, T>(vn, delta, ihd);
  const S l3 = entropy_fixed_abs<S, T>(vn + c, delta, ihd) * (pa + pb);
  const S sum = l1 + l3, dif = (l3 - l1) * c;
  const S ent = l2 * msub(T(2), pa, uR[0] - uL[0]), shr = l2 * rho, mass = sum + ent;
  Fh[0] = T(0.5) * ((uL[1 + k] + uR[1 + k]) - mass);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    S f = madd(uL[1 + j], L.vel[k], uR[1 + j] * R.vel[k]);
    f = msub(vel[j], mass, f);
    if (j == k) {
      f = f + ((L.p + R.p) - dif);
    } else {
      const S t = shr * dv[j];
      f = f - t;
      vt = madd(vel[j], t, vt);
    }
    Fh[1 + j] = T(0.5) * f;
  }
  S f = madd(uL[1 + k], L.h0, uR[1 + k] * R.h0) - vt;
  f = msub(h0, sum, f);
  f = msub(vn, dif, f);
  Fh[M - 1] = T(0.5) * msub(T(0.5) * q2, ent, f);
}
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void roe_flux(const S* uL, const S* uR, S* Fh, const Phys<T>& ph) {
  Prim<D, S> L, R;
  primitives<D, S, T>(uL, ph, L);
  primitives<D, S, T>(uR, ph, R);
  roe_flux<D, k, S, T>(uL, uR, L, R, Fh, ph);
}

// Pointwise physics of one face point, normal +e_k from L (its xi_k = +1 side)
// to R.  fp = Roe(uL, uR) + {F_v}.e_k; with jump = uL - uR, (mL, eL) and (mR,
// eR) are the entries (visc_rank1) of half the tensors K(uL), K(uR) (jump (x)
// e_k): twice their normal columns are the BR2 lifting integrands of eq. re,
// the tensors themselves the dual-consistency term of eq. dg_ns ((u+ - uhat) =
// jump/2).  The direction is a compile-time constant: no local array is
// indexed at run time.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void face_point_core(const S* uL, const S (*gL)[D], const S* uR, const S (*gR)[D],
                                                         const Phys<T>& ph, S* fp, S* mL, S* eL, S* mR, S* eR) {
  constexpr int M = D + 2;
  Prim<D, S> L, R;
  primitives<D, S, T>(uL, ph, L);
  primitives<D, S, T>(uR, ph, R);
  roe_flux<D, k, S, T>(uL, uR, L, R, fp, ph);
  add_visc_col<D, k, S, T>(L, gL, T(0.5), fp, ph);
  add_visc_col<D, k, S, T>(R, gR, T(0.5), fp, ph);
  S jump[M];
#pragma unroll
  for (int v = 0; v < M; ++v) jump[v] = uL[v] - uR[v];
  visc_rank1<D, k, S, T>(L, jump, T(0.5), mL, eL, ph);
  visc_rank1<D, k, S, T>(R, jump, T(0.5), mR, eR, ph);
}
template <int D, class S, class T>
__host__ __device__ __forceinline__ void face_point_core_k(int k, const S* uL, const S (*gL)[D], const S* uR,
                                                           const S (*gR)[D], const Phys<T>& ph, S* fp, S* mL, S* eL,
                                                           S* mR, S* eR) {
  if (k == 0) {
    face_point_core<D, 0, S, T>(uL, gL, uR, gR, ph, fp, mL, eL, mR, eR);
  } else if (k == 1) {
    face_point_core<D, 1, S, T>(uL, gL, uR, gR, ph, fp, mL, eL, mR, eR);
  } else {
    if constexpr (D == 3) face_point_core<D, 2, S, T>(uL, gL, uR, gR, ph, fp, mL, eL, mR, eR);
  }
}

// The same with full tensors: GLn/GRn = normal column of K(uL)/K(uR) (jump (x)
// e_k), DL/DR = half the full tensors.
template <int D, int k, class S, class T>
__host__ __device__ __forceinline__ void face_point(const S* uL, const S (*gL)[D], const S* uR,
                                                    const S (*gR)[D], const Phys<T>& ph, S* fp, S* GLn,
                                                    S* GRn, S (*DL)[D], S (*DR)[D]) {
  constexpr int M = D + 2;
  S mL[D], eL[D], mR[D], eR[D];
  face_point_core<D, k, S, T>(uL, gL, uR, gR, ph, fp, mL, eL, mR, eR);
  rank1_tensor<D, k, S, T>(mL, eL, DL);
  rank1_tensor<D, k, S, T>(mR, eR, DR);
#pragma unroll
  for (int v = 0; v < M; ++v) {
    GLn[v] = T(2) * DL[v][k];
    GRn[v] = T(2) * DR[v][k];
  }
}

template <int D, class S, class T>
__host__ __device__ __forceinline__ void face_point_k(int k, const S* uL, const S (*gL)[D], const S* uR,
                                                      const S (*gR)[D], const Phys<T>& ph, S* fp, S* GLn,
                                                      S* GRn, S (*DL)[D], S (*DR)[D]) {
  if (k == 0) {
    face_point<D, 0, S, T>(uL, gL, uR, gR, ph, fp, GLn, GRn, DL, DR);
  } else if (k == 1) {
    face_point<D, 1, S, T>(uL, gL, uR, gR, ph, fp, GLn, GRn, DL, DR);
  } else {
    if constexpr (D == 3) face_point<D, 2, S, T>(uL, gL, uR, gR, ph, fp, GLn, GRn, DL, DR);
  }
}

// rho > 0 and p > 0 of a point state (primal values), p / (gamma - 1) by the operations
// of primitives(): where the point's primitives are formed as well the compiler
// computes them once, and no product leaves the type's range (rho E does, in FP32,
// where rho is below 1e-22)
template <int D, class S, class T>
__host__ __device__ __forceinline__ bool physical(const S* u, T) {
  const T ir = T(1) / val(u[0]);
  T mv = val(u[1]) * (val(u[1]) * ir);
#pragma unroll
  for (int j = 1; j < D; ++j) mv = val(u[1 + j]) * (val(u[1 + j]) * ir) + mv;
  return val(u[0]) > T(0) && val(u[D + 1]) - T(0.5) * mv > T(0);
}

// ----------------------------------------------------------------- mesh view
template <class T>
struct MeshView {
  int d, m, nm, nb, nq, nqf, E;
  int n[3];
  const int* nbr;          // [E][d][2]   face neighbours (side 0: -e_k, side 1: +e_k)
  const T* vphiT;          // [nm][nq]    basis at volume points (transposed)
  const T* vdphiT;         // [d][nm][nq] physical gradients (transposed)
  const T* vphi;           // [nq][nm]
  const T* vdphi;          // [d][nq][nm]
  const T* vw;             // [nq]        weights * |J|
  const T* fphiT;          // [2d][nm][nqf] traces on local face f = 2k + side
  const T* fdphiT;         // [2d][d][nm][nqf]
  const T* fphi;           // [2d][nqf][nm]
  const T* fdphi;          // [2d][d][nqf][nm]
  const T* fw;             // [d][nqf]    face weights * |J_F|
  const T* lift;           // [2d][nqf q'][nqf q] BR2 lifting operator P[q][q'] (eq. re) incl. 1/(2|J|)
  const T* liftT;          // [2d][2][nqf][nm] lifted test functions of local face f:
                           //   sum_q fw(q) phi_i(q) P[q][q'], P = lift[2k+1] (c=0) or lift[2k] (c=1)
  const T* fpk;            // [2d][nm][nqf][4] (phi_i, d_0 phi_i, .., d_{d-1} phi_i, 0 ..) at face point q
  const T* fpw;            // [2d][nqf][nm][4] the same times the face weight fw(q)
  T detJ;
};

// padded length of a short vector of T in shared memory: a multiple of 16 bytes
__host__ __device__ constexpr int pad16(int n, int size) { return size == 4 ? ((n + 3) & ~3) : ((n + 1) & ~1); }

// N consecutive values from a 16-byte aligned address (N * sizeof(T) a
// multiple of 16): 16-byte loads
template <class T, int N>
__device__ __forceinline__ void ld_vec(const T* p, T* out) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int k = 0; k < N / 4; ++k) {
      const float4 t = reinterpret_cast<const float4*>(p)[k];
      out[4 * k] = t.x;
      out[4 * k + 1] = t.y;
      out[4 * k + 2] = t.z;
      out[4 * k + 3] = t.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
      const double2 t = reinterpret_cast<const double2*>(p)[k];
      out[2 * k] = t.x;
      out[2 * k + 1] = t.y;
    }
  }
}

// the same for stores
template <class T, int N>
__device__ __forceinline__ void st_vec(T* p, const T* v) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int k = 0; k < N / 4; ++k)
      reinterpret_cast<float4*>(p)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < N / 2; ++k) reinterpret_cast<double2*>(p)[k] = make_double2(v[2 * k], v[2 * k + 1]);
  }
}

}  // namespace dgk
