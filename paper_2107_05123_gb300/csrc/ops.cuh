// Element operators of the CHNS scheme (Sec. 4.1), each as a small struct with
//   load(...)  : gather the element's coefficient fields (hanging-interpolated) and prepare
//                per-quadrature-point data,
//   apply(...) : local y_e = A_e x_e for NC components.
// The same structs drive the matrix-free apply kernel and the exact diagonal kernel.
//
// In FP64 these forms are bound by the FP64 pipe (two operations per clock and SM on GB300), so they
// are written for few operations: unnormalised 1D interpolations of two FMAs whose factors go into
// constants, Kronecker products for the constant-coefficient terms, physical scalings on the 12
// compact gradient values instead of at 8 points, one reciprocal and one reciprocal square root
// per point by a third-order step from the hardware estimate, comparisons in integers. FP64 applies
// of all four operators on 156,640 leaves: 1,562 -> 923 us; the four FP64 right-hand sides and
// residuals on 314,672 leaves 4.82 -> 3.83 ms; FP32 momentum there 76.8 -> 55 us in
// the CTA-per-patch kernel (41.3 us as TileMom).
#pragma once

#include <type_traits>

#include "elem.cuh"

namespace chns {

template <class C>
struct CoefArgs {
  const C* phi;     // phi~ (bfloat16 storage holds 1 + phi~, see phi_shift)
  const C* u[3];    // advecting velocity (u_hat or u~)
  const C* mu;      // mu~
  float phi_shift;  // added to the stored phi values: -1 for bfloat16 storage, else 0
  const void* qd = nullptr;  // quadrature data of operators that precompute it (MomQK)
};

// Gather phi~ of an element. In bfloat16 storage the field is s = 1 + phi~, whose relative
// precision bounds the relative error of rho(phi) = alpha s + rho_- by 2^-8 even where
// rho_- << 1 (phi near -1); the shift is removed after interpolation (linear in s).
template <class T, class C>
__device__ __forceinline__ void gather_phi(const MeshDev& m, const int idx[8],
                                           const CoefArgs<C>& cf, T pe[8]) {
  gather<T, false>(m, idx, cf.phi, pe);
#pragma unroll
  for (int a = 0; a < 8; ++a) pe[a] += T(cf.phi_shift);
}

// ---------------------------------------------------------------- pressure Poisson
// (grad q, (1/rho(phi~*)) grad p) (Def. weak_VMS_disc_pp_vel, scalar test q), sum-factorised:
// r_a = sum_q c_q grad N_a(q) . grad u(q) with c = 1/rho.
template <class T, class C>
struct PoissonK {
  static constexpr bool QDATA = false;
  // CTAs of the patch apply resident per SM that the register allocation must allow (FP32: 5, i.e. at
  // most 51 registers; FP64: 3). Meshes of up to 8 patches per SM take this kernel in FP32: at 6 CTAs
  // and 40 registers it spills, 6.9 us on 77,932 leaves and 8.1 on 156,640 against 6.7 and 7.8.
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 5 : 3;
  static constexpr int NC = 1;
  static constexpr bool DIR = false;
  static constexpr bool DIAG_PER_COMP = false;
  static constexpr int NF = 1;  // coefficient fields: phi~
  T c[8];
  __device__ __forceinline__ void setup(const T f[NF][8], const Geo<T>&, const DevParams& p) {
    const PrmT<T>& k = p.get<T>();
    interp3<true>(f[0], c);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const T rho = mad(k.alpha, clamp1(c[q]), k.beta);
      if constexpr (sizeof(T) == 4)
        c[q] = __fdividef(1.f, rho);  // two ulp; the FP32 solves are refined in FP64
      else
        c[q] = recip(rho);
    }
  }
  __device__ __forceinline__ void load(const MeshDev& m, const DevParams& p, const CoefArgs<C>& cf,
                                       const int idx[8], const Geo<T>& g) {
    T f[NF][8];
    gather_phi(m, idx, cf, f[0]);
    setup(f, g, p);
  }
  __device__ __forceinline__ void apply(const Geo<T>& g, const DevParams&, const T x[NC][8],
                                        T r[NC][8]) const {
    stiff<false>(g, x[0], r[0]);
  }
  // apply and the element energy x . A_e x = sum_q c_q |grad x(q)|^2, formed from the per-axis
  // gradient data (a sum of non-negative terms, accurate in the working precision)
  static constexpr bool ENERGY = true;
  __device__ __forceinline__ T apply_energy(const Geo<T>& g, const DevParams&, const T x[NC][8],
                                            T r[NC][8]) const {
    return stiff<true>(g, x[0], r[0]);
  }

 private:
  template <bool E>
  __device__ __forceinline__ T stiff(const Geo<T>& g, const T u[8], T r[8]) const {
    constexpr double w = gauss_w<T>();
    GradC<T> d;
    d.eval(u);
    const T j = g.detJ * T(w * w * w * w);
    const T sc[3] = {j * g.ih[0] * g.ih[0], j * g.ih[1] * g.ih[1], j * g.ih[2] * g.ih[2]};
    T e[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // the two points that share a component: q and q + step
      const int qx = 2 * i, qy = (i & 1) + 4 * (i >> 1), qz = i;
      const T sx = d.x[i] * (c[qx] + c[qx + 1]), sy = d.y[i] * (c[qy] + c[qy + 2]),
              sz = d.z[i] * (c[qz] + c[qz + 4]);
      if (E) {
        e[0] = mad(d.x[i], sx, e[0]);
        e[1] = mad(d.y[i], sy, e[1]);
        e[2] = mad(d.z[i], sz, e[2]);
      }
      d.x[i] = sx;
      d.y[i] = sy;
      d.z[i] = sz;
    }
#pragma unroll
    for (int a = 0; a < 8; ++a) r[a] = T(0);
    d.transpose(sc, r);
    return mad(sc[0], e[0], mad(sc[1], e[1], sc[2] * e[2]));
  }
};

// ---------------------------------------------------------------- velocity update mass
// (w, rho~ u) per component (Def. weak_VMS_disc_vel_update); Dirichlet rows are identity.
template <class T, class C>
struct MassK {
  static constexpr bool QDATA = false;
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 5 : 3;
  static constexpr int NC = 3;
  static constexpr bool DIR = true;
  static constexpr bool DIAG_PER_COMP = false;
  static constexpr int NF = 1;  // phi~
  // FP32 keeps the normalised interpolation (rounding 5.6e-8 against 9.7e-8)
  static constexpr bool NORM = sizeof(T) == 4;
  T c[8];
  __device__ __forceinline__ void setup(const T f[NF][8], const Geo<T>& g, const DevParams& p) {
    constexpr double w = NORM ? 1.0 : gauss_w<T>();
    const PrmT<T>& k = p.get<T>();
    const T j = g.detJ * T(w * w * w * w * w * w);
    interp3<true>(f[0], c);
#pragma unroll
    for (int q = 0; q < 8; ++q) c[q] = j * mad(k.alpha, clamp1(c[q]), k.beta);
  }
  __device__ __forceinline__ void load(const MeshDev& m, const DevParams& p, const CoefArgs<C>& cf,
                                       const int idx[8], const Geo<T>& g) {
    T f[NF][8];
    gather_phi(m, idx, cf, f[0]);
    setup(f, g, p);
  }
  __device__ __forceinline__ void apply(const Geo<T>&, const DevParams&, const T x[NC][8],
                                        T r[NC][8]) const {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      T v[8];
      interp3<NORM>(x[k], v);
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] *= c[q];
      interp3<NORM>(v, r[k]);
    }
  }
};

// ---------------------------------------------------------------- shifted Laplacian
// sa (q, u) + sb (grad q, grad u) with constant sa, sb >= 0 (DevParams sa, sb): the operator of
// the inner solves of the Cahn-Hilliard Schur-complement preconditioner. No Dirichlet rows.
template <class T, class C>
struct ShiftK {
  static constexpr bool QDATA = false;
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 6 : 3;
  static constexpr int NC = 1;
  static constexpr bool DIR = false;
  static constexpr bool DIAG_PER_COMP = false;
  static constexpr int NF = 1;  // (phi~ gathered but unused: the patch kernel's layout)
  static constexpr bool IGNORES_FIELDS = true;
  // y = Px (cm B + cy C + cz E) + cx Dx B (see Kron)
  T cm, cx, cy, cz;
  __device__ __forceinline__ void setup(const T[NF][8], const Geo<T>& g, const DevParams& p) {
    const PrmT<T>& k = p.get<T>();
    const T V = T(8) * g.detJ;
    cm = k.sa * V * T(1.0 / 216.0);
    const T ks = k.sb * V * T(1.0 / 36.0);
    cx = ks * g.ih[0] * g.ih[0];
    cy = ks * g.ih[1] * g.ih[1];
    cz = ks * g.ih[2] * g.ih[2];
  }
  __device__ __forceinline__ void load(const MeshDev&, const DevParams& p, const CoefArgs<C>&,
                                       const int[8], const Geo<T>& g) {
    const T f[NF][8] = {};
    setup(f, g, p);
  }
  // sb = 0 (the mass M of the Schur preconditioner) skips the stiffness part: the branch is
  // uniform over the whole launch
  __device__ __forceinline__ void apply(const Geo<T>&, const DevParams&, const T x[NC][8],
                                        T r[NC][8]) const {
    Kron<T> k;
    T S[8];
    if (cx == T(0) && cy == T(0) && cz == T(0)) {
      k.mass(x[0]);
#pragma unroll
      for (int a = 0; a < 8; ++a) S[a] = cm * k.B[a];
    } else {
      k.eval(x[0]);
#pragma unroll
      for (int a = 0; a < 8; ++a) S[a] = mad(cm, k.B[a], mad(cy, k.c_at(a), cz * k.e_at(a)));
    }
    k.finish(S, cx, r[0]);
  }
};

// ---------------------------------------------------------------- Cahn-Hilliard Jacobian
// Newton Jacobian of Def. weak_VMS_disc_CH in (dphi, dmu), with phi~ the current iterate and
// u~ the advecting velocity (diffusion term with a plus sign, as in the strong form):
//   row phi: (q, dphi)/dt - 1/2 (grad q, u~ dphi) + 1/(2 Pe Cn) (grad q, grad dmu)
//   row mu : -1/2 (q, dmu) + 1/2 (q, psi''(phi~) dphi) + Cn^2/2 (grad q, grad dphi)
template <class T, class C>
struct ChK {
  static constexpr bool QDATA = false;
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 4 : 1;
  static constexpr int NC = 2;
  static constexpr bool DIR = false;
  static constexpr bool DIAG_PER_COMP = true;
  static constexpr int NF = 4;  // phi~, u~ (3)
  T pe[8];
  T ue[3][8];
  __device__ __forceinline__ void setup(const T f[NF][8], const Geo<T>&, const DevParams&) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      pe[a] = f[0][a];
      ue[0][a] = f[1][a];
      ue[1][a] = f[2][a];
      ue[2][a] = f[3][a];
    }
  }
  __device__ __forceinline__ void load(const MeshDev& m, const DevParams&, const CoefArgs<C>& cf,
                                       const int idx[8], const Geo<T>&) {
    gather_phi(m, idx, cf, pe);
#pragma unroll
    for (int d = 0; d < 3; ++d) gather<T, false>(m, idx, cf.u[d], ue[d]);
  }
  // The constant-coefficient terms are Kronecker products (Kron); the psi'' and advection terms are
  // evaluated at the Gauss points, sum-factorised.
  __device__ __forceinline__ void apply(const Geo<T>& g, const DevParams& p, const T x[NC][8],
                                        T r[NC][8]) const {
    constexpr double w = gauss_w<T>(), w3 = w * w * w;
    const PrmT<T>& pk = p.get<T>();
    const T J = g.detJ, V = T(8) * J;
    {
      const T cm = V * T(1.0 / 216.0), ks = V * T(1.0 / 36.0);
      const T kh[3] = {ks * g.ih[0] * g.ih[0], ks * g.ih[1] * g.ih[1], ks * g.ih[2] * g.ih[2]};
      Kron<T> f, m;
      f.eval(x[0]);
      m.eval(x[1]);
      T S[8];
      const T c0 = cm * pk.idt, c0y = pk.kmu * kh[1], c0z = pk.kmu * kh[2];
#pragma unroll
      for (int a = 0; a < 8; ++a)
        S[a] = mad(c0, f.B[a], mad(c0y, m.c_at(a), c0z * m.e_at(a)));
      m.finish(S, pk.kmu * kh[0], r[0]);
      const T c1 = T(-0.5) * cm, c1y = pk.kphi * kh[1], c1z = pk.kphi * kh[2];
#pragma unroll
      for (int a = 0; a < 8; ++a)
        S[a] = mad(c1, m.B[a], mad(c1y, f.c_at(a), c1z * f.e_at(a)));
      f.finish(S, pk.kphi * kh[0], r[1]);
    }
    T fv[8], s[8], t[8];
    interp3<false>(x[0], fv);
    interp3<false>(pe, t);
    // 1/2 (q, psi''(phi~) dphi), psi'' = 3 phi~^2 - 1
    const T cs = T(0.5 * w3 * w3) * J, c3 = T(3.0 * w3 * w3) * cs;
#pragma unroll
    for (int q = 0; q < 8; ++q) t[q] = mad(c3 * t[q], t[q], -cs) * fv[q];
    interp3<false>(t, s);
#pragma unroll
    for (int a = 0; a < 8; ++a) r[1][a] += s[a];
    // -1/2 (grad q, u~ dphi)
    GradC<T> d;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      interp3<false>(ue[k], t);
#pragma unroll
      for (int q = 0; q < 8; ++q) d.sum(q, k, t[q] * fv[q]);
    }
    const T ca = T(-0.5 * w3 * w3 * w * w) * J;
    const T sc[3] = {ca * g.ih[0], ca * g.ih[1], ca * g.ih[2]};
    d.transpose(sc, r[0]);
  }
};

// ---------------------------------------------------------------- velocity prediction (RBVMS)
// Per-quadrature-point coefficients of the momentum operator (Def. weak_VMS_disc):
//   rho~, eta~ from clamp(phi~); grad eta~ = gamma grad phi~ where |phi~| < 1;
//   J_hat = -(alpha/Cn) grad mu~; G = diag(4/h^2);
//   tau_m = (4/dt^2 + u.G.u + u.G.J/(rho Pe) + C_I (eta/(rho Re))^2 G:G)^(-1/2), the printed
//   radicand floored at 4/dt^2 (tau_m <= dt/2) where its mixed term would take it lower.
// The operator on one velocity component v (the same for each component):
//   s = rho/dt v + 1/2 rho u.grad v + 1/(2Pe) J.grad v                       (tested with N_a)
//   R = s - 1/(2Re) grad eta . grad v                                        (R^lin)
//   V = eta/(2Re) grad v + tau R (u/2 + J/(2 Pe rho))                       (tested with grad N_a)
template <class T>
struct VmsQ {
  T rho, ir, tau, a0, e, gge, b[3], bp[3], t[3];  // gge: gamma/(2Re) where |phi~| < 1, else 0
};

// What the points of an element share: G and the viscous term of tau_m's radicand.
template <class T>
struct VmsElem {
  T G[3], visc;
  __device__ __forceinline__ VmsElem(const Geo<T>& g, const PrmT<T>& k) {
#pragma unroll
    for (int d = 0; d < 3; ++d) G[d] = T(4) * g.ih[d] * g.ih[d];
    visc = k.C_I * k.inv_re * k.inv_re * (G[0] * G[0] + G[1] * G[1] + G[2] * G[2]);
  }
};

// The coefficients at one point from phi~ (pv), grad phi~ (gp), j = J_hat/(2 Pe) and u_hat (u).
template <class T>
__device__ __forceinline__ VmsQ<T> vms_point(T pv, const T gp[3], const T j[3], const T u[3],
                                             const VmsElem<T>& el, const PrmT<T>& k) {
  VmsQ<T> o;
  const T pc = clamp1(pv);
  o.rho = mad(k.alpha, pc, k.beta);
  const T eta = mad(k.gamma, pc, k.xi);
  o.gge = inside1(pv) ? k.h2re * k.gamma : T(0);
  o.ir = recip(o.rho);
  T ugu = k.four_idt2, ugj = T(0);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const T gu = el.G[d] * u[d];
    ugu = mad(gu, u[d], ugu);
    ugj = d == 0 ? gu * j[d] : mad(gu, j[d], ugj);
  }
  const T er = eta * o.ir;
  const T rad = mad(T(2) * o.ir, ugj, mad(er * er, el.visc, ugu));
  o.tau = inv_sqrt(rad > k.four_idt2 ? rad : k.four_idt2);
  o.a0 = o.rho * k.idt;
  o.e = eta * k.h2re;
  const T hr = T(0.5) * o.rho, ht = T(0.5) * o.tau, ti = o.tau * o.ir;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.b[d] = mad(hr, u[d], j[d]);
    o.bp[d] = mad(-o.gge, gp[d], o.b[d]);
    o.t[d] = mad(ht, u[d], ti * j[d]);
  }
  return o;
}

// phi~, grad phi~, J_hat/(2 Pe) and u_hat of an element at its Gauss points.
template <class T>
struct VmsFields {
  T pv[8], uq[3][8];
  GradC<T> gp, gj;
  __device__ __forceinline__ void eval(const T pe[8], const T me[8], const T ue[3][8],
                                       const Geo<T>& g, const PrmT<T>& k) {
    constexpr double w = gauss_w<T>();
    const T w2 = T(w * w), wj = w2 * k.h2pe * k.ka;
    const T cp[3] = {w2 * g.ih[0], w2 * g.ih[1], w2 * g.ih[2]};
    const T cj[3] = {wj * g.ih[0], wj * g.ih[1], wj * g.ih[2]};
    interp3<true>(pe, pv);
    gp.eval(pe, cp);
    gj.eval(me, cj);
#pragma unroll
    for (int d = 0; d < 3; ++d) interp3<true>(ue[d], uq[d]);
  }
  __device__ __forceinline__ VmsQ<T> at(int q, const VmsElem<T>& el, const PrmT<T>& k) const {
    const T p[3] = {gp.at(q, 0), gp.at(q, 1), gp.at(q, 2)};
    const T j[3] = {gj.at(q, 0), gj.at(q, 1), gj.at(q, 2)};
    const T u[3] = {uq[0][q], uq[1][q], uq[2][q]};
    return vms_point(pv[q], p, j, u, el, k);
  }
};

// The momentum operator on three components, point by point: coef(q, a0, b, bp, e, t) gives the
// coefficients of Gauss point q. All components are evaluated first (sum-factorised), the points'
// terms take the place of their values and sum up in compact gradient data, and the transposes
// follow, so that each point's coefficients are needed once.
template <class T, class F>
__device__ __forceinline__ void momentum_apply(const Geo<T>& g, const T x[3][8], T r[3][8], F&& coef) {
  constexpr double w = gauss_w<T>();
  // FP32 keeps the normalised interpolation of the values, as the mass operator does
  constexpr bool NORM = sizeof(T) == 4;
  const T cg[3] = {T(w * w) * g.ih[0], T(w * w) * g.ih[1], T(w * w) * g.ih[2]};
  const T w3 = T(NORM ? 1.0 : w * w * w), j3 = g.detJ * w3;
  T v[3][8];
  GradC<T> d[3], s[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    interp3<NORM>(x[k], v[k]);
    d[k].eval(x[k], cg);
  }
  for_qp([&](auto QC) {
    constexpr int Q = decltype(QC)::value;
    T a0, b[3], bp[3], e, t[3];
    coef(Q, a0, b, bp, e, t);
    a0 *= w3;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const T vg[3] = {d[k].at(Q, 0), d[k].at(Q, 1), d[k].at(Q, 2)};
      const T av = a0 * v[k][Q];
      const T R = mad(bp[0], vg[0], mad(bp[1], vg[1], mad(bp[2], vg[2], av)));
      v[k][Q] = j3 * mad(b[0], vg[0], mad(b[1], vg[1], mad(b[2], vg[2], av)));
#pragma unroll
      for (int i = 0; i < 3; ++i) s[k].sum(Q, i, mad(R, t[i], e * vg[i]));
    }
  });
  const T sc[3] = {g.detJ * cg[0], g.detJ * cg[1], g.detJ * cg[2]};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    interp3<NORM>(v[k], r[k]);
    s[k].transpose(sc, r[k]);
  }
}

// The same in packed FP32: the pair of Gauss points along x of line j = qy + 2 qz at once.
__device__ __forceinline__ VmsQ<F2> vms_point(F2 pv, const F2 gp[3], const F2 j[3], const F2 u[3],
                                              const VmsElem<float>& el, const PrmT<float>& k) {
  VmsQ<F2> o;
  const F2 pc = clamp_nan(pv, -1.f, 1.f);
  o.rho = mad(F2(k.alpha), pc, F2(k.beta));
  const F2 eta = mad(F2(k.gamma), pc, F2(k.xi));
  const float gge = k.h2re * k.gamma;
  o.gge = F2(inside1(pv.x) ? gge : 0.f, inside1(pv.y) ? gge : 0.f);
  o.ir = F2(recip(o.rho.x), recip(o.rho.y));
  F2 ugu(k.four_idt2), ugj(0.f);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const F2 gu = F2(el.G[d]) * u[d];
    ugu = mad(gu, u[d], ugu);
    ugj = d == 0 ? gu * j[d] : mad(gu, j[d], ugj);
  }
  const F2 er = eta * o.ir;
  const F2 rad = mad(F2(2.f) * o.ir, ugj, mad(er * er, F2(el.visc), ugu));
  o.tau = F2(inv_sqrt(rad.x > k.four_idt2 ? rad.x : k.four_idt2),
             inv_sqrt(rad.y > k.four_idt2 ? rad.y : k.four_idt2));
  o.a0 = o.rho * F2(k.idt);
  o.e = eta * F2(k.h2re);
  const F2 hr = F2(0.5f) * o.rho, ht = F2(0.5f) * o.tau, ti = o.tau * o.ir;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    o.b[d] = mad(hr, u[d], j[d]);
    o.bp[d] = mad(-o.gge, gp[d], o.b[d]);
    o.t[d] = mad(ht, u[d], ti * j[d]);
  }
  return o;
}

struct VmsFieldsP {
  F2 pv[4], uq[3][4];
  GradP gp, gj;
  __device__ __forceinline__ void eval(const float pe[8], const float me[8], const float ue[3][8],
                                       const Geo<float>& g, const PrmT<float>& k) {
    constexpr double w = gauss_w<float>();
    const float w2 = (float)(w * w), wj = w2 * k.h2pe * k.ka;
    const float cp[3] = {w2 * g.ih[0], w2 * g.ih[1], w2 * g.ih[2]};
    const float cj[3] = {wj * g.ih[0], wj * g.ih[1], wj * g.ih[2]};
    interp3<true>(pe, pv);
    gp.eval(pe, cp);
    gj.eval(me, cj);
#pragma unroll
    for (int d = 0; d < 3; ++d) interp3<true>(ue[d], uq[d]);
  }
  __device__ __forceinline__ VmsQ<F2> at(int q, const VmsElem<float>& el,
                                         const PrmT<float>& k) const {
    const F2 p[3] = {gp.at(q, 0), gp.at(q, 1), gp.at(q, 2)};
    const F2 j[3] = {gj.at(q, 0), gj.at(q, 1), gj.at(q, 2)};
    const F2 u[3] = {uq[0][q], uq[1][q], uq[2][q]};
    return vms_point(pv[q], p, j, u, el, k);
  }
};

// coef(j, ...) gives the coefficients of the point pair j
template <class F>
__device__ __forceinline__ void momentum_apply_pairs(const Geo<float>& g, const float x[3][8],
                                                     float r[3][8], F&& coef) {
  constexpr double w = gauss_w<float>();
  const float cg[3] = {(float)(w * w) * g.ih[0], (float)(w * w) * g.ih[1],
                       (float)(w * w) * g.ih[2]};
  F2 v[3][4];
  GradP d[3], s[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    interp3<true>(x[k], v[k]);
    d[k].eval(x[k], cg);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    F2 a0, b[3], bp[3], e, t[3];
    coef(q, a0, b, bp, e, t);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const F2 vg[3] = {d[k].at(q, 0), d[k].at(q, 1), d[k].at(q, 2)};
      const F2 av = a0 * v[k][q];
      const F2 R = mad(bp[0], vg[0], mad(bp[1], vg[1], mad(bp[2], vg[2], av)));
      v[k][q] = F2(g.detJ) * mad(b[0], vg[0], mad(b[1], vg[1], mad(b[2], vg[2], av)));
#pragma unroll
      for (int i = 0; i < 3; ++i) s[k].sum(q, i, mad(R, t[i], e * vg[i]));
    }
  }
  const float sc[3] = {g.detJ * cg[0], g.detJ * cg[1], g.detJ * cg[2]};
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    F2 o[4];
    interp3_t<true>(v[k], o);
    s[k].transpose(sc, o);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      r[k][2 * j] = o[j].x;
      r[k][2 * j + 1] = o[j].y;
    }
  }
}

template <class T, class C>
struct MomK {
  static constexpr bool QDATA = false;
  // FP32: two CTAs per SM (at most 128 registers)
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 2 : 1;
  static constexpr int NC = 3;
  static constexpr bool DIR = true;
  static constexpr bool DIAG_PER_COMP = false;
  static constexpr int NF = 5;  // phi~, u_hat (3), mu~
  T pe[8];
  T ue[3][8];
  T me[8];
  __device__ __forceinline__ void setup(const T f[NF][8], const Geo<T>&, const DevParams&) {
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      pe[a] = f[0][a];
      ue[0][a] = f[1][a];
      ue[1][a] = f[2][a];
      ue[2][a] = f[3][a];
      me[a] = f[4][a];
    }
  }
  __device__ __forceinline__ void load(const MeshDev& m, const DevParams&, const CoefArgs<C>& cf,
                                       const int idx[8], const Geo<T>&) {
    gather_phi(m, idx, cf, pe);
#pragma unroll
    for (int d = 0; d < 3; ++d) gather<T, false>(m, idx, cf.u[d], ue[d]);
    gather<T, false>(m, idx, cf.mu, me);
  }
  __device__ __forceinline__ void apply(const Geo<T>& g, const DevParams& p, const T x[NC][8],
                                        T r[NC][8]) const {
    const PrmT<T>& k = p.get<T>();
    const VmsElem<T> el(g, k);
    VmsFields<T> f;
    f.eval(pe, me, ue, g, k);
    momentum_apply(g, x, r, [&](int q, T& a0, T b[3], T bp[3], T& e, T t[3]) {
      const VmsQ<T> c = f.at(q, el, k);
      a0 = c.a0;
      e = c.e;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        b[d] = c.b[d];
        bp[d] = c.bp[d];
        t[d] = c.t[d];
      }
    });
  }
};

// Quadrature data of the momentum operator: per element and quadrature point the 11 values
// the linear operator needs (a0, b[3], bp[3], e, t[3] of VmsQ), computed once per solve while
// the coefficients are fixed, stored value-major, qd[(q * kMomQ + v) * n_elem + e], so that a
// warp's loads are coalesced. The apply then reads 88 values per element instead of
// re-evaluating tau_m and the RBVMS vectors at every quadrature point (FP64 arithmetic is the
// bound of that evaluation on GB300).
constexpr int kMomQ = 11;

template <class T, class C>
__global__ void __launch_bounds__(128)
k_mom_qdata(MeshDev m, DevParams p, CoefArgs<C> cf, T* __restrict__ qd) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  const PrmT<T>& pk = p.get<T>();
  int idx[8];
  load_corners(m, e, idx);
  const Geo<T> g = geometry<T>(m, e);
  MomK<T, C> k;
  k.load(m, p, cf, idx, g);
  const int64_t E = m.n_elem;
  const VmsElem<T> el(g, pk);
  VmsFields<T> f;
  f.eval(k.pe, k.me, k.ue, g, pk);
  for_qp([&](auto QC) {
    constexpr int Q = decltype(QC)::value;
    const VmsQ<T> c = f.at(Q, el, pk);
    T* q = qd + (int64_t)Q * kMomQ * E + e;
    q[0] = c.a0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      q[(1 + d) * E] = c.b[d];
      q[(4 + d) * E] = c.bp[d];
      q[(8 + d) * E] = c.t[d];
    }
    q[7 * E] = c.e;
  });
}

// The momentum operator from quadrature data (same arithmetic as MomK::apply).
template <class T, class C>
struct MomQK {
  static constexpr bool QDATA = true;
  static constexpr int MIN_CTAS = sizeof(T) == 4 ? 2 : 1;
  static constexpr int NC = 3;
  static constexpr bool DIR = true;
  static constexpr bool DIAG_PER_COMP = false;
  static constexpr int NF = 1;  // (phi~ only to keep the shared-memory layout of the kernel)
  const AccumT<T>* qd = nullptr;  // FP64 data for double-float
  int64_t ne = 0, e = 0;
  __device__ __forceinline__ void setup(const T[NF][8], const Geo<T>&, const DevParams&) {}
  __device__ __forceinline__ void load(const MeshDev&, const DevParams&, const CoefArgs<C>&,
                                       const int[8], const Geo<T>&) {}
  __device__ __forceinline__ void bind(const void* q, int64_t n_elem, int64_t elem) {
    qd = static_cast<const AccumT<T>*>(q);
    ne = n_elem;
    e = elem;
  }
  __device__ __forceinline__ void apply(const Geo<T>& g, const DevParams&, const T x[NC][8],
                                        T r[NC][8]) const {
    momentum_apply(g, x, r, [&](int q, T& a0, T b[3], T bp[3], T& ce, T t[3]) {
      const AccumT<T>* c = qd + (int64_t)q * kMomQ * ne + e;
      a0 = T(__ldg(c));
      ce = T(__ldg(c + 7 * ne));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        b[d] = T(__ldg(c + (1 + d) * ne));
        bp[d] = T(__ldg(c + (4 + d) * ne));
        t[d] = T(__ldg(c + (8 + d) * ne));
      }
    });
  }
};

// Operators that form the element energy x . A_e x alongside the apply (ENERGY = true).
template <class K, class = void>
struct HasEnergy : std::false_type {};
template <class K>
struct HasEnergy<K, std::void_t<decltype(K::ENERGY)>> : std::bool_constant<K::ENERGY> {};

// Operators whose element kernel never reads the coefficient fields it is handed (the shifted
// operator's coefficients are constants): the persistent apply gathers none for them.
template <class K, class = void>
struct IgnoresFields : std::false_type {};
template <class K>
struct IgnoresFields<K, std::void_t<decltype(K::IGNORES_FIELDS)>>
    : std::bool_constant<K::IGNORES_FIELDS> {};

}  // namespace chns
