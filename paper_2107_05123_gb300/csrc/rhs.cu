// Right-hand sides and nonlinear residuals of the time step (FP64), and the phi mass integral.
// These are the "vector assembly" traversals of the paper (Sec. 5.4), done matrix-free with the
// same gather / element quadrature / scatter-add skeleton as the operator applies.
#include <vector>

#include "ops.cuh"

namespace chns {

constexpr int kRhsThreads = 128;
// gravity direction g_hat = (0, -1, 0) (Sec. 3): the sign of the y component
__device__ __forceinline__ int ghat(int i) { return i == 1 ? -1 : 0; }

struct Ptr3 {
  const double* c[3];
};

// The kernels below are written for an arithmetic type A and run in FP64 (A = double): in
// double-float (dfloat.cuh) they measured about 3x slower, their register pressure and spills
// outweighing the FP32 issue rate. Fields are read from and results added to FP64 arrays.

// ---- CH residual at the new-time iterate (Def. weak_VMS_disc_CH):
//   F_phi = (q, (phi - phi_k)/dt) - (grad q, u~ phi~) + 1/(Pe Cn) (grad q, grad mu~)
//   F_mu  = -(q, mu~) + (q, psi'(phi~)) + Cn^2 (grad q, grad phi~)
template <class A>
__global__ void __launch_bounds__(kRhsThreads)
k_residual_ch(MeshDev m, DevParams p, const double* __restrict__ phi, const double* __restrict__ mu,
              const double* __restrict__ phik, const double* __restrict__ muk, Ptr3 u,
              double* __restrict__ f) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  const PrmT<A>& k = p.get<A>();
  int idx[8];
  load_corners(m, e, idx);
  const Geo<A> g = geometry<A>(m, e);
  A a[8], b[8], pt[8], mt[8], dp[8], ue[3][8];
  gather<A, false>(m, idx, phi, a);
  gather<A, false>(m, idx, phik, b);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    pt[i] = A(0.5) * (a[i] + b[i]);
    dp[i] = (a[i] - b[i]) * k.idt;
  }
  gather<A, false>(m, idx, mu, a);
  gather<A, false>(m, idx, muk, b);
#pragma unroll
  for (int i = 0; i < 8; ++i) mt[i] = A(0.5) * (a[i] + b[i]);
#pragma unroll
  for (int d = 0; d < 3; ++d) gather<A, false>(m, idx, u.c[d], ue[d]);
  // the constant-coefficient terms as Kronecker products (Kron), psi' and the advection at the
  // Gauss points
  constexpr double w = gauss_w<A>(), w3 = w * w * w;
  const A J = g.detJ, Vol = A(8) * J, cm = Vol * A(1.0 / 216.0), ks = Vol * A(1.0 / 36.0);
  const A kh[3] = {ks * g.ih[0] * g.ih[0], ks * g.ih[1] * g.ih[1], ks * g.ih[2] * g.ih[2]};
  A r0[8], r1[8], s[8];
  {
    Kron<A> kd, kp, kq;
    kd.mass(dp);
    kq.eval(mt);
    const A cy = k.inv_pecn * kh[1], cz = k.inv_pecn * kh[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = mad(cm, kd.B[i], mad(cy, kq.c_at(i), cz * kq.e_at(i)));
    kq.finish(s, k.inv_pecn * kh[0], r0);
    kp.eval(pt);
    const A py = k.cn2 * kh[1], pz = k.cn2 * kh[2];
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = mad(-cm, kq.B[i], mad(py, kp.c_at(i), pz * kp.e_at(i)));
    kp.finish(s, k.cn2 * kh[0], r1);
  }
  // phi~ normalised, so that a pure phase (phi = 1 or -1, mu = 0) has no residual, without rounding
  A pv[8];
  interp3<true>(pt, pv);
  const A c1 = J * A(w3);
#pragma unroll
  for (int q = 0; q < 8; ++q) s[q] = mad(c1 * pv[q], pv[q], -c1) * pv[q];
  A t[8];
  interp3<false>(s, t);
#pragma unroll
  for (int i = 0; i < 8; ++i) r1[i] += t[i];
  GradC<A> d;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    interp3<false>(ue[c], t);
#pragma unroll
    for (int q = 0; q < 8; ++q) d.sum(q, c, t[q] * pv[q]);
  }
  const A ca = J * A(-w3 * w * w);
  const A sc[3] = {ca * g.ih[0], ca * g.ih[1], ca * g.ih[2]};
  d.transpose(sc, r0);
  scatter<A, false>(m, idx, r0, f);
  scatter<A, false>(m, idx, r1, f + m.n_nodes);
}

// Mixed second derivatives of the trilinear interpolant (the pure ones vanish on box elements):
// H_xy depends on qz only, H_xz on qy, H_yz on qx. Forcing d_j(d_i phi d_j phi) at a point:
// F_i = sum_{j != i} H_ij d_j phi.
template <class A>
struct Forcing {
  A xy[2], xz[2], yz[2];
  __device__ __forceinline__ Forcing(const A u[8], const Geo<A>& g, const A& scale) {
    constexpr double w = gauss_w<A>();
    const A c = A(w) * scale;
    it(u[3] - u[2] - u[1] + u[0], u[7] - u[6] - u[5] + u[4], xy[0], xy[1]);
    it(u[5] - u[4] - u[1] + u[0], u[7] - u[6] - u[3] + u[2], xz[0], xz[1]);
    it(u[6] - u[4] - u[2] + u[0], u[7] - u[5] - u[3] + u[1], yz[0], yz[1]);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      xy[i] *= c * g.ih[0] * g.ih[1];
      xz[i] *= c * g.ih[0] * g.ih[2];
      yz[i] *= c * g.ih[1] * g.ih[2];
    }
  }
  // component i at point q, times the scale, added to v
  __device__ __forceinline__ A add(int q, int i, const A gp[3], A v) const {
    const A a = xy[q >> 2], b = xz[q >> 1 & 1], c = yz[q & 1];
    return i == 0   ? mad(a, gp[1], mad(b, gp[2], v))
           : i == 1 ? mad(a, gp[0], mad(c, gp[2], v))
                    : mad(b, gp[0], mad(c, gp[1], v));
  }
};

// ---- velocity-prediction right-hand side (Def. weak_VMS_disc), per component i:
//   (w, rho u_i/dt) - 1/2 (w, rho u.grad u_i) - 1/(2Pe) (w, J.grad u_i) - 1/(2Re) (grad w, eta grad u_i)
//   + Cn/We (d_j w, d_i phi d_j phi) - (w, d_i p) + (w, rho g_i/Fr) - (grad w . t, R0_i)
// with R0_i the part of R_m that does not depend on v^{k+1}.
// Every field's values and gradients at the 8 Gauss points come from interp3 / GradC. For each point
// the coefficients (tau_m and the advection and stabilisation vectors) are formed once and the
// three components' terms take the place of their values and sum up in compact gradient data; the
// transposes follow. Values and their transposes are interpolated normalised here and in the velocity
// update: unnormalised they cost 24 FP64 operations less per component (rhs of 314,672 leaves 3.75
// against 3.82 ms), but the right-hand sides' errors against an 80-bit reference were 9 and 7 % larger
// and constant states were no longer exact.
template <class A>
__global__ void __launch_bounds__(kRhsThreads)
k_rhs_momentum(MeshDev m, DevParams p, CoefArgs<double> cf, Ptr3 uk,
               const double* __restrict__ pk, double* __restrict__ b) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  constexpr double w = gauss_w<A>();
  const PrmT<A>& k = p.get<A>();
  int idx[8];
  load_corners(m, e, idx);
  const Geo<A> g = geometry<A>(m, e);
  const A J = g.detJ;
  const A cg[3] = {A(w * w) * g.ih[0], A(w * w) * g.ih[1], A(w * w) * g.ih[2]};
  const VmsElem<A> el(g, k);
  VmsFields<A> f;
  A pe[8];
  gather<A, false>(m, idx, cf.phi, pe);
  {
    A ue[3][8], me[8];
#pragma unroll
    for (int d = 0; d < 3; ++d) gather<A, false>(m, idx, cf.u[d], ue[d]);
    gather<A, false>(m, idx, cf.mu, me);
    f.eval(pe, me, ue, g, k);
  }
  const Forcing<A> fo(pe, g, k.cw);
  GradC<A> gpr, d[3], s[3];
  A v[3][8];
  {
    A t[8];
    gather<A, false>(m, idx, pk, t);
    gpr.eval(t, cg);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gather<A, false>(m, idx, uk.c[i], t);
      interp3<true>(t, v[i]);
      d[i].eval(t, cg);
    }
  }
  for_qp([&](auto QC) {
    constexpr int Q = decltype(QC)::value;
    const VmsQ<A> c = f.at(Q, el, k);
    const A gp[3] = {f.gp.at(Q, 0), f.gp.at(Q, 1), f.gp.at(Q, 2)};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const A vg[3] = {d[i].at(Q, 0), d[i].at(Q, 1), d[i].at(Q, 2)};
      // the part without advection, shared by both sums: a0 v - p_i + rho g_i / Fr
      A h = mad(c.a0, v[i][Q], -gpr.at(Q, i));
      if (ghat(i) != 0) h = mad(-c.rho, k.inv_fr, h);
      // R_0: b'.grad v + Cn/We F - h, and the tested value h - b.grad v
      const A r0 = fo.add(Q, i, gp, mad(c.bp[0], vg[0], mad(c.bp[1], vg[1], mad(c.bp[2], vg[2], -h))));
      v[i][Q] = J * mad(-c.b[0], vg[0], mad(-c.b[1], vg[1], mad(-c.b[2], vg[2], h)));
      const A cp = k.cw * gp[i];
#pragma unroll
      for (int n = 0; n < 3; ++n)
        s[i].sum(Q, n, mad(cp, gp[n], -mad(c.e, vg[n], c.t[n] * r0)));
    }
  });
  const A sc[3] = {J * cg[0], J * cg[1], J * cg[2]};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    A r[8];
    interp3<true>(v[i], r);
    s[i].transpose(sc, r);
    scatter<A, true>(m, idx, r, b + i * m.n_nodes);
  }
}

// The fields of the pressure-Poisson and velocity-update right-hand sides at the 8 Gauss points:
// v and the differences v - u_k, the gradients of v~ = (v + u_k)/2, and of p_k.
template <class A>
struct ProjFields {
  VmsFields<A> f;
  GradC<A> gpr, gt[3];
  A dv[3][8], vv[3][8];  // (v - u_k)/dt without gauss_w^3, v
  A div[8];
  A pe[8];
  __device__ __forceinline__ void load(const MeshDev& m, const int idx[8],
                                       const CoefArgs<double>& cf, const Ptr3& v, const Ptr3& uk,
                                       const double* pk, const Geo<A>& g, const PrmT<A>& k) {
    constexpr double w = gauss_w<A>();
    const A cg[3] = {A(w * w) * g.ih[0], A(w * w) * g.ih[1], A(w * w) * g.ih[2]};
    const A ch[3] = {A(0.5) * cg[0], A(0.5) * cg[1], A(0.5) * cg[2]};
    A t[8], u[8];
    gather<A, false>(m, idx, cf.phi, pe);
    {
      A ue[3][8];
#pragma unroll
      for (int d = 0; d < 3; ++d) gather<A, false>(m, idx, cf.u[d], ue[d]);
      gather<A, false>(m, idx, cf.mu, t);
      f.eval(pe, t, ue, g, k);
    }
    gather<A, false>(m, idx, pk, t);
    gpr.eval(t, cg);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      gather<A, false>(m, idx, v.c[i], t);
      gather<A, false>(m, idx, uk.c[i], u);
      interp3<true>(t, vv[i]);
      axis_gradient(t, i, cg[i]);
      A a[8];
#pragma unroll
      for (int n = 0; n < 8; ++n) a[n] = t[n] + u[n];
      gt[i].eval(a, ch);
#pragma unroll
      for (int n = 0; n < 8; ++n) a[n] = (t[n] - u[n]) * k.idt;
      interp3<false>(a, dv[i]);
    }
  }
  // R_m,i at point q (Def. of R_m)
  __device__ __forceinline__ A residual(int q, int i, const VmsQ<A>& c, const A adv[3],
                                        const A gp[3], const Forcing<A>& fo,
                                        const PrmT<A>& k) const {
    constexpr double w = gauss_w<A>();
    A r = mad(c.rho * A(w * w * w), dv[i][q], gpr.at(q, i));
#pragma unroll
    for (int d = 0; d < 3; ++d) r = mad(adv[d], gt[i].at(q, d), r);
    if (ghat(i) != 0) r = mad(c.rho, k.inv_fr, r);
    return fo.add(q, i, gp, r);
  }
  // coefficients, advection vector rho u + J/Pe - grad eta/Re = 2 b', and grad phi~ of point q
  __device__ __forceinline__ VmsQ<A> at(int q, const VmsElem<A>& el, const PrmT<A>& k, A adv[3],
                                        A gp[3]) const {
    const VmsQ<A> c = f.at(q, el, k);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      gp[d] = f.gp.at(q, d);
      adv[d] = A(2) * c.bp[d];
    }
    return c;
  }

 private:
  // div += the axis-i derivative of t, at the 8 points
  __device__ __forceinline__ void axis_gradient(const A t[8], int i, const A& c) {
    A e[4], o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int lo = i == 0 ? 2 * j : i == 1 ? (j & 1) + 4 * (j >> 1) : j;
      e[j] = t[lo + (1 << i)] - t[lo];
    }
    interp2(e, o);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int lo = i == 0 ? 2 * j : i == 1 ? (j & 1) + 4 * (j >> 1) : j;
      if (i == 0) {
        o[j] *= c;
        div[lo] = div[lo + 1] = o[j];
      } else {
        div[lo] = mad(c, o[j], div[lo]);
        div[lo + (1 << i)] = mad(c, o[j], div[lo + (1 << i)]);
      }
    }
  }
};

// ---- pressure-Poisson right-hand side (Def. weak_VMS_disc_pp_vel, scalar test q):
//   -(2/dt)(q, div v) - (2/dt)(grad q, tau R_m / rho~) + (grad q, grad p_k / rho~)
// With qvu, the velocity update's per-point terms J (rho~ v_i - tau R_m,i) (the same R_m) are
// stored as well, qvu[(q * 3 + i) * n_elem + e], for k_rhs_vu_q.
template <class A>
__global__ void __launch_bounds__(kRhsThreads)
k_rhs_poisson(MeshDev m, DevParams p, CoefArgs<double> cf, Ptr3 v, Ptr3 uk,
              const double* __restrict__ pk, double* __restrict__ b, double* __restrict__ qvu) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  int idx[8];
  load_corners(m, e, idx);
  const Geo<A> g = geometry<A>(m, e);
  constexpr double w = gauss_w<A>();
  const PrmT<A>& k = p.get<A>();
  const VmsElem<A> el(g, k);
  ProjFields<A> f;
  f.load(m, idx, cf, v, uk, pk, g, k);
  const Forcing<A> fo(f.pe, g, k.cw);
  const A J = g.detJ, js = -(J * k.k2dt) * A(w * w * w);
  GradC<A> d;
  for_qp([&](auto QC) {
    constexpr int Q = decltype(QC)::value;
    A adv[3], gp[3];
    const VmsQ<A> c = f.at(Q, el, k, adv, gp);
    const A kt = k.k2dt * c.tau, jr = J * c.rho, jt = J * c.tau;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const A R = f.residual(Q, i, c, adv, gp, fo, k);
      d.sum(Q, i, c.ir * mad(-kt, R, f.gpr.at(Q, i)));
      if (qvu)
        qvu[(int64_t)(Q * 3 + i) * m.n_elem + e] = (double)mad(-jt, R, jr * f.vv[i][Q]);
    }
    f.div[Q] *= js;
  });
  A r[8];
  interp3<false>(f.div, r);
  const A ca = J * A(w * w);
  const A sc[3] = {ca * g.ih[0], ca * g.ih[1], ca * g.ih[2]};
  d.transpose(sc, r);
  scatter<A, false>(m, idx, r, b);
}

// The velocity-update right-hand side from the per-point terms stored by k_rhs_poisson (same
// v, u_k, p_k and coefficients): only the pressure-difference term is evaluated here.
__global__ void __launch_bounds__(kRhsThreads)
k_rhs_vu_q(MeshDev m, DevParams p, const double* __restrict__ qvu, const double* __restrict__ pk,
           const double* __restrict__ pn, double* __restrict__ b) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  int idx[8];
  load_corners(m, e, idx);
  const Geo<double> g = geometry<double>(m, e);
  constexpr double w = gauss_w<double>();
  GradC<double> fd;  // dt/2 J grad (p_new - p_k)
  {
    double a[8], c0[8];
    gather<double, false>(m, idx, pn, a);
    gather<double, false>(m, idx, pk, c0);
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] -= c0[k];
    const double c = w * w * g.detJ * p.d.half_dt;
    const double cg[3] = {c * g.ih[0], c * g.ih[1], c * g.ih[2]};
    fd.eval(a, cg);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double s[8], r[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      s[q] = __ldg(qvu + (int64_t)(q * 3 + i) * m.n_elem + e) - fd.at(q, i);
    interp3<true>(s, r);
    scatter<double, true>(m, idx, r, b + i * m.n_nodes);
  }
}

// ---- velocity-update right-hand side (Def. weak_VMS_disc_vel_update), per component:
//   (w, rho~ v_i) - (w, tau R_m,i) - (dt/2)(w, d_i (p_new - p_k))
template <class A>
__global__ void __launch_bounds__(kRhsThreads)
k_rhs_vu(MeshDev m, DevParams p, CoefArgs<double> cf, Ptr3 v, Ptr3 uk,
         const double* __restrict__ pk, const double* __restrict__ pn, double* __restrict__ b) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= m.n_elem) return;
  int idx[8];
  load_corners(m, e, idx);
  const Geo<A> g = geometry<A>(m, e);
  constexpr double w = gauss_w<A>();
  const PrmT<A>& k = p.get<A>();
  const VmsElem<A> el(g, k);
  ProjFields<A> f;
  f.load(m, idx, cf, v, uk, pk, g, k);
  const Forcing<A> fo(f.pe, g, k.cw);
  GradC<A> fd;  // dt/2 grad (p_new - p_k)
  {
    A a[8], c0[8];
    gather<A, false>(m, idx, pn, a);
    gather<A, false>(m, idx, pk, c0);
#pragma unroll
    for (int n = 0; n < 8; ++n) a[n] = a[n] - c0[n];
    const A c = A(w * w) * k.half_dt;
    const A cg[3] = {c * g.ih[0], c * g.ih[1], c * g.ih[2]};
    fd.eval(a, cg);
  }
  const A J = g.detJ;
  for_qp([&](auto QC) {
    constexpr int Q = decltype(QC)::value;
    A adv[3], gp[3];
    const VmsQ<A> c = f.at(Q, el, k, adv, gp);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const A R = f.residual(Q, i, c, adv, gp, fo, k);
      f.vv[i][Q] = J * mad(c.rho, f.vv[i][Q], -mad(c.tau, R, fd.at(Q, i)));
    }
  });
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    A r[8];
    interp3<true>(f.vv[i], r);
    scatter<A, true>(m, idx, r, b + i * m.n_nodes);
  }
}

// ---- phi mass: sum_e detJ sum_q phi(q) = sum_e detJ sum_a phi_a (2-point Gauss weights sum to 1
// per corner). Block partial sums, then a deterministic final sum on the host.
__global__ void k_phi_mass(MeshDev m, const double* __restrict__ phi, double* __restrict__ part) {
  __shared__ double sh[kRhsThreads];
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double v = 0.0;
  if (e < m.n_elem) {
    int idx[8];
    load_corners(m, e, idx);
    const Geo<double> g = geometry<double>(m, e);
    double pe[8];
    gather<double, false>(m, idx, phi, pe);
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < 8; ++a) s += pe[a];
    v = g.detJ * s;
  }
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = kRhsThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

static unsigned nblk(const chns_mesh* m) {
  return (unsigned)((m->d.n_elem + kRhsThreads - 1) / kRhsThreads);
}

static chns_status need(bool ok, const char* what) {
  if (!ok) {
    set_error(what);
    return CHNS_EINVAL;
  }
  return CHNS_OK;
}

chns_status phi_mass(const chns_mesh* m, const double* phi, double* out, cudaStream_t s) {
  const unsigned nb = nblk(m);
  // The block partials (n_elem/128 <= 3N values) go to the last FP64 workspace vector. The
  // Chebyshev setup (cheb_bounds) also uses that vector as scratch; sharing it is safe because
  // this call reads the partials back and synchronises the stream before it returns, and it is
  // only called between solves (before and after a step), never inside one.
  double* part = m->ws.v64[kNumVec64 - 1];
  note_launch();
  k_phi_mass<<<nb, kRhsThreads, 0, s>>>(m->d, phi, part);
  CHNS_CUDA(cudaGetLastError());
  std::vector<double> h(nb);
  CHNS_CUDA(cudaMemcpyAsync(h.data(), part, nb * sizeof(double), cudaMemcpyDeviceToHost, s));
  CHNS_CUDA(cudaStreamSynchronize(s));
  double acc = 0.0;
  for (double v : h) acc += v;
  *out = acc;
  return CHNS_OK;
}

chns_status residual_ch(const chns_mesh* m, const chns_params* prm, const double* phi,
                        const double* mu, const double* phik, const double* muk,
                        const double* const u[3], double* f, cudaStream_t s) {
  const DevParams p = make_dev_params(*prm);
  Ptr3 up{{u[0], u[1], u[2]}};
  CHNS_CUDA(cudaMemsetAsync(f, 0, 2 * m->d.n_nodes * sizeof(double), s));
  note_launch();
  k_residual_ch<double><<<nblk(m), kRhsThreads, 0, s>>>(m->d, p, phi, mu, phik, muk, up, f);
  CHNS_CUDA(cudaGetLastError());
  return CHNS_OK;
}

static CoefArgs<double> cargs(const chns_coef* c) {
  CoefArgs<double> a;
  a.phi = static_cast<const double*>(c->phi_tilde);
  for (int d = 0; d < 3; ++d) a.u[d] = static_cast<const double*>(c->u_adv[d]);
  a.mu = static_cast<const double*>(c->mu_tilde);
  a.phi_shift = 0.0f;
  return a;
}

chns_status rhs_momentum(const chns_mesh* m, const chns_params* prm, const chns_coef* c,
                         const double* const uk[3], const double* pk, double* b, cudaStream_t s) {
  const DevParams p = make_dev_params(*prm);
  CHNS_CUDA(cudaMemsetAsync(b, 0, 3 * m->d.n_nodes * sizeof(double), s));
  note_launch();
  const Ptr3 u3{{uk[0], uk[1], uk[2]}};
  k_rhs_momentum<double><<<nblk(m), kRhsThreads, 0, s>>>(m->d, p, cargs(c), u3, pk, b);
  CHNS_CUDA(cudaGetLastError());
  return CHNS_OK;
}

chns_status rhs_poisson(const chns_mesh* m, const chns_params* prm, const chns_coef* c,
                        const double* const v[3], const double* const uk[3], const double* pk,
                        double* b, cudaStream_t s, double* qvu) {
  const DevParams p = make_dev_params(*prm);
  CHNS_CUDA(cudaMemsetAsync(b, 0, m->d.n_nodes * sizeof(double), s));
  note_launch();
  const Ptr3 v3{{v[0], v[1], v[2]}}, u3{{uk[0], uk[1], uk[2]}};
  k_rhs_poisson<double><<<nblk(m), kRhsThreads, 0, s>>>(m->d, p, cargs(c), v3, u3, pk, b, qvu);
  CHNS_CUDA(cudaGetLastError());
  return CHNS_OK;
}

chns_status rhs_vu(const chns_mesh* m, const chns_params* prm, const chns_coef* c,
                   const double* const v[3], const double* const uk[3], const double* pk,
                   const double* pn, double* b, cudaStream_t s) {
  const DevParams p = make_dev_params(*prm);
  CHNS_CUDA(cudaMemsetAsync(b, 0, 3 * m->d.n_nodes * sizeof(double), s));
  note_launch();
  const Ptr3 v3{{v[0], v[1], v[2]}}, u3{{uk[0], uk[1], uk[2]}};
  k_rhs_vu<double><<<nblk(m), kRhsThreads, 0, s>>>(m->d, p, cargs(c), v3, u3, pk, pn, b);
  CHNS_CUDA(cudaGetLastError());
  return CHNS_OK;
}

chns_status rhs_vu_from(const chns_mesh* m, const chns_params* prm, const double* qvu,
                        const double* pk, const double* pn, double* b, cudaStream_t s) {
  const DevParams p = make_dev_params(*prm);
  CHNS_CUDA(cudaMemsetAsync(b, 0, 3 * m->d.n_nodes * sizeof(double), s));
  note_launch();
  k_rhs_vu_q<<<nblk(m), kRhsThreads, 0, s>>>(m->d, p, qvu, pk, pn, b);
  CHNS_CUDA(cudaGetLastError());
  return CHNS_OK;
}

static bool coef_ok(const chns_coef* c) {
  return c && c->phi_tilde && c->u_adv[0] && c->u_adv[1] && c->u_adv[2] && c->mu_tilde;
}

}  // namespace chns

using namespace chns;

extern "C" chns_status chns_residual_ch(const chns_mesh* m, const chns_params* prm,
                                        const double* phi, const double* mu, const double* phik,
                                        const double* muk, const double* const u[3], double* f,
                                        void* stream) {
  chns_status st = need(m && prm && phi && mu && phik && muk && u && u[0] && u[1] && u[2] && f,
                        "chns_residual_ch: null argument");
  if (st != CHNS_OK) return st;
  return residual_ch(m, prm, phi, mu, phik, muk, u, f, as_stream(stream));
}

extern "C" chns_status chns_rhs_momentum(const chns_mesh* m, const chns_params* prm,
                                         const chns_coef* c, const double* const uk[3],
                                         const double* pk, double* b, void* stream) {
  chns_status st = need(m && prm && coef_ok(c) && uk && uk[0] && uk[1] && uk[2] && pk && b,
                        "chns_rhs_momentum: null argument");
  if (st != CHNS_OK) return st;
  return rhs_momentum(m, prm, c, uk, pk, b, as_stream(stream));
}

extern "C" chns_status chns_rhs_poisson(const chns_mesh* m, const chns_params* prm,
                                        const chns_coef* c, const double* const v[3],
                                        const double* const uk[3], const double* pk, double* b,
                                        void* stream) {
  chns_status st = need(m && prm && coef_ok(c) && v && v[0] && v[1] && v[2] && uk && uk[0] &&
                            uk[1] && uk[2] && pk && b,
                        "chns_rhs_poisson: null argument");
  if (st != CHNS_OK) return st;
  return rhs_poisson(m, prm, c, v, uk, pk, b, as_stream(stream));
}

extern "C" chns_status chns_rhs_velocity_update(const chns_mesh* m, const chns_params* prm,
                                                const chns_coef* c, const double* const v[3],
                                                const double* const uk[3], const double* pk,
                                                const double* pn, double* b, void* stream) {
  chns_status st = need(m && prm && coef_ok(c) && v && v[0] && v[1] && v[2] && uk && uk[0] &&
                            uk[1] && uk[2] && pk && pn && b,
                        "chns_rhs_velocity_update: null argument");
  if (st != CHNS_OK) return st;
  return rhs_vu(m, prm, c, v, uk, pk, pn, b, as_stream(stream));
}

extern "C" chns_status chns_phi_mass(const chns_mesh* m, const double* phi, double* out,
                                     void* stream) {
  chns_status st = need(m && phi && out, "chns_phi_mass: null argument");
  if (st != CHNS_OK) return st;
  return phi_mass(m, phi, out, as_stream(stream));
}
