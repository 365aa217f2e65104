// Device building blocks of the matrix-free operators: Q1 basis on box leaves with 2x2x2 Gauss
// quadrature (Sec. 4.1, r = 1), gather with hanging-node interpolation and the transposed
// scatter-add (the top-down copy / bottom-up accumulate of Sec. 5.4 "Traversal-based Vector
// Assembly", done here with flat index tables).
//
// Element-local numbering: corner a has bits (a&1, a>>1&1, a>>2&1) for (x, y, z); quadrature
// point q uses the same bit layout with xi = -1/sqrt(3) for bit 0 and +1/sqrt(3) for bit 1.
// Along one axis the Q1 basis at the Gauss points is B = [[W0, W1], [W1, W0]] (symmetric) and the
// reference derivative is (u1 - u0)/2 at both points.
#pragma once

#include "dfloat.cuh"
#include "f32x2.cuh"
#include "internal.h"

namespace chns {

constexpr double kW0 = 0.78867513459481288225;  // (1 + 1/sqrt(3)) / 2
constexpr double kW1 = 0.21132486540518711775;  // (1 - 1/sqrt(3)) / 2

// Physical parameters in device form (Sec. 3: rho(phi) = alpha phi + beta, eta = gamma phi + xi)
// with every quotient the kernels need precomputed on the host, in the kernel's own precision:
// the device code multiplies only (on GB300 an FP64 division inside an FP32 kernel costs more
// than the whole FP32 element computation around it).
template <class T>
struct PrmT {
  T alpha, beta, gamma, xi, C_I;
  T rho_m, eta_m;                       // rho_-, eta_- (phi = -1)
  T dt, idt, four_idt2, k2dt, half_dt;  // dt, 1/dt, 4/dt^2, 2/dt, dt/2
  T inv_re, h2re, inv_pe, h2pe;         // 1/Re, 1/(2Re), 1/Pe, 1/(2Pe)
  T inv_pecn, kmu, kphi, cn2;           // 1/(Pe Cn), 1/(2 Pe Cn), Cn^2/2, Cn^2
  T ka, cw, inv_fr;                     // -alpha/Cn, Cn/We, 1/Fr
  T sa, sb;  // constant-coefficient operator sa M + sb K (set per call by its apply, else 0)
};

struct DevParams {
  PrmT<double> d;
  PrmT<float> f;
  PrmT<DF> x;  // the FP64 values split into double-float
  template <class T>
  __host__ __device__ __forceinline__ const PrmT<T>& get() const;
};
template <>
__host__ __device__ __forceinline__ const PrmT<double>& DevParams::get<double>() const { return d; }
template <>
__host__ __device__ __forceinline__ const PrmT<float>& DevParams::get<float>() const { return f; }
template <>
__host__ __device__ __forceinline__ const PrmT<DF>& DevParams::get<DF>() const { return x; }

template <class T>
inline PrmT<T> make_prm(const chns_params& p) {
  const double rp = 1.0, rm = 1.0 / p.rho_ratio, ep = 1.0, em = 1.0 / p.eta_ratio;
  const double alpha = (rp - rm) / (2 * rp), beta = (rp + rm) / (2 * rp);
  const double gamma = (ep - em) / (2 * ep), xi = (ep + em) / (2 * ep);
  PrmT<T> q;
  q.alpha = (T)alpha;
  q.beta = (T)beta;
  q.gamma = (T)gamma;
  q.xi = (T)xi;
  q.C_I = (T)p.C_I;
  q.rho_m = (T)rm;
  q.eta_m = (T)em;
  q.dt = (T)p.dt;
  q.idt = (T)(1.0 / p.dt);
  q.four_idt2 = (T)(4.0 / (p.dt * p.dt));
  q.k2dt = (T)(2.0 / p.dt);
  q.half_dt = (T)(0.5 * p.dt);
  q.inv_re = (T)(1.0 / p.Re);
  q.h2re = (T)(0.5 / p.Re);
  q.inv_pe = (T)(1.0 / p.Pe);
  q.h2pe = (T)(0.5 / p.Pe);
  q.inv_pecn = (T)(1.0 / (p.Pe * p.Cn));
  q.kmu = (T)(0.5 / (p.Pe * p.Cn));
  q.kphi = (T)(0.5 * p.Cn * p.Cn);
  q.cn2 = (T)(p.Cn * p.Cn);
  q.ka = (T)(-alpha / p.Cn);
  q.cw = (T)(p.Cn / p.We);
  q.inv_fr = (T)(1.0 / p.Fr);
  q.sa = q.sb = (T)0;
  return q;
}

inline DevParams make_dev_params(const chns_params& p) {
  DevParams d;
  d.d = make_prm<double>(p);
  d.f = make_prm<float>(p);
  d.x = make_prm<DF>(p);
  return d;
}

// Storage type of values computed in arithmetic type T (FP64 for double-float) and the shared
// accumulator type of the patch applies (the same).
template <class T>
using AccumT = typename std::conditional<std::is_same<T, DF>::value, double, T>::type;

// GB300 executes two FP64 operations per clock and SM against 128 in FP32, and comparisons count:
// the FP64 helpers below use integer operations where they can.

// |v| < 1
template <class T>
__device__ __forceinline__ bool inside1(T v) {
  if constexpr (std::is_same<T, double>::value)
    return (__double2hiint(v) & 0x7fffffff) < 0x3ff00000;
  else
    return v < T(1) && v > T(-1);
}
// v clamped to [-1, 1]; NaN stays
template <class T>
__device__ __forceinline__ T clamp1(T v) {
  if constexpr (std::is_same<T, double>::value) {
    const int hi = __double2hiint(v);
    const bool out = (unsigned)((hi & 0x7fffffff) - 0x3ff00000) <= 0x40000000u;  // 1 <= |v| <= inf
    return out ? __hiloint2double((hi & (int)0x80000000) | 0x3ff00000, 0) : v;
  } else {
    return v > T(1) ? T(1) : (v < T(-1) ? T(-1) : v);
  }
}

// a b + c in one rounding where the type has it
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ DF mad(DF a, DF b, DF c) { return a * b + c; }

// 1/x for normal x up to 2^1021 in magnitude (densities, bounded away from 0; NaN stays): the
// hardware estimate y (about 20 bits) and one third-order step y (1 + e + e^2), e = 1 - x y
// (Householder's method): three operations, within 0.6 units of the last place (0.505 measured).
// FP64 applies of the four operators on 156,640 leaves 923 us, with divisions 932, and the same errors.
__device__ __forceinline__ double recip(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-x, y, 1.0);
  return ::fma(y, ::fma(e, e, e), y);
}
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
__device__ __forceinline__ DF recip(DF x) { return df_recip(x); }

// 1/sqrt(x) for normal x > 0 (0 for infinity; NaN stays), in FP64 likewise, within 1.1 units
// (0.98 measured): the binomial series of (1 - e)^(-1/2) up to its third term, y (1 + e/2 + 3 e^2 / 8), e = 1 - x y^2
__device__ __forceinline__ double inv_sqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-x * y, y, 1.0);
  const double z = ::fma(y * e, ::fma(0.375, e, 0.5), y);
  return __double2hiint(x) == 0x7ff00000 ? 0.0 : z;
}
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrt(x); }
__device__ __forceinline__ DF inv_sqrt(DF x) { return rsqrt(x); }

// ---- loads with conversion from the storage type
template <class T>
__device__ __forceinline__ T ldv(const double* p, int64_t i) { return (T)__ldg(p + i); }
template <class T>
__device__ __forceinline__ T ldv(const float* p, int64_t i) { return (T)__ldg(p + i); }
template <class T>
__device__ __forceinline__ T ldv(const __nv_bfloat16* p, int64_t i) {
  return (T)__bfloat162float(p[i]);
}

// ---- element geometry from the octant level (never stored): h_d = L_d 2^-level
template <class T>
struct Geo {
  T h[3];
  T ih[3];
  T detJ;  // h_x h_y h_z / 8 (Gauss weights are 1)
};

template <class T>
__device__ __forceinline__ Geo<T> level_geometry(const MeshDev& m, int level) {
  const LevelGeo& L = m.geo[level];
  Geo<T> g;
  if constexpr (std::is_same<T, double>::value) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      g.h[d] = L.h[d];
      g.ih[d] = L.ih[d];
    }
    g.detJ = L.detJ;
  } else if constexpr (std::is_same<T, DF>::value) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      g.h[d] = DF(L.h[d]);
      g.ih[d] = DF(L.ih[d]);
    }
    g.detJ = DF(L.detJ);
  } else {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      g.h[d] = L.hf[d];
      g.ih[d] = L.ihf[d];
    }
    g.detJ = L.detJf;
  }
  return g;
}

template <class T>
__device__ __forceinline__ Geo<T> geometry(const MeshDev& m, int64_t e) {
  return level_geometry<T>(m, m.level[e]);
}

__device__ __forceinline__ void load_corners(const MeshDev& m, int64_t e, int idx[8]) {
  int4 a = __ldg(m.enode + 2 * e);
  int4 b = __ldg(m.enode + 2 * e + 1);
  idx[0] = a.x; idx[1] = a.y; idx[2] = a.z; idx[3] = a.w;
  idx[4] = b.x; idx[5] = b.y; idx[6] = b.z; idx[7] = b.w;
}

// Value of one node reference (with Dirichlet flag) from a nodal array; DIR zeroes flagged nodes.
template <class T, bool DIR, class S>
__device__ __forceinline__ T node_val(const S* x, int v) {
  if (DIR && (v & kDirBit)) return T(0);
  return ldv<T>(x, v & kIdxMask);
}

// Gather the 8 corner values of an element; hanging corners are interpolated from their parents
// (edge midpoint: mean of 2, face centre: mean of 4).
template <class T, bool DIR, class S>
__device__ __forceinline__ void gather(const MeshDev& m, const int idx[8], const S* x, T out[8]) {
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    int v = idx[a];
    int j = v & kIdxMask;
    if (j < m.n_nodes) {
      out[a] = node_val<T, DIR>(x, v);
    } else {
      int4 h = __ldg(m.hang + (j - m.n_nodes));
      T s = node_val<T, DIR>(x, h.x) + node_val<T, DIR>(x, h.y);
      if (h.z < 0) {
        out[a] = T(0.5) * s;
      } else {
        s += node_val<T, DIR>(x, h.z) + node_val<T, DIR>(x, h.w);
        out[a] = T(0.25) * s;
      }
    }
  }
}

template <class S>
__device__ __forceinline__ void atomic_add(S* p, S v) { atomicAdd(p, v); }

// Transposed gather: add the element vector into the nodal output, distributing hanging corners
// to their parents with the same weights. DIR skips flagged (Dirichlet) rows.
template <class T, bool DIR, class S>
__device__ __forceinline__ void scatter(const MeshDev& m, const int idx[8], const T r[8], S* y) {
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    int v = idx[a];
    int j = v & kIdxMask;
    if (j < m.n_nodes) {
      if (!(DIR && (v & kDirBit))) atomic_add(y + j, (S)r[a]);
    } else {
      int4 h = __ldg(m.hang + (j - m.n_nodes));
      bool four = h.z >= 0;
      S w = (S)(four ? T(0.25) * r[a] : T(0.5) * r[a]);
      if (!(DIR && (h.x & kDirBit))) atomic_add(y + (h.x & kIdxMask), w);
      if (!(DIR && (h.y & kDirBit))) atomic_add(y + (h.y & kIdxMask), w);
      if (four) {
        if (!(DIR && (h.z & kDirBit))) atomic_add(y + (h.z & kIdxMask), w);
        if (!(DIR && (h.w & kDirBit))) atomic_add(y + (h.w & kIdxMask), w);
      }
    }
  }
}

// ---- sum-factorised Q1 kernels
// 1D interpolation to the Gauss points and its transpose (B is symmetric), divided by W0:
// o0 = a + r b, o1 = r a + b with r = W1 / W0, two operations. Every axis interpolated leaves a
// factor gauss_w<T>() to the caller, who folds it into a constant: that of the rounded ratio,
// 1 / (1 + r), so that constants are reproduced to the last rounding.
constexpr double kRat = 0.26794919243112270647;
template <class T>
constexpr double gauss_w() {
  if constexpr (std::is_same<T, double>::value || std::is_same<T, DF>::value)
    return kW0;
  else
    return 1.0 / (1.0 + (double)(float)kRat);
}
template <class T>
__device__ __forceinline__ void it(T a, T b, T& o0, T& o1) {
  o0 = mad(T(kRat), b, a);
  o1 = mad(T(kRat), a, b);
}
// Normalised form, o0 = a + W1 (b - a) and o1 = b - W1 (b - a): one more operation; reproduces
// constants exactly and halves the rounding error of a chain of them.
template <class T>
__device__ __forceinline__ void itn(T a, T b, T& o0, T& o1) {
  const T d = b - a;
  o0 = mad(T(kW1), d, a);
  o1 = mad(T(-kW1), d, b);
}
template <bool NORM, class T>
__device__ __forceinline__ void interp(T a, T b, T& o0, T& o1) {
  if constexpr (NORM)
    itn(a, b, o0, o1);
  else
    it(a, b, o0, o1);
}

// 3D interpolation of corner values to the 8 Gauss points (self-transpose).
template <bool NORM, class T>
__device__ __forceinline__ void interp3(const T u[8], T v[8]) {
  T t[8], s[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) interp<NORM>(u[2 * j], u[2 * j + 1], t[2 * j], t[2 * j + 1]);
#pragma unroll
  for (int z = 0; z < 2; ++z)
#pragma unroll
    for (int x = 0; x < 2; ++x)
      interp<NORM>(t[x + 4 * z], t[x + 2 + 4 * z], s[x + 4 * z], s[x + 2 + 4 * z]);
#pragma unroll
  for (int i = 0; i < 4; ++i) interp<NORM>(s[i], s[i + 4], v[i], v[i + 4]);
}
// 2D, 4 values (i0 + 2 i1)
template <class T>
__device__ __forceinline__ void interp2(const T in[4], T out[4]) {
  T t[4];
  it(in[0], in[1], t[0], t[1]);
  it(in[2], in[3], t[2], t[3]);
  it(t[0], t[2], out[0], out[2]);
  it(t[1], t[3], out[1], out[3]);
}

// Compact gradient data of an element: the x difference depends on (qy, qz) only, and so on; each
// is the bilinear interpolation of the 4 edge differences along its axis. True values are these
// times gauss_w^2 / h_d.
template <class T>
struct GradC {
  T x[4], y[4], z[4];  // [qy + 2 qz], [qx + 2 qz], [qx + 2 qy]
  __device__ __forceinline__ void eval(const T u[8]) {
    T d[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = u[2 * j + 1] - u[2 * j];
    interp2(d, x);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i) d[i + 2 * k] = u[i + 2 + 4 * k] - u[i + 4 * k];
    interp2(d, y);
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = u[j + 4] - u[j];
    interp2(d, z);
  }
  // physical gradients (c_d = gauss_w^2 / h_d, times whatever the caller folds in)
  __device__ __forceinline__ void eval(const T u[8], const T c[3]) {
    eval(u);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] *= c[0];
      y[j] *= c[1];
      z[j] *= c[2];
    }
  }
  // component d at Gauss point q
  __device__ __forceinline__ T at(int q, int d) const {
    return d == 0 ? x[q >> 1] : d == 1 ? y[(q & 1) + 2 * (q >> 2)] : z[q & 3];
  }
  // adds (FIRST: sets) the component d of a per-point vector at Gauss point q: the data whose
  // transpose is the sum over the points of grad N_a . V
  __device__ __forceinline__ void sum(int q, int d, T v) {
    T& s = d == 0 ? x[q >> 1] : d == 1 ? y[(q & 1) + 2 * (q >> 2)] : z[q & 3];
    const bool first = d == 0 ? !(q & 1) : d == 1 ? !(q & 2) : !(q & 4);
    s = first ? v : s + v;
  }
  // r_a += sum_d sc_d (transpose of eval)
  __device__ __forceinline__ void transpose(const T sc[3], T r[8]) const {
    T t[4];
    interp2(x, t);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      r[2 * j + 1] = mad(sc[0], t[j], r[2 * j + 1]);
      r[2 * j] = mad(-sc[0], t[j], r[2 * j]);
    }
    interp2(y, t);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        r[i + 2 + 4 * k] = mad(sc[1], t[i + 2 * k], r[i + 2 + 4 * k]);
        r[i + 4 * k] = mad(-sc[1], t[i + 2 * k], r[i + 4 * k]);
      }
    interp2(z, t);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      r[j + 4] = mad(sc[2], t[j], r[j + 4]);
      r[j] = mad(-sc[2], t[j], r[j]);
    }
  }
};

// One field of a constant-coefficient form on a box. The 2x2x2 Gauss rule is exact there and the
// element matrices are Kronecker products of the 1D matrices m = h/6 [[2, 1], [1, 2]] and
// k = 1/h [[1, -1], [-1, 1]]: with P(a, b) = (2a + b, a + 2b) and D(a, b) = (a - b, b - a) along
// one axis, M_e u = V/216 Px B and K_e u = V/36 (Px (C / h_y^2 + E / h_z^2) + Dx B / h_x^2), where
// B = Py Pz u, C = Dy Pz u, E = Py Dz u and V = h_x h_y h_z.
template <class T>
struct Kron {
  T B[8], C[4], E[4];  // C at y = 0 [x + 2 z] (y = 1: its negative), E at z = 0 [x + 2 y] (likewise)
  __device__ __forceinline__ void mass(const T u[8]) {
    T p[8];
    stage(u, p);
  }
  __device__ __forceinline__ void eval(const T u[8]) {
    T p[8], w[4];
    stage(u, p);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i) C[i + 2 * k] = p[i + 4 * k] - p[i + 2 + 4 * k];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = u[j] - u[j + 4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      E[i] = mad(T(2), w[i], w[i + 2]);
      E[i + 2] = mad(T(2), w[i + 2], w[i]);
    }
  }
  __device__ __forceinline__ T c_at(int a) const {
    const T v = C[(a & 1) + 2 * (a >> 2)];
    return a & 2 ? -v : v;
  }
  __device__ __forceinline__ T e_at(int a) const { return a & 4 ? -E[a & 3] : E[a & 3]; }
  // r = Px S + cx Dx B (of this field)
  __device__ __forceinline__ void finish(const T S[8], T cx, T r[8]) const {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T d = B[2 * j] - B[2 * j + 1];
      r[2 * j] = mad(cx, d, mad(T(2), S[2 * j], S[2 * j + 1]));
      r[2 * j + 1] = mad(-cx, d, mad(T(2), S[2 * j + 1], S[2 * j]));
    }
  }

 private:
  __device__ __forceinline__ void stage(const T u[8], T p[8]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      p[j] = mad(T(2), u[j], u[j + 4]);
      p[j + 4] = mad(T(2), u[j + 4], u[j]);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int a = i + 4 * k, b = a + 2;
        B[a] = mad(T(2), p[a], p[b]);
        B[b] = mad(T(2), p[b], p[a]);
      }
  }
};

// ---- the same in packed FP32 for one element: pairs over the Gauss points (or corners) along x,
// so that half the instructions do the work without a second element's registers. Index j = y + 2 z
// of the four x lines; the x stage is scalar, its two results land in one pair.
template <bool NORM>
__device__ __forceinline__ F2 it_x(float a, float b) {
  F2 o;
  interp<NORM>(a, b, o.x, o.y);
  return o;
}
template <bool NORM>
__device__ __forceinline__ void interp_yz(const F2 t[4], F2 v[4]) {
  F2 s[4];
#pragma unroll
  for (int z = 0; z < 4; z += 2) interp<NORM>(t[z], t[z + 1], s[z], s[z + 1]);
#pragma unroll
  for (int y = 0; y < 2; ++y) interp<NORM>(s[y], s[y + 2], v[y], v[y + 2]);
}
// corner values to the Gauss points
template <bool NORM>
__device__ __forceinline__ void interp3(const float u[8], F2 v[4]) {
  F2 t[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) t[j] = it_x<NORM>(u[2 * j], u[2 * j + 1]);
  interp_yz<NORM>(t, v);
}
// the transpose
template <bool NORM>
__device__ __forceinline__ void interp3_t(const F2 v[4], F2 r[4]) {
  F2 t[4];
  interp_yz<NORM>(v, t);
#pragma unroll
  for (int j = 0; j < 4; ++j) r[j] = it_x<NORM>(t[j].x, t[j].y);
}

// GradC in pairs along x
struct GradP {
  float x[4];     // [qy + 2 qz]
  F2 y[2], z[2];  // [qz], [qy]
  __device__ __forceinline__ void eval(const float u[8], const float c[3]) {
    float d[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = u[2 * j + 1] - u[2 * j];
    interp2(d, x);
    F2 l[4], t0, t1;
#pragma unroll
    for (int j = 0; j < 4; ++j) l[j] = F2(u[2 * j], u[2 * j + 1]);
    it(l[1] - l[0], l[3] - l[2], t0, t1);
    y[0] = F2(c[1]) * it_x<false>(t0.x, t0.y);
    y[1] = F2(c[1]) * it_x<false>(t1.x, t1.y);
    it(l[2] - l[0], l[3] - l[1], t0, t1);
    z[0] = F2(c[2]) * it_x<false>(t0.x, t0.y);
    z[1] = F2(c[2]) * it_x<false>(t1.x, t1.y);
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] *= c[0];
  }
  __device__ __forceinline__ F2 at(int j, int d) const {
    return d == 0 ? F2(x[j]) : d == 1 ? y[j >> 1] : z[j & 1];
  }
  __device__ __forceinline__ void sum(int j, int d, F2 v) {
    if (d == 0)
      x[j] = v.x + v.y;
    else if (d == 1)
      y[j >> 1] = j & 1 ? y[j >> 1] + v : v;
    else
      z[j & 1] = j & 2 ? z[j & 1] + v : v;
  }
  __device__ __forceinline__ void transpose(const float sc[3], F2 r[4]) const {
    float t[4];
    interp2(x, t);
#pragma unroll
    for (int j = 0; j < 4; ++j) r[j] = F2(fmaf(-sc[0], t[j], r[j].x), fmaf(sc[0], t[j], r[j].y));
    F2 a, b;
    it(it_x<false>(y[0].x, y[0].y), it_x<false>(y[1].x, y[1].y), a, b);  // z = 0, 1
    r[1] = mad(F2(sc[1]), a, r[1]);
    r[0] = mad(F2(-sc[1]), a, r[0]);
    r[3] = mad(F2(sc[1]), b, r[3]);
    r[2] = mad(F2(-sc[1]), b, r[2]);
    it(it_x<false>(z[0].x, z[0].y), it_x<false>(z[1].x, z[1].y), a, b);  // y = 0, 1
    r[2] = mad(F2(sc[2]), a, r[2]);
    r[0] = mad(F2(-sc[2]), a, r[0]);
    r[3] = mad(F2(sc[2]), b, r[3]);
    r[1] = mad(F2(-sc[2]), b, r[1]);
  }
};

// Compile-time loop over the 8 quadrature points.
template <int Q = 0, class F>
__device__ __forceinline__ void for_qp(F&& f) {
  if constexpr (Q < 8) {
    f(std::integral_constant<int, Q>{});
    for_qp<Q + 1>(f);
  }
}

}  // namespace chns
