// FP32 applies with two leaves per thread (FP32 vectors, FP32 or bfloat16 coefficients).
//
// A patch holds up to 256 Morton-consecutive leaves; a CTA of 128 threads computes a patch, a
// thread two leaves: x-neighbours of a brick (the 8 children of one octant, 87-97 % of the leaves
// of the adaptive workloads) or any two other leaves.
//  1. the values of the regular slots go to shared memory, then the hanging slots are
//     interpolated (mean of 2 or 4 parents);
//  2. each thread applies the element operator to its two leaves, sum-factorised, in packed FP32 pairs
//     (one issue slot for two operations): Poisson, mass and shifted to both leaves at once, CH and
//     momentum to one after the other with pairs of Gauss points;
//  3. the contributions are added to sums per slot in shared memory, one array per warp, by plain
//     read-add-write: the threads of a warp add the same corner of their leaves in the same step,
//     and a point is that corner of at most one leaf (the one that fills that octant around it),
//     so no two of them meet. That holds within the steps of one kind of pair; brick pairs and
//     others of a warp have different steps and add one kind after the other, with a barrier of
//     the whole warp in between. The leaves of a brick pair add up their four shared nodes first
//     (six additions per leaf);
//  4. the sums of the hanging slots are distributed to their parents with the same weights, and
//     each regular slot is written once: a plain store where the patch owns the node, a global
//     atomic add otherwise. y must be zero on entry.
// The CTAs are persistent and walk the patches blockIdx.x + k gridDim.x. The chain head -> node
// ids -> node values of a patch is spread over the two patches before it: while patch k is
// computed, the head of k + 2 and the ids of k + 1 are loaded, and before its hanging sums the
// values, parents and references of k + 1, all in registers, so that no phase waits for a load
// it has just issued.
//
// What bounds it: latency and issue together (Poisson on 1,429,744 leaves: 59 % of the issue slots,
// barrier and short scoreboard stalls), on large meshes also the index records (21 bytes per leaf of
// 35). Measured against one thread per leaf with shared-memory float atomics (a compare-and-swap loop on this part, 5.3 cycles
// per warp operation against 2.1 for the read-add-write and 26 against 9.6 in latency): Poisson
// on 6.9e6 leaves 185 -> 147 us, mass (bfloat16 coefficients) on 3.1e5 32.7 -> 28.0 us with the
// identity rows' kernel gone. Also measured, slower (Poisson, 6.9e6 leaves): one warp per patch
// and a lane per brick 190 us (150 registers leave 9 warps per SM); per-slot lists of contributions
// instead of sums in place 155 us (the lists double the traffic); shared atomics here 174 us; 6
// or 8 CTAs per SM 153 and 155 us. With the elements of both kinds of pair before the sums of either:
// 1,429,744 leaves, Poisson 32.9 -> 33.8 us and mass 74.9 -> 79.1 us in a CUDA graph.
#pragma once

#include "ops.cuh"
#include "reduce.cuh"

namespace chns {

constexpr float kRf = (float)kRat;
constexpr double kWr = gauss_w<F2>(), kWr2 = kWr * kWr;

// Element data by columns (col = ix + 2 iy): values interpolated along z (index qz) and z
// differences; the accumulators of the transposes are laid out the same way.

// column values of 4 columns -> the 8 Gauss points (qx + 2 qy + 4 qz)
template <bool NORM = false, class V>
__device__ __forceinline__ void cols_to_qp(const V s[4][2], V q[8]) {
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    V t0[2], t1[2];  // [qy] at ix = 0, 1
    interp<NORM>(s[0][z], s[2][z], t0[0], t0[1]);
    interp<NORM>(s[1][z], s[3][z], t1[0], t1[1]);
    interp<NORM>(t0[0], t1[0], q[4 * z], q[4 * z + 1]);
    interp<NORM>(t0[1], t1[1], q[4 * z + 2], q[4 * z + 3]);
  }
}
// the transpose
template <bool NORM = false, class V>
__device__ __forceinline__ void qp_to_cols(const V q[8], V s[4][2]) {
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    V a0, a1, b0, b1;
    interp<NORM>(q[4 * z], q[4 * z + 1], a0, a1);        // qy = 0: ix = 0, 1
    interp<NORM>(q[4 * z + 2], q[4 * z + 3], b0, b1);    // qy = 1
    interp<NORM>(a0, b0, s[0][z], s[2][z]);
    interp<NORM>(a1, b1, s[1][z], s[3][z]);
  }
}

// rho = alpha s + rho_- at the Gauss points from columns of s = 1 + phi~: relative accuracy where
// rho_- << 1, and phi = -1 gives rho_- exactly.
template <bool NORM = false, class V>
__device__ __forceinline__ void rho_qp(const V s[4][2], const PrmT<float>& k, V rho[8]) {
  constexpr double w = NORM ? 1.0 : kWr * kWr2;
  V q[8];
  cols_to_qp<NORM>(s, q);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    rho[i] = mad(V(k.alpha * (float)w), clamp_nan(q[i], 0.f, (float)(2.0 / w)), V(k.rho_m));
}

// Two Poisson elements from columns; A, AD: the transposes of the column values and differences.
// E: adds sum_q c |grad|^2 (non-negative terms) to *e.
template <class V, bool E>
__device__ __forceinline__ void poisson_cols(const V S[4][2], const V X[4][2], const V D[4],
                                             const V sc[3], const PrmT<float>& k, V A[4][2],
                                             V AD[4], V* e) {
  V c[8];
  rho_qp(S, k, c);
#pragma unroll
  for (int i = 0; i < 8; ++i) c[i] = rcp_approx(c[i]);
  V ee[3];
  {  // x: differences along x, interpolated in y
    V g[2][2];  // [qy][qz]
#pragma unroll
    for (int z = 0; z < 2; ++z) it(X[1][z] - X[0][z], X[3][z] - X[2][z], g[0][z], g[1][z]);
    if (E) ee[0] = V(0.f);
#pragma unroll
    for (int z = 0; z < 2; ++z) {
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        const V s = g[y][z] * (c[2 * y + 4 * z] + c[1 + 2 * y + 4 * z]);
        if (E) ee[0] = mad(g[y][z], s, ee[0]);
        g[y][z] = s;
      }
      V t0, t1;
      it(g[0][z], g[1][z], t0, t1);
      A[1][z] = sc[0] * t0;
      A[3][z] = sc[0] * t1;
      A[0][z] = -A[1][z];
      A[2][z] = -A[3][z];
    }
  }
  {  // y: differences along y, interpolated in x
    V g[2][2];  // [qx][qz]
#pragma unroll
    for (int z = 0; z < 2; ++z) it(X[2][z] - X[0][z], X[3][z] - X[1][z], g[0][z], g[1][z]);
    if (E) ee[1] = V(0.f);
#pragma unroll
    for (int z = 0; z < 2; ++z) {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const V s = g[x][z] * (c[x + 4 * z] + c[x + 2 + 4 * z]);
        if (E) ee[1] = mad(g[x][z], s, ee[1]);
        g[x][z] = s;
      }
      V t0, t1;
      it(g[0][z], g[1][z], t0, t1);
      A[0][z] = mad(-sc[1], t0, A[0][z]);
      A[2][z] = mad(sc[1], t0, A[2][z]);
      A[1][z] = mad(-sc[1], t1, A[1][z]);
      A[3][z] = mad(sc[1], t1, A[3][z]);
    }
  }
  {  // z: column differences, interpolated in x and y
    V t0[2], t1[2], g[2][2];  // g[qx][qy]
    it(D[0], D[2], t0[0], t0[1]);
    it(D[1], D[3], t1[0], t1[1]);
#pragma unroll
    for (int y = 0; y < 2; ++y) it(t0[y], t1[y], g[0][y], g[1][y]);
    if (E) ee[2] = V(0.f);
#pragma unroll
    for (int y = 0; y < 2; ++y)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const V s = g[x][y] * (c[x + 2 * y] + c[x + 2 * y + 4]);
        if (E) ee[2] = mad(g[x][y], s, ee[2]);
        g[x][y] = s;
      }
#pragma unroll
    for (int y = 0; y < 2; ++y) it(g[0][y], g[1][y], t0[y], t1[y]);  // [ix] at qy
    it(t0[0], t0[1], AD[0], AD[2]);
    it(t1[0], t1[1], AD[1], AD[3]);
  }
  if (E) *e = mad(sc[0], ee[0], mad(sc[1], ee[1], sc[2] * ee[2]));
}

// References of a thread's two leaves: byte offsets of their slots in 12 bits of 16. Brick pair
// (B): node ix + 3 (y + 2 z) of the 3 x 2 x 2 nodes in entry 0..11; others: corner a of the first
// leaf in entry a, of the second in 8 + a. The upper bits of entry 0 and, unless B, entry 8 hold the
// level of the first leaf and of the second above the patch's lowest; those of entry 6 say whether
// there is a second leaf.
template <bool B>
struct PairRefs {
  const uint32_t* w;
  __device__ __forceinline__ uint32_t operator()(int k) const {
    return k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xfffu;
  }
  __device__ __forceinline__ uint32_t nibble(int word) const { return w[word] >> 12 & 15u; }
  __device__ __forceinline__ float at(const float* base, int k) const {
    return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + (*this)(k));
  }
  // one step of additions by the threads of `mask` (see 3. above); the barrier orders it after
  // the step before
  template <int NC>
  __device__ __forceinline__ void add(float* base, int k, const float v[NC], unsigned mask) const {
    char* p = reinterpret_cast<char*>(base) + (*this)(k);
    __syncwarp(mask);
    float t[NC];
#pragma unroll
    for (int n = 0; n < NC; ++n)
      t[n] = *reinterpret_cast<volatile float*>(p + n * kPatchSlots * 4);
#pragma unroll
    for (int n = 0; n < NC; ++n)
      *reinterpret_cast<volatile float*>(p + n * kPatchSlots * 4) = t[n] + v[n];
  }
  // the nodes of x line j = y + 2 z at x = 0 and 1, first leaf and second
  __device__ __forceinline__ void line(const float* base, int j, F2& v0, F2& v1) const {
    if constexpr (B) {
      const float a = at(base, 3 * j), b = at(base, 3 * j + 1), c = at(base, 3 * j + 2);
      v0 = F2(a, b);
      v1 = F2(b, c);
    } else {
      v0 = F2(at(base, 2 * j), at(base, 8 + 2 * j));
      v1 = F2(at(base, 2 * j + 1), at(base, 9 + 2 * j));
    }
  }
  // lines interpolated along x (and, DIFF, their differences); the stage is scalar, so that the
  // node shared by the leaves of a brick pair needs no second register
  template <bool DIFF, bool NORM = false>
  __device__ __forceinline__ void load(const float* base, F2 s[4][2], F2 D[4]) const {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      F2 v0, v1;
      line(base, j, v0, v1);
      if constexpr (NORM) {
        itn(v0.x, v1.x, s[j][0].x, s[j][1].x);
        itn(v0.y, v1.y, s[j][0].y, s[j][1].y);
      } else {
        s[j][0] = F2(fmaf(kRf, v1.x, v0.x), fmaf(kRf, v1.y, v0.y));
        s[j][1] = F2(fmaf(kRf, v0.x, v1.x), fmaf(kRf, v0.y, v1.y));
      }
      if (DIFF) D[j] = F2(v1.x - v0.x, v1.y - v0.y);
    }
  }
  // contributions r[n][j][x] of component n, x line j
  template <int NC>
  __device__ __forceinline__ void store(const F2 r[NC][4][2], float* ys, unsigned mask,
                                        bool two) const {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v[4][NC];
#pragma unroll
      for (int n = 0; n < NC; ++n) {
        v[0][n] = r[n][j][0].x;
        v[1][n] = B ? r[n][j][1].x + r[n][j][0].y : r[n][j][1].x;
        v[2][n] = B ? r[n][j][1].y : r[n][j][0].y;
        v[3][n] = r[n][j][1].y;
      }
      if constexpr (B) {
#pragma unroll
        for (int i = 0; i < 3; ++i) add<NC>(ys, 3 * j + i, v[i], mask);
      } else {
        add<NC>(ys, 2 * j, v[0], mask);
        add<NC>(ys, 2 * j + 1, v[1], mask);
        if (!two)
#pragma unroll
          for (int n = 0; n < NC; ++n) v[2][n] = v[3][n] = 0.f;
        add<NC>(ys, 8 + 2 * j, v[2], mask);
        add<NC>(ys, 9 + 2 * j, v[3], mask);
      }
    }
  }
};

// Four constants of a level, for a thread's two leaves.
struct PairConst {
  F2 c[4];
};

// ---------------------------------------------------------------- operators
// NC components; NF coefficient fields: phi~ (ONE_PLUS: s = 1 + phi~), then the velocity, then mu~;
// consts(): four constants of a level; AHEAD: the next patch's values are loaded while a patch is
// computed. setup() computes what the components share and apply() the contributions of one
// component of a thread's two leaves at once (kPair); or leaf() computes one leaf after the other
// (kLeaf), in packed pairs of Gauss points, for operators whose state would not fit the registers
// twice.
enum class TileForm { kPair, kLeaf };
// "Columns" are the x lines here: the first stage runs along x, the in-plane axes are y and z.
template <bool E>
struct TilePoisson {
  static constexpr int NC = 1;
  static constexpr int NF = 1;
  static constexpr bool ONE_PLUS = true, AHEAD = true, DIR = false, ENERGY = E;
  static constexpr TileForm FORM = TileForm::kPair;
  static constexpr int CTAS = 7;  // resident CTAs per SM the register allocation allows
  static __device__ __forceinline__ float4 consts(const LevelGeo& g, const PrmT<float>&) {
    const float d = g.detJf * (float)(kWr2 * kWr2);
    return make_float4(d * g.ihf[1] * g.ihf[1], d * g.ihf[2] * g.ihf[2], d * g.ihf[0] * g.ihf[0],
                       0.f);
  }
  F2 S[4][2], sc[3];
  template <bool B>
  __device__ __forceinline__ void setup(const PairRefs<B>& pr, const float* fs,
                                        const PairConst& g, const PrmT<float>&) {
    pr.template load<false>(fs, S, nullptr);
#pragma unroll
    for (int i = 0; i < 3; ++i) sc[i] = g.c[i];
  }
  template <bool B>
  __device__ __forceinline__ void apply(const PrmT<float>& k, const PairRefs<B>& pr,
                                        const float* xs, F2 r[4][2], F2* e) const {
    F2 X[4][2], D[4], A[4][2], AD[4];
    pr.template load<true>(xs, X, D);
    poisson_cols<F2, E>(S, X, D, sc, k, A, AD, e);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      F2 o0, o1;
      it(A[j][0], A[j][1], o0, o1);
      r[j][0] = mad(-sc[2], AD[j], o0);
      r[j][1] = mad(sc[2], AD[j], o1);
    }
  }
};

// (w, rho~ u) per component
struct TileMass {
  static constexpr int NC = 3;
  static constexpr int NF = 1;
  static constexpr bool ONE_PLUS = true, AHEAD = true, DIR = true, ENERGY = false;
  static constexpr TileForm FORM = TileForm::kPair;
  static constexpr int CTAS = 5;
  static __device__ __forceinline__ float4 consts(const LevelGeo& g, const PrmT<float>&) {
    return make_float4(g.detJf, 0.f, 0.f, 0.f);
  }
  F2 c[8];
  template <bool B>
  __device__ __forceinline__ void setup(const PairRefs<B>& pr, const float* fs,
                                        const PairConst& g, const PrmT<float>& k) {
    F2 S[4][2];
    pr.template load<false, true>(fs, S, nullptr);
    rho_qp<true>(S, k, c);
#pragma unroll
    for (int q = 0; q < 8; ++q) c[q] *= g.c[0];
  }
  template <bool B>
  __device__ __forceinline__ void apply(const PrmT<float>&, const PairRefs<B>& pr, const float* xs,
                                        F2 r[4][2], F2*) const {
    F2 X[4][2], q[8];
    pr.template load<false, true>(xs, X, nullptr);
    cols_to_qp<true>(X, q);
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] *= c[i];
    qp_to_cols<true>(q, X);
#pragma unroll
    for (int j = 0; j < 4; ++j) itn(X[j][0], X[j][1], r[j][0], r[j][1]);
  }
};

// sa (q, u) + sb (grad q, grad u) with constants: Kronecker element matrices as in ShiftK, the
// first stage along x: y = Pz (cm B + cy C + cx E) + cz Dz B with B = Py Px u, C = Dy Px u,
// E = Py Dx u.
struct TileShift {
  static constexpr int NC = 1;
  static constexpr int NF = 0;
  static constexpr bool ONE_PLUS = false, AHEAD = true, DIR = false, ENERGY = false;
  static constexpr TileForm FORM = TileForm::kPair;
  static constexpr int CTAS = 7;
  static __device__ __forceinline__ float4 consts(const LevelGeo& g, const PrmT<float>& k) {
    const float V = 8.f * g.detJf, ks = k.sb * V * (float)(1.0 / 36.0);
    return make_float4(k.sa * V * (float)(1.0 / 216.0), ks * g.ihf[0] * g.ihf[0],
                       ks * g.ihf[1] * g.ihf[1], ks * g.ihf[2] * g.ihf[2]);
  }
  F2 cm, cx, cy, cz;
  template <bool B>
  __device__ __forceinline__ void setup(const PairRefs<B>&, const float*, const PairConst& g,
                                        const PrmT<float>&) {
    cm = g.c[0];
    cx = g.c[1];
    cy = g.c[2];
    cz = g.c[3];
  }
  static __device__ __forceinline__ void P(F2 a, F2 b, F2& o0, F2& o1) {
    o0 = mad(F2(2.f), a, b);
    o1 = mad(F2(2.f), b, a);
  }
  template <bool BR>
  __device__ __forceinline__ void apply(const PrmT<float>&, const PairRefs<BR>& pr,
                                        const float* xs, F2 r[4][2], F2*) const {
    F2 u[4][2], w[4];  // [j = y + 2 z][x]: Px u, and cx Dx u at x = 0 (x = 1: its negative)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      F2 v0, v1;
      pr.line(xs, j, v0, v1);
      u[j][0] = F2(fmaf(2.f, v0.x, v1.x), fmaf(2.f, v0.y, v1.y));
      u[j][1] = F2(fmaf(2.f, v1.x, v0.x), fmaf(2.f, v1.y, v0.y));
      w[j] = cx * F2(v0.x - v1.x, v0.y - v1.y);
    }
    F2 B[4][2], S[4][2];
#pragma unroll
    for (int z = 0; z < 4; z += 2) {
      F2 e0, e1;
      P(w[z], w[z + 1], e0, e1);
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        P(u[z][x], u[z + 1][x], B[z][x], B[z + 1][x]);
        const F2 dy = cy * (u[z][x] - u[z + 1][x]);
        S[z][x] = mad(cm, B[z][x], x ? dy - e0 : dy + e0);
        S[z + 1][x] = mad(cm, B[z + 1][x], -(x ? dy + e1 : dy - e1));
      }
    }
#pragma unroll
    for (int y = 0; y < 2; ++y)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const F2 dz = cz * (B[y][x] - B[y + 2][x]);
        P(S[y][x], S[y + 2][x], r[y][x], r[y + 2][x]);
        r[y][x] += dz;
        r[y + 2][x] -= dz;
      }
  }
};

// constants of a level for the operators in leaf form, and what they are
__device__ __forceinline__ float4 leaf_consts(const LevelGeo& g) {
  return make_float4(g.detJf, g.ihf[0], g.ihf[1], g.ihf[2]);
}
__device__ __forceinline__ Geo<float> leaf_geometry(const float4& c) {
  Geo<float> g;
  g.detJ = c.x;
  g.ih[0] = c.y;
  g.ih[1] = c.z;
  g.ih[2] = c.w;
  return g;
}

// Kron in pairs along x: B, C = Dy Pz u at y = 0 [z], E = Py Dz u at z = 0 [y]
struct KronP {
  F2 B[4], C[2], E[2];
  __device__ __forceinline__ void eval(const float u[8]) {
    F2 l[4], p[4], w[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) l[j] = F2(u[2 * j], u[2 * j + 1]);
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      p[y] = mad(F2(2.f), l[y], l[y + 2]);
      p[y + 2] = mad(F2(2.f), l[y + 2], l[y]);
      w[y] = l[y] - l[y + 2];
    }
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      B[2 * z] = mad(F2(2.f), p[2 * z], p[2 * z + 1]);
      B[2 * z + 1] = mad(F2(2.f), p[2 * z + 1], p[2 * z]);
      C[z] = p[2 * z] - p[2 * z + 1];
    }
    E[0] = mad(F2(2.f), w[0], w[1]);
    E[1] = mad(F2(2.f), w[1], w[0]);
  }
  // r = Px (cm B + c (kh_y C' + kh_z E')) + c kh_x Dx B' with the stiffness part of field o
  __device__ __forceinline__ void sum(float cm, const KronP& o, float c, const float kh[3],
                                      F2 r[4]) const {
    const F2 cy(c * kh[1]), cz(c * kh[2]);
    const float cx = c * kh[0];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const F2 yc = j & 1 ? -o.C[j >> 1] : o.C[j >> 1], ze = j & 2 ? -o.E[j & 1] : o.E[j & 1];
      const F2 S = mad(F2(cm), B[j], mad(cy, yc, cz * ze));
      const float d = cx * (o.B[j].x - o.B[j].y);
      r[j] = F2(fmaf(2.f, S.x, S.y) + d, fmaf(2.f, S.y, S.x) - d);
    }
  }
};

// The Cahn-Hilliard Jacobian (see ChK) in (dphi, dmu), one leaf after the other in packed pairs
// along x. Bound by latency (31 % of the issue slots with both leaves at once): five CTAs per SM at 96
// registers. FP32 on 1,429,744 leaves, in a CUDA graph: 72.1 us, CTA-per-patch kernel 85.8, both
// leaves at once in packed pairs 76.8 (four CTAs, 128 registers) and 81.4 (three, 149); six CTAs
// 81.0 (108 bytes of spills), the next patch's values loaded ahead 73.1.
struct TileCh {
  static constexpr int NC = 2;
  static constexpr int NF = 4;  // phi~, u~
  static constexpr bool ONE_PLUS = false, AHEAD = false, DIR = false, ENERGY = false;
  static constexpr TileForm FORM = TileForm::kLeaf;
  static constexpr int CTAS = 5;
  static __device__ __forceinline__ float4 consts(const LevelGeo& g, const PrmT<float>&) {
    return leaf_consts(g);
  }
  template <class At>
  static __device__ __forceinline__ void leaf(const float4& c, const PrmT<float>& k, const float* xs,
                                              const float* fs, const At& at, float (&r)[NC][8]) {
    constexpr double w = gauss_w<float>(), w3 = w * w * w;
    const Geo<float> g = leaf_geometry(c);
    const float J = g.detJ, *ih = g.ih;
    F2 R[2][4], fv[4], t[4], o[4];
    float v[8];
    auto get = [&](const float* base) {
#pragma unroll
      for (int a = 0; a < 8; ++a) v[a] = at(base, a);
    };
    get(xs);
    interp3<false>(v, fv);
    {
      const float cm = J * (float)(8.0 / 216.0), ks = J * (float)(8.0 / 36.0);
      const float kh[3] = {ks * ih[0] * ih[0], ks * ih[1] * ih[1], ks * ih[2] * ih[2]};
      KronP f, m;
      f.eval(v);
      get(xs + kPatchSlots);
      m.eval(v);
      f.sum(cm * k.idt, m, k.kmu, kh, R[0]);
      m.sum(-0.5f * cm, f, k.kphi, kh, R[1]);
    }
    // 1/2 (q, psi''(phi~) dphi), psi'' = 3 phi~^2 - 1
    get(fs);
    interp3<false>(v, t);
    const F2 cs((float)(0.5 * w3 * w3) * J), c3 = cs * F2((float)(3.0 * w3 * w3));
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = mad(c3 * t[j], t[j], -cs) * fv[j];
    interp3_t<false>(t, o);
#pragma unroll
    for (int j = 0; j < 4; ++j) R[1][j] += o[j];
    // -1/2 (grad q, u~ dphi)
    GradP d;
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      get(fs + (1 + n) * kPatchSlots);
      interp3<false>(v, t);
#pragma unroll
      for (int j = 0; j < 4; ++j) d.sum(j, n, t[j] * fv[j]);
    }
    const float ca = (float)(-0.5 * w3 * w3 * w * w) * J;
    const float sc[3] = {ca * ih[0], ca * ih[1], ca * ih[2]};
    d.transpose(sc, R[0]);
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        r[n][2 * j] = R[n][j].x;
        r[n][2 * j + 1] = R[n][j].y;
      }
  }
};

// The momentum operator with its coefficients evaluated on the fly (see MomK), one leaf after the
// other in packed pairs of Gauss points. Bound by latency (as CTA-per-patch kernel: 34 % of the issue
// slots, barriers 25 % and loads of the gather 20 % of the stalls): three CTAs of four warps at 168
// registers overlap their phases better than two of eight at 128, and the sums need no
// compare-and-swap loops, 24 per leaf. FP32 in a CUDA graph, CTA-per-patch kernel / this: 1,429,744
// leaves 210 / 148 us, 314,672 46.7 / 37.4, 77,932 19.4 / 15.5, 19,608 12.7 / 12.4; four CTAs at 128
// registers 194 us on the first (412 bytes of spills), in scalar arithmetic 178 us.
struct TileMom {
  static constexpr int NC = 3;
  static constexpr int NF = 5;  // phi~, u_hat, mu~
  static constexpr bool ONE_PLUS = false, AHEAD = false, DIR = true, ENERGY = false;
  static constexpr TileForm FORM = TileForm::kLeaf;
  static constexpr int CTAS = 3;
  static __device__ __forceinline__ float4 consts(const LevelGeo& g, const PrmT<float>&) {
    return leaf_consts(g);
  }
  template <class At>
  static __device__ __forceinline__ void leaf(const float4& c, const PrmT<float>& k, const float* xs,
                                              const float* fs, const At& at, float (&r)[NC][8]) {
    const Geo<float> g = leaf_geometry(c);
    VmsFieldsP f;
    {
      float pe[8], me[8], ue[3][8];
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        pe[a] = at(fs, a);
#pragma unroll
        for (int d = 0; d < 3; ++d) ue[d][a] = at(fs + (1 + d) * kPatchSlots, a);
        me[a] = at(fs + 4 * kPatchSlots, a);
      }
      f.eval(pe, me, ue, g, k);
    }
    float x[NC][8];
#pragma unroll
    for (int n = 0; n < NC; ++n)
#pragma unroll
      for (int a = 0; a < 8; ++a) x[n][a] = at(xs + n * kPatchSlots, a);
    const VmsElem<float> el(g, k);
    momentum_apply_pairs(g, x, r, [&](int q, F2& a0, F2 b[3], F2 bp[3], F2& e, F2 t[3]) {
      const VmsQ<F2> v = f.at(q, el, k);
      a0 = v.a0;
      e = v.e;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        b[d] = v.b[d];
        bp[d] = v.bp[d];
        t[d] = v.t[d];
      }
    });
  }
};

// ---------------------------------------------------------------- kernel
constexpr int kPreSlots = 3;  // regular slots per thread whose values are loaded ahead
constexpr int kPreHang = 2;   // hanging slots per thread whose parents are loaded ahead

// What a thread holds of a patch ahead of its turn. Indices beyond the last slot are clamped to
// it: such a lane repeats the last slot's loads and (equal) stores.
template <int NA>
struct TilePre {
  uint32_t id[kPreSlots];
  float v[kPreSlots][NA];  // components (CGP: p_old and z of the component), then fields
  uint2 par[kPreHang];
  uint32_t ref[8];
};

// A thread's two leaves one after the other (kLeaf). Bricks and other leaves need no separate steps:
// every thread adds corner a of its leaf in step a.
template <class Op>
__device__ __forceinline__ void tile_leaves(const PrmT<float>& k, const uint32_t ref[8],
                                            const float4* cst, bool brick, bool any,
                                            const float* xs, const float* fs, float* yw) {
  const PairRefs<true> pr{ref};
  // byte offsets of the corners of both leaves, x = 0 | x = 1 << 16, per x line
  uint32_t o0[4], o1[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t a = brick ? pr(3 * j) : pr(2 * j), b = brick ? pr(3 * j + 1) : pr(2 * j + 1),
                   c = brick ? b : pr(8 + 2 * j), d = brick ? pr(3 * j + 2) : pr(9 + 2 * j);
    o0[j] = a | b << 16;
    o1[j] = c | d << 16;
  }
  const bool two = any && (brick || pr.nibble(3) != 0);
  const uint32_t l0 = pr.nibble(0), l1 = brick ? l0 : pr.nibble(4);
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const bool active = s ? two : any;
    const unsigned mask = __ballot_sync(0xffffffffu, active);
    if (!active) continue;
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) o[j] = s ? o1[j] : o0[j];
    auto at = [&](const float* base, int a) {
      const uint32_t off = a & 1 ? o[a >> 1] >> 16 : o[a >> 1] & 0xffffu;
      return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + off);
    };
    float r[Op::NC][8];
    Op::leaf(cst[s ? l1 : l0], k, xs, fs, at, r);
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const uint32_t off = a & 1 ? o[a >> 1] >> 16 : o[a >> 1] & 0xffffu;
      char* p = reinterpret_cast<char*>(yw) + off;
      __syncwarp(mask);
      float t[Op::NC];
#pragma unroll
      for (int n = 0; n < Op::NC; ++n)
        t[n] = *reinterpret_cast<volatile float*>(p + n * kPatchSlots * 4);
#pragma unroll
      for (int n = 0; n < Op::NC; ++n)
        *reinterpret_cast<volatile float*>(p + n * kPatchSlots * 4) = t[n] + r[n][a];
    }
    __syncwarp(mask);
  }
}

template <class Op, class C, bool CGP>
__global__ void __launch_bounds__(kTileThreads, Op::CTAS)
k_apply_tile(MeshDev m, DevParams p, CoefArgs<C> cf, const float* __restrict__ x,
             float* __restrict__ y, double* __restrict__ S_cg, int par, int fcg,
             const float* __restrict__ zcg, float* __restrict__ pout) {
  constexpr int NC = Op::NC, NF = Op::NF, F0 = NC + (CGP ? 1 : 0), NA = F0 + NF;
  constexpr int kWarps = kTileThreads / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* ys = reinterpret_cast<float*>(smem_raw);   // [warps][NC][kPatchSlots] sums
  float* xb = ys + kWarps * NC * kPatchSlots;                      // [NC][kPatchSlots] node values
  float* fs = xb + NC * kPatchSlots;                // [NF][kPatchSlots] fields
  __shared__ float4 s_cst[CHNS_MAXD];
  __shared__ float s_beta;
  const int tid = threadIdx.x, G = gridDim.x;
  const int np = (int)m.n_patch, N = (int)m.n_nodes;
  const PrmT<float>& k = p.f;
  const float shift = (Op::ONE_PLUS ? 1.f : 0.f) + cf.phi_shift;
  if (CGP && tid == 0) {
    // CG direction update fused into the gather: p_new = z + beta p_old with
    // beta = rz_cur / rz_prev (fcg: Polak-Ribiere)
    double bn, bd;
    if (fcg) {
      bn = -S_cg[kFcgAlpha] * S_cg[kFcgZq0 + (par ^ 1)];
      bd = S_cg[kFcgRz0 + (par ^ 1)];
    } else {
      bn = S_cg[kCgRz0 + par];
      bd = S_cg[kCgRzPrev];
    }
    s_beta = (float)(bd != 0.0 ? bn / bd : 0.0);
    if (blockIdx.x == 0) {  // accumulators of the update kernel that follows
      S_cg[kCgRz0 + (par ^ 1)] = 0.0;
      S_cg[kCgRr0 + (par ^ 1)] = 0.0;
    }
  }
  if (tid >= 32 && tid < 32 + CHNS_MAXD) s_cst[tid - 32] = Op::consts(m.geo[tid - 32], k);
  for (int i = tid; i < kWarps * NC * kPatchSlots; i += kTileThreads) ys[i] = 0.f;  // (cleared as read)
  auto head_of = [&](int t) { return __ldg(m.patch_head + min(t, np - 1)); };
  auto rec_of = [&](const uint4& h) { return m.rec + 4 * (int64_t)h.x; };
  // values of the node with slot word id, in the order of TilePre::v
  auto load_values = [&](uint32_t id, float v[NA]) {
    const int g = (int)(id & kNodeMask);
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] = __ldg(x + (int64_t)c * N + g);
    if (CGP) v[NC] = __ldg(zcg + g);
    if constexpr (NF > 0) v[F0] = ldv<float>(cf.phi, g);
#pragma unroll
    for (int f = 1; f < NF; ++f) v[F0 + f] = ldv<float>(f < 4 ? cf.u[f - 1] : cf.mu, g);
  };
  auto load_ids = [&](const uint4& h, uint32_t id[kPreSlots]) {
    const int last = (int)(h.y & 0xffffu) - 1;
    const uint32_t* r = rec_of(h);
#pragma unroll
    for (int u = 0; u < kPreSlots; ++u) id[u] = __ldg(r + min(tid + kTileThreads * u, last));
  };
  // the parents of hanging slot i
  auto load_par = [&](const uint4& h, int i) {
    return __ldg(reinterpret_cast<const uint2*>(rec_of(h) + (((h.y & 0xffffu) + 3) & ~3u)) + i);
  };
  auto load_rest = [&](const uint4& h, TilePre<NA>& q) {
    const int nhang = (int)(h.y >> 16);
#pragma unroll
    for (int u = 0; u < kPreSlots; ++u) load_values(q.id[u], q.v[u]);
#pragma unroll
    for (int u = 0; u < kPreHang; ++u)
      if (tid + kTileThreads * u < nhang) q.par[u] = load_par(h, tid + kTileThreads * u);
    const int nb4 = 4 * (int)(h.z & 0xffffu), n2 = ((int)(h.z >> 16) + 1) >> 1;
    const uint32_t* gr = rec_of(h) + 4 * (h.w >> 16);
    if (tid < nb4) {
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const uint2 a = __ldg(reinterpret_cast<const uint2*>(gr) + j * nb4 + tid);
        q.ref[2 * j] = a.x;
        q.ref[2 * j + 1] = a.y;
      }
    } else if (tid < nb4 + n2) {
      const uint4* gs = reinterpret_cast<const uint4*>(gr + 6 * nb4) + (tid - nb4);
      const uint4 a = __ldg(gs), b = __ldg(gs + n2);
      q.ref[0] = a.x; q.ref[1] = a.y; q.ref[2] = a.z; q.ref[3] = a.w;
      q.ref[4] = b.x; q.ref[5] = b.y; q.ref[6] = b.z; q.ref[7] = b.w;
    }
  };
  DF en[1] = {df_zero()};
  int t = blockIdx.x;  // < np
  uint4 h = head_of(t), h1 = head_of(t + G);
  TilePre<NA> q;
  load_ids(h, q.id);
  if (Op::AHEAD) load_rest(h, q);
  if (CGP) __syncthreads();
  const float beta = CGP ? s_beta : 0.f;
  for (; t < np; t += G) {
    const int nreg = (int)(h.y & 0xffffu), nhang = (int)(h.y >> 16);
    const int nb4 = 4 * (int)(h.z & 0xffffu), nt = nb4 + (((int)(h.z >> 16) + 1) >> 1);
    if (!Op::AHEAD) load_rest(h, q);
    // 1. node values to shared memory
    auto put = [&](int i, uint32_t id, const float v[NA]) {
      const int g = (int)(id & kNodeMask);
      const bool dir = Op::DIR && (id & (uint32_t)kDirBit);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        float xv = v[c];
        if (CGP) {
          xv = fmaf(beta, xv, v[NC]);
          pout[g] = xv;  // patches sharing the node store the same value
        }
        if (dir) y[(int64_t)c * N + g] = xv;  // identity rows, likewise
        xb[c * kPatchSlots + i] = dir ? 0.f : xv;
      }
#pragma unroll
      for (int f = 0; f < NF; ++f) fs[f * kPatchSlots + i] = f == 0 ? v[F0] + shift : v[F0 + f];
    };
#pragma unroll
    for (int u = 0; u < kPreSlots; ++u)
      put(min(tid + kTileThreads * u, nreg - 1), q.id[u], q.v[u]);
    if (nreg > kTileThreads * kPreSlots)
      for (int i = tid + kTileThreads * kPreSlots; i < nreg; i += kTileThreads) {
        const uint32_t id = __ldg(rec_of(h) + i);
        float v[NA];
        load_values(id, v);
        put(i, id, v);
      }
    uint32_t id1[kPreSlots];
    const uint4 h2 = head_of(t + 2 * G);
    load_ids(h1, id1);
    __syncthreads();
    if (nhang) {  // hanging slots: (a + b) / 2 as (a + b + a + b) / 4
      for (int i = tid, u = 0; i < nhang; i += kTileThreads, ++u) {
        const uint2 w = u == 0 ? q.par[0] : u == 1 ? q.par[1] : load_par(h, i);
        const int a = w.x & 0xffffu, b = w.x >> 16, c = w.y & 0xffffu, d = w.y >> 16;
#pragma unroll
        for (int n = 0; n < NC; ++n) {
          float* v = xb + n * kPatchSlots;
          v[nreg + i] = 0.25f * ((v[a] + v[b]) + (v[c] + v[d]));
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          float* v = fs + f * kPatchSlots;
          v[nreg + i] = 0.25f * ((v[a] + v[b]) + (v[c] + v[d]));
        }
      }
      __syncthreads();
    }
    // 2.-3. elements
    float* yw = ys + (tid >> 5) * NC * kPatchSlots;
    if constexpr (Op::FORM == TileForm::kLeaf) {
      tile_leaves<Op>(k, q.ref, s_cst + (h.w & 0xffffu), tid < nb4, tid < nt, xb, fs, yw);
    } else {
      // brick pairs, then the others: a warp that has both takes them one after the other, with all
      // its lanes meeting in between, since a slot can be a corner of leaves of either kind
      const bool brick = tid < nb4, other = tid >= nb4 && tid < nt;
      const unsigned mask_b = __ballot_sync(0xffffffffu, brick);
      const unsigned mask_s = __ballot_sync(0xffffffffu, other);
      const uint32_t base = h.w & 0xffffu;
      if (brick) {
        F2 r[NC][4][2];
        Op op;
        PairConst pc;
        F2 e(0.f);
        const PairRefs<true> pr{q.ref};
        const float4 c = s_cst[base + pr.nibble(0)];
        pc.c[0] = F2(c.x); pc.c[1] = F2(c.y); pc.c[2] = F2(c.z); pc.c[3] = F2(c.w);
        op.setup(pr, fs, pc, k);
#pragma unroll
        for (int n = 0; n < NC; ++n) op.apply(k, pr, xb + n * kPatchSlots, r[n], &e);
        pr.template store<NC>(r, yw, mask_b, true);
        if (Op::ENERGY) {
          df_addf(en[0], e.x);
          df_addf(en[0], e.y);
        }
      }
      __syncwarp();
      if (other) {
        F2 r[NC][4][2];
        Op op;
        PairConst pc;
        F2 e(0.f);
        const PairRefs<false> pr{q.ref};
        const float4 c = s_cst[base + pr.nibble(0)], d = s_cst[base + pr.nibble(4)];
        pc.c[0] = F2(c.x, d.x); pc.c[1] = F2(c.y, d.y); pc.c[2] = F2(c.z, d.z); pc.c[3] = F2(c.w, d.w);
        const bool two = pr.nibble(3) != 0;
        op.setup(pr, fs, pc, k);
#pragma unroll
        for (int n = 0; n < NC; ++n) op.apply(k, pr, xb + n * kPatchSlots, r[n], &e);
        pr.template store<NC>(r, yw, mask_s, two);
        if (Op::ENERGY) {
          df_addf(en[0], e.x);
          if (two) df_addf(en[0], e.y);
        }
      }
    }
    __syncthreads();
    // the next patch's loads (its values replace this patch's, which are no longer needed)
    uint32_t id0[kPreSlots];
    uint2 par0[kPreHang];
#pragma unroll
    for (int u = 0; u < kPreSlots; ++u) {
      id0[u] = q.id[u];
      q.id[u] = id1[u];
    }
#pragma unroll
    for (int u = 0; u < kPreHang; ++u) par0[u] = q.par[u];
    if (Op::AHEAD) load_rest(h1, q);
    // the sum of slot i over the warps, cleared for the next patch
    auto take = [&](int n, int i) {
      float t[kWarps], v = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) {
        float* a = ys + (w * NC + n) * kPatchSlots + i;
        t[w] = *a;
        *a = 0.f;
      }
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += t[w];
      return v;
    };
    // 4. sums of the hanging slots to their parents
    if (nhang) {
      for (int i = tid, u = 0; i < nhang; i += kTileThreads, ++u) {
        const uint2 w = u == 0 ? par0[0] : u == 1 ? par0[1] : load_par(h, i);
        const bool two = w.x == w.y;
#pragma unroll
        for (int n = 0; n < NC; ++n) {
          float* a = ys + n * kPatchSlots;
          const float v = (two ? 0.5f : 0.25f) * take(n, nreg + i);
          atomicAdd(a + (w.x & 0xffffu), v);
          atomicAdd(a + (w.x >> 16), v);
          if (!two) {
            atomicAdd(a + (w.y & 0xffffu), v);
            atomicAdd(a + (w.y >> 16), v);
          }
        }
      }
      __syncthreads();
    }
    auto write = [&](int i, uint32_t id) {
#pragma unroll
      for (int n = 0; n < NC; ++n) {
        const float v = take(n, i);
        if (Op::DIR && (id & (uint32_t)kDirBit)) continue;
        float* dst = y + ((int64_t)n * N + (id & kNodeMask));
        if (id & (uint32_t)kOwnBit)
          *dst = v;
        else
          atomicAdd(dst, v);
      }
    };
#pragma unroll
    for (int u = 0; u < kPreSlots; ++u)
      if (tid + kTileThreads * u < nreg) write(tid + kTileThreads * u, id0[u]);
    if (nreg > kTileThreads * kPreSlots)
      for (int i = tid + kTileThreads * kPreSlots; i < nreg; i += kTileThreads)
        write(i, __ldg(rec_of(h) + i));
    h = h1;
    h1 = h2;
    // (a barrier of the next patch stands between these reads and the next sums)
  }
  if (Op::ENERGY) {
    double tot[1];
    block_sum<1, kTileThreads>(en, tot);
    if (tid == 0) atomicAdd(S_cg + kCgPq0 + par, tot[0]);
  }
}

}  // namespace chns
