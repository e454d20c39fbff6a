// Kernels for a caller-supplied two-dimensional Hermite lattice (LBM_HERMITE):
// the minimal square-symmetric rules of Sec. III.A (17 velocities, degree 7,
// truncation N = 3; 37 velocities, degree 9, N = 3 or 4) or any other such
// rule that integrates the Gaussian exactly to degree 2N.  The collision is the
// same Hermite-space CM-MRT as on the built-in 37-velocity lattice
// (h37::collide_coeffs: Eq. omega in the relative frame, K = 6 at order 4);
// only the projection onto and from the Hermite coefficients differs: it uses
// per-simulation tables passed by value instead of compiled-in constants.  One
// node per thread, AA pattern, FP64 or FP32 offsets from f_eq(1, 0, theta_ref).
// Velocities crossing the C ABI are in lattice units.
//
// Rules that are symmetric under e_x -> -e_x and e_y -> -e_y (every minimal rule
// is) go, in FP64, through hgen_orbit_kernel: raw moments of the reflection orbits
// (hgen_half_kernel on small grids).  Others, and FP32, take the dense tables
// (hgen_sweep_kernel).
#include <cmath>
#include <type_traits>

#include "h37_moments.cuh"
#include "pdl.cuh"
#include "reduce.cuh"

namespace lbm {

void hgen_build_tables(const HLattice& L, double theta_ref, HTables* t) {
  auto he = [](int n, double x) {
    return n == 0 ? 1.0 : n == 1 ? x : n == 2 ? x * x - 1.0 : n == 3 ? x * x * x - 3.0 * x
                                                                       : x * x * x * x - 6.0 * x * x + 3.0;
  };
  auto fct = [](int n) { return n <= 1 ? 1.0 : n == 2 ? 2.0 : n == 3 ? 6.0 : 24.0; };
  const double er = theta_ref - 1.0;
  auto aref = [&](int p, int q) {  // Hermite coefficients of f_eq(1, 0, theta_ref)
    auto g = [&](int n) { return n == 0 ? 1.0 : n == 2 ? er : n == 4 ? 3.0 * er * er : 0.0; };
    return g(p) * g(q);
  };
  const int nc = (L.order + 1) * (L.order + 2) / 2;
  t->q = L.q;
  t->nc = nc;
  t->c = L.c;
  for (int i = 0; i < L.q; ++i) {
    t->ex[i] = L.ex[i];
    t->ey[i] = L.ey[i];
    t->opp[i] = L.opp[i];
    const double x = L.c * L.ex[i], y = L.c * L.ey[i];
    double fr = 0.0;
    for (int k = 0; k < 15; ++k) {
      const int p = h37::cp(k), q = h37::cq(k);
      const double h = k < nc ? he(p, x) * he(q, y) : 0.0;
      t->H[k][i] = h;
      t->R[i][k] = k < nc ? L.w[i] * h / (fct(p) * fct(q)) : 0.0;
      if (k < nc) fr += aref(p, q) * t->R[i][k];
    }
    t->fref[i] = fr;
  }
}

namespace {

constexpr int kHgThreads = 128;

template <int S>
struct HStore;
template <>
struct HStore<LBM_F64> {
  using type = double;
};
template <>
struct HStore<LBM_F32> {
  using type = float;
};

struct HGrid {
  int nx, ny;
  int64_t N;
};

__device__ __forceinline__ uint32_t hnbr(const HGrid& g, int x, int y, int dx, int dy) {
  int xn = x + dx, yn = y + dy;
  xn = xn < 0 ? xn + g.nx : (xn >= g.nx ? xn - g.nx : xn);
  yn = yn < 0 ? yn + g.ny : (yn >= g.ny ? yn - g.ny : yn);
  return (uint32_t)xn + (uint32_t)g.nx * (uint32_t)yn;
}

// Offsets of node (x, y) in the state of the given parity.  Odd state: the
// population i of node x sits in slot (x - e_i, opp(i)).
template <typename T, int Q>
__device__ __forceinline__ void hgather(const T* __restrict__ f, const HGrid& g, const HTables& t, int x, int y,
                                        int odd, T (&v)[Q]) {
  const uint32_t node = (uint32_t)x + (uint32_t)g.nx * (uint32_t)y;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (!odd)
      v[i] = f[(size_t)i * g.N + node];
    else
      v[i] = f[(size_t)t.opp[i] * g.N + hnbr(g, x, y, -t.ex[i], -t.ey[i])];
  }
}

// Write the offsets of node (x, y) as the state of the given parity.
template <typename T, int Q>
__device__ __forceinline__ void hscatter(T* __restrict__ f, const HGrid& g, const HTables& t, int x, int y, int odd,
                                         const T (&v)[Q]) {
  const uint32_t node = (uint32_t)x + (uint32_t)g.nx * (uint32_t)y;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (!odd)
      f[(size_t)i * g.N + node] = v[i];
    else
      f[(size_t)t.opp[i] * g.N + hnbr(g, x, y, -t.ex[i], -t.ey[i])] = v[i];
  }
}

template <typename T, int Q, int NC>
__device__ __forceinline__ void to_coeffs(const HTables& t, const T (&v)[Q], T (&a)[NC]) {
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    T s = cst<T>(0.0);
#pragma unroll
    for (int i = 0; i < Q; ++i) s = fma_(v[i], (T)t.H[k][i], s);
    a[k] = s;
  }
}

template <typename T, int Q, int NC>
__device__ __forceinline__ void from_coeffs(const HTables& t, const T (&a)[NC], T (&v)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    T s = cst<T>(0.0);
#pragma unroll
    for (int k = 0; k < NC; ++k) s = fma_(a[k], (T)t.R[i][k], s);
    v[i] = s;
  }
}

// The projection tables as FP32 pairs hi + lo (hi = the FP32 rounding, lo = the
// FP32 rounding of the rest), for the correctly rounded FP32 transforms (see
// h37_common.cuh): built on the host from the FP64 tables at each launch.
struct HSplit {
  float Hh[15][kHQMax], Hl[15][kHQMax];
  float Rh[kHQMax][15], Rl[kHQMax][15];
};

void split_tables(const HTables& t, HSplit* out) {
  for (int k = 0; k < 15; ++k)
    for (int i = 0; i < kHQMax; ++i) {
      const double h = i < t.q ? t.H[k][i] : 0.0, r = i < t.q ? t.R[i][k] : 0.0;
      out->Hh[k][i] = (float)h;
      out->Hl[k][i] = (float)(h - (double)out->Hh[k][i]);
      out->Rh[i][k] = (float)r;
      out->Rl[i][k] = (float)(r - (double)out->Rh[i][k]);
    }
}

template <int Q, int NC>
__device__ __forceinline__ void to_coeffs_exact(const HSplit& t, const float (&v)[Q], float (&a)[NC]) {
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) h37::dot2_add_split(s, c, v[i], t.Hh[k][i], t.Hl[k][i]);
    a[k] = s + c;
  }
}

template <int Q, int NC>
__device__ __forceinline__ void from_coeffs_exact(const HSplit& t, const float (&a)[NC], float (&v)[Q]) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    float s = 0.f, c = 0.f;
#pragma unroll
    for (int k = 0; k < NC; ++k) h37::dot2_add_split(s, c, a[k], t.Rh[i][k], t.Rl[i][k]);
    v[i] = s + c;
  }
}

// EXACT: FP32 storage with the correctly rounded transforms (tables in sp).
template <int S, int Q, int NC, bool ODD, bool EXACT>
__global__ void __launch_bounds__(kHgThreads)
    hgen_sweep_kernel(typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, Rates r, h37::Model m,
                      int* __restrict__ status, const HSplit sp) {
  using T = typename HStore<S>::type;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= g.nx) return;
  const int y = blockIdx.y;
  T om[5];
#pragma unroll
  for (int n = 0; n < 5; ++n) om[n] = (T)r.w[n];
  T v[Q];
  const uint32_t node = (uint32_t)x + (uint32_t)g.nx * (uint32_t)y;
  // even state: population i of node x in slot (x, i); odd state: in slot (x - e_i, opp(i))
#pragma unroll
  for (int i = 0; i < Q; ++i)
    v[i] = ODD ? f[(size_t)t.opp[i] * g.N + hnbr(g, x, y, -t.ex[i], -t.ey[i])] : f[(size_t)i * g.N + node];
  T a[NC];
  if constexpr (EXACT)
    to_coeffs_exact<Q, NC>(sp, v, a);
  else
    to_coeffs<T, Q, NC>(t, v, a);
  if (!h37::collide_coeffs<T, NC>(a, om, m)) atomicOr(status, 1);
  if constexpr (EXACT)
    from_coeffs_exact<Q, NC>(sp, a, v);
  else
    from_coeffs<T, Q, NC>(t, a, v);
  // even sweep: population i to slot (x, opp(i)); odd sweep: to slot (x + e_i, i)
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (!ODD)
      f[(size_t)t.opp[i] * g.N + node] = v[i];
    else
      f[(size_t)i * g.N + hnbr(g, x, y, t.ex[i], t.ey[i])] = v[i];
  }
}

// ---- reflection orbits --------------------------------------------------------
// The velocities of a rule with both reflections are the rest velocity, pairs
// (+-a, 0) and (0, +-a), and quadruples (+-a, +-b).  The raw moments M_pq (lattice
// units; h37_moments.cuh has the collision on them) need each orbit only as its
// sums of even and odd parity in x and y: with 37 velocities and N = 4 that takes
// 180 FP64 operations in and 181 out, against 555 each way through the dense
// tables, which bound this kernel (FP64 runs at 1 / 76 of the FP32 rate).
// Shear wave on 80^2, rule E9-A, FP64: 48.2 -> 24.6 us a step (23.4 with
// chained launches; 18 of them are the FP64 pipe: one warp on each of
// 200 of the 608 SM partitions, 64 cycles per FP64 warp instruction).
template <int NA, int NQ>
struct Orbits {
  int rest, xp[NA], xm[NA], yp[NA], ym[NA], pp[NQ], mp[NQ], pm[NQ], mm[NQ];  // velocity indices
  int da[NA], qa[NQ], qb[NQ];                                                // |e| of pairs, |e_x| and |e_y| of quadruples
  double w0, pw[NA], qw[NQ];                                                 // weights
  double p1[NA], p2[NA], p3[NA], p4[NA];                                     // powers of a
  double a1[NQ], a2[NQ], a3[NQ], a4[NQ], b1[NQ], b2[NQ], b3[NQ], b4[NQ];     // a^p b^q of quadruples
  double ab[NQ], a2b[NQ], ab2[NQ], a2b2[NQ], a3b[NQ], ab3[NQ];
  double vp1[NA], vp2[NA], vp3[NA], vp4[NA];  // the same times the weight
  double va1[NQ], va2[NQ], va3[NQ], va4[NQ], vb1[NQ], vb2[NQ], vb3[NQ], vb4[NQ];
  double vab[NQ], va2b[NQ], vab2[NQ], va2b2[NQ], va3b[NQ], vab3[NQ];
};

// Fills o from the rule; false if the rule lacks a reflection, has other numbers of
// orbits, or weights that differ within an orbit.
template <int NA, int NQ>
bool make_orbits(const HLattice& L, Orbits<NA, NQ>* o) {
  int at[7][7];
  for (auto& r : at)
    for (int& k : r) k = -1;
  for (int i = 0; i < L.q; ++i) at[L.ey[i] + 3][L.ex[i] + 3] = i;
  auto idx = [&](int x, int y) { return at[y + 3][x + 3]; };
  auto same = [&](int i, int j) { return i >= 0 && j >= 0 && L.w[i] == L.w[j]; };
  int na = 0, nq = 0;
  o->rest = idx(0, 0);
  if (o->rest < 0) return false;
  o->w0 = L.w[o->rest];
  for (int a = 1; a <= 3; ++a) {
    const int xp = idx(a, 0), xm = idx(-a, 0), yp = idx(0, a), ym = idx(0, -a);
    if (xp < 0 && xm < 0 && yp < 0 && ym < 0) continue;
    if (!same(xp, xm) || !same(yp, ym) || !same(xp, yp) || na == NA) return false;
    o->xp[na] = xp;
    o->xm[na] = xm;
    o->yp[na] = yp;
    o->ym[na] = ym;
    o->da[na] = a;
    const double w = L.w[xp], d = a;
    o->pw[na] = w;
    o->p1[na] = d;
    o->p2[na] = d * d;
    o->p3[na] = d * d * d;
    o->p4[na] = d * d * d * d;
    o->vp1[na] = w * d;
    o->vp2[na] = w * d * d;
    o->vp3[na] = w * d * d * d;
    o->vp4[na] = w * d * d * d * d;
    ++na;
  }
  for (int b = 1; b <= 3; ++b)
    for (int a = 1; a <= 3; ++a) {
      const int pp = idx(a, b), mp = idx(-a, b), pm = idx(a, -b), mm = idx(-a, -b);
      if (pp < 0 && mp < 0 && pm < 0 && mm < 0) continue;
      if (!same(pp, mp) || !same(pp, pm) || !same(pp, mm) || nq == NQ) return false;
      const int k = nq++;
      o->pp[k] = pp;
      o->mp[k] = mp;
      o->pm[k] = pm;
      o->mm[k] = mm;
      o->qa[k] = a;
      o->qb[k] = b;
      const double w = L.w[pp], x = a, y = b;
      o->qw[k] = w;
      o->a1[k] = x;
      o->a2[k] = x * x;
      o->a3[k] = x * x * x;
      o->a4[k] = x * x * x * x;
      o->b1[k] = y;
      o->b2[k] = y * y;
      o->b3[k] = y * y * y;
      o->b4[k] = y * y * y * y;
      o->ab[k] = x * y;
      o->a2b[k] = x * x * y;
      o->ab2[k] = x * y * y;
      o->a2b2[k] = x * x * y * y;
      o->a3b[k] = x * x * x * y;
      o->ab3[k] = x * y * y * y;
      o->va1[k] = w * x;
      o->va2[k] = w * x * x;
      o->va3[k] = w * x * x * x;
      o->va4[k] = w * x * x * x * x;
      o->vb1[k] = w * y;
      o->vb2[k] = w * y * y;
      o->vb3[k] = w * y * y * y;
      o->vb4[k] = w * y * y * y * y;
      o->vab[k] = w * x * y;
      o->va2b[k] = w * x * x * y;
      o->vab2[k] = w * x * y * y;
      o->va2b2[k] = w * x * x * y * y;
      o->va3b[k] = w * x * x * x * y;
      o->vab3[k] = w * x * y * y * y;
    }
  return na == NA && nq == NQ && 1 + 4 * NA + 4 * NQ == L.q;
}

// Node values by orbit, and calls of fn(value, velocity index, signed e_x, signed e_y, index of
// the opposite velocity) for each.
template <int NA, int NQ>
struct OrbitValues {
  double r, xp[NA], xm[NA], yp[NA], ym[NA], pp[NQ], mp[NQ], pm[NQ], mm[NQ];
  template <typename F>
  __device__ __forceinline__ void each(const Orbits<NA, NQ>& o, F fn) {
    fn(r, o.rest, 0, 0, o.rest);
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      fn(xp[k], o.xp[k], o.da[k], 0, o.xm[k]);
      fn(xm[k], o.xm[k], -o.da[k], 0, o.xp[k]);
      fn(yp[k], o.yp[k], 0, o.da[k], o.ym[k]);
      fn(ym[k], o.ym[k], 0, -o.da[k], o.yp[k]);
    }
#pragma unroll
    for (int k = 0; k < NQ; ++k) {
      fn(pp[k], o.pp[k], o.qa[k], o.qb[k], o.mm[k]);
      fn(mp[k], o.mp[k], -o.qa[k], o.qb[k], o.pm[k]);
      fn(pm[k], o.pm[k], o.qa[k], -o.qb[k], o.mp[k]);
      fn(mm[k], o.mm[k], -o.qa[k], -o.qb[k], o.pp[k]);
    }
  }
};

template <int NA, int NQ, int NC>
__device__ __forceinline__ void orbit_moments(const Orbits<NA, NQ>& o, const OrbitValues<NA, NQ>& v, double (&M)[NC]) {
  using h37::cidx;
#pragma unroll
  for (int c = 0; c < NC; ++c) M[c] = 0.0;
  M[0] = v.r;
  auto acc = [&](int c, double k, double x) { M[c] = fma_(k, x, M[c]); };
#pragma unroll
  for (int k = 0; k < NQ; ++k) {
    const double s1 = v.pp[k] + v.mm[k], d1 = v.pp[k] - v.mm[k], s2 = v.pm[k] + v.mp[k], d2 = v.pm[k] - v.mp[k];
    const double ee = s1 + s2, oo = s1 - s2, oe = d1 + d2, eo = d1 - d2;
    M[0] = M[0] + ee;
    acc(cidx(2, 0), o.a2[k], ee);
    acc(cidx(0, 2), o.b2[k], ee);
    acc(cidx(1, 0), o.a1[k], oe);
    acc(cidx(3, 0), o.a3[k], oe);
    acc(cidx(1, 2), o.ab2[k], oe);
    acc(cidx(0, 1), o.b1[k], eo);
    acc(cidx(0, 3), o.b3[k], eo);
    acc(cidx(2, 1), o.a2b[k], eo);
    acc(cidx(1, 1), o.ab[k], oo);
    if constexpr (NC == 15) {
      acc(cidx(4, 0), o.a4[k], ee);
      acc(cidx(0, 4), o.b4[k], ee);
      acc(cidx(2, 2), o.a2b2[k], ee);
      acc(cidx(3, 1), o.a3b[k], oo);
      acc(cidx(1, 3), o.ab3[k], oo);
    }
  }
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    const double sx = v.xp[k] + v.xm[k], dx = v.xp[k] - v.xm[k], sy = v.yp[k] + v.ym[k], dy = v.yp[k] - v.ym[k];
    M[0] = M[0] + (sx + sy);
    acc(cidx(1, 0), o.p1[k], dx);
    acc(cidx(2, 0), o.p2[k], sx);
    acc(cidx(3, 0), o.p3[k], dx);
    acc(cidx(0, 1), o.p1[k], dy);
    acc(cidx(0, 2), o.p2[k], sy);
    acc(cidx(0, 3), o.p3[k], dy);
    if constexpr (NC == 15) {
      acc(cidx(4, 0), o.p4[k], sx);
      acc(cidx(0, 4), o.p4[k], sy);
    }
  }
}

// w P(e) at every velocity
template <int NA, int NQ, int NC>
__device__ __forceinline__ void orbit_values(const Orbits<NA, NQ>& o, const double (&b)[NC], OrbitValues<NA, NQ>& v) {
  using h37::cidx;
  auto w0 = [&](double w, double x) { return w * x; };
  auto add = [&](double k, int c, double x) { return fma_(k, b[c], x); };
  auto mul = [&](double k, int c) { return k * b[c]; };
  v.r = w0(o.w0, b[0]);
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    const double z = w0(o.pw[k], b[0]);
    double ex = add(o.vp2[k], cidx(2, 0), z), ey = add(o.vp2[k], cidx(0, 2), z);
    if constexpr (NC == 15) {
      ex = add(o.vp4[k], cidx(4, 0), ex);
      ey = add(o.vp4[k], cidx(0, 4), ey);
    }
    const double ox = add(o.vp3[k], cidx(3, 0), mul(o.vp1[k], cidx(1, 0)));
    const double oy = add(o.vp3[k], cidx(0, 3), mul(o.vp1[k], cidx(0, 1)));
    v.xp[k] = ex + ox;
    v.xm[k] = ex - ox;
    v.yp[k] = ey + oy;
    v.ym[k] = ey - oy;
  }
#pragma unroll
  for (int k = 0; k < NQ; ++k) {
    double ee = add(o.va2[k], cidx(2, 0), add(o.vb2[k], cidx(0, 2), w0(o.qw[k], b[0])));
    double oo = mul(o.vab[k], cidx(1, 1));
    if constexpr (NC == 15) {
      ee = add(o.va2b2[k], cidx(2, 2), add(o.va4[k], cidx(4, 0), add(o.vb4[k], cidx(0, 4), ee)));
      oo = add(o.va3b[k], cidx(3, 1), add(o.vab3[k], cidx(1, 3), oo));
    }
    const double oe = add(o.va3[k], cidx(3, 0), add(o.vab2[k], cidx(1, 2), mul(o.va1[k], cidx(1, 0))));
    const double eo = add(o.vb3[k], cidx(0, 3), add(o.va2b[k], cidx(2, 1), mul(o.vb1[k], cidx(0, 1))));
    const double s1 = ee + oo, s2 = ee - oo, t1 = oe + eo, t2 = oe - eo;
    v.pp[k] = s1 + t1;
    v.mm[k] = s1 - t1;
    v.pm[k] = s2 + t2;
    v.mp[k] = s2 - t2;
  }
}

// The constants of h37::to_polynomial for the rule's c.
struct HMap {
  double v[13];
  __device__ __forceinline__ double ns() const { return v[0]; }
  __device__ __forceinline__ double ns3() const { return v[1]; }
  __device__ __forceinline__ double ns6() const { return v[2]; }
  __device__ __forceinline__ double s2() const { return v[3]; }
  __device__ __forceinline__ double s2x3() const { return v[4]; }
  __device__ __forceinline__ double n1() const { return v[5]; }
  __device__ __forceinline__ double n2() const { return v[6]; }
  __device__ __forceinline__ double n2h() const { return v[7]; }
  __device__ __forceinline__ double n3h() const { return v[8]; }
  __device__ __forceinline__ double n3s() const { return v[9]; }
  __device__ __forceinline__ double n4q() const { return v[10]; }
  __device__ __forceinline__ double n4s() const { return v[11]; }
  __device__ __forceinline__ double n4f() const { return v[12]; }
};
template <int NA, int NQ>
struct OrbitRule {
  Orbits<NA, NQ> o;
  HMap map;
};

template <int NA, int NQ, int NC>
__device__ __forceinline__ bool orbit_update(const OrbitRule<NA, NQ>& rule, OrbitValues<NA, NQ>& v,
                                             const h37::MomentModel<double>& m) {
  double M[NC], H[NC], inc[NC];
  orbit_moments(rule.o, v, M);
  h37::to_basis<double, NC>(M, H, m);
  const bool ok = h37::moment_increments<double, NC>(H, inc, m);
#pragma unroll
  for (int k = 3; k < NC; ++k) M[k] += inc[k];
  h37::to_polynomial<double, NC>(M, rule.map);
  orbit_values(rule.o, M, v);
  return ok;
}

template <bool ODD, int NA, int NQ>
__device__ __forceinline__ void orbit_load(const double* __restrict__ f, const HGrid& g, const OrbitRule<NA, NQ>& rule,
                                           int x, int y, OrbitValues<NA, NQ>& v) {
  const uint32_t node = (uint32_t)x + (uint32_t)g.nx * (uint32_t)y;
  v.each(rule.o, [&](double& val, int i, int ex, int ey, int opp) {
    val = ODD ? f[(size_t)opp * g.N + hnbr(g, x, y, -ex, -ey)] : f[(size_t)i * g.N + node];
  });
}
template <bool ODD, int NA, int NQ>
__device__ __forceinline__ void orbit_store(double* __restrict__ f, const HGrid& g, const OrbitRule<NA, NQ>& rule, int x,
                                            int y, OrbitValues<NA, NQ>& v) {
  const uint32_t node = (uint32_t)x + (uint32_t)g.nx * (uint32_t)y;
  v.each(rule.o, [&](double& val, int i, int ex, int ey, int opp) {
    if (ODD)
      f[(size_t)i * g.N + hnbr(g, x, y, ex, ey)] = val;
    else
      f[(size_t)opp * g.N + node] = val;
  });
}

// The sweep of hgen_sweep_kernel by orbits, threads walking the nodes in one dimension.
template <int NC, int NA, int NQ, bool ODD>
__global__ void __launch_bounds__(kHgThreads)
    hgen_orbit_kernel(double* __restrict__ f, HGrid g, const __grid_constant__ OrbitRule<NA, NQ> rule,
                      const __grid_constant__ h37::MomentModel<double> m, int* __restrict__ status) {
  const uint32_t node = blockIdx.x * blockDim.x + threadIdx.x;
  chain_wait();
  if (node >= (uint32_t)g.N) return;
  const int y = (int)(node / (uint32_t)g.nx), x = (int)(node - (uint32_t)y * (uint32_t)g.nx);
  OrbitValues<NA, NQ> v;
  orbit_load<ODD>(f, g, rule, x, y, v);
  if (!orbit_update<NA, NQ, NC>(rule, v, m)) atomicOr(status, 1);
  orbit_store<ODD>(f, g, rule, x, y, v);
}

// The FP64 sweep with two threads per node, for grids that leave SM partitions empty: a
// partition issues one FP64 warp instruction per 64 cycles however few of its lanes are
// active, so more warps of shorter streams are faster while partitions are free.  The
// first thread of a node takes the x pairs and half of the quadruples; the second takes
// the y pairs and the other half, with x and y exchanged, so that both run the same
// code.  Each adds the other's sums to its own (102 FP64 operations in and 91 out,
// against 180 and 181); both compute the collision, from the same bits.  Shear wave on
// 80^2, rule E9-A, with its amplitude records: 23.4 -> 19.3 us a step.
template <int NA, int NH>
struct HalfOrbits {
  struct Pair {
    int i[2], a;         // +, -; |e|
    double c[5], v[5];   // a^n, w a^n
  } p[NA];
  struct Quad {
    int i[4], a, b;         // (a, b), (-a, b), (a, -b), (-a, -b); a = 0: none
    double c[15], v[15];    // a^p b^q, w a^p b^q
  } q[NH];
};
template <int NA, int NH>
struct HalfRule {
  HalfOrbits<NA, NH> half[2];
  HMap map;
  int rest;
  double w0;
};

template <int NA, int NQ>
void split_orbits(const OrbitRule<NA, NQ>& r, HalfRule<NA, (NQ + 1) / 2>* out) {
  const auto& o = r.o;
  *out = HalfRule<NA, (NQ + 1) / 2>{};
  out->map = r.map;
  out->rest = o.rest;
  out->w0 = o.w0;
  for (int h = 0; h < 2; ++h) {
    for (int k = 0; k < NA; ++k) {
      auto& p = out->half[h].p[k];
      p.i[0] = h ? o.yp[k] : o.xp[k];
      p.i[1] = h ? o.ym[k] : o.xm[k];
      p.a = o.da[k];
      for (int n = 0; n < 5; ++n) {
        p.c[n] = n ? p.c[n - 1] * p.a : 1.0;
        p.v[n] = o.pw[k] * p.c[n];
      }
    }
    for (int k = 0; k < (NQ + 1) / 2; ++k) {
      auto& q = out->half[h].q[k];
      const int j = 2 * k + h;
      if (j >= NQ) {
        for (int& i : q.i) i = o.rest;
        continue;
      }
      q.i[0] = o.pp[j];
      q.i[1] = h ? o.pm[j] : o.mp[j];
      q.i[2] = h ? o.mp[j] : o.pm[j];
      q.i[3] = o.mm[j];
      q.a = h ? o.qb[j] : o.qa[j];
      q.b = h ? o.qa[j] : o.qb[j];
      for (int c = 0; c < 15; ++c) {
        q.c[c] = 1.0;  // small integers: exact
        for (int n = 0; n < h37::cp(c); ++n) q.c[c] *= q.a;
        for (int n = 0; n < h37::cq(c); ++n) q.c[c] *= q.b;
        q.v[c] = o.qw[j] * q.c[c];
      }
    }
  }
}

template <int NC, int NA, int NH, bool ODD>
__global__ void __launch_bounds__(32)
    hgen_half_kernel(double* __restrict__ f, HGrid g, const __grid_constant__ HalfRule<NA, NH> rule,
                     const __grid_constant__ h37::MomentModel<double> m, int* __restrict__ status) {
  using h37::cidx;
  using h37::cp;
  using h37::cq;
  const uint32_t id = blockIdx.x * 32 + threadIdx.x;
  const int h = (int)(id & 1);
  const HalfOrbits<NA, NH>& o = rule.half[h];
  chain_wait();
  const bool in = (id >> 1) < (uint32_t)g.N;
  // threads past the grid take part in the exchange, with the last node's values: it is of
  // their own warp, whose stores come after all of its loads
  const uint32_t node = in ? id >> 1 : (uint32_t)g.N - 1u;
  const int y = (int)(node / (uint32_t)g.nx), x = (int)(node - (uint32_t)y * (uint32_t)g.nx);
  auto nbr = [&](int ex, int ey) { return h ? hnbr(g, x, y, ey, ex) : hnbr(g, x, y, ex, ey); };
  auto load = [&](int i, int ex, int ey, int opp) {
    return ODD ? f[(size_t)opp * g.N + nbr(-ex, -ey)] : f[(size_t)i * g.N + node];
  };
  auto store = [&](double v, int i, int ex, int ey, int opp) {
    if (ODD)
      f[(size_t)i * g.N + nbr(ex, ey)] = v;
    else
      f[(size_t)opp * g.N + node] = v;
  };
  double vr = load(rule.rest, 0, 0, rule.rest), vp[NA][2], vq[NH][4];
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    vp[k][0] = load(o.p[k].i[0], o.p[k].a, 0, o.p[k].i[1]);
    vp[k][1] = load(o.p[k].i[1], -o.p[k].a, 0, o.p[k].i[0]);
  }
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const int a = o.q[k].a, b = o.q[k].b;
    vq[k][0] = load(o.q[k].i[0], a, b, o.q[k].i[3]);
    vq[k][1] = load(o.q[k].i[1], -a, b, o.q[k].i[2]);
    vq[k][2] = load(o.q[k].i[2], a, -b, o.q[k].i[1]);
    vq[k][3] = load(o.q[k].i[3], -a, -b, o.q[k].i[0]);
    if (a == 0) vq[k][0] = vq[k][1] = vq[k][2] = vq[k][3] = 0.0;
  }
  double M[NC], H[NC], inc[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) M[c] = 0.0;
  if (h == 0) M[0] = vr;
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const double s1 = vq[k][0] + vq[k][3], d1 = vq[k][0] - vq[k][3], s2 = vq[k][2] + vq[k][1], d2 = vq[k][2] - vq[k][1];
    const double z[4] = {s1 + s2, d1 + d2, d1 - d2, s1 - s2};  // parities (even, even), (odd, even), (even, odd), (odd, odd)
    M[0] += z[0];
#pragma unroll
    for (int c = 1; c < NC; ++c) M[c] = fma_(o.q[k].c[c], z[(cp(c) & 1) + 2 * (cq(c) & 1)], M[c]);
  }
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    const double sx = vp[k][0] + vp[k][1], dx = vp[k][0] - vp[k][1];
    M[0] += sx;
#pragma unroll
    for (int n = 1; n <= (NC == 15 ? 4 : 3); ++n) M[cidx(n, 0)] = fma_(o.p[k].c[n], n & 1 ? dx : sx, M[cidx(n, 0)]);
  }
  {
    double other[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) other[c] = __shfl_xor_sync(0xffffffffu, M[cidx(cq(c), cp(c))], 1);
#pragma unroll
    for (int c = 0; c < NC; ++c) M[c] += other[c];
  }
  h37::to_basis<double, NC>(M, H, m);
  const bool ok = h37::moment_increments<double, NC>(H, inc, m);
  // the second thread's increments are the first's: its own may differ in the last bits
#pragma unroll
  for (int c = 3; c < NC; ++c) {
    const double first = __shfl_sync(0xffffffffu, inc[c], threadIdx.x & 30);
    H[c] = first;
  }
#pragma unroll
  for (int c = 3; c < NC; ++c) M[c] += h ? H[cidx(cq(c), cp(c))] : H[c];
  h37::to_polynomial<double, NC>(M, rule.map);
  if (!in) return;
  if (!ok) atomicOr(status, 1);
  if (h == 0) store(rule.w0 * M[0], rule.rest, 0, 0, rule.rest);
#pragma unroll
  for (int k = 0; k < NA; ++k) {
    const auto& p = o.p[k];
    double e = fma_(p.v[2], M[cidx(2, 0)], p.v[0] * M[0]);
    if constexpr (NC == 15) e = fma_(p.v[4], M[cidx(4, 0)], e);
    const double od = fma_(p.v[3], M[cidx(3, 0)], p.v[1] * M[cidx(1, 0)]);
    store(e + od, p.i[0], p.a, 0, p.i[1]);
    store(e - od, p.i[1], -p.a, 0, p.i[0]);
  }
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const auto& q = o.q[k];
    double z[4] = {q.v[0] * M[0], q.v[1] * M[1], q.v[2] * M[2], q.v[cidx(1, 1)] * M[cidx(1, 1)]};
#pragma unroll
    for (int c = 3; c < NC; ++c) {
      if (c == cidx(1, 1)) continue;
      double& t = z[(cp(c) & 1) + 2 * (cq(c) & 1)];
      t = fma_(q.v[c], M[c], t);
    }
    const double s1 = z[0] + z[3], s2 = z[0] - z[3], t1 = z[1] + z[2], t2 = z[1] - z[2];
    if (q.a == 0) continue;
    store(s1 + t1, q.i[0], q.a, q.b, q.i[3]);
    store(s1 - t1, q.i[3], -q.a, -q.b, q.i[0]);
    store(s2 + t2, q.i[2], q.a, -q.b, q.i[1]);
    store(s2 - t2, q.i[1], -q.a, q.b, q.i[2]);
  }
}

__device__ __forceinline__ void hxy_of(const HGrid& g, int64_t n, int& x, int& y) {
  const uint32_t nn = (uint32_t)n, nx = (uint32_t)g.nx;
  y = (int)(nn / nx);
  x = (int)(nn - (uint32_t)y * nx);
}

template <int S, int Q, int NC, typename F>
__global__ void hgen_init_kernel(typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, double eps_ref,
                                 const F* __restrict__ rho, const F* __restrict__ u, const F* __restrict__ theta,
                                 int64_t n0, int64_t cnt, int64_t ld) {
  using T = typename HStore<S>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  int x, y;
  hxy_of(g, n0 + k, x, y);
  const T ux = (T)((double)u[k] * t.c), uy = (T)((double)u[ld + k] * t.c);
  const T eps = theta ? (T)((double)theta[k] - 1.0) : cst<T>(0.0);
  T gx[5], gy[5];
  h37::g_forms<T>(ux, eps, gx);
  h37::g_forms<T>(uy, eps, gy);
  T a[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c)
    a[c] = (T)rho[k] * gx[h37::cp(c)] * gy[h37::cq(c)] - h37::aref<T>(c, (T)eps_ref);
  T v[Q];
  from_coeffs<T, Q, NC>(t, a, v);
  hscatter<T, Q>(f, g, t, x, y, 0, v);
}

// rho - 1, u (Hermite units) and theta - 1 of one node from its offsets
template <typename T, int Q, int NC>
__device__ __forceinline__ void hnode_macro(const HTables& t, const T (&v)[Q], double eps_ref, int thermal, T& drho,
                                            T& ux, T& uy, T& eps) {
  T a[NC];
  to_coeffs<T, Q, NC>(t, v, a);
  drho = a[0];
  const T irho = cst<T>(1.0) / (cst<T>(1.0) + drho);
  ux = a[h37::cidx(1, 0)] * irho;
  uy = a[h37::cidx(0, 1)] * irho;
  eps = thermal ? cst<T>(0.5) * ((cst<T>(2.0 * eps_ref) + a[h37::cidx(2, 0)] + a[h37::cidx(0, 2)]) * irho -
                                 (ux * ux + uy * uy))
                : cst<T>(0.0);
}

template <int S, int Q, int NC, typename F>
__global__ void hgen_moments_kernel(const typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, int odd,
                                    double eps_ref, int thermal, F* __restrict__ rho, F* __restrict__ u,
                                    F* __restrict__ theta, int64_t n0, int64_t cnt, int64_t ld) {
  using T = typename HStore<S>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  int x, y;
  hxy_of(g, n0 + k, x, y);
  T v[Q];
  hgather<T, Q>(f, g, t, x, y, odd, v);
  // the moments in the wider of the storage and the output type, so that FP64
  // fields of FP32 storage carry no FP32 rounding of their own
  using M = typename std::conditional<(sizeof(F) > sizeof(T)), F, T>::type;
  M vm[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) vm[i] = (M)v[i];
  M drho, ux, uy, eps;
  hnode_macro<M, Q, NC>(t, vm, eps_ref, thermal, drho, ux, uy, eps);
  rho[k] = (F)(cst<M>(1.0) + drho);
  u[k] = (F)((double)ux / t.c);
  u[ld + k] = (F)((double)uy / t.c);
  if (theta) theta[k] = (F)(cst<M>(1.0) + eps);
}

template <int S, int Q>
__global__ void hgen_get_pops_kernel(const typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, int odd,
                                     double* __restrict__ out, int64_t n0, int64_t cnt, int64_t ld) {
  using T = typename HStore<S>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  int x, y;
  hxy_of(g, n0 + k, x, y);
  T v[Q];
  hgather<T, Q>(f, g, t, x, y, odd, v);
#pragma unroll
  for (int i = 0; i < Q; ++i) out[i * ld + k] = t.fref[i] + (double)v[i];
}

template <int S, int Q>
__global__ void hgen_set_pops_kernel(typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, int odd,
                                     const double* __restrict__ in, int64_t n0, int64_t cnt, int64_t ld) {
  using T = typename HStore<S>::type;
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= cnt) return;
  int x, y;
  hxy_of(g, n0 + k, x, y);
  T v[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) v[i] = (T)(in[i * ld + k] - t.fref[i]);
  hscatter<T, Q>(f, g, t, x, y, odd, v);
}

// Grid totals {sum (rho - 1), sum rho u_x, sum rho u_y, 0, sum rho |u|^2 / 2}, lattice units.
template <int S, int Q, int NC>
__global__ void __launch_bounds__(kAuxThreads)
    hgen_reduce_kernel(const typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, int odd,
                       double eps_ref, double* __restrict__ partials) {
  using T = typename HStore<S>::type;
  double acc[5] = {0, 0, 0, 0, 0};
  for (int y = blockIdx.x; y < g.ny; y += gridDim.x)
    for (int x = threadIdx.x; x < g.nx; x += blockDim.x) {
      T v[Q];
      hgather<T, Q>(f, g, t, x, y, odd, v);
      T drho, ux, uy, eps;
      hnode_macro<T, Q, NC>(t, v, eps_ref, 0, drho, ux, uy, eps);
      const double r = 1.0 + (double)drho, vx = (double)ux / t.c, vy = (double)uy / t.c;
      acc[0] += (double)drho;
      acc[1] += r * vx;
      acc[2] += r * vy;
      acc[4] += 0.5 * r * (vx * vx + vy * vy);
    }
  block_sum<5>(acc);
  if (threadIdx.x == 0)
    for (int k = 0; k < 5; ++k) partials[(size_t)blockIdx.x * 8 + k] = acc[k];
}

// Mode amplitude of field 0 = rho - 1, 1/2 = u_x/u_y (lattice units), 3 = theta - 1,
// 4 = rho theta - 1.
template <int S, int Q, int NC>
__global__ void __launch_bounds__(kAuxThreads)
    hgen_mode_kernel(const typename HStore<S>::type* __restrict__ f, HGrid g, const HTables t, int odd, double eps_ref,
                     int thermal, int field, long long mx, long long my, double* __restrict__ partials) {
  using T = typename HStore<S>::type;
  double acc[2] = {0, 0};
  const long long ax = ((mx % g.nx) + g.nx) % g.nx, ay = ((my % g.ny) + g.ny) % g.ny;
  for (int y = blockIdx.x; y < g.ny; y += gridDim.x) {
    double sr, cr;
    sincospi(2.0 * (double)((ay * y) % g.ny) / g.ny, &sr, &cr);
    double ar = 0, ai = 0;
    for (int x = threadIdx.x; x < g.nx; x += blockDim.x) {
      T v[Q];
      hgather<T, Q>(f, g, t, x, y, odd, v);
      T drho, ux, uy, eps;
      hnode_macro<T, Q, NC>(t, v, eps_ref, thermal, drho, ux, uy, eps);
      double q;
      if (field == 0) q = (double)drho;
      else if (field == 1) q = (double)ux / t.c;
      else if (field == 2) q = (double)uy / t.c;
      else if (field == 3) q = (double)eps;
      else q = (double)drho + (double)eps + (double)drho * (double)eps;  // (1 + drho)(1 + eps) - 1
      double sn, cs;
      sincospi(2.0 * (double)((ax * x) % g.nx) / g.nx, &sn, &cs);
      ar += q * cs;
      ai -= q * sn;
    }
    acc[0] += ar * cr + ai * sr;
    acc[1] += ai * cr - ar * sr;
  }
  block_sum<2>(acc);
  if (threadIdx.x == 0) {
    partials[(size_t)blockIdx.x * 8 + 0] = acc[0];
    partials[(size_t)blockIdx.x * 8 + 1] = acc[1];
  }
}

inline HGrid hgrid(const Sim* s) { return HGrid{(int)s->nx, (int)s->ny, s->N}; }
inline unsigned hblocks(int64_t cnt) { return (unsigned)((cnt + kAuxThreads - 1) / kAuxThreads); }

inline h37::Model hmodel(const Sim* s) {
  h37::Model m;
  m.thermal = (s->flags & LBM_THERMAL) ? 1 : 0;
  m.raw = 0;
  m.kfac = 1.0f;
  m.eps_ref = s->theta_ref - 1.0;
  m.sround = 0;
  m.seed = 0;
  return m;
}

void fill_map(double c2, HMap* k) {
  const double s = 1.0 / c2, n = c2;
  const double v[13] = {-s, -3.0 * s, -6.0 * s, s * s, 3.0 * s * s, n, n * n, 0.5 * n * n, 0.5 * n * n * n,
                        n * n * n / 6.0, 0.25 * n * n * n * n, n * n * n * n / 6.0, n * n * n * n / 24.0};
  for (int i = 0; i < 13; ++i) k->v[i] = v[i];
}
template <int NA, int NQ>
bool fill_rule(const HLattice& L, OrbitRule<NA, NQ>* r) {
  fill_map(L.c * L.c, &r->map);
  return make_orbits(L, &r->o);
}
h37::MomentModel<double> hmoment_model(const Sim* s) {
  h37::MomentModel<double> m;
  const double sl = 1.0 / (s->hl.c * s->hl.c), tau = h37::basis_temperature(s->theta_ref * sl);
  for (int n = 0; n < 5; ++n) m.no[n] = -s->rates.w[n];
  m.s = sl;
  m.basis = tau;
  m.basis2x3 = 3.0 * tau * tau;
  m.th_ref = s->theta_ref * sl - tau;
  m.th_iso = sl - tau;
  m.kext = 0;
  m.usq_max = 4.0 * sl;
  m.thermal = (s->flags & LBM_THERMAL) ? 1 : 0;
  m.raw = 0;
  return m;
}

// The orbit sweep if the rule has NA and NQ orbits of each kind; *taken says so.
template <int NC, int NA, int NQ>
cudaError_t orbit_sweep(Sim* s, int odd, bool* taken) {
  OrbitRule<NA, NQ> rule;
  *taken = fill_rule(s->hl, &rule);
  if (!*taken) return cudaSuccess;
  double* f = static_cast<double*>(s->pop);
  // two threads per node while that leaves at most one warp per SM partition: beyond, a
  // partition would issue two shorter streams instead of one (us a step, one thread and
  // two: 80^2 22.3 and 18.6, 64 x 152 22.3 and 18.1, 100^2 22.4 and 23.9, 139^2 25.4 and 33.1;
  // 17 velocities on 80^2: E7-D 9.1 and 8.7, E7-A, whose 3 quadruples do not halve, 9.5 and 9.6)
  if (s->N <= (int64_t)4 * 152 * 16) {
    constexpr int NH = (NQ + 1) / 2;
    HalfRule<NA, NH> half;
    split_orbits(rule, &half);
    return launch_chained(odd ? hgen_half_kernel<NC, NA, NH, true> : hgen_half_kernel<NC, NA, NH, false>,
                          dim3((unsigned)((2 * s->N + 31) / 32)), dim3(32), 0, s->stream, f, hgrid(s), half,
                          hmoment_model(s), status_word(s));
  }
  // the largest of 128, 64, 32 threads that gives every SM two blocks: small grids spread over all of them
  int t = kHgThreads;
  while (t > 32 && s->N < (int64_t)t * 2 * 152) t /= 2;
  const unsigned blocks = (unsigned)((s->N + t - 1) / t);
  return launch_chained(odd ? hgen_orbit_kernel<NC, NA, NQ, true> : hgen_orbit_kernel<NC, NA, NQ, false>, dim3(blocks),
                        dim3(t), 0, s->stream, f, hgrid(s), rule, hmoment_model(s), status_word(s));
}

template <int S, int Q, int NC, bool EXACT>
cudaError_t sweep_e(Sim* s, int odd, const HSplit& sp) {
  using E = typename HStore<S>::type;
  dim3 grid((unsigned)((s->nx + kHgThreads - 1) / kHgThreads), (unsigned)s->ny);
  E* f = static_cast<E*>(s->pop);
  if (odd)
    hgen_sweep_kernel<S, Q, NC, true, EXACT><<<grid, kHgThreads, 0, s->stream>>>(f, hgrid(s), *s->ht, s->rates,
                                                                                 hmodel(s), status_word(s), sp);
  else
    hgen_sweep_kernel<S, Q, NC, false, EXACT><<<grid, kHgThreads, 0, s->stream>>>(f, hgrid(s), *s->ht, s->rates,
                                                                                  hmodel(s), status_word(s), sp);
  return cudaGetLastError();
}

// FP32 storage takes the correctly rounded transforms unless LBM_FAST_TRANSFORMS.
template <int S, int Q, int NC>
cudaError_t sweep_t(Sim* s, int odd) {
  // FP64 only: FP32 populations keep the roundings of the tables' collision
  if constexpr (S == LBM_F64) {
    // the orbit counts of the minimal rules: 37 velocities have three axis shells, 17 one or two
    bool taken = false;
    cudaError_t e;
    if constexpr (Q == 37) {
      e = orbit_sweep<NC, 3, 6>(s, odd, &taken);
      if (taken) return e;
    } else {
      e = orbit_sweep<NC, 2, 2>(s, odd, &taken);
      if (taken) return e;
      e = orbit_sweep<NC, 1, 3>(s, odd, &taken);
      if (taken) return e;
    }
  }
  // host staging of the split tables, one per host thread (the launch copies its parameters)
  thread_local static HSplit sp;
  if constexpr (S == LBM_F32) {
    if (!(s->flags & LBM_FAST_TRANSFORMS)) {
      split_tables(*s->ht, &sp);
      return sweep_e<S, Q, NC, true>(s, odd, sp);
    }
  }
  return sweep_e<S, Q, NC, false>(s, odd, sp);
}

template <int S, int Q, int NC>
cudaError_t init_t(Sim* s, const void* rho, const void* u, const void* th, int dtype, int64_t n0, int64_t cnt,
                   int64_t ld) {
  using E = typename HStore<S>::type;
  if (cnt <= 0) return cudaSuccess;
  E* f = static_cast<E*>(s->pop);
  const double er = s->theta_ref - 1.0;
  if (dtype == LBM_DTYPE_F64)
    hgen_init_kernel<S, Q, NC, double><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
        f, hgrid(s), *s->ht, er, static_cast<const double*>(rho), static_cast<const double*>(u),
        static_cast<const double*>(th), n0, cnt, ld);
  else
    hgen_init_kernel<S, Q, NC, float><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
        f, hgrid(s), *s->ht, er, static_cast<const float*>(rho), static_cast<const float*>(u),
        static_cast<const float*>(th), n0, cnt, ld);
  return cudaGetLastError();
}

template <int S, int Q, int NC>
cudaError_t moments_t(Sim* s, void* rho, void* u, void* th, int dtype, int64_t n0, int64_t cnt, int64_t ld) {
  using E = typename HStore<S>::type;
  if (cnt <= 0) return cudaSuccess;
  const E* f = static_cast<const E*>(s->pop);
  const int odd = (int)(s->step & 1);
  const int thermal = (s->flags & LBM_THERMAL) ? 1 : 0;
  if (dtype == LBM_DTYPE_F64)
    hgen_moments_kernel<S, Q, NC, double><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
        f, hgrid(s), *s->ht, odd, s->theta_ref - 1.0, thermal, static_cast<double*>(rho), static_cast<double*>(u),
        static_cast<double*>(th), n0, cnt, ld);
  else
    hgen_moments_kernel<S, Q, NC, float><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
        f, hgrid(s), *s->ht, odd, s->theta_ref - 1.0, thermal, static_cast<float*>(rho), static_cast<float*>(u),
        static_cast<float*>(th), n0, cnt, ld);
  return cudaGetLastError();
}

template <int S, int Q, int NC>
cudaError_t get_pops_t(Sim* s, double* out, int64_t n0, int64_t cnt, int64_t ld) {
  using E = typename HStore<S>::type;
  if (cnt <= 0) return cudaSuccess;
  hgen_get_pops_kernel<S, Q><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
      static_cast<const E*>(s->pop), hgrid(s), *s->ht, (int)(s->step & 1), out, n0, cnt, ld);
  return cudaGetLastError();
}

template <int S, int Q, int NC>
cudaError_t set_pops_t(Sim* s, const double* in, int64_t n0, int64_t cnt, int64_t ld) {
  using E = typename HStore<S>::type;
  if (cnt <= 0) return cudaSuccess;
  hgen_set_pops_kernel<S, Q><<<hblocks(cnt), kAuxThreads, 0, s->stream>>>(
      static_cast<E*>(s->pop), hgrid(s), *s->ht, (int)(s->step & 1), in, n0, cnt, ld);
  return cudaGetLastError();
}

template <int S, int Q, int NC>
cudaError_t reduce_into_t(Sim* s, double* partials, int nblocks, double* result) {
  using E = typename HStore<S>::type;
  hgen_reduce_kernel<S, Q, NC><<<nblocks, kAuxThreads, 0, s->stream>>>(
      static_cast<const E*>(s->pop), hgrid(s), *s->ht, (int)(s->step & 1), s->theta_ref - 1.0, partials);
  finalize_kernel<<<1, kAuxThreads, 0, s->stream>>>(partials, nblocks, 5, result);
  return cudaGetLastError();
}

template <int S, int Q, int NC>
cudaError_t mode_into_t(Sim* s, int field, const int64_t m[3], double* out2) {
  using E = typename HStore<S>::type;
  hgen_mode_kernel<S, Q, NC><<<kRedBlocks, kAuxThreads, 0, s->stream>>>(
      static_cast<const E*>(s->pop), hgrid(s), *s->ht, (int)(s->step & 1), s->theta_ref - 1.0,
      (s->flags & LBM_THERMAL) ? 1 : 0, field, (long long)m[0], (long long)m[1], partials_buf(s));
  finalize_kernel<<<1, kAuxThreads, 0, s->stream>>>(partials_buf(s), kRedBlocks, 2, out2);
  return cudaGetLastError();
}

// storage (FP64 / FP32) x (Q, NC) in {(17, 10), (37, 10), (37, 15)}
#define LBM_HGEN_DISPATCH(FN, ...)                                                        \
  do {                                                                                    \
    const int key = s->hl.q * 100 + s->ht->nc;                                            \
    if (s->storage == LBM_F64) {                                                          \
      if (key == 1710) return FN<LBM_F64, 17, 10>(s, __VA_ARGS__);                        \
      if (key == 3710) return FN<LBM_F64, 37, 10>(s, __VA_ARGS__);                        \
      if (key == 3715) return FN<LBM_F64, 37, 15>(s, __VA_ARGS__);                        \
    } else if (s->storage == LBM_F32) {                                                   \
      if (key == 1710) return FN<LBM_F32, 17, 10>(s, __VA_ARGS__);                        \
      if (key == 3710) return FN<LBM_F32, 37, 10>(s, __VA_ARGS__);                        \
      if (key == 3715) return FN<LBM_F32, 37, 15>(s, __VA_ARGS__);                        \
    }                                                                                     \
    return cudaErrorInvalidValue;                                                         \
  } while (0)

}  // namespace

cudaError_t hgen_launch_sweep(Sim* s, int odd) { LBM_HGEN_DISPATCH(sweep_t, odd); }
cudaError_t hgen_launch_init(Sim* s, const void* rho, const void* u, const void* theta, int dtype, int64_t n0,
                             int64_t cnt, int64_t ld) {
  LBM_HGEN_DISPATCH(init_t, rho, u, theta, dtype, n0, cnt, ld);
}
cudaError_t hgen_launch_moments(Sim* s, void* rho, void* u, void* theta, int dtype, int64_t n0, int64_t cnt,
                                int64_t ld) {
  LBM_HGEN_DISPATCH(moments_t, rho, u, theta, dtype, n0, cnt, ld);
}
cudaError_t hgen_launch_get_pops(Sim* s, double* f, int64_t n0, int64_t cnt, int64_t ld) {
  LBM_HGEN_DISPATCH(get_pops_t, f, n0, cnt, ld);
}
cudaError_t hgen_launch_set_pops(Sim* s, const double* f, int64_t n0, int64_t cnt, int64_t ld) {
  LBM_HGEN_DISPATCH(set_pops_t, f, n0, cnt, ld);
}
cudaError_t hgen_launch_reduce_into(Sim* s, double* partials, int nblocks, double* result) {
  LBM_HGEN_DISPATCH(reduce_into_t, partials, nblocks, result);
}
cudaError_t hgen_launch_mode_into(Sim* s, int field, const int64_t mode[3], double* out2) {
  LBM_HGEN_DISPATCH(mode_into_t, field, mode, out2);
}

}  // namespace lbm
