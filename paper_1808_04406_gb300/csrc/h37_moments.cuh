// The 37-velocity node update through raw moments in lattice units.
//
// The collision of Sec. II.C only needs the 15 moments of the truncated
// distribution up to order 4.  Written with the integer velocities e (xi = c e),
// they are M_pq = sum_i f_i e_ix^p e_iy^q, and the velocities are rows of a 7 x 7
// grid (7, 7, 5 and 3 nodes wide for |e_y| = 0, 1, 2, 3).  So the projection is
// done per axis: every row is folded at e_x = 0 and summed with the weights
// 1, 4, 9, 16, 81 / 1, 2, 3, 8, 27, the rows are folded at e_y = 0 and summed
// likewise: 136 additions and FMAs for all 15 moments.  The way back evaluates
// the polynomial P(e) = sum b_pq e_x^p e_y^q with f_i = w_i P(e_i) row by row:
// 131 operations, after a 45-operation map from the moments to b.  The dense
// products with the 37 x 15 Hermite tables this replaces took 315 each way (with
// +- pairs folded).  Arithmetic and instruction fetch bound these kernels (all of
// an update is straight-line code, 96 KB of it for the FP32 sweep with
// compensated table sums, whose warps waited for instructions 78 % of the time).
// Microseconds a step, before and after, FP32 (correctly rounded): 512^2 66.5 and
// 20.3, 128^2 14.3 and 6.1 (18.2 and 4.0 since the steps are chained launches).
//
// FP64, and FP32 with error-free sums, only: plain FP32 sums of raw moments drift
// twice as fast as the tables' (h37.cu).
#pragma once

#include <cmath>

#include "h37_common.cuh"

namespace lbm {
namespace h37 {

// velocity index of (ex, ey), -1 where the rule has none
__host__ __device__ constexpr int vidx(int ex, int ey) {
  for (int i = 0; i < kQ; ++i)
    if (ex_of(i) == ex && ey_of(i) == ey) return i;
  return -1;
}
__host__ __device__ constexpr int row_half(int ey) {  // widest |e_x| of a row
  const int a = ey < 0 ? -ey : ey;
  return a < 2 ? 3 : a == 2 ? 2 : 1;
}
__host__ __device__ constexpr double w_at(int ex, int ey) { return w_of(vidx(ex, ey)); }
constexpr double kS = 1.0 / (kC * kC);  // unit temperature in lattice units

// m + k x, a plain addition for k = 1
template <typename T>
__device__ __forceinline__ T axpy(double k, T x, T m) {
  return k == 1.0 ? m + x : fma_(x, cst<T>(k), m);
}

// x moments 0..4 of row EY
template <typename T, int EY>
__device__ __forceinline__ void row_moments(const T (&v)[kQ], T (&r)[5]) {
  constexpr int H = row_half(EY);
  const T s1 = v[vidx(1, EY)] + v[vidx(-1, EY)], d1 = v[vidx(1, EY)] - v[vidx(-1, EY)];
  r[0] = s1 + v[vidx(0, EY)];
  r[1] = r[3] = d1;
  r[2] = r[4] = s1;
  if constexpr (H >= 2) {
    const T s2 = v[vidx(2, EY)] + v[vidx(-2, EY)], d2 = v[vidx(2, EY)] - v[vidx(-2, EY)];
    r[0] = r[0] + s2;
    r[1] = axpy(2.0, d2, r[1]);
    r[2] = axpy(4.0, s2, r[2]);
    r[3] = axpy(8.0, d2, r[3]);
    r[4] = axpy(16.0, s2, r[4]);
  }
  if constexpr (H >= 3) {
    const T s3 = v[vidx(3, EY)] + v[vidx(-3, EY)], d3 = v[vidx(3, EY)] - v[vidx(-3, EY)];
    r[0] = r[0] + s3;
    r[1] = axpy(3.0, d3, r[1]);
    r[2] = axpy(9.0, s3, r[2]);
    r[3] = axpy(27.0, d3, r[3]);
    r[4] = axpy(81.0, s3, r[4]);
  }
}

// add rows +B and -B to the moments
template <typename T, int B>
__device__ __forceinline__ void add_rows(const T (&v)[kQ], T (&M)[kNC]) {
  T a[5], b[5];
  row_moments<T, B>(v, a);
  row_moments<T, -B>(v, b);
  constexpr bool narrow = row_half(B) == 1;  // then r2 = r4 and r1 = r3
  T e[5], o[4];
#pragma unroll
  for (int p = 0; p < 5; ++p) e[p] = narrow && p > 2 ? e[p - 2] : a[p] + b[p];
#pragma unroll
  for (int p = 0; p < 4; ++p) o[p] = narrow && p > 2 ? o[p - 2] : a[p] - b[p];
#pragma unroll
  for (int p = 0; p < 5; ++p) M[cidx(p, 0)] = M[cidx(p, 0)] + e[p];
#pragma unroll
  for (int p = 0; p < 4; ++p) M[cidx(p, 1)] = axpy(B, o[p], M[cidx(p, 1)]);
#pragma unroll
  for (int p = 0; p < 3; ++p) M[cidx(p, 2)] = axpy(B * B, e[p], M[cidx(p, 2)]);
#pragma unroll
  for (int p = 0; p < 2; ++p) M[cidx(p, 3)] = axpy(B * B * B, o[p], M[cidx(p, 3)]);
  M[cidx(0, 4)] = axpy(B * B * B * B, e[0], M[cidx(0, 4)]);
}

// rows +1 and -1 start the sums over e_y != 0 (so that no addition to zero is left)
template <typename T>
__device__ __forceinline__ void to_moments(const T (&v)[kQ], T (&M)[kNC]) {
  T r[5];
  row_moments<T, 0>(v, r);
#pragma unroll
  for (int p = 0; p < 5; ++p) M[cidx(p, 0)] = r[p];
  T a[5], b[5];
  row_moments<T, 1>(v, a);
  row_moments<T, -1>(v, b);
#pragma unroll
  for (int p = 0; p < 5; ++p) {
    const T e = a[p] + b[p];
    M[cidx(p, 0)] = M[cidx(p, 0)] + e;
    if (p < 3) M[cidx(p, 2)] = e;
    if (p == 0) M[cidx(0, 4)] = e;
    if (p < 4) {
      const T o = a[p] - b[p];
      M[cidx(p, 1)] = o;
      if (p < 2) M[cidx(p, 3)] = o;
    }
  }
  add_rows<T, 2>(v, M);
  add_rows<T, 3>(v, M);
}

// Row EY and -EY of the populations from the polynomial's coefficients.
template <typename T, bool SCALED, int B>
__device__ __forceinline__ void eval_row(const T (&C)[5], int ey, T (&v)[kQ]) {
  constexpr int H = row_half(B);
  auto put = [&](int ex, T x) {
    v[vidx(ex, ey)] = SCALED ? x : x * cst<T>(w_at(ex, B));
  };
  put(0, C[0]);
#pragma unroll
  for (int a = 1; a <= H; ++a) {
    T ev, od;
    if (a == 1) {
      ev = C[0] + (C[2] + C[4]);
      od = C[1] + C[3];
    } else {
      ev = fma_(fma_(C[4], cst<T>(a * a), C[2]), cst<T>(a * a), C[0]);
      od = fma_(C[3], cst<T>(a * a * a), C[1] * cst<T>(a));
    }
    put(a, ev + od);
    put(-a, ev - od);
  }
}

template <typename T, bool SCALED, int B>
__device__ __forceinline__ void eval_rows(const T (&b)[kNC], T (&v)[kQ]) {
  auto at = [&](int p, int q) { return b[cidx(p, q)]; };
  const T E0 = axpy(B * B, axpy(B * B, at(0, 4), at(0, 2)), at(0, 0));
  const T E1 = axpy(B * B, at(1, 2), at(1, 0));
  const T E2 = axpy(B * B, at(2, 2), at(2, 0));
  T O0, O1;
  if constexpr (B == 1) {
    O0 = at(0, 1) + at(0, 3);
    O1 = at(1, 1) + at(1, 3);
  } else {
    O0 = fma_(at(0, 3), cst<T>(B * B * B), at(0, 1) * cst<T>(B));
    O1 = fma_(at(1, 3), cst<T>(B * B * B), at(1, 1) * cst<T>(B));
  }
  {
    const T C[5] = {E0 + O0, E1 + O1, axpy(B, at(2, 1), E2), axpy(B, at(3, 1), at(3, 0)), at(4, 0)};
    eval_row<T, SCALED, B>(C, B, v);
  }
  {
    const T C[5] = {E0 - O0, E1 - O1, B == 1 ? E2 - at(2, 1) : fma_(at(2, 1), cst<T>(-B), E2),
                    B == 1 ? at(3, 0) - at(3, 1) : fma_(at(3, 1), cst<T>(-B), at(3, 0)), at(4, 0)};
    eval_row<T, SCALED, B>(C, -B, v);
  }
}

template <typename T, bool SCALED>
__device__ __forceinline__ void from_polynomial(const T (&b)[kNC], T (&v)[kQ]) {
  {
    const T C[5] = {b[cidx(0, 0)], b[cidx(1, 0)], b[cidx(2, 0)], b[cidx(3, 0)], b[cidx(4, 0)]};
    eval_row<T, SCALED, 0>(C, 0, v);
  }
  eval_rows<T, SCALED, 1>(b, v);
  eval_rows<T, SCALED, 2>(b, v);
  eval_rows<T, SCALED, 3>(b, v);
}

// The constants of the map below, s = 1 / c^2: compiled in for the built-in rule.
template <typename T>
struct BuiltInMap {
  static __device__ __forceinline__ T ns() { return cst<T>(-kS); }
  static __device__ __forceinline__ T ns3() { return cst<T>(-3.0 * kS); }
  static __device__ __forceinline__ T ns6() { return cst<T>(-6.0 * kS); }
  static __device__ __forceinline__ T s2() { return cst<T>(kS * kS); }
  static __device__ __forceinline__ T s2x3() { return cst<T>(3.0 * kS * kS); }
  static __device__ __forceinline__ T n1() { return cst<T>(1.0 / kS); }
  static __device__ __forceinline__ T n2() { return cst<T>(1.0 / (kS * kS)); }
  static __device__ __forceinline__ T n2h() { return cst<T>(0.5 / (kS * kS)); }
  static __device__ __forceinline__ T n3h() { return cst<T>(0.5 / (kS * kS * kS)); }
  static __device__ __forceinline__ T n3s() { return cst<T>(1.0 / (6.0 * kS * kS * kS)); }
  static __device__ __forceinline__ T n4q() { return cst<T>(0.25 / (kS * kS * kS * kS)); }
  static __device__ __forceinline__ T n4s() { return cst<T>(1.0 / (6.0 * kS * kS * kS * kS)); }
  static __device__ __forceinline__ T n4f() { return cst<T>(1.0 / (24.0 * kS * kS * kS * kS)); }
};

// Moments to the polynomial's coefficients (in place): the Hermite coefficients
// in lattice units, B_pq = A_pq / (s^(p+q) p! q!), first, so that what the
// reference state contributes cancels before anything is scaled up; then
// their monomials.
template <typename T, int NC, typename K>
__device__ __forceinline__ void to_polynomial(T (&M)[NC], const K& k) {
  const T m00 = M[0], m20 = M[cidx(2, 0)], m02 = M[cidx(0, 2)], m11 = M[cidx(1, 1)];
  const T m10 = M[cidx(1, 0)], m01 = M[cidx(0, 1)];
  const T B20 = k.n2h() * fma_(k.ns(), m00, m20), B02 = k.n2h() * fma_(k.ns(), m00, m02);
  M[0] = fma_(k.ns(), B20 + B02, m00);
  M[cidx(2, 0)] = B20;
  M[cidx(0, 2)] = B02;
  M[cidx(1, 1)] = k.n2() * m11;
  const T B30 = k.n3s() * fma_(k.ns3(), m10, M[cidx(3, 0)]), B12 = k.n3h() * fma_(k.ns(), m10, M[cidx(1, 2)]);
  const T B03 = k.n3s() * fma_(k.ns3(), m01, M[cidx(0, 3)]), B21 = k.n3h() * fma_(k.ns(), m01, M[cidx(2, 1)]);
  M[cidx(1, 0)] = fma_(k.ns(), B12, fma_(k.ns3(), B30, k.n1() * m10));
  M[cidx(0, 1)] = fma_(k.ns(), B21, fma_(k.ns3(), B03, k.n1() * m01));
  M[cidx(3, 0)] = B30;
  M[cidx(1, 2)] = B12;
  M[cidx(0, 3)] = B03;
  M[cidx(2, 1)] = B21;
  if constexpr (NC == 15) {
    const T B40 = k.n4f() * fma_(k.s2x3(), m00, fma_(k.ns6(), m20, M[cidx(4, 0)]));
    const T B04 = k.n4f() * fma_(k.s2x3(), m00, fma_(k.ns6(), m02, M[cidx(0, 4)]));
    const T B22 = k.n4q() * fma_(k.s2(), m00, fma_(k.ns(), m20 + m02, M[cidx(2, 2)]));
    const T B31 = k.n4s() * fma_(k.ns3(), m11, M[cidx(3, 1)]), B13 = k.n4s() * fma_(k.ns3(), m11, M[cidx(1, 3)]);
    M[0] = fma_(k.s2x3(), B40 + B04, fma_(k.s2(), B22, M[0]));
    M[cidx(2, 0)] = fma_(k.ns6(), B40, fma_(k.ns(), B22, B20));
    M[cidx(0, 2)] = fma_(k.ns6(), B04, fma_(k.ns(), B22, B02));
    M[cidx(1, 1)] = fma_(k.ns3(), B31 + B13, M[cidx(1, 1)]);
    M[cidx(4, 0)] = B40;
    M[cidx(0, 4)] = B04;
    M[cidx(2, 2)] = B22;
    M[cidx(3, 1)] = B31;
    M[cidx(1, 3)] = B13;
  }
}

// What a sweep needs of the model, in the precision it computes in (FP64
// conversions run at the FP64 rate, so they are done once on the host).
template <typename R>
struct MomentModel {
  R no[5];      // minus the rates of orders 2..4
  R s;          // 1 / c^2
  R basis;      // temperature tau of the Hermite basis the collision takes its moments in (0: plain moments)
  R basis2x3;   // 3 tau^2
  R th_ref;     // theta_ref / c^2 - tau
  R th_iso;     // temperature of isothermal runs, 1 / c^2 - tau
  R kext;       // 4th-order coupling beyond that of the central moments themselves: (1 - K / 6), 1 with raw
  R usq_max;    // the largest |u|^2 the collision is defined on
  int thermal;
  int raw;      // relax in the absolute frame (the shifts to and from the relative frame are left out)
};

template <typename T>
__device__ __forceinline__ T spread(T x) {
  return x;
}
template <typename T>
__device__ __forceinline__ T spread(typename std::enable_if<std::is_same<T, f2>::value, float>::type x) {
  return pack2(x, x);
}

__device__ __forceinline__ bool in_range(float rho, float th, float usq, float lim) {
  return rho > 0.f && th > 0.f && usq < lim;
}
__device__ __forceinline__ bool in_range(double rho, double th, double usq, double lim) {
  return rho > 0.0 && th > 0.0 && usq < lim;
}

// theta rounded to 11 significant bits
inline double basis_temperature(double theta) {
  int e;
  const double f = std::frexp(theta, &e);
  return std::ldexp(std::nearbyint(f * 2048.0), e - 11);
}

// Moments in the Hermite basis of temperature tau: H_20 = M_20 - tau M_00, H_30 =
// M_30 - 3 tau M_10, ... with tau = theta_ref / c^2 rounded to 11 bits (so that its
// multiples below are exact in FP32).  A state near the reference has small H:
// what the collision subtracts from them then cancels little, and the rounding
// errors it leaves in stress and heat flux (which recur every step on a slowly
// varying state) are those of small numbers.
template <typename T, int NC>
__device__ __forceinline__ void to_basis(const T (&M)[NC], T (&H)[NC], const MomentModel<T>& m) {
  const T t = m.basis, nt = neg_(t), nt3 = cst<T>(3.0) * nt, nt6 = nt3 + nt3;
  H[0] = M[0];
  H[1] = M[1];
  H[2] = M[2];
  H[cidx(1, 1)] = M[cidx(1, 1)];
  H[cidx(2, 0)] = fma_(nt, M[0], M[cidx(2, 0)]);
  H[cidx(0, 2)] = fma_(nt, M[0], M[cidx(0, 2)]);
  H[cidx(3, 0)] = fma_(nt3, M[cidx(1, 0)], M[cidx(3, 0)]);
  H[cidx(1, 2)] = fma_(nt, M[cidx(1, 0)], M[cidx(1, 2)]);
  H[cidx(2, 1)] = fma_(nt, M[cidx(0, 1)], M[cidx(2, 1)]);
  H[cidx(0, 3)] = fma_(nt3, M[cidx(0, 1)], M[cidx(0, 3)]);
  if constexpr (NC == 15) {
    // x^4 - 6 tau x^2 + 3 tau^2 = x^4 - 6 tau (x^2 - tau) - 3 tau^2, and so on
    const T q = m.basis2x3, t2 = t * t;
    H[cidx(4, 0)] = fma_(neg_(q), M[0], fma_(nt6, H[cidx(2, 0)], M[cidx(4, 0)]));
    H[cidx(0, 4)] = fma_(neg_(q), M[0], fma_(nt6, H[cidx(0, 2)], M[cidx(0, 4)]));
    H[cidx(2, 2)] = fma_(neg_(t2), M[0], fma_(nt, H[cidx(2, 0)] + H[cidx(0, 2)], M[cidx(2, 2)]));
    H[cidx(3, 1)] = fma_(nt3, M[cidx(1, 1)], M[cidx(3, 1)]);
    H[cidx(1, 3)] = fma_(nt3, M[cidx(1, 1)], M[cidx(1, 3)]);
  }
}

// The collision: what it adds to the moments of the offsets f - f_ref (lattice
// units, orders 2..N; orders 0 and 1 are conserved).  M: the offsets' moments in
// the basis of temperature tau, in which the Maxwellian's have the form of the
// plain ones with theta - tau for theta.  With M1 = M - (M_eq - M_ref) the non-equilibrium moments,
// K their central moments about u, every K of order n >= 2 changes by -omega_n K
// (Eq. omega: the relaxation of central monomial moments; K = 6 at order 4 is
// what it amounts to for Hermite coefficients, any other K adds kext terms).
// Only these increments are shifted back, so the conserved moments keep their
// bits.  The trace of K_2 is zero by the definition of the temperature (nonzero
// in isothermal runs only), so order 2 is relaxed as half trace and half
// difference: the collision then conserves the energy exactly too.
template <typename T, int NC>
__device__ __forceinline__ bool moment_increments(const T (&M)[NC], T (&inc)[NC], const MomentModel<T>& m) {
  static_assert(NC == 10 || NC == 15, "truncation N = 3 or 4");
  const T thr = m.th_ref;
  const T drho = M[0];
  const T rho = cst<T>(1.0) + drho;
  const T irho = rcp_(rho);
  const T jx = M[cidx(1, 0)], jy = M[cidx(0, 1)];
  T ux = jx * irho, uy = jy * irho;
  const T ux2 = ux * ux, uy2 = uy * uy;
  const T usq = ux2 + uy2;
  const T half = cst<T>(0.5);
  // theta - theta_ref from the trace: rho (u^2 + 2 theta) = M_20 + M_02 + 2 theta_ref
  const T tr = fma_(cst<T>(-2.0) * thr, drho, M[cidx(2, 0)] + M[cidx(0, 2)]);
  T de, ht = cst<T>(0.0);
  if (m.thermal) {
    de = half * fma_(tr, irho, neg_(usq));
  } else {
    de = m.th_iso - thr;
    ht = half * fma_(neg_(jx), ux, fma_(neg_(jy), uy, tr)) - rho * de;
  }
  const T hd = half * fma_(neg_(jx), ux, fma_(jy, uy, M[cidx(2, 0)] - M[cidx(0, 2)]));
  const T th = thr + de;
  // one-axis moments r_n of the Maxwellian, and their increments over the reference's (r_n(0, theta_ref))
  const T th3 = cst<T>(3.0) * th, d3 = cst<T>(3.0) * de;
  T rx[5], ry[5], dx[5], dy[5];
  rx[1] = dx[1] = ux;
  ry[1] = dy[1] = uy;
  rx[2] = ux2 + th;
  ry[2] = uy2 + th;
  dx[2] = ux2 + de;
  dy[2] = uy2 + de;
  rx[3] = dx[3] = ux * (ux2 + th3);
  ry[3] = dy[3] = uy * (uy2 + th3);
  if constexpr (NC == 15) {
    const T th6 = th3 + th3, thth = th3 * th, dd = d3 * (th + thr);
    const T px = ux2 * (ux2 + th6), py = uy2 * (uy2 + th6);
    rx[4] = px + thth;
    ry[4] = py + thth;
    dx[4] = px + dd;
    dy[4] = py + dd;
  }
  // M1 for orders 2 (2, 0 and 0, 2 above) to N: M_eq - M_ref = (drho r_p + d_p) r_q + r_p(0, theta_ref) d_q
  T A[NC];
  A[cidx(2, 0)] = ht + hd;
  A[cidx(0, 2)] = ht - hd;
#pragma unroll
  for (int c = 4; c < NC; ++c) {
    if (c == 5) continue;
    const int p = cp(c), q = cq(c);
    T d0;
    if (p == 0) {
      d0 = fma_(drho, ry[q], dy[q]);
    } else {
      const T t = fma_(drho, rx[p], dx[p]);
      if (q == 0)
        d0 = t;
      else if (p == 2)
        d0 = fma_(t, ry[q], thr * dy[q]);
      else
        d0 = t * ry[q];
    }
    A[c] = M[c] - d0;
  }
  if (m.raw) ux = uy = cst<T>(0.0);
  const T u3x = cst<T>(3.0) * ux, u3y = cst<T>(3.0) * uy, u2x = ux + ux, u2y = uy + uy;
  const T o2 = m.no[2], o3 = m.no[3];
  const T a20 = A[cidx(2, 0)], a11 = A[cidx(1, 1)], a02 = A[cidx(0, 2)];
  // order 2: the shift leaves it
  const T k20 = o2 * a20, k11 = o2 * a11, k02 = o2 * a02;
  inc[cidx(2, 0)] = k20;
  inc[cidx(1, 1)] = k11;
  inc[cidx(0, 2)] = k02;
  // order 3: K = A - [3] u A2; the increment -omega_3 K + [3] u (-omega_2 A2)
  const T a30 = A[cidx(3, 0)], a21 = A[cidx(2, 1)], a12 = A[cidx(1, 2)], a03 = A[cidx(0, 3)];
  const T s30 = u3x * a20, s21 = fma_(u2x, a11, uy * a20), s12 = fma_(u2y, a11, ux * a02), s03 = u3y * a02;
  const T k30 = o3 * (a30 - s30), k21 = o3 * (a21 - s21), k12 = o3 * (a12 - s12), k03 = o3 * (a03 - s03);
  const T i30 = fma_(o2, s30, k30), i21 = fma_(o2, s21, k21), i12 = fma_(o2, s12, k12), i03 = fma_(o2, s03, k03);
  inc[cidx(3, 0)] = i30;
  inc[cidx(2, 1)] = i21;
  inc[cidx(1, 2)] = i12;
  inc[cidx(0, 3)] = i03;
  if constexpr (NC == 15) {
    if (m.basis != 0) {  // order 4 as plain moments
      const T t = m.basis, t3 = cst<T>(3.0) * t, t6 = t3 + t3;
      A[cidx(4, 0)] = fma_(t6, a20, A[cidx(4, 0)]);
      A[cidx(3, 1)] = fma_(t3, a11, A[cidx(3, 1)]);
      A[cidx(2, 2)] = fma_(t, a20 + a02, A[cidx(2, 2)]);
      A[cidx(1, 3)] = fma_(t3, a11, A[cidx(1, 3)]);
      A[cidx(0, 4)] = fma_(t6, a02, A[cidx(0, 4)]);
    }
    // order 4: K = A4 - [4] u A3 + [6] u u A2, back with [4] u K3 + [6] u u K2
    const T o4 = m.no[4];
    const T u4x = u2x + u2x, u4y = u2y + u2y;
    const T x1 = ux * ux, y1 = uy * uy, xx = u3x * ux, yy = u3y * uy, xx6 = xx + xx, yy6 = yy + yy;
    const T xy3 = u3x * uy, xy4 = u4x * uy;
    // [4] u P3 + [6] u u P2
    auto lift = [&](const T (&P3)[4], const T (&P2)[3], T (&out)[5]) {
      out[0] = fma_(u4x, P3[0], xx6 * P2[0]);
      out[1] = fma_(u3x, P3[1], fma_(uy, P3[0], fma_(xx, P2[1], xy3 * P2[0])));
      out[2] = fma_(u2x, P3[2], fma_(u2y, P3[1], fma_(x1, P2[2], fma_(xy4, P2[1], y1 * P2[0]))));
      out[3] = fma_(u3y, P3[2], fma_(ux, P3[3], fma_(yy, P2[1], xy3 * P2[2])));
      out[4] = fma_(u4y, P3[3], yy6 * P2[2]);
    };
    T up[5], dn[5];
    {
      const T P3[4] = {a30, a21, a12, a03}, P2[3] = {neg_(a20), neg_(a11), neg_(a02)};
      lift(P3, P2, up);
    }
    {
      const T P3[4] = {k30, k21, k12, k03}, P2[3] = {k20, k11, k02};
      lift(P3, P2, dn);
    }
    T k4[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) k4[q] = fma_(o4, A[10 + q] - up[q], dn[q]);
    if (m.kext != 0) {  // K other than 6, or the absolute-frame relaxation of Hermite coefficients
      const T e = m.kext * m.s * (o2 - o4);
      k4[0] = fma_(e, cst<T>(6.0) * a20, k4[0]);
      k4[1] = fma_(e, cst<T>(3.0) * a11, k4[1]);
      k4[2] = fma_(e, a20 + a02, k4[2]);
      k4[3] = fma_(e, cst<T>(3.0) * a11, k4[3]);
      k4[4] = fma_(e, cst<T>(6.0) * a02, k4[4]);
    }
#pragma unroll
    for (int q = 0; q < 5; ++q) inc[10 + q] = k4[q];
  }
  return in_range(rho, th + m.basis, usq, m.usq_max);
}

// ---- correctly rounded transforms (FP32 storage) ----------------------------
// Plain FP32 transforms drift: their constants, rounded once, are not exact
// inverses of each other, and every addition rounds; both errors recur at every
// step on a slowly varying state, and the conserved moments accumulate them
// (1e-5 relative on the velocity after 1000 steps).  Here every moment and every
// population is computed to ~2^-37 of the node's largest value and rounded once.
//
// In raw moments the transform's own constants are small integers, so the sums
// are made exact instead of compensated: each value x is cut at a quantum common
// to the node, hi = (sigma + x) - sigma and lo = x - hi (exact, sigma a power of
// two), with sigma so large that the integer combinations of the hi parts never
// need more than 24 bits.  The hi and lo parts ride in the two lanes of packed
// FP32 arithmetic: the plain transform, once.  Only the map between moments and
// polynomial takes error-free products and sums (the compensated dot product of
// Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26, 2005), 47 terms of it with the
// constants as FP32 pairs hi + lo.

// sigma = 2^(bits + 1) times the power of two at or below mx: a power of two
// at least 2^bits times every |x| <= mx.  Parts of values cut at it are
// multiples of 2^-24 sigma, so integer combinations of them whose coefficients
// sum up to at most 2^bits are exact.
__device__ __forceinline__ float cut_at(float mx, int bits) {
  return __uint_as_float((__float_as_uint(fminf(mx, 0x1p100f)) & 0x7f800000u) + ((unsigned)(bits + 1) << 23));
}
__device__ __forceinline__ f2 cut(float x, float sigma) {
  const float hi = __fsub_rn(__fadd_rn(sigma, x), sigma);
  return pack2(hi, __fsub_rn(x, hi));
}

// The map's constants b = G^-1 M (the inverse Gram matrix of the monomials up to
// order 4 under the rule's weights), as multiples of powers of c^2.
enum MapTerm {
  kT0, kT0_2, kT2_2, kT22, kT0_4, kT0_22, kT2_4, kT4_4, kT22_22, kT1, kT1_3, kT3_3, kT3_12, kT11, kT11_31, kT31_31,
  kMapTerms
};
__host__ __device__ constexpr double map_term(int t, double n) {  // n = c^2
  return t == kT0 ? 3.0
       : t == kT0_2 ? -1.5 * n
       : t == kT2_2 ? 2.25 * n * n
       : t == kT22 ? 0.25 * n * n
       : t == kT0_4 ? 0.125 * n * n
       : t == kT0_22 ? 0.25 * n * n
       : t == kT2_4 ? -0.25 * n * n * n
       : t == kT4_4 ? n * n * n * n / 24.0
       : t == kT22_22 ? 0.25 * n * n * n * n
       : t == kT1 ? 3.0 * n
       : t == kT1_3 ? -0.5 * n * n
       : t == kT3_3 ? n * n * n / 6.0
       : t == kT3_12 ? 0.5 * n * n * n
       : t == kT11 ? 4.0 * n * n
       : t == kT11_31 ? -0.5 * n * n * n
                      : n * n * n * n / 6.0;
}
struct Split {
  float h, l;
};
__host__ __device__ constexpr Split split_of(double x) { return Split{(float)x, (float)(x - (double)(float)x)}; }
__device__ __forceinline__ Split map_split(int t) { return split_of(map_term(t, kC * kC)); }

// s + c = sum of products of (x + xl) and h, s the rounded sum and c its error to second
// order (the error terms are those of the rounded products)
template <typename T>
struct Dot2 {
  T s, c;
  __device__ __forceinline__ Dot2(T x, T xl, Split h) {
    const T hh = spread<T>(h.h);
    s = mul_apart(x, hh);
    c = fma_(xl, hh, fma_(x, spread<T>(h.l), fma_(x, hh, neg_(s))));
  }
  __device__ __forceinline__ void add(T x, T xl, Split h) {
    const T hh = spread<T>(h.h);
    const T p = mul_apart(x, hh);
    const T t = s + p;
    const T z = t - s;
    const T e = (s - (t - z)) + (p - z);
    s = t;
    c = c + fma_(xl, hh, fma_(x, spread<T>(h.l), fma_(x, hh, neg_(p)) + e));
  }
};

// The polynomial's coefficients of the moments M + L (FP32 pairs) as unevaluated
// sums s + c.  Pairs that only swap x and y share packed instructions.
__device__ __forceinline__ void to_polynomial_exact(const float (&M)[kNC], const float (&L)[kNC], float (&s)[kNC],
                                                    float (&c)[kNC]) {
  auto dot = [&](int i, int t) { return Dot2<float>(M[i], L[i], map_split(t)); };
  auto add = [&](Dot2<float>& d, int i, int t) { d.add(M[i], L[i], map_split(t)); };
  auto dot2 = [&](int i, int j, int t) { return Dot2<f2>(pack2(M[i], M[j]), pack2(L[i], L[j]), map_split(t)); };
  auto add2 = [&](Dot2<f2>& d, int i, int j, int t) { d.add(pack2(M[i], M[j]), pack2(L[i], L[j]), map_split(t)); };
  auto put = [&](int i, const Dot2<float>& d) {
    s[i] = d.s;
    c[i] = d.c;
  };
  auto put2 = [&](int i, int j, const Dot2<f2>& d) {
    unpack2(d.s, s[i], s[j]);
    unpack2(d.c, c[i], c[j]);
  };
  constexpr int i20 = cidx(2, 0), i02 = cidx(0, 2), i11 = cidx(1, 1), i10 = cidx(1, 0), i01 = cidx(0, 1);
  constexpr int i30 = cidx(3, 0), i03 = cidx(0, 3), i21 = cidx(2, 1), i12 = cidx(1, 2);
  Dot2<float> b00 = dot(0, kT0);
  add(b00, i20, kT0_2);
  add(b00, i02, kT0_2);
  Dot2<f2> b2 = dot2(0, 0, kT0_2);
  add2(b2, i20, i02, kT2_2);
  Dot2<float> b11 = dot(i11, kT11);
  Dot2<f2> b1 = dot2(i10, i01, kT1);
  add2(b1, i30, i03, kT1_3);
  add2(b1, i12, i21, kT1_3);
  put2(i10, i01, b1);
  Dot2<f2> b3 = dot2(i30, i03, kT3_3);
  add2(b3, i10, i01, kT1_3);
  put2(i30, i03, b3);
  Dot2<f2> b12 = dot2(i12, i21, kT3_12);
  add2(b12, i10, i01, kT1_3);
  put2(i12, i21, b12);
  constexpr int i40 = cidx(4, 0), i04 = cidx(0, 4), i22 = cidx(2, 2), i31 = cidx(3, 1), i13 = cidx(1, 3);
  add(b00, i40, kT0_4);
  add(b00, i04, kT0_4);
  add(b00, i22, kT0_22);
  add2(b2, i02, i20, kT22);
  add2(b2, i40, i04, kT2_4);
  add2(b2, i22, i22, kT2_4);
  add(b11, i31, kT11_31);
  add(b11, i13, kT11_31);
  Dot2<f2> b4 = dot2(0, 0, kT0_4);
  add2(b4, i20, i02, kT2_4);
  add2(b4, i40, i04, kT4_4);
  put2(i40, i04, b4);
  Dot2<float> b22 = dot(0, kT0_22);
  add(b22, i20, kT2_4);
  add(b22, i02, kT2_4);
  add(b22, i22, kT22_22);
  put(i22, b22);
  Dot2<f2> b31 = dot2(i31, i13, kT31_31);
  add2(b31, i11, i11, kT11_31);
  put2(i31, i13, b31);
  put(0, b00);
  put2(i20, i02, b2);
  put(i11, b11);
}

// hi + lo parts of the sums as M + L, M rounded
__device__ __forceinline__ void round_parts(const f2 (&M2)[kNC], float (&M)[kNC], float (&L)[kNC]) {
#pragma unroll
  for (int k = 0; k < kNC; ++k) {
    float hi, lo;
    unpack2(M2[k], hi, lo);
    M[k] = hi + lo;
    L[k] = lo - (M[k] - hi);
  }
}

constexpr int kMomentBits = 10;      // sum of e_x^4 over the rule: 660
constexpr int kPolynomialBits = 8;   // sum of |e_x^p e_y^q| over p + q <= 4 at (3, 1): 179

__device__ __forceinline__ void cut_polynomial(const float (&s)[kNC], const float (&c)[kNC], f2 (&b)[kNC]) {
  float mx = fabsf(s[0]);
#pragma unroll
  for (int k = 1; k < kNC; ++k) mx = fmaxf(mx, fabsf(s[k]));
  const float sigma = cut_at(mx, kPolynomialBits);
#pragma unroll
  for (int k = 0; k < kNC; ++k) {
    float hi, lo;
    unpack2(cut(s[k], sigma), hi, lo);
    b[k] = pack2(hi, lo + c[k]);
  }
}

// w (hi + lo), rounded once
__device__ __forceinline__ float weigh(f2 p, Split w) {
  float hi, lo;
  unpack2(p, hi, lo);
  return __fmaf_rn(w.h, hi, __fmaf_rn(w.h, lo, w.l * hi));
}

// to_basis of the moments M + L, each H rounded once
__device__ __forceinline__ void to_basis_exact(const float (&M)[kNC], const float (&L)[kNC], float (&H)[kNC],
                                               const MomentModel<float>& m) {
  const float t = m.basis, t3 = 3.f * t, t6 = 6.f * t;
  auto sub = [&](float& h, float& l, float k, int i) {  // h + l -= k (M_i + L_i), k of at most 24 bits
    const float p = mul_apart(k, M[i]), d = h - p;
    l += (two_sum_err(h, -p, d) - __fmaf_rn(k, M[i], -p)) - k * L[i];
    h = d;
  };
  auto less = [&](int c, float k, int i) {
    float h = M[c], l = L[c];
    sub(h, l, k, i);
    H[c] = h + l;
  };
  H[0] = M[0];
  H[1] = M[1];
  H[2] = M[2];
  H[cidx(1, 1)] = M[cidx(1, 1)];
  less(cidx(2, 0), t, 0);
  less(cidx(0, 2), t, 0);
  less(cidx(3, 0), t3, cidx(1, 0));
  less(cidx(1, 2), t, cidx(1, 0));
  less(cidx(2, 1), t, cidx(0, 1));
  less(cidx(0, 3), t3, cidx(0, 1));
  less(cidx(3, 1), t3, cidx(1, 1));
  less(cidx(1, 3), t3, cidx(1, 1));
  auto fourth = [&](int c, float k1, int i1, float k2, int i2, float k0) {
    float h = M[c], l = L[c];
    sub(h, l, k1, i1);
    if (i2 >= 0) sub(h, l, k2, i2);
    sub(h, l, -k0, 0);
    H[c] = h + l;
  };
  fourth(cidx(4, 0), t6, cidx(2, 0), 0.f, -1, m.basis2x3);
  fourth(cidx(0, 4), t6, cidx(0, 2), 0.f, -1, m.basis2x3);
  fourth(cidx(2, 2), t, cidx(2, 0), t, cidx(0, 2), t * t);
}

// M + L <- M + L + inc for the orders that the collision changes
__device__ __forceinline__ void add_increments(float (&M)[kNC], float (&L)[kNC], const float (&inc)[kNC]) {
#pragma unroll
  for (int k = 3; k < kNC; ++k) {
    const float t = __fadd_rn(M[k], inc[k]);
    L[k] += two_sum_err(M[k], inc[k], t);
    M[k] = t;
  }
}

// The moments keep their low parts L through the collision (which computes its
// increments in plain FP32 from M), so the conserved ones come back unrounded.
__device__ __forceinline__ bool collide_exact(float (&v)[kQ], const MomentModel<float>& m) {
  float M[kNC], L[kNC], inc[kNC], s[kNC], c[kNC];
  {
    float mx = fabsf(v[0]);
#pragma unroll
    for (int i = 1; i < kQ; ++i) mx = fmaxf(mx, fabsf(v[i]));
    const float sigma = cut_at(mx, kMomentBits);
    f2 x[kQ], M2[kNC];
#pragma unroll
    for (int i = 0; i < kQ; ++i) x[i] = cut(v[i], sigma);
    to_moments(x, M2);
    round_parts(M2, M, L);
  }
  float H[kNC];
  to_basis_exact(M, L, H, m);
  const bool ok = moment_increments<float, kNC>(H, inc, m);
  add_increments(M, L, inc);
  to_polynomial_exact(M, L, s, c);
  f2 b[kNC], x[kQ];
  cut_polynomial(s, c, b);
  from_polynomial<f2, true>(b, x);
#pragma unroll
  for (int i = 0; i < kQ; ++i) v[i] = weigh(x[i], split_of(w_of(i)));
  return ok;
}

// One node of the built-in rule, in FP64.  v: offsets, in and out.
__device__ __forceinline__ bool collide_rows(double (&v)[kQ], const MomentModel<double>& m) {
  double M[kNC], H[kNC], inc[kNC];
  to_moments(v, M);
  to_basis<double, kNC>(M, H, m);
  const bool ok = moment_increments<double, kNC>(H, inc, m);
#pragma unroll
  for (int k = 3; k < kNC; ++k) M[k] = M[k] + inc[k];
  to_polynomial<double, kNC>(M, BuiltInMap<double>());
  from_polynomial<double, false>(M, v);
  return ok;
}

}  // namespace h37
}  // namespace lbm
