// PDE terms of Eq. 1 (dQ/dt + div F(Q) + B(Q).grad Q = S(Q)) as device functors.
//
// Each system provides, per voxel, the derived quantities W (computed once per
// voxel and shared by all directions), the flux F_d, the largest
// characteristic speed lambda_d, the non-conservative product B_d(Qb).dQ and
// the source S.  The direction d may be a run-time value: it is only used in
// selects, never to index a register array, so the same code serves interior
// voxels (d unrolled) and halo voxels of either direction without divergence.
#pragma once

#include <type_traits>
#include <utility>

#include "dh_internal.cuh"

namespace dh {

// f(integral_constant<int, 0>), f(integral_constant<int, 1>), ..: a loop whose index is a constant.
template <class F, int... I>
__device__ __forceinline__ void for_seq(F f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void for_n(F f) {
  for_seq(f, std::make_integer_sequence<int, N>{});
}

__device__ __forceinline__ double sel3(int d, double a, double b, double c) {
  return d == 0 ? a : (d == 1 ? b : c);
}

// GB300 issues FP64 fused multiply-adds with register operands at 2.0 per
// clock per SM, but DADD, DMUL and FP64 instructions with a constant-bank
// operand (a kernel parameter or a literal) at 1.68 (measured).  The FV stage
// therefore writes its adds, subtractions and products as FMAs whose extra
// operand is 1, -1 or 0 from its parameters (values the compiler cannot see,
// so it cannot turn them back into DADD/DMUL), and its kernels copy those
// parameters into registers once per thread (a shuffle hides them from the
// compiler, which would fold them into constant-bank operands).  The FD stage
// keeps plain operations (the FMA form measured 7% slower there with
// constant-bank operands, and no faster with register operands).  The results are bitwise those of a + b, a - b and a * b (a
// product that is -0 comes out as +0).
__device__ __forceinline__ double ADD(const DevParams& P, double a, double b) { return fma(a, P.one, b); }
__device__ __forceinline__ double SUB(const DevParams& P, double a, double b) { return fma(b, P.mone, a); }
__device__ __forceinline__ double MUL(const DevParams& P, double a, double b) { return fma(a, b, P.zero); }

// The kernels' arithmetic constants as register values: the constants that the adds, subtractions and
// products written as FMAs use and the gas constants are copied into registers once per thread; a
// shuffle hides their values from the compiler, which would otherwise fold them back into constant-bank
// operands.
__device__ __forceinline__ double opaque_reg(double v) { return __shfl_sync(0xffffffffu, v, 0); }
template <class Args>
__device__ __forceinline__ Args with_reg_params(const Args& A) {
  Args L = A;
  L.P.one = opaque_reg(A.P.one);
  L.P.mone = opaque_reg(A.P.mone);
  L.P.zero = opaque_reg(A.P.zero);
  L.P.half = opaque_reg(A.P.half);
  L.P.gamma = opaque_reg(A.P.gamma);
  L.P.gm1 = opaque_reg(A.P.gm1);
  L.P.Gamma = opaque_reg(A.P.Gamma);
  L.P.Gq = opaque_reg(A.P.Gq);
  return L;
}

// 1/a for a normal, finite, positive or negative a: the hardware reciprocal
// estimate y (PTX rcp.approx.ftz.f64, relative error below 2^-19.9 over 2^28
// sampled mantissas and exponents on GB300) refined by one step of the
// third-order (Householder, order 2) iteration for f(y) = 1/y - a:
// with e = 1 - a y, 1/a = y / (1 - e) = y (1 + e + e^2 + e^3 + ...), and
// y (1 + e + e^2) leaves a relative error of e^3 < 2^-59.  Three FMAs instead of
// a full IEEE division (about 5.7 FMA times); the result is within one unit
// in the last place of the correctly rounded reciprocal (checked against 1.0/a
// by the GPU tests).
__device__ __forceinline__ double recip_nr(double a) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-a, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// 1/sqrt(x) for normal, finite x > 0: the hardware estimate y (PTX
// rsqrt.approx.ftz.f64, relative error below 1e-6 over 2^22 samples spanning the
// normal range on GB300) refined by one third-order step of the binomial series
// (1 - e)^(-1/2) = 1 + e/2 + 3e^2/8 + 5e^3/16 + ...  with e = 1 - x y^2 (formed by an
// FMA): y (1 + e/2 + 3e^2/8) leaves a relative error of about 5e^3/16 < 1e-18, so
// the result is within two units in the last place of the correctly rounded value
// (checked by the GPU tests).  Five FP64 operations.
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// 1/sqrt(x): rsqrt_nr for normal, finite x > 0; zero, subnormal, negative, infinite and NaN
// arguments take rsqrt itself (bit tests on the integer pipe).
__device__ __forceinline__ double rsqrt_pos(double x) {
  const long long b = __double_as_longlong(x);
  return (b >= 0x0010000000000000ll && b < 0x7ff0000000000000ll) ? rsqrt_nr(x) : rsqrt(x);
}

// sqrt(x) for finite x > 0 from the same estimate: with s = x y and e = 1 - s y,
// sqrt(x) = s (1 - e)^(-1/2) = s (1 + e/2 + 3e^2/8 + ...), the same third-order step
// (five FP64 operations; within two units in the last place of the correctly rounded
// square root, checked by the GPU tests).  Zero, subnormal, negative, infinite and NaN
// arguments take sqrt itself.  The bit tests run on the integer pipe.
__device__ __forceinline__ double sqrt_pos(double x) {
  const long long b = __double_as_longlong(x);
  if (b >= 0x0010000000000000ll && b < 0x7ff0000000000000ll) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double s = x * y;
    const double e = fma(-s, y, 1.0);
    return fma(s * e, fma(0.375, e, 0.5), s);
  }
  return sqrt(x);
}

// |a| by clearing the sign bit on the integer pipe (fabs as an operand of an FMA is an FP64
// operation of its own).
__device__ __forceinline__ double abs_int(double a) {
  int h;
  asm("and.b32 %0, %1, 0x7fffffff;" : "=r"(h) : "r"(__double2hiint(a)));
  return __hiloint2double(h, __double2loint(a));
}

// Whether a is positive and within about 2^-500 and 2^500 (integer pipe).
__device__ __forceinline__ bool mid_range(double a) {
  return (unsigned)(__double2hiint(a) - (523 << 20)) <= (unsigned)(1000 << 20);
}

// max(a, b) for a, b >= +0 (characteristic speeds): non-negative doubles order
// like their bit patterns read as signed 64-bit integers, so the comparison
// runs on the integer pipe instead of the FP64 pipe.
__device__ __forceinline__ double max_nn(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  return __longlong_as_double(ia > ib ? ia : ib);
}

// ---------------------------------------------------------------- advection
// dq/dt + div(a q) = 0 with material velocity a (M = 3).  F_d = a_d q, lambda_d = |a_d|.
struct PdeAdvFlux {
  static constexpr int N = 1, M = 3, NW = 1, DIM = 3;
  static constexpr bool FLUX = true, NCP = false, SRC = false, HYDRO = false;
  __device__ static constexpr bool moves(int) { return true; }
  __device__ static double vel(int d, const double* q, const double*) { return sel3(d, q[1], q[2], q[3]); }
  template <bool>
  __device__ static void edge(int d, const double* q, const DevParams&, double& u, double& p, double& lam) {
    u = sel3(d, q[1], q[2], q[3]);
    p = 0.0;
    lam = fabs(u);
  }
  __device__ static void prims(const double*, const DevParams&, double*) {}
  __device__ static void flux(int d, const double* q, const double*, const DevParams& P, double* F) {
    F[0] = MUL(P, sel3(d, q[1], q[2], q[3]), q[0]);
  }
  __device__ static double speed(int d, const double* q, const double*, const DevParams&) {
    return fabs(sel3(d, q[1], q[2], q[3]));
  }
  __device__ static void ncp(int, const double*, const double*, const DevParams&, double*) {}
  __device__ static void source(const double*, const double*, const DevParams&, double*) {}
};

// dq/dt + a . grad q = 0 (non-conservative form, F = 0): B_d = a_d.
struct PdeAdvNcp {
  static constexpr int N = 1, M = 3, NW = 1, DIM = 3;
  static constexpr bool FLUX = false, NCP = true, SRC = false, HYDRO = false;
  __device__ static constexpr bool moves(int) { return false; }
  __device__ static double vel(int d, const double* q, const double*) { return sel3(d, q[1], q[2], q[3]); }
  __device__ static constexpr bool needs_grad(int, int v) { return v == 0; }
  __device__ static void prims(const double*, const DevParams&, double*) {}
  __device__ static void flux(int, const double*, const double*, const DevParams&, double*) {}
  __device__ static double speed(int d, const double* q, const double*, const DevParams&) {
    return fabs(sel3(d, q[1], q[2], q[3]));
  }
  // qb holds N + M midpoint values (evolved then material).
  __device__ static void ncp(int d, const double* qb, const double* dq, const DevParams& P, double* D) {
    D[0] = MUL(P, sel3(d, qb[1], qb[2], qb[3]), dq[0]);
  }
  __device__ static void source(const double*, const double*, const DevParams&, double*) {}
};

// ---------------------------------------------------------------- Euler
// Ideal-gas Euler equations in DIM dimensions: Q = (rho, rho u_k, E).
// W = (u_0 .. u_{DIM-1}, p, c): one reciprocal and one square root per voxel.
template <int D_>
struct PdeEuler {
  static constexpr int DIM = D_, N = D_ + 2, M = 0, NW = D_ + 2;
  static constexpr bool FLUX = true, NCP = false, SRC = false, HYDRO = true;
  // F_d = Q u_d + p e_d + (p u_d) e_E: every quantity moves with u_d; the pressure terms are the
  // cell values press and cross.
  __device__ static constexpr bool moves(int) { return true; }
  __device__ static double vel(int d, const double*, const double* w) {
    return (DIM == 3) ? sel3(d, w[0], w[1], w[DIM == 3 ? 2 : 0]) : (d == 0 ? w[0] : w[1]);
  }
  __device__ static double press(const double* w) { return w[DIM]; }
  __device__ static double cross(const double*, double u, const double* w, const DevParams& P) { return MUL(P, w[DIM], u); }
  __device__ static void prims(const double* q, const DevParams& P, double* w) {
    const double r = recip_nr(q[0]);
    w[0] = MUL(P, q[1], r);
    double kin = MUL(P, q[1], w[0]);
#pragma unroll
    for (int k = 1; k < DIM; ++k) {
      w[k] = MUL(P, q[1 + k], r);
      kin = fma(q[1 + k], w[k], kin);
    }
    const double p = MUL(P, P.gm1, fma(-0.5, kin, q[DIM + 1]));
    w[DIM] = p;
    w[DIM + 1] = sqrt_pos(MUL(P, MUL(P, P.gamma, p), r));
  }
  __device__ static void flux(int d, const double* q, const double* w, const DevParams& P, double* F) {
    const double u = vel(d, q, w), p = w[DIM];
#pragma unroll
    for (int v = 0; v < N; ++v) F[v] = v == 1 + d ? fma(q[v], u, p) : MUL(P, q[v], u);
    F[N - 1] = MUL(P, ADD(P, q[N - 1], p), u);
  }
  // Velocity, pressure and speed along d of a state whose other velocities are not needed (18 FP64
  // operations).  The squares of the momenta stay in range while density and energy lie within
  // 2^-500 and 2^500 (m^2 <= 2 rho E); WIDE forms the velocities first, as prims does.
  template <bool WIDE>
  __device__ static void edge(int d, const double* q, const DevParams& P, double& u, double& p, double& lam) {
    const double r = recip_nr(q[0]);
    double kin = WIDE ? MUL(P, q[1], MUL(P, q[1], r)) : MUL(P, q[1], q[1]);
#pragma unroll
    for (int k = 1; k < DIM; ++k) kin = fma(q[1 + k], WIDE ? MUL(P, q[1 + k], r) : q[1 + k], kin);
    if (!WIDE) kin = MUL(P, kin, r);
    u = MUL(P, (DIM == 3) ? sel3(d, q[1], q[2], q[DIM == 3 ? 3 : 1]) : (d == 0 ? q[1] : q[2]), r);
    p = MUL(P, P.gm1, fma(-P.half, kin, q[DIM + 1]));
    lam = ADD(P, abs_int(u), sqrt_pos(MUL(P, MUL(P, P.gamma, p), r)));
  }
  __device__ static double speed(int d, const double*, const double* w, const DevParams& P) {
    return ADD(P, abs_int(vel(d, nullptr, w)), w[DIM + 1]);
  }
  __device__ static void ncp(int, const double*, const double*, const DevParams&, double*) {}
  __device__ static void source(const double*, const double*, const DevParams&, double*) {}
};

using PdeEuler2 = PdeEuler<2>;
using PdeEuler3 = PdeEuler<3>;

// ---------------------------------------------------------------- SRHD
// Special-relativistic hydrodynamics, Q = (D, S_x, S_y, S_z, tau), ideal gas Gamma.
// The material slots carry the primitives (rho, v_x, v_y, v_z, p) recovered by
// con2prim.  W = (v_x, v_y, v_z, p, 1 - cs^2, cs^2 (1 - v^2), 1 - v^2 cs^2,
// 1/(1 - v^2 cs^2)): the direction-independent factors of the speeds.
//   F_d = (D v_d, S v_d + p e_d, S_d - D v_d)
//   lambda_pm = [v_d (1 - cs^2) +- cs sqrt((1 - v^2)(1 - v^2 cs^2 - v_d^2 (1 - cs^2)))] / (1 - v^2 cs^2)
//   max(|lambda_+|, |lambda_-|) = (|v_d| (1 - cs^2) + sqrt(cs^2 (1 - v^2)(...))) / (1 - v^2 cs^2)
// (cs is folded under the square root: one square root per direction, none per voxel).
struct PdeSRHD {
  static constexpr int N = 5, M = 5, NW = 8, DIM = 3;
  static constexpr bool FLUX = true, NCP = false, SRC = false, HYDRO = true;
  // D and S move with v_d; the flux S_d - D v_d of tau is a cell value (cross), and so is p.
  __device__ static constexpr bool moves(int v) { return v < 4; }
  __device__ static double vel(int d, const double*, const double* w) { return sel3(d, w[0], w[1], w[2]); }
  __device__ static double press(const double* w) { return w[3]; }
  __device__ static double cross(double D, double Sd, double v) { return fma(-D, v, Sd); }
  __device__ static void prims(const double* q, const DevParams& P, double* w) {
    const double rho = q[5], vx = q[6], vy = q[7], vz = q[8], p = q[9];
    const double v2 = fma(vx, vx, fma(vy, vy, MUL(P, vz, vz)));
    const double rhoh = fma(P.Gq, p, rho);
    const double cs2 = MUL(P, MUL(P, P.Gamma, p), recip_nr(rhoh));
    const double c0 = fma(-v2, cs2, P.one);
    w[0] = vx; w[1] = vy; w[2] = vz; w[3] = p;
    w[4] = SUB(P, P.one, cs2);
    w[5] = MUL(P, cs2, SUB(P, P.one, v2));
    w[6] = c0;
    w[7] = recip_nr(c0);
  }
  __device__ static void flux(int d, const double* q, const double* w, const DevParams& P, double* F) {
    const double v = sel3(d, w[0], w[1], w[2]), p = w[3], Sd = sel3(d, q[1], q[2], q[3]);
    F[0] = MUL(P, q[0], v);
#pragma unroll
    for (int k = 0; k < 3; ++k) F[1 + k] = k == d ? fma(q[1 + k], v, p) : MUL(P, q[1 + k], v);
    F[4] = cross(q[0], Sd, v);
  }
  __device__ static double speed(int d, const double*, const double* w, const DevParams& P) {
    const double v = sel3(d, w[0], w[1], w[2]), omc = w[4];
    const double disc = MUL(P, w[5], fma(-MUL(P, v, v), omc, w[6]));
    return MUL(P, fma(abs_int(v), omc, sqrt_pos(disc)), w[7]);
  }
  // The largest speed over the three directions.  For |v_d| < 1 (and cs^2 < 1) the speed
  // increases with |v_d|:
  // with a = 1 - cs^2, b = cs^2 (1 - v^2), c = 1 - v^2 cs^2 = a + b, d lambda / d|v_d| has the sign
  // of sqrt(c - v_d^2 a) - |v_d| sqrt(b), i.e. of c (1 - v_d^2) > 0.  So the maximum is the speed
  // of the direction of the largest |v_d|: one square root instead of three, and the value is
  // that direction's speed bit for bit (the max over separately rounded speeds can differ from
  // it only between directions whose |v_d| agree to a few units in the last place).
  __device__ static double max_speed(const double* w, const DevParams& P) {
    const double u = max_nn(max_nn(fabs(w[0]), fabs(w[1])), fabs(w[2]));
    const double omc = w[4];
    const double disc = MUL(P, w[5], fma(-MUL(P, u, u), omc, w[6]));
    return MUL(P, fma(u, omc, sqrt_pos(disc)), w[7]);
  }
  __device__ static void ncp(int, const double*, const double*, const DevParams&, double*) {}
  __device__ static void source(const double*, const double*, const DevParams&, double*) {}
};

// ---------------------------------------------------------------- wave system
// First-order reduction of the damped scalar wave equation with speed c(x):
//   d_t phi = Pi,  d_t Pi = c^2 div psi - gamma Pi,  d_t psi_i = d_i Pi
// as Eq. 1: F = 0; B_d has (row Pi, col psi_d) = -c^2 and (row psi_d, col Pi) = -1;
// S = (Pi, -gamma Pi, 0, 0, 0).  Material: c (M = 1).  lambda_d = c.
struct PdeWave {
  static constexpr int N = 5, M = 1, NW = 1, DIM = 3;
  static constexpr bool FLUX = false, NCP = true, SRC = true;
  __device__ static constexpr bool needs_grad(int d, int v) { return v == 1 || v == 2 + d; }
  __device__ static void prims(const double*, const DevParams&, double*) {}
  __device__ static void flux(int, const double*, const double*, const DevParams&, double*) {}
  __device__ static double speed(int, const double* q, const double*, const DevParams&) { return q[5]; }
  __device__ static void ncp(int d, const double* qb, const double* dq, const DevParams& P, double* D) {
    const double c2 = MUL(P, qb[5], qb[5]);
    D[0] = 0.0;
    D[1] = MUL(P, -c2, sel3(d, dq[2], dq[3], dq[4]));
    D[2] = d == 0 ? -dq[1] : 0.0;
    D[3] = d == 1 ? -dq[1] : 0.0;
    D[4] = d == 2 ? -dq[1] : 0.0;
  }
  __device__ static void source(const double* q, const double*, const DevParams& P, double* S) {
    S[0] = q[1];
    S[1] = MUL(P, -P.damp, q[1]);
    S[2] = 0.0; S[3] = 0.0; S[4] = 0.0;
  }
};

// ---------------------------------------------------------------- GW59 stand-in
// 11 first-order scalar waves (phi_a, Pi_a, psi_a,xyz) coupled to a lapse alpha
// and shift beta (59 unknowns):
//   d_t phi_a   = alpha Pi_a + beta^k psi_a,k
//   d_t Pi_a    = alpha d_k psi_a,k + beta^k d_k Pi_a + alpha sum_b C_ab phi_b Pi_b
//   d_t psi_a,i = alpha d_i Pi_a + Pi_a d_i alpha + beta^k d_k psi_a,i
//   d_t alpha   = -kappa alpha^2 sum_a Pi_a^2
//   d_t beta^i  = 3/4 sum_a psi_a,i Pi_a
// F = 0; every gradient term is part of B(Q).grad Q.  Layout: field a at 5a..5a+4,
// alpha at 55, beta at 56..58.  lambda_d = alpha + |beta^d|.
struct PdeGW59 {
  static constexpr int N = 59, M = 0, NW = 1, DIM = 3;
  static constexpr bool FLUX = false, NCP = true, SRC = true;
  __device__ static void prims(const double*, const DevParams&, double*) {}
  __device__ static double speed(int d, const double* q, const double*, const DevParams&) {
    return q[55] + fabs(sel3(d, q[56], q[57], q[58]));
  }
};

// The cell value that a system adds to the face differences of its last quantity (the flux of the
// energy beyond its transport): p u_d for Euler, S_d - D v_d for SRHD (q: N quantities, u = vel).
template <class PDE>
__device__ __forceinline__ double cross_term(int d, const double* q, double u, const double* w, const DevParams& P) {
  if constexpr (std::is_same<PDE, PdeSRHD>::value) return PdeSRHD::cross(q[0], sel3(d, q[1], q[2], q[3]), u);
  else if constexpr (PDE::HYDRO) return PDE::cross(q, u, w, P);
  else return 0.0;
}

// The part of twice the Rusanov flux that needs both sides of a face,
//   F_L + F_R - s (Q_R - Q_L) = Q_L (u_L + s) + Q_R (u_R - s) + cell terms,  s = max(lambda_L, lambda_R):
// two operations per quantity that moves with the velocity u (and s (Q_L - Q_R) for the others).
// The cell terms (pressure, cross_term) enter the sums over a voxel's faces directly (fx_sum),
// where those of the voxel itself cancel.
// It rounds at Q s: a face between equal quantities leaves a residue of at most u Q s (u = 2^-53) where
// s (Q_R - Q_L) is exactly 0.  With a time step within the CFL limit (dt s/dx <= 1/6 along each axis) the six of
// a voxel move the result by less than u Q/2, below the rounding of its update: a contact at rest keeps
// its energy and momentum to the bit.  R.m.s. error of a stage on smooth fields (replayed on the CPU), the two
// fluxes and the difference formed apart -> this: density 5.0e-17 -> 5.2e-17, energy 4.9e-17 -> 5.1e-17, momenta 1.0e-16 ->
// 6.1e-17 (they round at their own size, not at the pressure's).
template <class PDE>
__device__ __forceinline__ void rusanov(const DevParams& P, const double* qL, double uL, double lL, const double* qR,
                                        double uR, double lR, double* H) {
  const double s = max_nn(lL, lR);
  const double a = ADD(P, uL, s), b = SUB(P, uR, s);
#pragma unroll
  for (int v = 0; v < PDE::N; ++v)
    H[v] = PDE::moves(v) ? fma(qR[v], b, MUL(P, qL[v], a)) : MUL(P, s, SUB(P, qL[v], qR[v]));
}

// The largest characteristic speed of a voxel over its dim directions (SRHD: the speed of the
// direction of the largest |v_d|, which is the largest).
template <class PDE>
__device__ __forceinline__ double max_speed_dirs(const double* u, const double* W, const DevParams& P, int dim) {
  if constexpr (std::is_same<PDE, PdeSRHD>::value) {
    return PdeSRHD::max_speed(W, P);
  } else {
    double l = fmax(PDE::speed(0, u, W, P), PDE::speed(1, u, W, P));
    if (dim == 3) l = fmax(l, PDE::speed(2, u, W, P));
    return l;
  }
}

}  // namespace dh
