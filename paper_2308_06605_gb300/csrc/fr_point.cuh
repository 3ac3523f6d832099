// Pointwise device functions shared by the hexahedral and prismatic kernels: gas dynamics (normal
// inviscid flux with the Rusanov wave-speed bound, viscous flux with optional eddy viscosity) and
// the output / RK44 stage update of one solution point.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "df32.cuh"
#include "fr_device.hpp"

namespace frx {

template <typename T> __device__ __forceinline__ const PhysT<T> &phys_of(const DevPhys &p);
template <> __device__ __forceinline__ const PhysT<double> &phys_of<double>(const DevPhys &p) { return p.d; }
template <> __device__ __forceinline__ const PhysT<df32> &phys_of<df32>(const DevPhys &p) { return p.f; }
template <> __device__ __forceinline__ const PhysT<float> &phys_of<float>(const DevPhys &p) { return p.s; }

// ------------------------------------------------------------------------------------------
// Gas dynamics (ideal gas, Stokes hypothesis, constant mu, Fourier heat flux).
// ------------------------------------------------------------------------------------------
// Normal inviscid flux F(q).n and (|u.n^| + c)|n|, in FP64 (pressure/energy recovery); nn = |n|.
__device__ __forceinline__ void normal_inviscid(const double q[5], const double n[3], double nn, double g,
                                                double out[5], double &un_abs_plus_c_n) {
  const double ri = 1.0 / q[0];
  const double u = q[1] * ri, v = q[2] * ri, w = q[3] * ri;
  const double p = (g - 1.0) * (q[4] - 0.5 * (q[1] * u + q[2] * v + q[3] * w));
  const double un = u * n[0] + v * n[1] + w * n[2];
  out[0] = q[0] * un;
  out[1] = q[1] * un + p * n[0];
  out[2] = q[2] * un + p * n[1];
  out[3] = q[3] * un + p * n[2];
  out[4] = (q[4] + p) * un;
  un_abs_plus_c_n = fabs(un) + sqrt(g * p * ri) * nn;      // (|u.n^| + c) |n|
}

// Double-float normal flux with the pressure recovery p = (gamma-1)(E - m.u/2) in FP64.
__device__ __forceinline__ void normal_inviscid(const df32 q[5], const df32 n[3], df32 nn, const DevPhys &dph,
                                                df32 out[5], df32 &un_abs_plus_c_n) {
  const PhysT<df32> &ph = dph.f;
  const df32 ri = reciprocal(q[0]);
  const df32 u[3] = {q[1] * ri, q[2] * ri, q[3] * ri};
  const double pd = (dph.gamma - 1.0) *
                    (to_double(q[4]) - 0.5 * to_double(dot3(q[1], u[0], q[2], u[1], q[3], u[2])));
  const df32 p = df_from(pd);
  const df32 un = dot3(u[0], n[0], u[1], n[1], u[2], n[2]);
  out[0] = q[0] * un;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    Dot<df32> f(q[1 + c], un);
    f.add(p, n[c]);
    out[1 + c] = f.raw();
  }
  out[4] = (q[4] + p) * un;
  un_abs_plus_c_n = fabs(un) + sqrt(ph.gamma * p * ri) * nn;
}

// FP64 overload with the same signature shape (the FP64 path's arithmetic).
__device__ __forceinline__ void normal_inviscid(const double q[5], const double n[3], double nn, const DevPhys &dph,
                                                double out[5], double &s) {
  normal_inviscid(q, n, nn, dph.gamma, out, s);
}

// Roe's approximate Riemann flux (Roe 1981) through the area-scaled normal n (|n| = nn), FP64:
// 1/2 (F(qL) + F(qR)).n - 1/2 |n| sum_k |lambda_k| alpha_k r_k over the waves of the Jacobian at the
// Roe average (density-weighted velocity and total enthalpy): acoustic waves u.n^ -/+ c with
// strengths (dp -/+ rho c du_n) / (2 c^2), entropy wave u.n^ with drho - dp / c^2, shear wave u.n^
// carrying rho (du - du_n n^).  Harten's entropy fix on the acoustic waves: |lambda| below
// d = 0.1 c becomes (lambda^2 + d^2) / (2 d).
__device__ __forceinline__ void roe_flux(const double qL[5], const double qR[5], const double n[3], double nn,
                                         double g, double F[5]) {
  // Five reciprocals and three square roots: on this FP64 pipe a division costs about ten additions.
  const double inn = 1.0 / nn, iL = 1.0 / qL[0], iR = 1.0 / qR[0];
  const double nh[3] = {n[0] * inn, n[1] * inn, n[2] * inn};
  const double rL = qL[0], rR = qR[0];
  const double uL[3] = {qL[1] * iL, qL[2] * iL, qL[3] * iL}, uR[3] = {qR[1] * iR, qR[2] * iR, qR[3] * iR};
  const double pL = (g - 1.0) * (qL[4] - 0.5 * (qL[1] * uL[0] + qL[2] * uL[1] + qL[3] * uL[2]));
  const double pR = (g - 1.0) * (qR[4] - 0.5 * (qR[1] * uR[0] + qR[2] * uR[1] + qR[3] * uR[2]));
  const double eL = qL[4] + pL, eR = qR[4] + pR;
  const double sl = sqrt(rL), sr = sqrt(rR), w = 1.0 / (sl + sr);
  const double r = sl * sr, wl = sl * w, wr = sr * w;
  double u[3], du[3], q2 = 0.0, un = 0.0, dun = 0.0, nL = 0.0, nR = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    u[c] = wl * uL[c] + wr * uR[c];
    du[c] = uR[c] - uL[c];
    q2 += u[c] * u[c];
    un += u[c] * nh[c];
    dun += du[c] * nh[c];
    nL += uL[c] * n[c];
    nR += uR[c] * n[c];
  }
  const double H = wl * (eL * iL) + wr * (eR * iR);
  const double c2 = (g - 1.0) * (H - 0.5 * q2), c = sqrt(c2), ic2 = 1.0 / c2;
  const double dp = pR - pL, dr = rR - rL, rcd = r * c * dun, h2 = 0.5 * ic2;
  const double a1 = (dp - rcd) * h2, a2 = dr - dp * ic2, a3 = (dp + rcd) * h2;
  // Harten's fix with d = 0.1 c: (lam^2 + d^2) / (2 d), 1 / (2 d) = 5 / c = 5 c / c^2.
  const double d = 0.1 * c, i2d = 5.0 * c * ic2;
  auto fix = [d, i2d](double lam) {
    const double a = fabs(lam);
    return a < d ? (lam * lam + d * d) * i2d : a;
  };
  const double l1 = fix(un - c) * a1, l2 = fabs(un), l3 = fix(un + c) * a3;
  const double la = l1 + l3, lc = (l3 - l1) * c, m2 = l2 * a2, mr = l2 * r;
  double D[5], ush = 0.0;
  D[0] = la + m2;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double sh = du[k] - dun * nh[k];     // shear, times r
    ush += u[k] * sh;
    D[1 + k] = D[0] * u[k] + lc * nh[k] + mr * sh;
  }
  D[4] = la * H + lc * un + m2 * 0.5 * q2 + mr * ush;
  const double ps = pL + pR;
  F[0] = 0.5 * (rL * nL + rR * nR - nn * D[0]);
#pragma unroll
  for (int k = 0; k < 3; ++k) F[1 + k] = 0.5 * (qL[1 + k] * nL + qR[1 + k] * nR + ps * n[k] - nn * D[1 + k]);
  F[4] = 0.5 * (eL * nL + eR * nR - nn * D[4]);
}

// Transport coefficients of one viscous-flux evaluation (molecular, or with an eddy viscosity).
template <typename T>
struct Visc {
  T mu, m2mu3, kappa;   // mu, -2 mu / 3, kappa
};

template <typename T>
__device__ __forceinline__ Visc<T> visc_of(const PhysT<T> &ph) {
  return Visc<T>{ph.mu, ph.m2mu3, ph.kappa};
}

// Closure: mu + rho nu_t, kappa + rho nu_t cp / Pr_t (nu_t = 0 gives the molecular values exactly).
template <typename T>
__device__ __forceinline__ Visc<T> visc_with(const PhysT<T> &ph, T rho_nu, const DevPhys &dph) {
  if (!dph.closure) return visc_of(ph);
  const T mu = ph.mu + rho_nu;
  return Visc<T>{mu, ph.m2mu3 + from_double<T>(-2.0 / 3.0) * rho_nu, ph.kappa + from_double<T>(dph.cp_prt) * rho_nu};
}

// Viscous flux through the normal n: tn = tau . n and en = u . tn + kappa dT/dn, of the state q and
// gradient g(j * 5 + v) = dQ_v/dx_j.  Both enter through their ratio only (and u, E/rho), so a pair of
// sides passes the sums of its states and gradients, and no factor 1/2 is spent on the mean.  The
// columns of the gradient are read one at a time (five values live) and the 3 x 3 stress is never
// formed: 80 FP64 operations with the sums, where the full flux and its projection take 190.
template <typename T, typename GetG>
__device__ __forceinline__ void viscous_normal(const T q[5], GetG g, const T n[3], const PhysT<T> &ph,
                                               const Visc<T> &vc, T tn[3], T &en) {
  const T ri = reciprocal(q[0]);
  const T u[3] = {q[1] * ri, q[2] * ri, q[3] * ri};
  const T eo = q[4] * ri;
  T z[3], div;        // z[j] = sum_i n_i rho du_i/dx_j
  Dot<T> w[3], h;     // w[i] = sum_j n_j rho du_i/dx_j, h = sum_j n_j (dE/dx_j - E/rho drho/dx_j)
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const T g0 = g(j * 5);
    T a[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) a[i] = muladd(g(j * 5 + 1 + i), -u[i], g0);
    z[j] = dot3(n[0], a[0], n[1], a[1], n[2], a[2]);
    const T e = muladd(g(j * 5 + 4), -eo, g0);
    if (j == 0) {
      div = a[0];
      h = Dot<T>(n[0], e);
    } else {
      div = div + a[j];
      h.add(n[j], e);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (j == 0)
        w[i] = Dot<T>(n[0], a[i]);
      else
        w[i].add(n[j], a[i]);
    }
  }
  const T t = vc.mu * ri, ld = vc.m2mu3 * ri * div;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const T wi = w[i].raw();
    h.add(-u[i], wi);
    tn[i] = muladd(t * (wi + z[i]), ld, n[i]);
  }
  en = muladd(dot3(u[0], tn[0], u[1], tn[1], u[2], tn[2]), vc.kappa * (ph.cT * ri), h.raw());
}

// Viscous stress tau = mu (du_i/dx_j + du_j/dx_i) + delta_ij lambda div u, packed (xx, yy, zz, xy,
// xz, yz), and heat-flux term hq[j] = kappa dT/dx_j of state q with gradient G[j*5 + v] = dQ_v/dx_j.  Works on
// rho du_i/dx_j = G[j][1+i] - u_i G[j][0] and puts the factor 1/rho into the coefficients: 40 FP64 operations, 450 FP32 instructions in double-float (57 and 700 with
// du_i/dx_j itself).
template <typename T>
__device__ __forceinline__ void viscous_stress(const T q[5], const T u[3], T ri, const T *G, const PhysT<T> &ph,
                                               const Visc<T> &vc, T tau[6], T hq[3]) {
  const T eo = q[4] * ri, kc = vc.kappa * (ph.cT * ri), t = vc.mu * ri, t2 = scale2(t, 2.f);
  T a[3][3];   // a[i][j] = rho du_i/dx_j
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) a[i][j] = muladd(G[j * 5 + 1 + i], -u[i], G[j * 5]);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    Dot<T> d(G[j * 5 + 4]);
    d.add(-eo, G[j * 5]);
#pragma unroll
    for (int i = 0; i < 3; ++i) d.add(-u[i], a[i][j]);
    hq[j] = kc * d.raw();
  }
  const T lam = vc.m2mu3 * ri * (a[0][0] + a[1][1] + a[2][2]);
#pragma unroll
  for (int i = 0; i < 3; ++i) tau[i] = muladd(lam, t2, a[i][i]);
  tau[3] = t * (a[0][1] + a[1][0]);
  tau[4] = t * (a[0][2] + a[2][0]);
  tau[5] = t * (a[1][2] + a[2][1]);
}

// Physical flux F - Fv of Eq. 1 in the three directions: the momentum part is the symmetric tensor
// m = rho u u + p I - tau (packed xx, yy, zz, xy, xz, yz), the energy part
// en_j = (E + p) u_j - sum_i u_i tau_ij - hq_j, the mass part rho u itself.  With its transforms
// (transformed_flux: 15 three-term products) 105 FP64 operations or 1300 FP32 instructions in
// double-float, where the contravariant form (U_d = S_d . u, then S_d tau and S_d hq for each direction d)
// takes 150 and 1900 with the stress.  Volume kernel, GB300, double-float 48^3 p = 4: 3.80 -> 3.43 ms;
// FP64 32^3 p = 4: 4.16 -> 3.79 ms.
//
// FP64 holds the pressure in the tensor's diagonal.  The double-float forms leave it out, and their transforms add
// S p by itself: with the pressure in the tensor it is rounded there and again in the transform, and at low Mach
// number it is much the largest part (momentum residual's error at Ma 0.1 3 to 8 % larger on hexahedra of p = 2 to 7;
// volume launch 48^3 p = 4 3.134 ms for 3.184).
template <typename T> constexpr bool kPressureInTensor = std::is_same<T, double>::value;

template <typename T>
__device__ __forceinline__ void physical_flux(const T q[5], const T u[3], T p, bool viscous, const T tau[6],
                                              const T hq[3], T m[6], T en[3]) {
  const T H = q[4] + p;
  if (!viscous) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if constexpr (kPressureInTensor<T>)
        m[i] = muladd(p, q[1 + i], u[i]);
      else
        m[i] = q[1 + i] * u[i];
      en[i] = H * u[i];
    }
    m[3] = q[1] * u[1];
    m[4] = q[1] * u[2];
    m[5] = q[2] * u[2];
    return;
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if constexpr (kPressureInTensor<T>) {
      Dot<T> d(p);
      d.add(q[1 + i], u[i]);
      d.plus(-tau[i]);
      m[i] = d.raw();
    } else {
      m[i] = muladd(-tau[i], q[1 + i], u[i]);
    }
  }
  m[3] = muladd(-tau[3], q[1], u[1]);
  m[4] = muladd(-tau[4], q[1], u[2]);
  m[5] = muladd(-tau[5], q[2], u[2]);
  // Row j of tau, packed.
  const int row[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    Dot<T> d(-hq[j]);
    d.add(H, u[j]);
#pragma unroll
    for (int i = 0; i < 3; ++i) d.add(-tau[row[j][i]], u[i]);
    en[j] = d.raw();
  }
}

// Inviscid transformed flux of reference direction d in FP64, from the contravariant velocity: 12 operations per
// direction where the tensor above and its transform take 18 (the viscous part is what the tensor saves on).  Every
// FP64 element kernel without a viscous branch uses it, each with the same operations.
__device__ __forceinline__ void inviscid_transformed(const double q[5], const double u[3], double p, const double Sd[3],
                                                     double f[5]) {
  const double Ud = fma(Sd[2], u[2], fma(Sd[1], u[1], Sd[0] * u[0]));
  f[0] = q[0] * Ud;
#pragma unroll
  for (int i = 0; i < 3; ++i) f[1 + i] = fma(q[1 + i], Ud, Sd[i] * p);
  f[4] = __dadd_rn(q[4], p) * Ud;
}

// Transformed flux of reference direction d, F^_d = sum_j S[d][j] (F - Fv)_j (Eq. 1); Sd = S[d][0..2].
template <typename T>
__device__ __forceinline__ void transformed_flux(const T q[5], const T m[6], const T en[3], T p, const T Sd[3], T f[5]) {
  f[0] = dot3(Sd[0], q[1], Sd[1], q[2], Sd[2], q[3]);
  f[1] = dot3(Sd[0], m[0], Sd[1], m[3], Sd[2], m[4]);
  f[2] = dot3(Sd[0], m[3], Sd[1], m[1], Sd[2], m[5]);
  f[3] = dot3(Sd[0], m[4], Sd[1], m[5], Sd[2], m[2]);
  f[4] = dot3(Sd[0], en[0], Sd[1], en[1], Sd[2], en[2]);
  if constexpr (!kPressureInTensor<T>)
#pragma unroll
    for (int i = 0; i < 3; ++i) f[1 + i] = muladd(f[1 + i], Sd[i], p);
}

// ------------------------------------------------------------------------------------------
// Coefficients of one stage, formed once per launch on the host (a product with dt or a conversion in
// each thread would cost FP64 slots, of which the correction kernels are short).
// ------------------------------------------------------------------------------------------
struct StageCoef {
  int mode, stage, last;   // last: the step's final stage
  double b, a;             // RK44: b_k dt, a_{k+1} dt; SSP(3,3): b_k, a_k; SSP(10,4): b = dt/6 or dt/10
  double dt;
  float a_hi, a_lo;        // a as double-float (RK44)
};

__host__ __device__ __forceinline__ StageCoef stage_coef(int mode, int stage, double dt) {
  StageCoef c{mode, stage, 0, 0.0, 0.0, dt, 0.f, 0.f};
  if (mode == MODE_RK) {
    // b_k = (1/6, 1/3, 1/3, 1/6), next-stage a = (1/2, 1/2, 1).
    c.last = stage == 3;
    c.b = ((stage == 0 || stage == 3) ? 1.0 / 6.0 : 1.0 / 3.0) * dt;
    c.a = c.last ? 0.0 : (stage < 2 ? 0.5 : 1.0) * dt;
    c.a_hi = (float)c.a;
    c.a_lo = (float)(c.a - (double)c.a_hi);
  } else if (mode == MODE_SSP33) {
    c.last = stage == 2;
    c.a = stage == 0 ? 0.0 : (stage == 1 ? 0.75 : 1.0 / 3.0);
    c.b = stage == 0 ? 1.0 : (stage == 1 ? 0.25 : 2.0 / 3.0);
  } else if (mode == MODE_SSP104) {
    c.last = stage == 9;
    c.b = c.last ? 0.1 * dt : dt / 6.0;
  }
  return c;
}

// ------------------------------------------------------------------------------------------
// Output or Runge-Kutta stage update of one value o (flat index over points and variables).  rs is the
// residual without source terms in the element arithmetic, src its source term (FP64; SRC: a template
// parameter, because as a select its addition and conversion would be paid for by every value).
// MODE_RESIDUAL writes R; the other modes update the FP64 registers (acc, U_n) and the stage state
// (FP64 Q, and on the mixed path its double-float copy Qc).  x1 and x2 are the old register values the
// stage reads (stage_inputs).  Returns true for a non-finite value at the last stage.
// ------------------------------------------------------------------------------------------
// The two arrays a stage reads besides the residual, as 8-byte words (null: not read).  RK44: acc after the
// first stage, and U_n (its double-float copy for a mixed stage state); SSP(3,3): Q, U_n; SSP(10,4): Q, and
// U_n or acc where the registers recombine.
struct StageIn {
  const double *x1, *x2;
};
template <typename T>
__device__ __forceinline__ StageIn stage_inputs(const StageCoef &c, const double *Q, const double *Un, const T *Unc,
                                                const double *acc) {
  if (c.mode == MODE_RESIDUAL) return StageIn{nullptr, nullptr};
  if (c.mode == MODE_RK) {
    const double *u = Un;
    if constexpr (std::is_same<T, df32>::value)
      if (!c.last) u = reinterpret_cast<const double *>(Unc);
    return StageIn{c.stage > 0 ? acc : nullptr, u};
  }
  if (c.mode == MODE_SSP33) return StageIn{Q, Un};
  return StageIn{Q, c.last ? acc : (c.stage == 4 ? Un : nullptr)};
}
__device__ __forceinline__ df32 as_df32(double x) { return *reinterpret_cast<df32 *>(&x); }

template <typename T, bool SRC>
__device__ __forceinline__ bool finish_value(int64_t o, T rs, double src, const StageCoef &c, double x1, double x2,
                                             double *__restrict__ Rout, double *__restrict__ Q, T *__restrict__ Qc,
                                             double *__restrict__ Un, T *__restrict__ Unc, double *__restrict__ acc) {
  // Products and sums that the compiler could contract in more than one way are written as the operations they
  // are: the staged kernel and the one with a thread per point have to give the same bits.
  double rd = to_double(rs);
  if constexpr (SRC) rd = __dadd_rn(rd, src);
  if (c.mode == MODE_RESIDUAL) {
    Rout[o] = rd;
    return false;
  }
  if (c.mode == MODE_RK) {
    if constexpr (std::is_same<T, df32>::value) {
      // Mixed path: acc and U_n are FP64; the next stage state, read only by the element kernels, is
      // formed in double-float from the df32 copy of U_n (with a source term from the FP64 residual,
      // which includes it).
      if (!c.last) {
        acc[o] = fma(c.b, rd, x1);
        if constexpr (SRC)
          Qc[o] = as_df32(x2) + df(c.a_hi, c.a_lo) * from_double<T>(rd);
        else
          Qc[o] = as_df32(x2) + df(c.a_hi, c.a_lo) * rs;
        return false;
      }
      const double nv = fma(c.b, rd, x2 + x1);
      Un[o] = nv;
      Q[o] = nv;
      const T nc = from_double<T>(nv);
      Unc[o] = nc;
      Qc[o] = nc;
      return !isfinite(nv);
    } else {
      if (!c.last) {
        acc[o] = fma(c.b, rd, x1);
        Q[o] = fma(c.a, rd, x2);
        return false;
      }
      const double nv = fma(c.b, rd, x2 + x1);
      Un[o] = nv;
      Q[o] = nv;
      return !isfinite(nv);
    }
  }
  // FP64 registers on both paths: U_n (start of the step), Q (stage state) and, for the ten-stage
  // scheme, acc (its second register); the mixed path also refreshes the double-float copy Qc.
  //   SSP(3,3):  Q <- a_k U_n + b_k (Q + dt R), (a, b) = (0, 1), (3/4, 1/4), (1/3, 2/3).
  //   SSP(10,4): Q <- Q + dt/6 R at stages 0..8; after stage 4 the registers recombine,
  //              q2 = U_n/25 + 9/25 Q, Q <- 15 q2 - 5 Q; stage 9: Q <- q2 + 3/5 Q + dt/10 R.
  const double q = x1;
  double nq;
  if (c.mode == MODE_SSP33) {
    nq = fma(c.b, fma(c.dt, rd, q), __dmul_rn(c.a, x2));
  } else if (!c.last) {
    nq = fma(c.b, rd, q);
    if (c.stage == 4) {
      const double q2 = fma(9.0 / 25.0, nq, x2 / 25.0);
      acc[o] = q2;
      nq = fma(15.0, q2, -5.0 * nq);
    }
  } else {
    nq = fma(c.b, rd, fma(0.6, q, x2));
  }
  Q[o] = nq;
  if constexpr (std::is_same<T, df32>::value) Qc[o] = from_double<T>(nq);
  if (!c.last) return false;
  Un[o] = nq;
  if constexpr (std::is_same<T, df32>::value) Unc[o] = from_double<T>(nq);
  return !isfinite(nq);
}

// Source term of solution point t at the state the residual was evaluated on (the element kernels'
// input): body acceleration and sponge.
template <typename T>
__device__ __forceinline__ void point_source(int64_t t, const double *__restrict__ Q, const T *__restrict__ Qc,
                                             const DevPhys &dph, double src[5]) {
  double q[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    q[v] = Qc ? to_double(Qc[t * 5 + v]) : Q[t * 5 + v];
    src[v] = 0.0;
  }
  if (dph.src_body) {
    src[1] = q[0] * dph.accel[0];
    src[2] = q[0] * dph.accel[1];
    src[3] = q[0] * dph.accel[2];
    src[4] = fma(q[3], dph.accel[2], fma(q[2], dph.accel[1], q[1] * dph.accel[0]));
  }
  if (dph.src_sponge) {
    const double sg = dph.sigma[t];
#pragma unroll
    for (int v = 0; v < 5; ++v) src[v] = fma(-sg, q[v] - dph.Q_ref[t * 5 + v], src[v]);
  }
}

// finish_value for the five values of solution point t; rv is the bracket of Eq. 3, s = -1/|J|.
template <typename T>
__device__ __forceinline__ void finish_point(int64_t t, const T rv[5], T s, const StageCoef &c,
                                             double *__restrict__ Rout, double *__restrict__ Q, T *__restrict__ Qc,
                                             double *__restrict__ Un, T *__restrict__ Unc, double *__restrict__ acc,
                                             int *__restrict__ flag, const DevPhys &dph) {
  bool bad = false;
  const StageIn in = stage_inputs<T>(c, Q, Un, Unc, acc);
  double x1[5], x2[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    x1[v] = in.x1 ? in.x1[t * 5 + v] : 0.0;
    x2[v] = in.x2 ? in.x2[t * 5 + v] : 0.0;
  }
  if (dph.src_body || dph.src_sponge) {
    double src[5];
    point_source<T>(t, Q, Qc, dph, src);
#pragma unroll
    for (int v = 0; v < 5; ++v)
      bad |= finish_value<T, true>(t * 5 + v, rv[v] * s, src[v], c, x1[v], x2[v], Rout, Q, Qc, Un, Unc, acc);
  } else {
#pragma unroll
    for (int v = 0; v < 5; ++v)
      bad |= finish_value<T, false>(t * 5 + v, rv[v] * s, 0.0, c, x1[v], x2[v], Rout, Q, Qc, Un, Unc, acc);
  }
  if (bad) atomicOr(flag, 1);
}

// Correction kernels of kCorrectThreads threads, one point each, with every access to the [point][5]
// arrays (partial residual, registers, states) made by consecutive threads on consecutive values: the
// partial residual is staged through shared memory (sr, 5 values per thread), the thread of a
// point replaces its five entries by the residual, and the update runs over the block's values.  With
// a thread reading its own point's values each 8-byte access of a warp touches ten 128-byte lines.
// The copies into shared memory (cp.async: partial residual and the stage's two old register values) are in
// flight while the double-float kernel gathers the fluxes.  Double-float 48^3 p = 4 1.07 -> 0.80 ms per launch (0.93 with
// the partial residual alone staged by plain loads; 0.757 since to_double runs on the integer pipe), FP64 32^3 p = 4
// 0.447 -> 0.398 ms; bound by the FP64 pipe (an addition and an FMA per value, the last stage a split into
// double-float) beside 3.5 GB of traffic (0.51 ms at 48^3).  FP64 6 blocks per SM (40 registers), double-float 5 (48; 6 measured the same).
constexpr int kCorrectThreads = 256;

// Shared memory of a block: the partial residual (replaced by the residual), the stage's two old register
// values, and with source terms their five FP64 values per point.
struct CorrectSmem {
  double *r, *x1, *x2, *src;
  __device__ __forceinline__ explicit CorrectSmem(double *p)
      : r(p), x1(p + 5 * kCorrectThreads), x2(p + 10 * kCorrectThreads), src(p + 15 * kCorrectThreads) {}
};

__device__ __forceinline__ void copy_async8(double *dst, const double *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// Start the copies of everything the block reads by value; the lifted fluxes are gathered meanwhile.  base:
// first value of the block in the registers, part: of its partial residual, n: points.
template <typename T>
__device__ __forceinline__ void stage_begin(const CorrectSmem &sm, const T *part, int64_t base, int n,
                                            const StageIn &in) {
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int i = threadIdx.x + k * kCorrectThreads;
    if (i < n * 5) {
      copy_async8(sm.r + i, reinterpret_cast<const double *>(part) + i);
      if (in.x1) copy_async8(sm.x1 + i, in.x1 + base + i);
      if (in.x2) copy_async8(sm.x2 + i, in.x2 + base + i);
    }
  }
}
__device__ __forceinline__ void stage_arrive() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
}

// Double-float gathers and lifts the fluxes while the copies arrive and adds the partial residual last; in
// FP64 that addition is one more operation per value on the pipe that bounds the kernel (0.399 -> 0.447 ms
// at 32^3 p = 4), so there the sum starts from the staged residual.
template <typename T> constexpr bool kGatherFirst = std::is_same<T, df32>::value;

// first: flat index of the block's first point in the registers, n: points of the block; this thread's lifted
// fluxes rv (FP64: with the partial residual), a second part of them that is added after the residual (may be
// null) and s = -1/|J| (used if threadIdx.x < n).
template <typename T, bool SRC>
__device__ __forceinline__ void finish_block(int64_t first, int n, const CorrectSmem &sm, Dot<T> rv[5],
                                             const Dot<T> *last, T s, const StageCoef &c, const StageIn &in,
                                             double *__restrict__ Rout, double *__restrict__ Q, T *__restrict__ Qc, double *__restrict__ Un,
                                             T *__restrict__ Unc, double *__restrict__ acc, int *__restrict__ flag,
                                             const DevPhys &dph) {
  const int me = threadIdx.x;
  T *sr = reinterpret_cast<T *>(sm.r);
  if constexpr (kGatherFirst<T>) stage_arrive();
  if (me < n) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      if constexpr (kGatherFirst<T>) rv[v].plus(sr[me * 5 + v]);
      if (last) rv[v].join(last[v]);
      sr[me * 5 + v] = rv[v].get() * s;
    }
    if constexpr (SRC) {
      double src[5];
      point_source<T>(first + me, Q, Qc, dph, src);
#pragma unroll
      for (int v = 0; v < 5; ++v) sm.src[me * 5 + v] = src[v];
    }
  }
  __syncthreads();
  bool bad = false;
#pragma unroll 5
  for (int i = me; i < n * 5; i += kCorrectThreads)
    bad |= finish_value<T, SRC>(first * 5 + i, sr[i], SRC ? sm.src[i] : 0.0, c, in.x1 ? sm.x1[i] : 0.0,
                                in.x2 ? sm.x2[i] : 0.0, Rout, Q, Qc, Un, Unc, acc);
  if (bad) atomicOr(flag, 1);
}

inline bool has_source(const DevPhys &ph) { return ph.src_body || ph.src_sponge; }
inline size_t correct_smem(const DevPhys &ph) {
  return sizeof(double) * 5 * kCorrectThreads * (has_source(ph) ? 4 : 3);
}

}  // namespace frx
