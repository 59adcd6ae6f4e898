// rhs.cuh -- device right-hand side dY/dt of one constant-(rho, e) cell.
//
// Per evaluation: temperature from (e, Y) by Newton on NASA-7 (Eq. 10; calculate_T of
// Table 1), species Gibbs functions, Arrhenius / third-body / Troe forward rates,
// reverse rates from equilibrium constants (Sec. 2.1.2), law of mass action (Eq. 16),
// and F_k = W_k wdot_k / rho (Eq. 14, 20 at constant density).
//
// Arithmetic layout (an FP64 instruction occupies a warp's sub-partition for 64 cycles on
// GB300, an integer one for 2, a wide multiply for 5; the FP64 pipe bounds the kernels):
//   - exponentials run in fixed point on the integer pipe (exp2_q52, fastmath.cuh), the Arrhenius
//     exponent with them: log2 A + b log2 T - (Ta / ln2) / T in 64-bit integers, no FP64
//     instruction and at most 0.6 ulp off, for T in (128, 32768) K and coefficients within the
//     forms' range; anything else takes the table-driven exp_t (production_rates_any).  The
//     36 exponentials of an evaluation were 430 of its ~1040 FP64 instructions: with them gone
//     the 1M-cell detonation slice takes 49.2 instead of 83.2 ms, a single warp's step 27 % less;
//   - g_k / RT comes from one combined NASA-7 polynomial per species (6 FMAs);
//   - Newton works on mixture coefficients m_i = sum_k Y_k (ec_ki / W_k), assembled once
//     per evaluation (54 FMAs), so each iteration is two Horner chains and a reciprocal;
//   - equilibrium constants come from per-species G_k = exp(-g_k / RT):
//     1/K_c,j = prod_reactants G * prod_products (1/G) * (R_u T / p_ref)^(sum nu), i.e.
//     18 exponentials per evaluation (G and 1/G) instead of one per
//     reaction; with a_k = c_k / G_k the net rate of progress is
//     k_f (prod_reactants c - prod_reactants G * prod_products a * (R_u T / p_ref)^(sum nu)),
//     one FMA for the reverse direction;
//   - reciprocals are Newton-Raphson-refined hardware approximations (rcp1 / rcp2), ~3.5
//     and ~5.7 FP64-pipe slots against ~9 for an IEEE divide; compares, clamps and
//     fp32 <-> fp64 conversions run on the integer pipe (fastmath.cuh);
//   - forward rates are one exponential per reaction (none for temperature-independent rates
//     or A T^-1, A T^-2 with no activation).
#pragma once

#include <cmath>
#include <utility>

#include "fastmath.cuh"
#include "mech.cuh"

namespace chem {

// Mixture internal-energy coefficients from mass fractions, shifted by the target:
// e/R_u - eR = T (m0 + T (m1 + T (m2 + T (m3 + T m4)))) + m5
__device__ __forceinline__ void mix_ecoef(const MechTables &mt, int range, const double (&Y)[NSP],
                                          double eR, double (&m)[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NSP; ++k) s = fma(Y[k], mt.ecw[range][k][i], s);
    m[i] = s;
  }
  m[5] -= eR;
}

__device__ __forceinline__ double e_over_R(const double (&m)[6], double T) {
  return fma(T, fma(T, fma(T, fma(T, fma(T, m[4], m[3]), m[2]), m[1]), m[0]), m[5]);
}

// cv/R = d(e/R)/dT from the scaled coefficients d = {m0, 2 m1, 3 m2, 4 m3, 5 m4}
__device__ __forceinline__ double cv_over_R(const double (&d)[5], double T) {
  return fma(T, fma(T, fma(T, fma(T, d[4], d[3]), d[2]), d[1]), d[0]);
}

__device__ __forceinline__ void cv_coef(const double (&m)[6], double (&d)[5]) {
  d[0] = m[0];
  d[1] = 2.0 * m[1];
  d[2] = 3.0 * m[2];
  d[3] = 4.0 * m[3];
  d[4] = 5.0 * m[4];
}

// Temperature from e/R_u and the mass fractions Y.  T: in = starting guess (1500 K if not
// positive and finite), out = root.  Newton stops at |dT| <= 1e-12 T, or as soon as the
// quadratic convergence bound guarantees that (dT^2 <= newton_sq T: the remaining error
// is then below 1e-12 T / 2), within 30 iterations; on a non-positive / non-finite
// iterate or no convergence, bisection on [200, 6000] K.  The step divides by c_v through
// a reciprocal with relative error ~2^-40 (a perturbed Newton step converges the same
// way), the stop test runs in fp32 on the rounded dT and T (it only decides when to
// stop), and the range and sign tests run on the integer pipe.
__device__ __forceinline__ bool solve_T(const MechTables &mt, const double (&Y)[NSP], double eR,
                                        double &T) {
  double Tn = pos_normal(T) ? T : 1500.0;
  int range = ge_nonneg(Tn, mt.T_mid);
  double m[6], d[5];
  mix_ecoef(mt, range, Y, eR, m);
  cv_coef(m, d);
  for (int it = 0; it < 30; ++it) {
    const int r = ge_nonneg(Tn, mt.T_mid);
    if (r != range) {
      range = r;
      mix_ecoef(mt, range, Y, eR, m);
      cv_coef(m, d);
    }
    const double dT = e_over_R(m, Tn) * rcp1(cv_over_R(d, Tn));
    Tn -= dT;
    if (!pos_normal(Tn)) break;
    const float dTf = d2f(dT), Tf = d2f(Tn);
    if (fabsf(dTf) <= 1e-12f * Tf || dTf * dTf <= mt.f.newton_sq * Tf) {
      T = Tn;
      return true;
    }
  }
  // bracketed fallback
  double lo = 200.0, hi = 6000.0, mlo[6], mhi[6];
  mix_ecoef(mt, lo >= mt.T_mid, Y, eR, mlo);
  mix_ecoef(mt, hi >= mt.T_mid, Y, eR, mhi);
  if (e_over_R(mlo, lo) > 0.0 || e_over_R(mhi, hi) < 0.0) return false;
  for (int it = 0; it < 200 && hi - lo > 1e-13 * hi; ++it) {
    const double mid = 0.5 * (lo + hi);
    mix_ecoef(mt, mid >= mt.T_mid, Y, eR, m);
    if (e_over_R(m, mid) > 0.0) hi = mid; else lo = mid;
  }
  T = 0.5 * (lo + hi);
  return true;
}

// Quantities shared by every reaction of one evaluation.
struct RateInputs {
  double lnT, invT, RTP, PRT, ctot;
  long long lT, iT;  // log2 T (Q58), 1 / T (Q70): the fixed-point form's
  double c[NSP];     // clamped concentrations, mol/m^3
  double G[NSP];     // exp(-g_k / (R_u T))
  double iG[NSP];    // c_k / G_k
};

// Temperatures of the fixed-point form: (128, 32768), on the high word.
__device__ __forceinline__ bool fixed_range(double T) {
  return (uint32_t)__double2hiint(T) - 0x40600001u < 0x40e00000u - 0x40600001u;
}

// Troe broadening factor (Gilbert, Luther & Troe 1983).
template <int J, bool kFixed>
__device__ __forceinline__ double troe_F(const MechTables &mt, double T, double invT, double Pr) {
  constexpr int n = kRx[J].troe_n;
  if constexpr (n == 0) {
    return 1.0;
  } else {
    const double a = mt.troe_a[J];
    double Fc;
    if constexpr (kFixed) {
      Fc = (1.0 - a) * exp2_lim(-T * mt.troe_q3[J]) + a * exp2_lim(-T * mt.troe_q1[J]);
      if constexpr (n == 4) Fc += exp2_lim(-mt.troe_q2[J] * invT);
    } else {
      Fc = (1.0 - a) * exp_t(-T * mt.troe_i3[J]) + a * exp_t(-T * mt.troe_i1[J]);
      if constexpr (n == 4) Fc += exp_t(-mt.troe_T2[J] * invT);
    }
    const double lFc = log10_t(Fc);
    const double cc = -0.4 - 0.67 * lFc;
    const double nn = 0.75 - 1.27 * lFc;
    const double x = log10_t(Pr) + cc;
    const double f1 = x * rcp2(nn - 0.14 * x);
    const double lF = lFc * rcp2(1.0 + f1 * f1);
    if constexpr (kFixed) return exp2_lim(lF * kLog2_10);
    else return exp10_t(lF);
  }
}

// Rate of progress of reaction J added into wdot (law of mass action, Eq. 16).  kFixed: the
// exponentials in fixed point.
template <int J, bool kFixed>
__device__ __forceinline__ void reaction(const MechTables &mt, const RateInputs &in, double T,
                                         double (&wdot)[NSP]) {
  constexpr RxStruct R = kRx[J];
  constexpr int dnu = n_prod(R) - n_reac(R);
  static_assert(dnu >= -1 && dnu <= 1, "compiled structure assumes |sum nu| <= 1");
  // kconst: 0 Arrhenius exponential; 1 constant (b = Ea = 0); 2, 3: A T^-1, A T^-2 (Ea = 0)
  const int kc = mt.kconst[J];
  double kf;
  if (kc == 0) {
    if constexpr (kFixed) kf = exp2_q52(limit_q52(arrhenius_log2(mt.qA[J], mt.qB[J], mt.qH[J], in.lT, in.iT)));
    else kf = exp_t(fma(mt.beta[J], in.lnT, mt.lnA[J]) - mt.Ta[J] * in.invT);
  } else if (kc == 1) kf = mt.A[J];
  else if (kc == 2) kf = mt.A[J] * in.invT;
  else kf = mt.A[J] * in.invT * in.invT;
  double M = 0.0;
  if constexpr (R.type != ELEM) {
    M = in.ctot;
    if (mt.has_eff[J]) {
#pragma unroll
      for (int k = 0; k < NSP; ++k)
        if ((mt.eff_mask[J] >> k) & 1) M = fma(mt.effm1[J][k], in.c[k], M);
    }
  }
  if constexpr (R.type == FALLOFF) {
    double k0;
    if constexpr (kFixed) k0 = exp2_q52(limit_q52(arrhenius_log2(mt.qA0[J], mt.qB0[J], mt.qH0[J], in.lT, in.iT)));
    else k0 = exp_t(fma(mt.beta0[J], in.lnT, mt.lnA0[J]) - mt.Ta0[J] * in.invT);
    const double Pr = k0 * M * rcp2(kf);
    kf = (Pr > 0.0) ? kf * (Pr * rcp2(1.0 + Pr)) * troe_F<J, kFixed>(mt, T, in.invT, Pr) : 0.0;
  }
  // q = k_f (prod c_reactants - prod G_reactants prod (c / G)_products (R_u T / p)^dnu),
  // the same net rate as k_f prod c - k_r prod c with k_r = k_f / K_c
  double cf = in.c[R.r0];
  if constexpr (R.r1 >= 0) cf *= in.c[R.r1];
  if (mt.reversible[J]) {
    double gr = in.G[R.r0];
    if constexpr (R.r1 >= 0) gr *= in.G[R.r1];
    if constexpr (dnu == 1) gr *= in.RTP;
    if constexpr (dnu == -1) gr *= in.PRT;
    double ap = in.iG[R.p0];
    if constexpr (R.p1 >= 0) ap *= in.iG[R.p1];
    cf = fma(-gr, ap, cf);
  }
  double q = kf * cf;
  if constexpr (R.type == THIRD_BODY) q *= M;
  wdot[R.r0] -= q;
  if constexpr (R.r1 >= 0) wdot[R.r1] -= q;
  wdot[R.p0] += q;
  if constexpr (R.p1 >= 0) wdot[R.p1] += q;
}

template <bool kFixed, int... J>
__device__ __forceinline__ void all_reactions(const MechTables &mt, const RateInputs &in, double T,
                                              double (&wdot)[NSP], std::integer_sequence<int, J...>) {
  (reaction<J, kFixed>(mt, in, T, wdot), ...);
}

// Molar production rates wdot (mol/m^3/s) at temperature T and clamped concentrations c.
template <bool kFixed>
__device__ __forceinline__ void production_rates(const MechTables &mt, double T,
                                                 const double (&c)[NSP], double (&wdot)[NSP]) {
  RateInputs in;
  in.lnT = log_t(T);
  in.invT = rcp2(T);
  in.RTP = (R_U / P_REF) * T;
  in.PRT = (P_REF / R_U) * in.invT;
  if constexpr (kFixed) {
    in.lT = (long long)abs_q<58>(in.lnT * kLog2E);
    in.iT = (long long)abs_q<70>(in.invT);
  }
  const double oml = 1.0 - in.lnT;
  const int range = ge_nonneg(T, mt.T_mid);
  double ctot = 0.0;
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    in.c[k] = c[k];
    ctot += c[k];
    const double *gc = kFixed ? mt.gc_q[range][k] : mt.gc[range][k];
    double g = fma(T, fma(T, fma(T, fma(T, gc[4], gc[3]), gc[2]), gc[1]), fma(gc[5], in.invT, gc[6]));
    g = fma(gc[0], oml, g);
    // the limits keep G finite far outside the tables' range
    if constexpr (kFixed) {
      const long long y = to_q52(g);
      in.G[k] = exp2_q52(y);
      in.iG[k] = c[k] * exp2_q52(-y);
    } else {
      g = clamp_abs(g, 700.0);
      in.G[k] = exp_t(-g);
      in.iG[k] = c[k] * rcp2(in.G[k]);
    }
    wdot[k] = 0.0;
  }
  in.ctot = ctot;
  all_reactions<kFixed>(mt, in, T, wdot, std::make_integer_sequence<int, NRX>{});
}

// The form on exp_t, for temperatures or coefficients outside the fixed-point form's range;
// out of line, as few evaluations come here.
static __device__ __noinline__ void production_rates_any(const MechTables &mt, double T, const double *c,
                                                         double *wdot) {
  double cc[NSP], w[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) cc[k] = c[k];
  production_rates<false>(mt, T, cc, w);
#pragma unroll
  for (int k = 0; k < NSP; ++k) wdot[k] = w[k];
}

// dY/dt of one cell at fixed (rho, e).  T: in = Newton guess, out = solved T.
// Returns false when the temperature solve fails.
__device__ __forceinline__ bool cell_rhs(const MechTables &mt, const double (&Y)[NSP], double rho,
                                         double invRho, double eR, double &T, double (&F)[NSP]) {
  if (!solve_T(mt, Y, eR, T)) return false;
  double c[NSP], wdot[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) c[k] = clamp_nonneg(rho * (Y[k] * mt.invW[k]));
  if (mt.fixed_ok && fixed_range(T)) {
    production_rates<true>(mt, T, c, wdot);
  } else {
    double cc[NSP], w[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) cc[k] = c[k];
    production_rates_any(mt, T, cc, w);
#pragma unroll
    for (int k = 0; k < NSP; ++k) wdot[k] = w[k];
  }
#pragma unroll
  for (int k = 0; k < NSP; ++k) F[k] = wdot[k] * mt.W[k] * invRho;
  return true;
}

}  // namespace chem
