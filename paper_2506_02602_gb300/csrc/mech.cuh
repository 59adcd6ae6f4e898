// mech.cuh -- compile-time structure of the reaction mechanism and the per-context
// coefficient tables the kernels read.
//
// The kernels are specialised to the stoichiometry of one hydrogen mechanism (Eq. 15):
// every species index and stoichiometric coefficient is a compile-time constant, so the
// law of mass action (Eq. 16) unrolls into straight register code with no per-reaction
// branching on data.  The structure comes from a generated header (gen_mech.py): the
// 9-species / 21-reaction mechanism, or the 13-species / 27-reaction one of the paper's
// size.  The coefficients (Arrhenius,
// efficiencies, Troe, NASA-7) are runtime data: chem_setup packs them into MechTables,
// which every launch passes by value as a __grid_constant__ parameter, so the tables
// sit in the constant bank, are read with uniform (broadcast) accesses and need no
// global state -- several contexts with different coefficients can coexist.
#pragma once

#include <cstdint>

namespace chem {

constexpr double R_U = 8.31446261815324;  // J/(mol K)
constexpr double P_REF = 101325.0;        // Pa, standard state of the equilibrium constants

enum RxType : int { ELEM = 0, THIRD_BODY = 1, FALLOFF = 2 };

// Reaction structure: up to two reactant and two product molecules (a repeated
// species appears twice), reaction type, number of Troe parameters.
struct RxStruct {
  int r0, r1, p0, p1, type, troe_n;
};

}  // namespace chem

// The compiled structure (NSP, NRX, the species enum Sp and the reaction table kRx),
// generated by gen_mech.py from the mechanism description.  One library is built per
// structure: the 9-species / 21-reaction mechanism by default, the 13-species /
// 27-reaction one with CHEM_MECH_H2O2_13.
#if defined(CHEM_MECH_H2O2_13)
#include "mech_h2o2_13.cuh"
#else
#include "mech_h2o2_9.cuh"
#endif

namespace chem {

__host__ __device__ constexpr int n_reac(const RxStruct &r) { return (r.r0 >= 0) + (r.r1 >= 0); }
__host__ __device__ constexpr int n_prod(const RxStruct &r) { return (r.p0 >= 0) + (r.p1 >= 0); }

// fp32 copies of the rate coefficients for the mixed-precision variant.
struct MechTablesF32 {
  float A[NRX];
  float W[NSP];
  float invW[NSP];
  float lnA[NRX], beta[NRX], Ta[NRX];
  float lnA0[NRX], beta0[NRX], Ta0[NRX];
  float troe_a[NRX], troe_i3[NRX], troe_i1[NRX], troe_T2[NRX];
  float effm1[NRX][NSP];
  // fp32 thermo for the surrogate's error test (all-fp32 right-hand side)
  float ec[2][NSP][6];
  float gc[2][NSP][7];
  float T_mid, ln_R_over_Pref;
  float newton_sq;  // the fp64 Newton's stop constant (below), tested in fp32
  // fp32 pairs (value = [0] + [1] to ~2^-49) of ecw, gc, T_mid and ln_R_over_Pref below,
  // for the mixed right-hand side's double-float arithmetic (ff.cuh)
  float ecw2[2][NSP][6][2];
  float gc2[2][NSP][7][2];
  float T_mid2[2], ln_R_over_Pref2[2];
};

// A coefficient in fixed point: h 2^32 plus the top bits l of the lower half (2^2 l, or 2^4 l in qgt;
// in qe the lower half is signed and its limb 2 l)
struct QCoef { int32_t h, l; };

// Per-context tables (host-built from chem_mechanism by build_tables()).
struct MechTables {
  double T_mid;
  double W[NSP];
  double invW[NSP];
  // e_k W_k / R_u = sum_i ec[i] T^(i+1) + ec[5]: {a1 - 1, a2/2, a3/3, a4/4, a5/5, a6}
  double ec[2][NSP][6];
  // the same per unit mass fraction (ec / W_k): mixture coefficients sum_k Y_k ecw_k
  double ecw[2][NSP][6];
  // g_k / (R_u T) = h/RT - s/R = gc0 (1 - ln T) + gc1 T + gc2 T^2 + gc3 T^3 + gc4 T^4
  //                 + gc5 / T + gc6  with {a1, -a2/2, -a3/6, -a4/12, -a5/20, a6, -a7}
  double gc[2][NSP][7];
  // Arrhenius: k = exp(lnA + beta ln T - Ta / T); Ta = Ea / R_u.  kconst selects a form
  // without the exponential when Ea == 0: 1 for b == 0 (k = A), 2 for b == -1 (A / T),
  // 3 for b == -2 (A / T^2); 0 otherwise.
  double lnA[NRX], beta[NRX], Ta[NRX], A[NRX];
  int32_t kconst[NRX];
  int32_t reversible[NRX];
  // fall-off low-pressure limit and Troe parameters (alpha, 1/T***, 1/T*, T**)
  double lnA0[NRX], beta0[NRX], Ta0[NRX];
  double troe_a[NRX], troe_i3[NRX], troe_i1[NRX], troe_T2[NRX];
  // The fixed-point form's tables (rhs_fixed.cuh); fixed_ok: every coefficient is in its range.
  // Rates: log2 A (Q52), b (Q58), -Ta / ln2 (Q46) of both limits; Troe temperatures' factors
  // times log2(e).
  int64_t qA[NRX], qA0[NRX];
  QCoef qB[NRX], qH[NRX], qB0[NRX], qH0[NRX];
  double troe_q3[NRX], troe_q1[NRX], troe_q2[NRX];
  // t = T 2^-S per range, S = q_log2[range]: ecw (Q q_res + 2) times 2^(S (i+1)), the Gibbs functions
  // times -log2(e) by log2 T (Q56), 1/T (Q44), t .. t^4 (Q57) and 1 (Q50)
  QCoef qe[2][NSP][6];
  QCoef qg[2][NSP][2], qgt[2][NSP][4];
  int64_t qg1[2][NSP];
  int64_t qT_mid, qRP;  // T_mid (Q50), log2(R_u / p_ref) (Q50)
  int32_t q_log2[2], q_res[2];
  int32_t fixed_ok;
  // third-body efficiencies minus one: [M] = sum_k c_k + sum_k effm1 c_k
  double effm1[NRX][NSP];
  int32_t has_eff[NRX];
  int32_t eff_mask[NRX];  // bit k set where effm1[j][k] != 0 (the fp64 sums skip the rest)
  // the same as short lists: [M] = m_base sum_k c_k + sum_i m_c[i] c[m_k[i]], m_base 1 or 0,
  // whichever makes the shorter list of m_n entries
  double m_c[NRX][NSP];
  int32_t m_base[NRX], m_n[NRX];
  int8_t m_k[NRX][NSP];
  double ln_R_over_Pref;  // ln(R_u / p_ref): ln(R_u T / p_ref) = ln T + this
  // Newton's quadratic-convergence stop: after a step dT the remaining error is at most
  // (C / 2) dT^2 with C = max |c_v' / c_v| of the tables on [200, 6000] K, so a step with
  // dT^2 <= newton_sq T, newton_sq = 1e-12 / C, already leaves T within 1e-12 T / 2
  double newton_sq;
  // element mass fraction (H, O, N) per unit mass fraction of species k:
  // n_ke A_e / sum_e' n_ke' A_e' (columns sum to 1, so conserving elements conserves sum Y)
  double Emat[3][NSP];
  MechTablesF32 f;
};

// kernel parameters may take up to 32,764 bytes (sm_70 and later, CUDA 12.1 and later)
static_assert(sizeof(MechTables) < 32000, "MechTables must fit a kernel parameter block");

}  // namespace chem
