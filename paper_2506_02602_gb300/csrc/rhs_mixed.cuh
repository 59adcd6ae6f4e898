// rhs_mixed.cuh -- mixed-precision right-hand side of one constant-(rho, e) cell.
//
// The same right-hand side as rhs.cuh (Eq. 10, 14-16), split by precision:
//   double-float (pairs of fp32, ~48 bits, ff.cuh): the temperature solve (Newton on the
//         mixture NASA-7 coefficients), ln T, the Gibbs functions g_k / RT and
//         ln(R_u T / p_ref): the part whose accuracy decides the temperature and the
//         equilibrium state;
//   fp32: forward rate coefficients, third-body sums, Troe fall-off, reverse rates
//         k_r = exp(ln k_f + ln(1 / K_c)), the law-of-mass-action products, production
//         rates and F.
// What reaches the fp32 part is T, ln T, 1/T and the equilibrium exponents
// ln(1 / K_c,j) = sum_k nu_jk g_k + (sum_k nu_jk) ln(R_u T / p_ref), each rounded once to
// fp32.  They are to be no less exact than fp64 values rounded once, and a rounding test (Ziv,
// ACM TOMS 17 (1991) 410-423) sees to it: where the double-float value lies near the middle between
// two fp32 numbers, the cell's temperature and Gibbs functions
// are evaluated again in fp64 (solve_gibbs_fp64; 0.4 % of the cells' evaluations).
// The exponents are summed from fp32 hi parts on a 2^-12 grid (exact in fp32) and lo parts, in fp64
// as here; it is the lo parts' rounding that limits both.  Over 200,000 temperatures from 250 to
// 4500 K an exponent of fp64 Gibbs functions is up to 4.6e-11 beyond half an fp32 ulp off, one of
// double-float functions 5.4e-11, and one that passed the test, at kLnKcErr = 2.4e-11, thus at most
// 3.0e-11.  (The two are still other fp32 numbers now and then, neither of them nearer: see there.)
//
// On GB300 an FP64 instruction costs a warp 64 cycles of its sub-partition whatever else the
// warp does, a double-float multiply-add about 13 (6 with the packed f32x2 forms).  With the
// temperature solve and the Gibbs functions in fp64 the FP64 pipe was 82 % busy and the issue
// slots 26 %; now the pipe is 51 % busy (the solution and error registers, the norm, the
// evaluations in fp64) and issue 53 %.  What bounds the kernel is the latency of dependent
// fp32 operations at 16 warps an SM, and it runs the 1M-cell detonation slice in 7.9 ms
// instead of 16.1 (the 151,979-cell 13-species slice in 2.46 instead of 3.40).
//
// Straight-line code is fetched at no more than two instructions a clock and SM, and code that
// exceeds the instruction caches (the unrolled form: 64 KB) at the speed of the L2; so the
// loops over species and reactions stay rolled, over per-thread columns in shared memory
// (stride ST) and tables in shared memory, and the rare fp64 path is compact.  (Unrolled
// register code: 8.2 ms without the rounding test, with fetch stalls 41 % of all; rolled: 7.0
// without the test and 7.9 with it.)
#pragma once

#include <math_constants.h>

#include "ff.cuh"
#include "rhs.cuh"

namespace chem {

// Species with an equilibrium role: 1 + the largest index in a reaction (the inert ones,
// N2 and the colliders, come last).
__host__ __device__ constexpr int n_reactive() {
  int m = 0;
  for (int j = 0; j < NRX; ++j) {
    const int v[4] = {kRx[j].r0, kRx[j].r1, kRx[j].p0, kRx[j].p1};
    for (int i = 0; i < 4; ++i) m = v[i] > m ? v[i] : m;
  }
  return m + 1;
}
constexpr int NGB = n_reactive();

// The reactions of one type before reaction j (j = NRX: all of them).
__host__ __device__ constexpr int count_before(int j, int type) {
  int m = 0;
  for (int i = 0; i < j; ++i) m += kRx[i].type == type;
  return m;
}
constexpr int NFO = count_before(NRX, FALLOFF);
constexpr int NRL = NRX - NFO;                         // reactions of the rolled loop
constexpr int NM = NFO + count_before(NRX, THIRD_BODY);  // reactions with a third-body sum
static_assert(NFO > 0 && NRX <= 31, "one bit per reaction");
// Slot of reaction j: the loop's reactions in order, then the fall-off ones.
__host__ __device__ constexpr int rx_slot(int j) {
  const int f = count_before(j, FALLOFF);
  return kRx[j].type == FALLOFF ? NRL + f : j - f;
}
// Position of reaction j among those with a third-body sum: the fall-off ones, then the rest.
__host__ __device__ constexpr int m_index(int j) {
  return kRx[j].type == FALLOFF ? count_before(j, FALLOFF) : NFO + count_before(j, THIRD_BODY);
}

// Per-thread columns of the mixed variant, ST threads apart in dynamic shared memory: per
// species the Gibbs function's hi and lo parts G and the pair CU of the concentration and
// the stage state U (each with a row for an absent molecule: 0 and c = 1), the rates of progress
// Q (the derivative F takes their place), the advancing solution X
// and the error register E: 388 bytes a thread for 9 species.  In shared memory the rolled
// loops index them without local memory, and every access is conflict-free.
struct MixedCols {
  float2 *G, *CU;
  float *Q;
  double *X, *E;
};
static_assert(NRX >= NSP, "F takes Q's place");
constexpr size_t mixed_cols_bytes(int block) { return (size_t)block * (8 * 2 * (NSP + 1) + 8 * 2 * NSP + 4 * NRX); }
template <int ST>
__device__ __forceinline__ MixedCols mixed_cols() {
  extern __shared__ double s_cols[];
  MixedCols c;
  c.X = s_cols + threadIdx.x;
  c.E = c.X + NSP * ST;
  c.G = reinterpret_cast<float2 *>(s_cols + 2 * NSP * ST) + threadIdx.x;
  c.CU = c.G + (NSP + 1) * ST;
  c.Q = reinterpret_cast<float *>(s_cols + (4 * NSP + 2) * ST) + threadIdx.x;
  return c;
}
// The rows of an absent molecule; once per thread before the first evaluation.
template <int ST>
__device__ __forceinline__ void init_mixed_cols(const MixedCols &m) {
  m.G[NSP * ST] = make_float2(0.0f, 0.0f);
  m.CU[NSP * ST] = make_float2(1.0f, 0.0f);
}

// Per-block tables: ecw2 as pairs of coefficients {h0, h1, l0, l1}, gc2 as pairs of species
// (both of a lane's own NASA-7 range), and the loop's reactions: the byte offsets of the
// reactants' and products' rows (an absent second reactant, and an absent FIRST product, is
// row NSP: the net rate is then the same single FMA with one product or two), {ln A, beta,
// Ta, sum nu} and {s, a, t}: k_f = s exp(ln k_f) + a (s, a = 1, 0, or 0, A for a constant) and
// k_r is kept where k_f > t (t = 0, or infinity for an irreversible reaction).
__shared__ float4 s_ecw[2][NSP][3];
__shared__ float4 s_gc[2][(NGB + 1) / 2][7];
__shared__ int4 s_rx_row[NRX];
__shared__ float4 s_rx_k[NRX];
__shared__ float4 s_rx_f[NRX];
// Fall-off: {ln A0, beta0, Ta0, Troe parameter count} and {alpha, 1/T***, 1/T*, T**}; third-body
// efficiencies minus one, species by reaction; {1/W, W} per species.
__shared__ float4 s_fo_k[NFO];
__shared__ float4 s_fo_t[NFO];
__shared__ float s_eff[NSP][(NM + 3) / 4 * 4];
__shared__ float2 s_w[NSP];

template <int J, int ST>
__device__ __forceinline__ void load_rx(const MechTables &mt) {
  constexpr RxStruct R = kRx[J];
  constexpr int i = rx_slot(J), b = ST * 8;
  s_rx_row[i] = make_int4(R.r0 * b, (R.r1 >= 0 ? R.r1 : NSP) * b, (R.p1 >= 0 ? R.p0 : NSP) * b,
                          (R.p1 >= 0 ? R.p1 : R.p0) * b);
  s_rx_k[i] = make_float4(mt.f.lnA[J], mt.f.beta[J], mt.f.Ta[J], (float)(n_prod(R) - n_reac(R)));
  const bool fixed = mt.kconst[J] == 1;
  s_rx_f[i] = make_float4(fixed ? 0.0f : 1.0f, fixed ? mt.f.A[J] : 0.0f, mt.reversible[J] ? 0.0f : CUDART_INF_F, 0.0f);
  if constexpr (R.type == FALLOFF) {
    s_fo_k[i - NRL] = make_float4(mt.f.lnA0[J], mt.f.beta0[J], mt.f.Ta0[J], (float)R.troe_n);
    s_fo_t[i - NRL] = make_float4(mt.f.troe_a[J], mt.f.troe_i3[J], mt.f.troe_i1[J], mt.f.troe_T2[J]);
  }
  if constexpr (R.type != ELEM)
    for (int k = 0; k < NSP; ++k) s_eff[k][m_index(J)] = mt.f.effm1[J][k];
}
template <int ST, int... J>
__device__ __forceinline__ void load_rxs(const MechTables &mt, std::integer_sequence<int, J...>) {
  ((threadIdx.x == J % 32 ? load_rx<J, ST>(mt) : (void)0), ...);
}

// Fills the tables (and ff_log's); every kernel that calls cell_rhs_mixed or gibbs_hl starts
// with it (all threads).
template <int ST>
__device__ __forceinline__ void load_mixed_tables(const MechTables &mt) {
  for (int i = threadIdx.x; i < 2 * NSP; i += blockDim.x) {
    const int r = i / NSP, k = i % NSP;
    const float(*e)[2] = mt.f.ecw2[r][k];
    for (int q = 0; q < 3; ++q) s_ecw[r][k][q] = make_float4(e[2 * q][0], e[2 * q + 1][0], e[2 * q][1], e[2 * q + 1][1]);
    if (k % 2 == 0 && k < NGB) {
      const float(*g)[2] = mt.f.gc2[r][k], (*g1)[2] = mt.f.gc2[r][k + 1 < NSP ? k + 1 : k];
      for (int q = 0; q < 7; ++q) s_gc[r][k / 2][q] = make_float4(g[q][0], g1[q][0], g[q][1], g1[q][1]);
    }
  }
  load_ln_ff();
  for (int i = threadIdx.x; i < 65; i += blockDim.x) {
    s_log_inv[i] = k_log_inv[i];
    s_log_tab[i] = k_log_tab[i];
    s_log_tab_m1[i] = k_log_tab_m1[i];
  }
  for (int k = threadIdx.x; k < NSP; k += blockDim.x) s_w[k] = make_float2(mt.f.invW[k], mt.f.W[k]);
  load_rxs<ST>(mt, std::make_integer_sequence<int, NRX>{});
  __syncthreads();
}

struct RateTempsF {
  float lnT, invT, T;
};
// for the fp32 estimators
struct RateInputsF : RateTempsF {
  float ctot;
  float c[NSP];
};

// Troe broadening factor in fp32 on the fast intrinsics (hardware base-2 exponential and
// logarithm, approximate division; relative errors ~1e-6 on these arguments), for the
// estimators: the surrogate's error test, which compares with a tolerance of ~5e-4 T, and the
// batched path's stiffness key.
template <int J>
__device__ __forceinline__ float troe_F_f32(const MechTables &mt, float T, float invT, float Pr) {
  constexpr int n = kRx[J].troe_n;
  if constexpr (n == 0) {
    return 1.0f;
  } else {
    const float a = mt.f.troe_a[J];
    float Fc = (1.0f - a) * __expf(-T * mt.f.troe_i3[J]) + a * __expf(-T * mt.f.troe_i1[J]);
    if constexpr (n == 4) Fc += __expf(-mt.f.troe_T2[J] * invT);
    const float lFc = __log10f(Fc);
    const float cc = -0.4f - 0.67f * lFc;
    const float nn = 0.75f - 1.27f * lFc;
    const float x = __log10f(Pr) + cc;
    const float f1 = __fdividef(x, nn - 0.14f * x);
    return __exp10f(__fdividef(lFc, 1.0f + f1 * f1));
  }
}

// The ingredients of ln(1/K_c,j) = sum_k nu_jk g_k + (sum_k nu_jk) ln(R_u T / p_ref).
// Mixed variant: g_k / RT (in the columns) and ln(R_u T / p_ref) as fp32 hi/lo pairs; the hi parts
// sum exactly in fp32 and the lo parts carry the rest (to within ~1e-11).
// GibbsF (the error test's all-fp32 right-hand side): plain fp32.
struct GibbsF {
  float g[NSP];
  float r;
};

// The hi / lo split of a pair, as split_hilo makes it of an fp64 value: hi = x
// truncated to a multiple of 2^-12 (for |x| < 2^10, where every g_k above ~70 K lies; a
// neighbouring multiple beyond), lo the rest.
__device__ __forceinline__ float2 split_grid(ff x) {
  float h = fsub(fadd(x.h, 3072.0f), 3072.0f);
  float r = fadd(fsub(x.h, h), x.l);
  const float step = copysignf(2.44140625e-4f, x.h);
  if (__float_as_int(r) != 0 && r * step < 0.0f) {  // rounded away from zero
    h = fsub(h, step);
    r = fadd(fsub(x.h, h), x.l);
  }
  return make_float2(h, r);
}

__device__ __forceinline__ bool ge_mid(const MechTables &mt, ff T) {
  return T.h > mt.f.T_mid2[0] || (T.h == mt.f.T_mid2[0] && T.l >= mt.f.T_mid2[1]);
}

// g_k / RT = a1 (1 - ln T) - a2 T / 2 - ... - a5 T^4 / 20 + a6 / T - a7 (NASA-7, with the
// coefficients pre-combined per range into gc2) of the reactive species and
// ln(R_u T / p_ref), evaluated in double-float as sums of products with the functions of T
// (error-free products and two-sums; error ~1e-12 for terms of a few hundred), two species at
// a time, and split; species k's parts go to g[k ST].
template <int ST>
__device__ __forceinline__ void gibbs_hl(const MechTables &mt, ff T, ff lnT, ff invT, float2 *g, float2 &r) {
  const int range = ge_mid(mt, T);
  const ff2 oml = both(ff_norm(ff_acc(ff{1.0f, 0.0f}, ff{-lnT.h, -lnT.l})));
  const ff q2 = ff_norm(ff_mul(T, T));
  const ff2 T1 = both(T), T2 = both(q2), T3 = both(ff_norm(ff_mul(q2, T))), T4 = both(ff_norm(ff_mul(q2, q2)));
  const ff2 iT = both(invT);
#pragma unroll 1
  for (int k = 0; k < NGB; k += 2) {
    const float4 *c = s_gc[range][k >> 1];
    auto coef = [&](int i) {
      const float4 v = c[i];
      return ff2{make_float2(v.x, v.y), make_float2(v.z, v.w)};
    };
    ff2 s = ff_acc(coef(6), ff_mul(iT, coef(5)));
    s = ff_acc(s, ff_mul(oml, coef(0)));
    ff2 q = ff_acc(ff_mul(T3, coef(3)), ff_mul(T4, coef(4)));
    q = ff_acc(ff_mul(T2, coef(2)), q);
    q = ff_acc(ff_mul(T1, coef(1)), q);
    s = ff_acc(s, q);
    g[k * ST] = split_grid(ff{s.h.x, s.l.x});
    if (NGB % 2 == 0 || k + 1 < NGB) g[(k + 1) * ST] = split_grid(ff{s.h.y, s.l.y});
  }
  r = split_grid(ff_acc(lnT, ff{mt.f.ln_R_over_Pref2[0], mt.f.ln_R_over_Pref2[1]}));
}

// The same functions evaluated entirely in fp32 (the error test's right-hand side).
__device__ __forceinline__ void gibbs_f(const MechTables &mt, float T, float lnT, float invT, GibbsF &g) {
  const float oml = 1.0f - lnT;
  const int range = T >= mt.f.T_mid;
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    const float *gc = mt.f.gc[range][k];
    const float gk = fmaf(T, fmaf(T, fmaf(T, fmaf(T, gc[4], gc[3]), gc[2]), gc[1]), fmaf(gc[5], invT, gc[6]));
    g.g[k] = fmaf(gc[0], oml, gk);
  }
  g.r = lnT + mt.f.ln_R_over_Pref;
}

// Whether x.h + x.l rounds to the same fp32 number anywhere within +-d.
__device__ __forceinline__ bool rounds_safely(ff x, float d) {
  return fadd(x.h, fadd(x.l, d)) == fadd(x.h, fsub(x.l, d));
}

template <int J>
__device__ __forceinline__ float ln_inv_kc(const GibbsF &g) {
  constexpr RxStruct R = kRx[J];
  constexpr int dnu = n_prod(R) - n_reac(R);
  float q = g.g[R.p0] - g.g[R.r0];
  if constexpr (R.p1 >= 0) q += g.g[R.p1];
  if constexpr (R.r1 >= 0) q -= g.g[R.r1];
  if constexpr (dnu == 1) q += g.r;
  if constexpr (dnu == -1) q -= g.r;
  return q;
}

// One reaction in fp32 on the fast intrinsics, added into wdot.  With kDestr, the one-way
// fluxes that consume each species are also summed into dflux (the stiffness key).
template <int J, bool kDestr>
__device__ __forceinline__ void reaction_f32(const MechTables &mt, const RateInputsF &in, const GibbsF &g,
                                             float (&wdot)[NSP], float *dflux) {
  constexpr RxStruct R = kRx[J];
  float lnkf = fmaf(mt.f.beta[J], in.lnT, mt.f.lnA[J]) - mt.f.Ta[J] * in.invT;
  float kf = mt.kconst[J] == 1 ? mt.f.A[J] : __expf(lnkf);
  float M = 0.0f;
  if constexpr (R.type != ELEM) {
    M = in.ctot;
    if (mt.has_eff[J]) {
#pragma unroll
      for (int k = 0; k < NSP; ++k) M = fmaf(mt.f.effm1[J][k], in.c[k], M);
    }
  }
  if constexpr (R.type == FALLOFF) {
    const float k0 = __expf(fmaf(mt.f.beta0[J], in.lnT, mt.f.lnA0[J]) - mt.f.Ta0[J] * in.invT);
    const float Pr = __fdividef(k0 * M, kf);
    kf = (Pr > 0.0f) ? kf * __fdividef(Pr, 1.0f + Pr) * troe_F_f32<J>(mt, in.T, in.invT, Pr) : 0.0f;
    lnkf = __logf(kf);
  }
  float qf = kf * in.c[R.r0];
  if constexpr (R.r1 >= 0) qf *= in.c[R.r1];
  float q = qf, qr = 0.0f;
  if (mt.reversible[J]) {
    const float kr = (kf > 0.0f) ? __expf(lnkf + ln_inv_kc<J>(g)) : 0.0f;
    qr = kr * in.c[R.p0];
    if constexpr (R.p1 >= 0) qr *= in.c[R.p1];
    q = qf - qr;
  }
  if constexpr (R.type == THIRD_BODY) q *= M;
  wdot[R.r0] -= q;
  if constexpr (R.r1 >= 0) wdot[R.r1] -= q;
  wdot[R.p0] += q;
  if constexpr (R.p1 >= 0) wdot[R.p1] += q;
  if constexpr (kDestr) {
    const float m = (R.type == THIRD_BODY) ? M : 1.0f;
    dflux[R.r0] += m * qf;
    if constexpr (R.r1 >= 0) dflux[R.r1] += m * qf;
    dflux[R.p0] += m * qr;
    if constexpr (R.p1 >= 0) dflux[R.p1] += m * qr;
  }
}

template <bool kDestr, int... J>
__device__ __forceinline__ void all_reactions_f32(const MechTables &mt, const RateInputsF &in, const GibbsF &g,
                                                  float (&wdot)[NSP], float *dflux,
                                                  std::integer_sequence<int, J...>) {
  (reaction_f32<J, kDestr>(mt, in, g, wdot, dflux), ...);
}

// What the rates need of the temperature, in fp64: T from the guess by solve_T, T, ln T and
// 1/T rounded to fp32, and the split Gibbs functions.  Out of line and rolled up (a few
// hundred instructions in all), as few cells come here and straight-line code would evict the
// main path from the instruction caches.
struct Fp64Out {
  double T;
  float2 r;
  float lnT, invT;
};
// solve_T, for what the compact Newton below leaves.
template <int ST>
static __device__ __noinline__ bool solve_T_full(const MechTables &mt, const float2 *CU, double eR, double *T) {
  double Y[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) Y[k] = f2d(CU[k * ST].y);
  return solve_T(mt, Y, eR, *T);
}
// The same Newton iteration as solve_T's (operation for operation) while the iterates stay in
// the guess's NASA-7 range; anything else goes to solve_T.
template <int ST>
static __device__ __noinline__ bool solve_gibbs_fp64(const MechTables &mt, const float2 *CU, double eR, double guess,
                                                     float2 *g, Fp64Out *out) {
  double T = pos_normal(guess) ? guess : 1500.0;
  const int range = ge_nonneg(T, mt.T_mid);
  double m[6] = {};
#pragma unroll 1
  for (int k = 0; k < NSP; ++k) {
    const double y = f2d(CU[k * ST].y);
    const double *c = mt.ecw[range][k];
#pragma unroll
    for (int i = 0; i < 6; ++i) m[i] = fma(y, c[i], m[i]);
  }
  m[5] -= eR;
  double d[5];
  cv_coef(m, d);
  bool done = false;
#pragma unroll 1
  for (int it = 0; it < 30 && !done; ++it) {
    const double dT = e_over_R(m, T) * rcp1(cv_over_R(d, T));
    T -= dT;
    if (!pos_normal(T) || ge_nonneg(T, mt.T_mid) != range) break;
    const float dTf = d2f(dT), Tf = d2f(T);
    done = fabsf(dTf) <= 1e-12f * Tf || dTf * dTf <= mt.f.newton_sq * Tf;
  }
  if (!done) {
    T = guess;
    if (!solve_T_full<ST>(mt, CU, eR, &T)) return false;
  }
  const double lnT = log_tab(T), invT = rcp1(T), oml = 1.0 - lnT;
  const int rg = ge_nonneg(T, mt.T_mid);
#pragma unroll 1
  for (int k = 0; k < NGB; ++k) {
    const double *gc = mt.gc[rg][k];
    const double gk = fma(T, fma(T, fma(T, fma(T, gc[4], gc[3]), gc[2]), gc[1]), fma(gc[5], invT, gc[6]));
    split_hilo(fma(gc[0], oml, gk), g[k * ST].x, g[k * ST].y);
  }
  split_hilo(lnT + mt.ln_R_over_Pref, out->r.x, out->r.y);
  out->T = T;
  out->lnT = d2f(lnT);
  out->invT = d2f(invT);
  return true;
}

// solve_T in double-float: T from e/R_u = eR and the fp32 mass fractions (CU.y), by Newton from
// T (in).  The mixture coefficients and the residual are double-float (error about 2^-45 of
// e), c_v is fp32: first iterations entirely in fp32 to within ~1e-4 K, then with the
// double-float residual until the remaining error (the quadratic term C dT^2 / 2 and the
// fp32 derivative's 3e-7 dT) is below 1e-13 T, a tenth of solve_T's own bound.  False, with T
// unchanged, for a guess that is not positive, a large or failing step, a root on the other
// side of the NASA-7 switch or no convergence: the caller then takes the fp64 path.
template <int ST>
__device__ __forceinline__ bool solve_T_ff(const MechTables &mt, const float2 *CU, ff eR, ff &T) {
  const int range = ge_mid(mt, T);
  ff2 m01{}, m23{}, m45{make_float2(0.0f, -eR.h), make_float2(0.0f, -eR.l)};
#pragma unroll 1
  for (int k = 0; k < NSP; ++k) {
    const float4 a = s_ecw[range][k][0], b = s_ecw[range][k][1], c = s_ecw[range][k][2];
    const float2 y = both(CU[k * ST].y);
    m01 = ff_acc(m01, ff_mul(ff2{make_float2(a.x, a.y), make_float2(a.z, a.w)}, y));
    m23 = ff_acc(m23, ff_mul(ff2{make_float2(b.x, b.y), make_float2(b.z, b.w)}, y));
    m45 = ff_acc(m45, ff_mul(ff2{make_float2(c.x, c.y), make_float2(c.z, c.w)}, y));
  }
  m01 = ff_norm(m01);
  m23 = ff_norm(m23);
  m45 = ff_norm(m45);
  const ff m[6] = {{m01.h.x, m01.l.x}, {m01.h.y, m01.l.y}, {m23.h.x, m23.l.x},
                   {m23.h.y, m23.l.y}, {m45.h.x, m45.l.x}, {m45.h.y, m45.l.y}};
  const float d1 = 2.0f * m[1].h, d2 = 3.0f * m[2].h, d3 = 4.0f * m[3].h, d4 = 5.0f * m[4].h;
  auto cv = [&](float t) {
    return __fmaf_rn(t, __fmaf_rn(t, __fmaf_rn(t, __fmaf_rn(t, d4, d3), d2), d1), m[0].h);
  };
  float t = T.h;
  bool ok = t > 0.0f, done = false;
#pragma unroll 1
  for (int it = 0; it < 8 && ok && !done; ++it) {
    const float r = __fmaf_rn(
        t, __fmaf_rn(t, __fmaf_rn(t, __fmaf_rn(t, __fmaf_rn(t, m[4].h, m[3].h), m[2].h), m[1].h), m[0].h), m[5].h);
    const float dt = __fdividef(r, cv(t));
    ok = fabsf(dt) <= 0.25f * t;
    t = fsub(t, dt);
    done = fabsf(dt) <= 2e-4f * t;
  }
  ff x{t, 0.0f};
  ok &= done;
  done = false;
#pragma unroll 1
  for (int it = 0; it < 6 && ok && !done; ++it) {
    ff r = m[4];
#pragma unroll
    for (int i = 3; i >= 0; --i) r = ff_acc(m[i], ff_mul(r, x));
    r = ff_acc(m[5], ff_mul(r, x));
    const float dt = __fdividef(fadd(r.h, r.l), cv(x.h));
    x = ff_norm(ff_acc(x, ff{-dt, 0.0f}));
    ok = fabsf(dt) <= 1e-2f * x.h;
    done = dt * dt <= 0.1f * mt.f.newton_sq * x.h && fabsf(dt) <= 3e-7f * x.h;
  }
  if (!(ok && done && ge_mid(mt, x) == range)) return false;
  T = x;
  return true;
}

// Rounding test of the exponents: the double-float sums are within ~2e-12 of the fp64
// ones, but their lo parts may round to the other neighbour on the 2^-36 grid that fp32 gives
// them (four terms, seldom more than one of them); kLnKcErr covers one of them, not several at
// once.  On an AMR batch of 3.5 M cells (65 evaluations a cell and more) 1.6e-11 leaves 110 cells
// in which some exponent is another fp32 number than from fp64 functions, 2.4e-11 40 and 4e-11 15;
// each step costs about 4 % of the kernel's time.
constexpr float kLnKcErr = 2.4e-11f;

// k_f c_r0 c_r1 - k_r c_p0 c_p1 with k_r = exp(ln k_f + ln(1 / K_c)), k_f > t else 0, given
// the four molecules' concentrations and the exponent's parts.
__device__ __forceinline__ float net_rate(float kf, float lnkf, float t, float2 x, float r0, float r1, float p0,
                                          float p1) {
  const float kr = kf > t ? expf(fadd(lnkf, fadd(x.x, x.y))) : 0.0f;
  return __fmaf_rn(-fmul(kr, p0), p1, fmul(fmul(kf, r0), r1));
}

// The exponent ln(1 / K_c) of the reaction with rows o and sum nu dn, in two parts.
template <int ST>
__device__ __forceinline__ float2 slot_exponent(int4 o, float dn, float2 rt, const MixedCols &m) {
  const char *g = reinterpret_cast<const char *>(m.G);
  auto row = [&](int off) { return *reinterpret_cast<const float2 *>(g + off); };
  return __ffma2_rn(rt, both(dn), sub2(add2(sub2(row(o.z), row(o.x)), row(o.w)), row(o.y)));
}

// The net rate of the reaction in slot i (without a third-body factor) into Q, for k_f and its
// logarithm; returns whether the exponent may round either way.
template <int ST>
__device__ __forceinline__ bool slot_rate(int i, float kf, float lnkf, float dn, float t, float2 rt, const MixedCols &m) {
  constexpr int kC = (NSP + 1) * ST * 8;  // from a row of G to the same row of CU
  const char *c = reinterpret_cast<const char *>(m.G) + kC;
  const int4 o = s_rx_row[i];
  auto conc = [&](int off) { return *reinterpret_cast<const float *>(c + off); };
  const float2 x = slot_exponent<ST>(o, dn, rt, m);
  m.Q[i * ST] = net_rate(kf, lnkf, t, x, conc(o.x), conc(o.y), conc(o.z), conc(o.w));
  return !rounds_safely(ff{x.x, x.y}, kLnKcErr);
}

__device__ __forceinline__ float ln_kf(float4 k, float lnT, float invT) {
  return __fmaf_rn(-k.z, invT, __fmaf_rn(k.y, lnT, k.x));
}

// Troe broadening of fall-off reaction f (n: parameter count).
__device__ __forceinline__ float troe_rolled(float4 p, float n, float T, float invT, float Pr) {
  const float a = p.x;
  float Fc = (1.0f - a) * expf(-T * p.y) + a * expf(-T * p.z);
  if (n == 4.0f) Fc += expf(-p.w * invT);
  const float lFc = log10f(Fc);
  const float cc = -0.4f - 0.67f * lFc;
  const float nn = 0.75f - 1.27f * lFc;
  const float x = log10f(Pr) + cc;
  const float f1 = x / (nn - 0.14f * x);
  return n == 0.0f ? 1.0f : exp10f(lFc / (1.0f + f1 * f1));
}

// Rate of progress (without the third-body factor) of fall-off reaction f (slot NRL + f) and of
// the loop's reaction i; returns whether the exponent may round either way.
template <int ST>
__device__ __forceinline__ bool falloff_rate(int f, const RateTempsF &in, const float (&M)[NM], float2 rt,
                                             const MixedCols &m) {
  const int i = NRL + f;
  const float4 k = s_rx_k[i], kk = s_rx_f[i], k0 = s_fo_k[f];
  float Mf = M[0];
#pragma unroll
  for (int q = 1; q < NFO; ++q) Mf = f == q ? M[q] : Mf;
  float kf = __fmaf_rn(expf(ln_kf(k, in.lnT, in.invT)), kk.x, kk.y);
  const float Pr = (expf(ln_kf(k0, in.lnT, in.invT)) * Mf) / kf;
  kf = (Pr > 0.0f) ? kf * (Pr / (1.0f + Pr)) * troe_rolled(s_fo_t[f], k0.w, in.T, in.invT, Pr) : 0.0f;
  return slot_rate<ST>(i, kf, logf(kf), k.w, kk.z, rt, m);
}
template <int ST>
__device__ __forceinline__ bool loop_rate(int i, float lnT, float invT, float2 rt, const MixedCols &m) {
  const float4 k = s_rx_k[i], kk = s_rx_f[i];
  const float lnkf = ln_kf(k, lnT, invT);
  return slot_rate<ST>(i, __fmaf_rn(expf(lnkf), kk.x, kk.y), lnkf, k.w, kk.z, rt, m);
}

// Every reaction's, rolled.  Returns the bits whose exponents may round either way.
template <int ST>
__device__ __forceinline__ unsigned all_rates(const RateTempsF &in, const float (&M)[NM], float2 rt, const MixedCols &m) {
  unsigned doubt = 0;
#pragma unroll 1
  for (int f = 0; f < NFO; ++f)
    if (falloff_rate<ST>(f, in, M, rt, m)) doubt |= 1u << (NRL + f);
#pragma unroll 1
  for (int i = 0; i < NRL; ++i)
    if (loop_rate<ST>(i, in.lnT, in.invT, rt, m)) doubt |= 1u << i;
  return doubt;
}
// Those of the bits in todo, out of line.
template <int ST>
static __device__ __noinline__ void some_rates(const RateTempsF *in, const float *M, float2 rt, unsigned todo) {
  const MixedCols m = mixed_cols<ST>();
  float Mr[NM];
#pragma unroll
  for (int j = 0; j < NM; ++j) Mr[j] = M[j];
#pragma unroll 1
  for (; todo; todo &= todo - 1u) {
    const int i = __ffs(todo) - 1;
    if (i < NRL) loop_rate<ST>(i, in->lnT, in->invT, rt, m);
    else falloff_rate<ST>(i - NRL, *in, Mr, rt, m);
  }
}

// The reactions' production rates from their rates of progress.
template <int J>
__device__ __forceinline__ void add_progress(float q, const float (&M)[NM], float (&wdot)[NSP]) {
  constexpr RxStruct R = kRx[J];
  if constexpr (R.type == THIRD_BODY) {
    const float m = M[m_index(J)];
    wdot[R.r0] = __fmaf_rn(-q, m, wdot[R.r0]);
    if constexpr (R.r1 >= 0) wdot[R.r1] = __fmaf_rn(-q, m, wdot[R.r1]);
    wdot[R.p0] = __fmaf_rn(q, m, wdot[R.p0]);
    if constexpr (R.p1 >= 0) wdot[R.p1] = __fmaf_rn(q, m, wdot[R.p1]);
  } else {
    wdot[R.r0] = fsub(wdot[R.r0], q);
    if constexpr (R.r1 >= 0) wdot[R.r1] = fsub(wdot[R.r1], q);
    wdot[R.p0] = fadd(wdot[R.p0], q);
    if constexpr (R.p1 >= 0) wdot[R.p1] = fadd(wdot[R.p1], q);
  }
}
template <int ST, int... J>
__device__ __forceinline__ void all_progress(const float *Q, const float (&M)[NM], float (&wdot)[NSP],
                                             std::integer_sequence<int, J...>) {
  (add_progress<J>(Q[rx_slot(J) * ST], M, wdot), ...);
}

// dY/dt (fp32) of one cell at fixed (rho, e) from the fp32 stage state (CU.y), into the
// column Q.  T: in = Newton guess, out = solved T.  Returns false when the temperature solve fails.
template <int ST>
__device__ __forceinline__ bool cell_rhs_mixed(const MechTables &mt, const MixedCols &m, float rho_f, float invRho_f,
                                               ff eR, ff &T) {
  RateTempsF in;
  const ff guess = T;
  float2 rt = make_float2(0.0f, 0.0f);  // ln(R_u T / p_ref)
  constexpr unsigned kAll = (1u << NRX) - 1u;
  const bool fast = solve_T_ff<ST>(mt, m.CU, eR, T);
  bool unsafe = false;
  if (fast) {
    const ff lnT = ff_log(T);
    const double invTd = rcp1(ff2d(T));
    in.T = T.h;
    in.lnT = lnT.h;
    in.invT = d2f(invTd);
    gibbs_hl<ST>(mt, T, lnT, d2ff(invTd), m.G, rt);
    // T within solve_T's own 1e-12 T / 2, ln T within 1e-12, 1/T as T
    const float e = 6e-13f;
    unsafe = !(rounds_safely(T, e * T.h) && rounds_safely(lnT, 1e-12f) && rounds_safely(d2ff(invTd), e * in.invT));
  }
  float ctot = 0.0f;
#pragma unroll 1
  for (int k = 0; k < NSP; ++k) {
    const float c = fmaxf(rho_f * m.CU[k * ST].y * s_w[k].x, 0.0f);
    m.CU[k * ST].x = c;
    ctot += c;
  }
  float M[NM];
#pragma unroll
  for (int j = 0; j < NM; ++j) M[j] = ctot;
#pragma unroll 1
  for (int k = 0; k < NSP; ++k) {
    const float c = m.CU[k * ST].x;
#pragma unroll
    for (int j = 0; j < NM; ++j) M[j] = __fmaf_rn(s_eff[k][j], c, M[j]);
  }
  unsigned doubt = kAll;
  if (fast) {
    doubt = all_rates<ST>(in, M, rt, m);
    if (unsafe) doubt = kAll;
  }
  if (doubt) {  // the rates in doubt, from fp64 values
    Fp64Out o;
    if (!solve_gibbs_fp64<ST>(mt, m.CU, ff2d(eR), ff2d(guess), m.G, &o)) return false;
    T = ff_norm(d2ff(o.T));
    RateTempsF in2;
    in2.T = d2f(o.T);
    in2.lnT = o.lnT;
    in2.invT = o.invT;
    float M2[NM];
#pragma unroll
    for (int j = 0; j < NM; ++j) M2[j] = M[j];
    some_rates<ST>(&in2, M2, o.r, doubt);
  }
  float wdot[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) wdot[k] = 0.0f;
  all_progress<ST>(m.Q, M, wdot, std::make_integer_sequence<int, NRX>{});
#pragma unroll
  for (int k = 0; k < NSP; ++k) m.Q[k * ST] = wdot[k] * s_w[k].y * invRho_f;
  return true;
}

// Temperature from e/R_u and Y/W entirely in fp32 (for the error test): Newton from T
// (1500 K if not positive and finite), |dT| <= 2e-6 T within 12 iterations; false on
// no convergence or a non-positive / non-finite iterate (the test then rejects).
__device__ __forceinline__ bool solve_T_f32(const MechTables &mt, const float (&yw)[NSP], float eR, float &T) {
  float Tn = (isfinite(T) && T > 0.0f) ? T : 1500.0f;
  int range = -1;
  float m[6], d[5];
  for (int it = 0; it < 12; ++it) {
    const int r = Tn >= mt.f.T_mid;
    if (r != range) {
      range = r;
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        float s = 0.0f;
#pragma unroll
        for (int k = 0; k < NSP; ++k) s = fmaf(yw[k], mt.f.ec[range][k][i], s);
        m[i] = s;
      }
      d[0] = m[0];
      d[1] = 2.0f * m[1];
      d[2] = 3.0f * m[2];
      d[3] = 4.0f * m[3];
      d[4] = 5.0f * m[4];
    }
    const float eT = fmaf(Tn, fmaf(Tn, fmaf(Tn, fmaf(Tn, fmaf(Tn, m[4], m[3]), m[2]), m[1]), m[0]), m[5]);
    const float cv = fmaf(Tn, fmaf(Tn, fmaf(Tn, fmaf(Tn, d[4], d[3]), d[2]), d[1]), d[0]);
    const float dT = __fdividef(eT - eR, cv);
    Tn -= dT;
    if (!isfinite(Tn) || Tn <= 0.0f) return false;
    if (fabsf(dT) <= 2e-6f * Tn) {
      T = Tn;
      return true;
    }
  }
  return false;
}

// dY/dt of one cell entirely in fp32 (temperature, Gibbs functions and ln(1/K_c)
// included) with the fast intrinsics: the right-hand side of the surrogate's error test and of
// the stiffness key, estimators that need relative accuracy far coarser than fp32's.  T: in =
// guess, out = solved T.  kDestr: also the consumption rates per unit concentration, D (0
// where there is nothing to consume).
template <bool kDestr = false>
__device__ __forceinline__ bool cell_rhs_f32(const MechTables &mt, const float (&U)[NSP], float rho,
                                             float invRho, float eR, float &T, float (&F)[NSP], float *D = nullptr) {
  float yw[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) yw[k] = U[k] * mt.f.invW[k];
  if (!solve_T_f32(mt, yw, eR, T)) return false;
  const float lnT = __logf(T);
  const float invT = __fdividef(1.0f, T);
  GibbsF g;
  gibbs_f(mt, T, lnT, invT, g);
  RateInputsF in;
  in.lnT = lnT;
  in.invT = invT;
  in.T = T;
  float ctot = 0.0f, wdot[NSP];
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    in.c[k] = fmaxf(rho * yw[k], 0.0f);
    ctot += in.c[k];
    wdot[k] = 0.0f;
    if constexpr (kDestr) D[k] = 0.0f;
  }
  in.ctot = ctot;
  all_reactions_f32<kDestr>(mt, in, g, wdot, D, std::make_integer_sequence<int, NRX>{});
#pragma unroll
  for (int k = 0; k < NSP; ++k) {
    F[k] = wdot[k] * mt.f.W[k] * invRho;
    if constexpr (kDestr) D[k] = in.c[k] > 1e-30f ? __fdividef(D[k], in.c[k]) : 0.0f;
  }
  return true;
}

}  // namespace chem
