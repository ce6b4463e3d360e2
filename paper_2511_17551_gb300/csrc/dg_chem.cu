// Finite-rate chemistry source on the device (appendix, Chemical Kinetics: Eqs. nrp,
// forward_rate, backward, kedef, calc_prod), one thread per node: in FP64 in the FP64 form
// (chem_node); in the mixed form (chem_node_dd) the thermodynamics in FP64 and the kinetics in
// double-FP32 pairs, the source rounded to FP32.
//
// Concentrations c_s = 1e-6 rho_s / W_s (mol/cm^3, the units of Park-type constants);
// k_f = exp(ln A + beta ln T - theta/T); k_b = k_f / K_c with
// ln K_c = -sum dnu_s g_s/(R_u T) + (sum dnu_s) ln(1e-6 p0 / (R_u T)), p0 = 101325 Pa,
// g/(RT) = h/(RT) - s/R from each species' polynomial; rate of progress
// R_r = (k_f prod c^nu' - k_b prod c^nu'') (times sum eff_s c_s for third-body steps);
// omega_s = 1e6 W_s sum_r dnu_sr R_r (kg/m^3/s); point-implicit source
// S_s = omega_s / (1 + dt max(0, -d omega_s/d rho_s)) with the analytic diagonal
// Jacobian at fixed T, dt = the running RK step (0 outside RK stepping).
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

#include "../../include/dg.h"
#include "dg_dd.cuh"
#include "dg_internal.h"
#include "dg_launch.cuh"
#include "dg_mlp.cuh"
#include "dg_mlp_tc5.cuh"
#include "dg_thermo.h"

#define NSPEC 5
#define DG_RU 8.314462618
#define DG_P0 101325.0

namespace {

// Device tables (built by dg_chem_init from the species and reaction arrays):
// species rows [16]: 1e-6/W, 1e6 W, g/(RT) = h/(RT) - s/R as the coefficients of 1, T, T^2,
//   T^3, T^4 (from a1..a5 and a7), the 1/T coefficient a6 and the ln T coefficient a1,
//   1e-6 p0 / R_u and its reciprocal, slots 11-13 unused, ln(1e-6 p0 / R_u), 0;
// reaction rows [32]: nu'(5), nu''(5), third_body, eff(5), ln A, beta, theta,
//   dn = sum dnu, dnu(5), then (slot 25, as raw bits) the integer form of the row, and
//   dnu_s eff_s (5, slots 26-30); the integer form holds 2 bits
//   per species of nu' in {0..3} (bits 0-9) and nu'' (bits 10-19), the third-body flag (bit 20) and
//   one bit per species with dnu != 0 (bits 21-25), and, where k_b may be formed as a product
//   (sum |dnu_s| <= 15 and |dn| <= 3), sum |dnu_s| (bits 26-29) with bit 30 set.  The
//   integer form drives the uniform
//   branches of the reaction loop, so that no FP64 compare or conversion is spent on them.
#define SP_W 16
#define RX_W 32
#define RX_META 25

// c^nu for the stoichiometric coefficients nu in {1, 2, 3} (c2 = c c)
__device__ __forceinline__ double pow123(int nu, double c, double c2) {
  return nu == 1 ? c : (nu == 2 ? c2 : c2 * c);
}

// x^n for n in {-3..3} \ {0} from x and 1/x
__device__ __forceinline__ double ipow_pm3(int n, double x, double xi) {
  const double b = n > 0 ? x : xi;
  const int m = n > 0 ? n : -n;
  return m == 1 ? b : (m == 2 ? b * b : b * b * b);
}

// Plain FP64 source at one node: omega_s (kg/m^3/s) and the point-implicit terms
// jpi_s = max(0, -d omega_s / d rho_s) of the analytic diagonal Jacobian at fixed T.
// uu points at the node's first species density, stride np between variables.
// The Jacobian of reaction r with respect to c_s is M (nu'_s pf - nu''_s pb) / c_s plus, for
// third-body reactions, eff_s (pf - pb); the first part is summed over the reactions and
// divided by c_s once after the loop (c_s > 0), the explicit products are kept for c_s = 0.
template <typename T>
__device__ __forceinline__ void chem_node(const T* uu, int np, double Tk, const double* sp,
                                          const double* reac, int nr, double* om, double* jpi) {
  const double lnT = log(Tk), iT = 1.0 / Tk;
  // ln(1e-6 p0 / (R_u T)) = ln(1e-6 p0 / R_u) - ln T (the constant sits in species row 0)
  const double lnP = sp[14] - lnT;
  double c[NSPEC], c2[NSPEC], g[NSPEC], jd[NSPEC], j1[NSPEC];
  bool pos[NSPEC];
  double gmax = 0.0;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    const double* q = sp + SP_W * s;
    c[s] = q[0] * (double)uu[s * np];
    c2[s] = c[s] * c[s];
    pos[s] = c[s] > 0.0;
    // g/(RT) = h/(RT) - s/R as one polynomial in T plus the 1/T and ln T terms
    g[s] = q[2] + Tk * (q[3] + Tk * (q[4] + Tk * (q[5] + Tk * q[6]))) + q[7] * iT - q[8] * lnT;
    gmax = fmax(gmax, fabs(g[s]));
    om[s] = 0.0;
    jd[s] = 0.0;
    j1[s] = 0.0;
  }
  // k_b = k_f X with X = exp(sum dnu_s g_s) P^-dn, P = 1e-6 p0 / (R_u T): from E_s = exp(g_s)
  // taken once per node, X is a product of powers of E_s, 1/E_s and P.  A reaction takes it
  // when every partial product stays inside the double range: sum |dnu_s| max|g_s| < 650
  // (the integer gcap bounds sum |dnu_s|; |P^-dn| adds at most e^42 for |dn| <= 3 and
  // 200 K <= T <= 10^4 K) and k_f is a normal number; otherwise one exp of the whole exponent.
  double E[NSPEC], Ei[NSPEC];
  const double P = sp[9] * iT, Pi = Tk * sp[10];
  const int gcap = gmax < 650.0 ? (gmax > 0.0 ? (int)fmin(650.0 / gmax, 64.0) : 64) : 0;
  if (gcap) {
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      E[s] = exp(g[s]);
      Ei[s] = 1.0 / E[s];
    }
  }
#pragma unroll 1
  for (int r = 0; r < nr; ++r) {
    const double* row = reac + RX_W * r;
    const int meta = (int)__double_as_longlong(row[RX_META]);
    const double lnkf = row[16] + row[17] * lnT - row[18] * iT;
    const double kf = exp(lnkf);
    double kb;
    // bits 26-29: sum |dnu_s|; bit 30: |dn| <= 3 (set at init)
    if ((meta >> 30) & 1 && ((meta >> 26) & 15) <= gcap && lnkf > -700.0) {
      double X = 1.0;
      int dn = 0;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) {
        const int ds = ((meta >> (10 + 2 * s)) & 3) - ((meta >> (2 * s)) & 3);
        dn += ds;
        if (ds) X *= ipow_pm3(ds, E[s], Ei[s]);
      }
      if (dn) X *= ipow_pm3(-dn, P, Pi);
      kb = kf * X;
    } else {
      double dg = 0.0;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s)
        if (meta & (1 << (21 + s))) dg += row[20 + s] * g[s];
      kb = exp(lnkf + dg - row[19] * lnP);
    }
    double pf = kf, pb = kb;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      const int a = (meta >> (2 * s)) & 3, b = (meta >> (10 + 2 * s)) & 3;
      if (a) pf *= pow123(a, c[s], c2[s]);
      if (b) pb *= pow123(b, c[s], c2[s]);
    }
    double M = 1.0;
    const bool tb = meta & (1 << 20);
    if (tb) {
      M = 0.0;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) M += row[11 + s] * c[s];
    }
    const double dp = pf - pb, Rr = dp * M;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      if (!(meta & (1 << (21 + s)))) continue;  // the same for every node: no divergence
      const double d = row[20 + s];
      om[s] += d * Rr;
      if (tb) jd[s] += row[26 + s] * dp;  // dnu_s eff_s (pf - pb)
      const int a = (meta >> (2 * s)) & 3, b = (meta >> (10 + 2 * s)) & 3;
      if (!(a | b)) continue;
      if (pos[s]) {
        // nu'_s pf - nu''_s pb (the stoichiometric coefficients are exact small integers)
        const double t = row[s] * pf - row[5 + s] * pb;
        j1[s] += (tb ? d * M : d) * t;
      } else {
        // c_s = 0: the explicit products for nu = 1 (higher powers have zero derivative)
        double dpf = 0.0, dpb = 0.0;
        if (a == 1) {
          dpf = kf;
#pragma unroll
          for (int q = 0; q < NSPEC; ++q)
            if (q != s) {
              const int aq = (meta >> (2 * q)) & 3;
              if (aq) dpf *= pow123(aq, c[q], c2[q]);
            }
        }
        if (b == 1) {
          dpb = kb;
#pragma unroll
          for (int q = 0; q < NSPEC; ++q)
            if (q != s) {
              const int bq = (meta >> (10 + 2 * q)) & 3;
              if (bq) dpb *= pow123(bq, c[q], c2[q]);
            }
        }
        jd[s] += d * (dpf - dpb) * M;
      }
    }
  }
  // omega in kg/(m^3 s); d omega_s / d rho_s = 1e6 W_s (1e-6 / W_s) d(...)/dc_s = jd_s
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    if (pos[s]) jd[s] += j1[s] / c[s];
    om[s] *= sp[SP_W * s + 1];
    jpi[s] = -jd[s] > 0.0 ? -jd[s] : 0.0;
  }
}

// element and node of a global node index; the 64-bit division (about 70 instructions) only
// where the index needs it
__device__ __forceinline__ void split_node(int64_t i, int np, int64_t& k, int& node) {
  if (i >> 32) {
    k = i / np;
    node = (int)(i - k * np);
  } else {
    const unsigned q = (unsigned)i / (unsigned)np;
    k = q;
    node = (int)((unsigned)i - q * (unsigned)np);
  }
}

// ------------------------------------------------------------------ mixed form
// Tables of the double-FP32 evaluation (pairs): the same numbers as the FP64 rows above, passed
// by value so that they sit in the constant bank (uniform loads and branches; as a table in
// shared memory the loop spent a quarter of its issue slots on loading and decoding it).
constexpr int MAXR = 64;
constexpr int SCALE2 = 60;  // rates are carried times 2^60 (see chem_node_dd)
struct ChemRow32 {
  dgdd::dd lnA, beta, mtheta, eff[NSPEC];
  // nu'_s, dnu_s, and the factors of r_f and r_b in the Jacobian, nu'_s dnu_s and -nu''_s dnu_s
  float nf[NSPEC], dn[NSPEC], jf[NSPEC], jb[NSPEC];
  // bits s, 5 + s, 10 + s, 15 + s: these are not zero; bit 20: third body
  int mask;
  // bits s: nu''_s > 0; 5 + s, 10 + s: nu'_s, nu''_s odd; 15 + s, 20 + s: nu'_s, nu''_s one
  int mask2;
  double dn64[NSPEC];
};
struct ChemTab32 {
  dgdd::dd cw[NSPEC], ow[NSPEC];     // 1e-6 / W; 1e6 W 2^-60
  ChemRow32 row[MAXR];
  int n;                             // rows; reactions switched off (A = 0) are left out
};
static_assert(sizeof(ChemTab32) < 16 * 1024, "a kernel argument");

// The rates of chem_node with the thermodynamics in FP64 and the kinetics in double-FP32 pairs
// (48 bits; the source is rounded to FP32's 24 afterwards).  FP32 has no room for the exponents of
// k_f, k_b and the concentration products, so the two rates of a reaction are formed from their
// logarithms,
//   ln r_f = ln k_f + sum nu'_s ln c_s,   ln r_b = ln r_f + delta,   delta = sum dnu_s w_s,
//   w_s = g_s/(R T) + ln c_s - ln(1e-6 p0 / (R_u T)),
// and carried times 2^60: rates from 2^-160 mol/cm^3/s (flushed to zero below: their source
// is below FP32's range) to 2^66.  Near equilibrium r_f and r_b cancel to -r_f (e^delta - 1): delta is a
// difference of numbers up to 100, so w and delta stay in FP64, and where |delta| < 1/16 the
// difference comes from delta itself.  Measured against FP64 on states with rates from cold to 9000 K
// and after 50 steps: the same relative L2 to three digits (2.5e-8, the rounding of the result).
// What bounds it: about 200 FP64 operations and 8,000 others per node, on two pipes; 1,063 FP64
// operations before.  4.6 M nodes: 10.17 -> 2.28 ms, and 1.74 ms since the conversions to and from
// pairs are integer work (as instructions they took a quarter of the FP64 pipe's time).  All of it in
// pairs, logarithms, g and delta too, missed the FP64 source by a tenfold larger maximum near
// equilibrium.
//
// GEN = false holds where every concentration lies between 1e-24 and 1e6 mol/cm^3.  GEN = true takes
// absent species (c = 0), negative ones (overshoots next to a front) and concentrations down to
// 9e-43 mol/cm^3 as well: ln |c_s| (of 2^60 |c_s| where |c_s| < 1e-24), 0 for an absent species, so that
// the exponentials give the products without it; a direction that consumes an absent species has
// rate zero, a negative species gives its sign by the parity of nu, and for both the derivative
// is the explicit product without c_s for nu = 1 and zero for higher powers, as in chem_node.  For
// other species the values are those of GEN = false.
// Returns false where the pairs do not hold (other concentrations, or a result that is not
// finite).
template <bool GEN>
__device__ __forceinline__ bool chem_node_dd(const float* uu, int np, double Td, const ChemTab32& t,
                                             const dgdd::dd* exp2, const double* sp, dgdd::dd* om, dgdd::dd* jpi) {
  using namespace dgdd;
  constexpr float UP = 1152921504606846976.0f;  // 2^60
  dd c[NSPEC], lc[NSPEC], jd[NSPEC], j1[NSPEC];
  double w[NSPEC];
  int none = 0, minus = 0, tiny = 0;  // GEN: bit s of an absent, a negative, a scaled species
  bool ok = true;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    const float us = uu[s * np];
    c[s] = mul(t.cw[s], GEN ? fabsf(us) : us);
    if (GEN) {
      if (us < 0.f) minus |= 1 << s;
      if (us == 0.f) {
        none |= 1 << s;
        c[s] = make(1.f, 0.f);
      } else if (c[s].h < 1e-24f) {
        tiny |= 1 << s;
        c[s] = mul(make(t.cw[s].h * UP, t.cw[s].l * UP), fabsf(us));
      }
    }
    ok = ok && c[s].h >= 1e-24f && c[s].h <= 1e6f;
  }
  if (!ok) return false;
  // (ln T is multiplied by the species' a1 in g: the FP64 logarithm; ln c_s good to 2^-45)
  const double lnTd = log(Td), iTd = 1.0 / Td, mlnP = lnTd - sp[14];
  const dd lnT = from_double(lnTd), iT = from_double(iTd);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    const double* q = sp + SP_W * s;
    double l;
    lc[s] = log_(c[s], exp2, &l);
    if (GEN && (tiny >> s & 1)) {
      constexpr double ln_up = 60.0 * 0.69314718055994530942;
      lc[s] = add(lc[s], make(-(float)ln_up, -(float)(ln_up - (double)(float)ln_up)));
      l -= ln_up;
    }
    w[s] = (q[2] + Td * (q[3] + Td * (q[4] + Td * (q[5] + Td * q[6]))) + q[7] * iTd - q[8] * lnTd) + l + mlnP;
    om[s] = jd[s] = j1[s] = make(0.f, 0.f);
  }
#pragma unroll 1
  for (int r = 0; r < t.n; ++r) {
    const ChemRow32& row = t.row[r];
    const int mask = row.mask;  // the same for every node: no divergence below
    double dl = 0.0;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s)
      if (mask & (1 << (5 + s))) dl += row.dn64[s] * w[s];
    dd tf = row.lnA;
    acc_mul(tf, row.beta, lnT);
    acc_mul(tf, row.mtheta, iT);
#pragma unroll
    for (int s = 0; s < NSPEC; ++s)
      if (mask & (1 << s)) acc_mul(tf, lc[s], row.nf[s]);
    const dd delta = from_double(dl);
    tf = norm(tf);
    dd pf = exp_scaled(tf, SCALE2, exp2);
    dd pb = exp_scaled(add(tf, delta), SCALE2, exp2), dp = add(pf, neg(pb));
    if (fabsf(delta.h) < 0.0625f) {
      dp = neg(mul(pf, expm1_small(delta)));
      pb = add(pf, neg(dp));
    }
    // GEN: pf and pb are the products over the species that are there; their signs, 0 where a
    // species of theirs is absent
    float sf = 1.f, sb = 1.f;
    const dd qf = pf, qb = pb;
    if (GEN) {
      if (__popc(minus & row.mask2 >> 5) & 1) sf = -1.f;
      if (__popc(minus & row.mask2 >> 10) & 1) sb = -1.f;
      pf = none & mask & 31 ? make(0.f, 0.f) : make(sf * qf.h, sf * qf.l);
      pb = none & row.mask2 & 31 ? make(0.f, 0.f) : make(sb * qb.h, sb * qb.l);
      if (none & (mask | row.mask2) & 31 || sf != sb || sf < 0.f)
        dp = none & (mask | row.mask2) & 31 || sf != sb ? add(pf, neg(pb)) : neg(dp);
    }
    dd Rr = dp, pfM = pf, pbM = pb, M = make(1.f, 0.f);
    if (mask & (1 << 20)) {
      // (GEN: the concentrations themselves; adding a zero changes nothing)
      auto conc = [&](int s) {
        if (!GEN) return c[s];
        const float f = none >> s & 1 ? 0.f : (minus >> s & 1 ? -1.f : 1.f) * (tiny >> s & 1 ? 1.f / UP : 1.f);
        return make(f * c[s].h, f * c[s].l);
      };
      M = mul(row.eff[0], conc(0));
#pragma unroll
      for (int s = 1; s < NSPEC; ++s) acc_mul(M, row.eff[s], conc(s));
      M = norm(M);
      Rr = mul(dp, M);
      pfM = mul(pf, M);
      pbM = mul(pb, M);
#pragma unroll
      for (int s = 0; s < NSPEC; ++s)
        if (mask & (1 << (5 + s))) acc_mul(jd[s], mul(row.eff[s], dp), row.dn[s]);
    }
    // dnu_s (nu'_s r_f - nu''_s r_b) M goes to j1, divided by c_s after the loop; one of nu'_s and
    // nu''_s is mostly zero
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      if (mask & (1 << (5 + s))) acc_mul(om[s], Rr, row.dn[s]);
      if (mask & (1 << (10 + s))) acc_mul(j1[s], pfM, row.jf[s]);
      if (mask & (1 << (15 + s))) acc_mul(j1[s], pbM, row.jb[s]);
    }
    if (GEN) {  // absent and negative species: the explicit products (j1 is not used for them)
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) {
        const int b = 1 << s;
        if (!((none | minus) & mask >> 5 & b)) continue;
        dd e = make(0.f, 0.f);
        const float up = tiny & b ? -UP : -1.f;  // 1 / c_s = up / |scaled c_s|
        if (row.mask2 >> 15 & b && !(none & mask & 31 & ~b)) {
          const dd q = none & b ? make(sf * qf.h, sf * qf.l) : div(pf, c[s]);
          e = none & b ? q : make(up * q.h, up * q.l);
        }
        if (row.mask2 >> 20 & b && !(none & row.mask2 & 31 & ~b)) {
          const dd q = none & b ? make(sb * qb.h, sb * qb.l) : div(pb, c[s]);
          e = add(e, none & b ? neg(q) : make(-up * q.h, -up * q.l));
        }
        acc_mul(jd[s], mul(e, M), row.dn[s]);
      }
    }
  }
  const float down = bits((uint32_t)(127 - SCALE2) << 23);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    om[s] = mul(norm(om[s]), t.ow[s]);
    dd j = norm(jd[s]);
    if (!GEN) {
      j = add(j, div(norm(j1[s]), c[s]));
    } else if (!((none | minus) >> s & 1)) {
      const dd q = div(norm(j1[s]), c[s]);
      const float up = tiny >> s & 1 ? UP : 1.f;
      j = add(j, make(up * q.h, up * q.l));
    }
    ok = ok && isfinite(om[s].h) && isfinite(j.h);
    jpi[s] = j.h < 0.f ? make(fmul(-j.h, down), fmul(-j.l, down)) : make(0.f, 0.f);
  }
  return ok;
}

// the FP64 evaluation of a mixed-form node that the pairs cannot hold
__device__ __noinline__ void chem_node_rare(const float* uu, int np, double Tk, const double* sp, const double* reac,
                                            int nr, dgdd::dd* om, dgdd::dd* jpi) {
  double o[NSPEC], j[NSPEC];
  chem_node<float>(uu, np, Tk, sp, reac, nr, o, j);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {  // (subnormals kept)
    split_f64(o[s], om[s].h, om[s].l);
    split_f64(j[s], jpi[s].h, jpi[s].l);
  }
}

// a node outside the usual range of concentrations.  A function of its own, so that the kernels keep
// the registers of the usual case.  576,000 nodes, one of five species absent everywhere: 346 us (all
// present: 237; every node in FP64: 1,274); absent in every second node, so that a warp runs both, 640.
__device__ __noinline__ void chem_node_general(const float* uu, int np, double Tk, const ChemTab32& t,
                                               const dgdd::dd* exp2, const double* sp, const double* reac, int nr,
                                               dgdd::dd* om, dgdd::dd* jpi) {
  if (!chem_node_dd<true>(uu, np, Tk, t, exp2, sp, om, jpi)) chem_node_rare(uu, np, Tk, sp, reac, nr, om, jpi);
}

// The plain source of one node in the two forms: the rates in the form's arithmetic, and
// S_s = omega_s / (1 + dt jpi_s) rounded to the form.  Every kernel that evaluates the plain
// source for a step goes through these, so that they agree bit for bit (the training samples of
// chem_sample_kernel are FP64 in both forms).
struct Chem64 {  // FP64 form
  struct Tab {};
  struct Args {};  // the pairs' table is no argument of this form's kernels
  double om[NSPEC], jpi[NSPEC];
  __device__ __forceinline__ static void stage(Tab&, const dgdd::dd*) {}
  __device__ __forceinline__ void rates(const double* uu, int np, double Tk, const Tab&, const Args&,
                                        const double* sp, const double* reac, int nr) {
    chem_node<double>(uu, np, Tk, sp, reac, nr, om, jpi);
  }
  __device__ __forceinline__ double source(int s, double dt) const { return om[s] / (1.0 + dt * jpi[s]); }
};
struct Chem32 {  // mixed form
  typedef ChemTab32 Args;
  struct Tab {
    dgdd::dd exp2[dgdd::EXP_TAB];  // 2^(j/128), in shared memory
  };
  dgdd::dd om[NSPEC], jpi[NSPEC];
  __device__ __forceinline__ static void stage(Tab& t, const dgdd::dd* src) {
    for (int j = threadIdx.x; j < dgdd::EXP_TAB; j += blockDim.x) t.exp2[j] = src[j];
    __syncthreads();
  }
  __device__ __forceinline__ void rates(const float* uu, int np, double Tk, const Tab& e, const ChemTab32& t,
                                        const double* sp, const double* reac, int nr) {
    if (!chem_node_dd<false>(uu, np, Tk, t, e.exp2, sp, om, jpi)) {
      dgdd::dd o[NSPEC], j[NSPEC];
      chem_node_general(uu, np, Tk, t, e.exp2, sp, reac, nr, o, j);
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) {
        om[s] = o[s];
        jpi[s] = j[s];
      }
    }
  }
  __device__ __forceinline__ float source(int s, dgdd::dd dt) const {
    using namespace dgdd;
    return div(om[s], mul_add(dt, jpi[s], make(1.f, 0.f))).h;
  }
};
template <typename T> struct ChemForm;
template <> struct ChemForm<double> { typedef Chem64 type; typedef double step; };
template <> struct ChemForm<float> { typedef Chem32 type; typedef dgdd::dd step; };
template <typename T> using ChemArgs = typename ChemForm<T>::type::Args;
// (Launch bounds of the kernels below: the FP64 instances are held to 168 registers, three CTAs of 128 on
// an SM; unbounded they took 178 to 186 and two: plain 1,255 -> 1,247 us at 576,000 nodes, refreshes
// 1,309 -> 1,280.)
__device__ __forceinline__ void form_step(double dt, double& out) { out = dt; }
__device__ __forceinline__ void form_step(double dt, dgdd::dd& out) { out = dgdd::from_double(dt); }

template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 6 : 3)
chem_kernel(const T* u, const double* Tc, int64_t K, int np, int dim, const double* sp_raw, const double* reac,
            int nr, const __grid_constant__ ChemArgs<T> tab, const dgdd::dd* exp2, const double* dtp, T* src) {
  typedef typename ChemForm<T>::type Form;
  __shared__ typename Form::Tab t;
  Form::stage(t, exp2);
  pdl_wait();
  if (sizeof(T) == 4) pdl_trigger();
  const int nv = NSPEC + dim + 1;
  typename ChemForm<T>::step dt;
  form_step(dtp ? *dtp : 0.0, dt);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < K * np;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t k;
    int node;
    split_node(i, np, k, node);
    Form f;
    f.rates(u + k * nv * np + node, np, Tc[i], t, tab, sp_raw, reac, nr);
    T* so = src + k * NSPEC * np + node;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) so[s * np] = f.source(s, dt);
  }
}

// ------------------------------------------------------------------ learned source
// Surrogate of (omega, jpi): 7 -> 64 -> 64 -> 10 perceptron on standardised features
// (Y_1..Y_5, ln rho, T); outputs are the standardised asinh images
// z_s = asinh(omega_s / omega_ref), z_{5+s} = asinh(jpi_s / jpi_ref).
// Acceptance, per tile of 32 nodes (one warp): every node inside the training box, every
// node's raw rates mass-balanced (|sum omega| <= tol_mass sum|omega| + floor), every
// node's learned update positive (rho_s + dt S_s >= 0), and one sampled node per tile
// (moved each call) within tol_check of the plain source; otherwise the tile's source
// is recomputed plainly.  Accepted rates are projected onto exact mass balance:
// omega_s -= |omega_s| sum(omega) / sum|omega|.
// With a refresh period (plain correction): a refresh evaluation takes the plain source at
// every node and stores, per node, the plain rates minus the network's decoded ones; the
// evaluations until the next refresh add those differences to the decoded rates before the
// tests, so the corrected network is exact at the refresh state.
struct DgChemStats {
  float mean[7], inv_std[7], muY[10], sdY[10], lo[7], hi[7];
  float w_ref, j_ref, tol_mass, floor32;
};
struct __align__(16) DgChemMlp {
  DgMlpW<10> w;
  DgChemStats st;
  double tol_check, floor;
};
constexpr int CHEM_NR = 1;  // rows per thread of the tile engine (the decode needs the registers)

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// raw features of one node: Y_1..Y_5, ln rho, T, each rounded to FP32 once
template <typename T>
__device__ __forceinline__ void chem_features(const T* uu, int np, double Tk, const dgdd::dd*, float* x) {
  double r[NSPEC], rho = 0.0;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    r[s] = (double)uu[s * np];
    rho += r[s];
  }
  const double ir = 1.0 / rho;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) x[s] = (float)(r[s] * ir);
  x[5] = (float)log(rho);
  x[6] = (float)Tk;
}
// the mixed form's in pairs (tab: the table of exp_scaled): one FP64 logarithm and division per
// node took half of the network kernel's time
__device__ __forceinline__ void chem_features(const float* uu, int np, double Tk, const dgdd::dd* tab, float* x) {
  using namespace dgdd;
  float r[NSPEC];
  dd rho = make(0.f, 0.f);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    r[s] = uu[s * np];
    acc(rho, make(r[s], 0.f));
  }
  rho = norm(rho);
  if (!(rho.h > 1e-30f && rho.h < 1e30f)) {  // out of the pairs' range
    chem_features<float>(uu, np, Tk, tab, x);
    return;
  }
  const dd ir = rcp(rho);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) x[s] = mul(ir, r[s]).h;
  x[5] = log_(rho, tab).h;
  x[6] = (float)Tk;
}

// sinh(z): its Taylor series to z^9 below 1 (the next term is under 3e-8 of it), (e^a - e^-a) / 2
// above; half the instructions of sinhf, whose branches both run in a mixed warp
__device__ __forceinline__ float sinh_pair(float z) {
  const float a = fabsf(z), a2 = a * a;
  const float lo = a + a * a2 * (1.f / 6.f + a2 * (1.f / 120.f + a2 * (1.f / 5040.f + a2 * (1.f / 362880.f))));
  const float E = expf(a);
  const float hi = 0.5f * E - __fdividef(0.5f, E);
  return copysignf(a < 1.f ? lo : hi, z);
}

// the node of tile t that evaluation `call` checks
__device__ __forceinline__ int64_t sampled_node(int64_t t, int64_t total, uint64_t call) {
  const int64_t in_tile = total - t * 32 < 32 ? total - t * 32 : 32;
  return t * 32 + (int64_t)(splitmix64(call * 0x100000001B3ull + (uint64_t)t) % (uint64_t)in_tile);
}

// The learned source on the fifth-generation tensor cores: CTAs of 128 threads take
// 128-node tiles through the tcgen05 tile engine (dg_mlp_tc5.cuh); each thread forms its
// node's features (and the trust-box test) before the two tensor-core layers and decodes
// its node's ten outputs after them (species sources, mass-balance test).  Flags per
// 32-node (warp) tile: 0 accepted, 1 rejected; a tile whose tensor-core waits ran out is
// rejected too, so the plain fallback recomputes it.
// corr ([10][K np], FP32) with cmode 1: the decoded rates are corrected by the stored
// plain-minus-network differences before the tests (omega_s + c_s, max(0, jpi'_s + c_5+s));
// cmode 2 (refresh): only the decoded rates (jpi' before its clamp) are written to corr,
// for chem_refresh_kernel to turn into corrections.
// The first `checks` CTAs of the grid evaluate the plain source at every tile's sampled node
// instead (one thread per tile, S into `sampled`) for the next kernel to compare with: a chain
// of one evaluation that fills a fraction of the GPU (28 us as a kernel of its own at 18,000
// tiles) runs beside the network.  In the FP64 form there are none (checks = 0): both sides need the
// FP64 pipe, so nothing is hidden, and tiles that the other tests reject would be evaluated too (18,000
// tiles: all accepted 235 against 220 us, all rejected 1,439 against 1,368).
template <typename T>
__global__ void __launch_bounds__(dgtc5::THREADS, sizeof(T) == 4 ? 5 : 3)
chem_mlp_tc5_kernel(const T* u, const double* Tc, int64_t K, int np, int dim, const double* sp_raw,
                    const double* reac, int nr, const __grid_constant__ ChemArgs<T> tab, const dgdd::dd* exp2,
                    const DgChemMlp* mlp, const double* dtp, T* src, unsigned char* flags, float* corr,
                    const unsigned char* trust, int cmode, int checks, T* sampled, uint64_t call,
                    unsigned long long* stats) {
  typedef typename ChemForm<T>::type Form;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int nv = NSPEC + dim + 1;
  const int64_t total = K * np;
  // behind the wait for the preceding kernel; tables and weights, which no kernel writes, come before it
  auto enter = [&]() {
    pdl_wait();
    if (cmode != 2 && blockIdx.x == 0 && threadIdx.x == 0) stats[2] = 0;  // chem_fallback_kernel's tile counter
  };
  if (sizeof(T) == 4 && (int)blockIdx.x < checks) {
    typename Form::Tab& tb = *reinterpret_cast<typename Form::Tab*>(smem_raw);
    Form::stage(tb, exp2);
    enter();
    const int64_t t = blockIdx.x * (int64_t)dgtc5::THREADS + threadIdx.x;
    if (t * 32 >= total || (cmode == 1 && !trust[t])) return;
    typename ChemForm<T>::step dt;
    form_step(dtp ? *dtp : 0.0, dt);
    int64_t k;
    int node;
    const int64_t i = sampled_node(t, total, call);
    split_node(i, np, k, node);
    Form f;
    f.rates(u + k * nv * np + node, np, Tc[i], tb, tab, sp_raw, reac, nr);
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) sampled[NSPEC * t + s] = f.source(s, dt);
    return;
  }
  dgtc5::Smem<10, CHEM_NR>& s = *reinterpret_cast<dgtc5::Smem<10, CHEM_NR>*>(smem_raw);
  dgtc5::alloc_tmem<10, CHEM_NR>(s);
  __shared__ DgChemStats m;
  __shared__ dgdd::dd e2[sizeof(T) == 4 ? dgdd::EXP_TAB : 1];
  if (threadIdx.x < sizeof(m) / 4)
    reinterpret_cast<int*>(&m)[threadIdx.x] = reinterpret_cast<const int*>(&mlp->st)[threadIdx.x];
  if (sizeof(T) == 4)
    for (int j = threadIdx.x; j < dgdd::EXP_TAB; j += dgtc5::THREADS) e2[j] = exp2[j];
  dgtc5::load_weights<10, CHEM_NR>(s, mlp->w);
  enter();
  __syncthreads();
  const float dt = dtp ? (float)*dtp : 0.f;
  auto prod = [&](int64_t i, float* x, int) {
    float raw[7];
    bool ok = true;
    if (i < total) {
      int64_t k;
      int node;
      split_node(i, np, k, node);
      chem_features(u + k * nv * np + node, np, Tc[i], e2, raw);
#pragma unroll
      for (int q = 0; q < 7; ++q) ok = ok && raw[q] >= m.lo[q] && raw[q] <= m.hi[q];
    } else {
#pragma unroll
      for (int q = 0; q < 7; ++q) raw[q] = m.mean[q];
    }
#pragma unroll
    for (int q = 0; q < 7; ++q) x[q] = (raw[q] - m.mean[q]) * m.inv_std[q];
    x[7] = 0.f;
    return ok;
  };
  auto cons = [&](int64_t i, const float* y, bool ok, bool valid, int) {
    if (cmode == 2) {  // uniform over the grid: no lane reaches the vote below
      if (i < total && valid) {
#pragma unroll
        for (int q = 0; q < NSPEC; ++q) {
          corr[q * total + i] = m.w_ref * sinh_pair(m.muY[q] + m.sdY[q] * y[q]);
          corr[(5 + q) * total + i] = m.j_ref * sinh_pair(m.muY[5 + q] + m.sdY[5 + q] * y[5 + q]);
        }
      }
      return;
    }
    ok = ok && valid;
    if (i < total && valid) {
      int64_t k;
      int node;
      split_node(i, np, k, node);
      float om[NSPEC], jp[NSPEC], msum = 0.f, asum = 0.f;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) {
        om[q] = m.w_ref * sinh_pair(m.muY[q] + m.sdY[q] * y[q]);
        float jr = m.j_ref * sinh_pair(m.muY[5 + q] + m.sdY[5 + q] * y[5 + q]);
        if (cmode == 1) {
          om[q] += corr[q * total + i];
          jr += corr[(5 + q) * total + i];
        }
        jp[q] = fmaxf(0.f, jr);
        msum += om[q];
        asum += fabsf(om[q]);
      }
      ok = ok && isfinite(asum) && fabsf(msum) <= m.tol_mass * asum + m.floor32;
      const float f = asum > 0.f ? msum / asum : 0.f;
      T* so = src + k * NSPEC * np + node;
      // positivity of the learned update: rho_s + dt S_s >= 0 (the plain point-implicit
      // source never consumes a species faster than the step allows; a learned one can)
      const T* uu = u + k * nv * np + node;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) {
        const float Sq = (om[q] - fabsf(om[q]) * f) / (1.f + dt * jp[q]);
        ok = ok && ((float)uu[q * np] + dt * Sq >= 0.f);
        so[q * np] = (T)Sq;
      }
    }
    const bool tile_ok = __all_sync(0xffffffffu, ok);
    const int64_t base = i - (threadIdx.x & 31);  // first node of this warp's 32-node tile
    if ((threadIdx.x & 31) == 0 && base < total) {
      // with corrections, a tile whose network missed the plain source at the last refresh
      // is not trusted until the next one
      const bool trusted = cmode != 1 || trust[base >> 5];
      flags[base >> 5] = !trusted ? 4 : (tile_ok ? 0 : 1);
    }
  };
  // with corrections, a tile none of whose warps is trusted needs no network
  auto skip = [&](int64_t row0) {
    if (cmode != 1) return false;
    bool need = false;
#pragma unroll
    for (int r = 0; r < CHEM_NR; ++r) {
      const int64_t t = (row0 + r * dgtc5::ROWS) >> 5;  // this warp's 32-node tile
      need = need || (t * 32 < total && trust[t]);
    }
    if (__syncthreads_or(need)) return false;
#pragma unroll
    for (int r = 0; r < CHEM_NR; ++r) {
      const int64_t t = (row0 + r * dgtc5::ROWS) >> 5;
      if ((threadIdx.x & 31) == 0 && t * 32 < total) flags[t] = 4;
    }
    return true;
  };
  dgtc5::run_tiles<10, CHEM_NR>(s, total, prod, cons, skip, checks);
}

// the FP64 form's check evaluations: the plain source at the sampled node of each tile that is
// still accepted, one thread per tile
__global__ void __launch_bounds__(128, 3)
chem_sampled_kernel(const double* u, const double* Tc, int64_t K, int np, int dim, const double* sp_raw,
                    const double* reac, int nr, const double* dtp, const unsigned char* flags, double* sampled,
                    uint64_t call) {
  pdl_wait();
  const int nv = NSPEC + dim + 1;
  const int64_t total = K * np, t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t * 32 >= total || flags[t]) return;
  int64_t k;
  int node;
  const int64_t i = sampled_node(t, total, call);
  split_node(i, np, k, node);
  Chem64 f;
  f.rates(u + k * nv * np + node, np, Tc[i], Chem64::Tab(), Chem64::Args(), sp_raw, reac, nr);
  const double dt = dtp ? *dtp : 0.0;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) sampled[NSPEC * t + s] = f.source(s, dt);
}

// a warp at a time takes the next tile (stats[2] counts them, set to zero by chem_mlp_tc5_kernel):
// the sampled check if it is still accepted (the learned source at the sampled node against the
// plain one in `sampled`), then, if rejected, the plain source at its nodes;
// counts nodes.  Rejected tiles cluster where the rates are large; with a fixed share of the tiles
// per warp a learned evaluation takes 5 % longer (18,000 tiles, 44 % rejected).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 3)
chem_fallback_kernel(const T* u, const double* Tc, int64_t K, int np, int dim, const double* sp_raw,
                     const double* reac, int nr, const __grid_constant__ ChemArgs<T> tab, const dgdd::dd* exp2,
                     const DgChemMlp* mlp, const double* dtp, T* src, unsigned char* flags, const T* sampled,
                     uint64_t call, unsigned long long* stats) {
  typedef typename ChemForm<T>::type Form;
  __shared__ typename Form::Tab tb;
  Form::stage(tb, exp2);
  pdl_wait();
  const int nv = NSPEC + dim + 1;
  const int lane = threadIdx.x & 31;
  const int64_t total = K * np, ntiles = (total + 31) / 32;
  // (a tolerance above the form's range stays finite: infinity times a zero scale accepts nothing)
  const T tol = (T)fmin(mlp->tol_check, sizeof(T) == 4 ? 3.4028234663852886e38 : 1.7976931348623157e308);
  const T floor_ = (T)mlp->floor;
  typename ChemForm<T>::step dt;
  form_step(dtp ? *dtp : 0.0, dt);
  unsigned long long n_ok = 0, n_fb = 0;
  for (;;) {
    unsigned long long next = 0;
    if (lane == 0) next = atomicAdd(&stats[2], 1ull);
    const int64_t t = (int64_t)__shfl_sync(0xffffffffu, next, 0);
    if (t >= ntiles) break;
    int flag = flags[t];
    if (!flag) {
      int64_t k;
      int node;
      split_node(sampled_node(t, total, call), np, k, node);
      T Sp[NSPEC], scale = 0;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) {
        Sp[s] = sampled[NSPEC * t + s];
        scale += fabs(Sp[s]);
      }
      bool ok = true;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) {
        const T Sm = src[(k * NSPEC + s) * np + node];
        ok = ok && fabs(Sm - Sp[s]) <= tol * scale + floor_;
      }
      if (!ok) {  // the same in all lanes
        flag = 2;
        __syncwarp();
        if (lane == 0) flags[t] = 2;
      }
    }
    const int64_t i = t * 32 + lane;
    if (i < total) {
      if (!flag) {
        ++n_ok;
      } else {
        ++n_fb;
        int64_t k;
        int node;
        split_node(i, np, k, node);
        Form f;
        f.rates(u + k * nv * np + node, np, Tc[i], tb, tab, sp_raw, reac, nr);
        T* so = src + k * NSPEC * np + node;
#pragma unroll
        for (int s = 0; s < NSPEC; ++s) so[s * np] = f.source(s, dt);
      }
    }
    __syncwarp();
  }
  for (int o = 16; o > 0; o >>= 1) {
    n_ok += __shfl_xor_sync(0xffffffffu, n_ok, o);
    n_fb += __shfl_xor_sync(0xffffffffu, n_fb, o);
  }
  if (lane == 0 && (n_ok | n_fb)) {
    atomicAdd(&stats[0], n_ok);
    atomicAdd(&stats[1], n_fb);
  }
}

// refresh of the corrections: every node takes the plain source, and corr (holding
// the network's decoded rates of this state, written by chem_mlp_tc5_kernel in cmode 2)
// becomes the plain-minus-network differences; every tile is flagged 3 (plain).  The full
// check: each node's uncorrected learned source (projection, point-implicit factor) against
// the plain one with the sampled check's test; a tile is trusted until the next refresh when
// all of its nodes pass.  Threads are grouped in warps over whole 32-node tiles.
__device__ __forceinline__ bool refresh_node(const Chem64& p, double dt, double tol, double floor_, int64_t total,
                                             float* corr, double* S) {
  double oh[NSPEC], jh[NSPEC], scale = 0.0, msum = 0.0, asum = 0.0;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    S[s] = p.source(s, dt);
    scale += fabs(S[s]);
    oh[s] = (double)corr[s * total];
    jh[s] = (double)corr[(5 + s) * total];
    msum += oh[s];
    asum += fabs(oh[s]);
  }
  const double f = asum > 0.0 ? msum / asum : 0.0;
  bool ok = isfinite(asum);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    const double Sl = (oh[s] - fabs(oh[s]) * f) / (1.0 + dt * fmax(0.0, jh[s]));
    ok = ok && fabs(Sl - S[s]) <= tol * scale + floor_;
    corr[s * total] = (float)(p.om[s] - oh[s]);
    corr[(5 + s) * total] = (float)(p.jpi[s] - jh[s]);
  }
  return ok;
}
// the same in pairs (the comparison itself in FP32: both sides carry 48 bits up to it)
__device__ __forceinline__ bool refresh_node(const Chem32& p, dgdd::dd dt, double tol, double floor_, int64_t total,
                                             float* corr, float* S) {
  using namespace dgdd;
  dd Sp[NSPEC], msum = make(0.f, 0.f), asum = msum, scale = msum;
  float oh[NSPEC], jh[NSPEC];
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    Sp[s] = div(p.om[s], mul_add(dt, p.jpi[s], make(1.f, 0.f)));
    S[s] = Sp[s].h;
    acc(scale, Sp[s].h < 0.f ? neg(Sp[s]) : Sp[s]);
    oh[s] = corr[s * total];
    jh[s] = corr[(5 + s) * total];
    acc(msum, make(oh[s], 0.f));
    acc(asum, make(fabsf(oh[s]), 0.f));
  }
  bool ok = isfinite(asum.h);
  const dd f = asum.h > 0.f ? div(norm(msum), norm(asum)) : make(0.f, 0.f);
  const float bound = (float)(tol * to_double(norm(scale)) + floor_);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
    const dd Sl = div(add(neg(mul(f, fabsf(oh[s]))), oh[s]), add(mul(dt, fmaxf(0.f, jh[s])), 1.f));
    ok = ok && fabsf(add(Sl, neg(Sp[s])).h) <= bound;
    corr[s * total] = add(p.om[s], -oh[s]).h;
    corr[(5 + s) * total] = add(p.jpi[s], -jh[s]).h;
  }
  return ok;
}

template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 3)
chem_refresh_kernel(const T* u, const double* Tc, int64_t K, int np, int dim, const double* sp_raw,
                    const double* reac, int nr, const __grid_constant__ ChemArgs<T> tab, const dgdd::dd* exp2,
                    const DgChemMlp* mlp, const double* dtp, T* src, float* corr, unsigned char* flags,
                    unsigned char* trust) {
  typedef typename ChemForm<T>::type Form;
  __shared__ typename Form::Tab tb;
  Form::stage(tb, exp2);
  pdl_wait();
  const int nv = NSPEC + dim + 1;
  const int64_t total = K * np;
  typename ChemForm<T>::step dt;
  form_step(dtp ? *dtp : 0.0, dt);
  const double tol = mlp->tol_check, floor_ = mlp->floor;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;  // a multiple of 32
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i - lane < total; i += stride) {
    bool ok = true;
    if (i < total) {
      int64_t k;
      int node;
      split_node(i, np, k, node);
      Form p;
      p.rates(u + k * nv * np + node, np, Tc[i], tb, tab, sp_raw, reac, nr);
      T S[NSPEC];
      ok = refresh_node(p, dt, tol, floor_, total, corr + i, S);
      T* so = src + k * NSPEC * np + node;
#pragma unroll
      for (int s = 0; s < NSPEC; ++s) so[s * np] = S[s];
    }
    const bool tile_ok = __all_sync(0xffffffffu, ok);
    if (lane == 0) {
      flags[i >> 5] = 3;
      trust[i >> 5] = tile_ok ? 1 : 0;
    }
  }
}

// training data: raw features and the plain (omega, jpi) at counter-sampled nodes
template <typename T>
__global__ void chem_sample_kernel(const T* u, const double* Tc, int64_t K, int np, int dim,
                                   const double* sp_raw, const double* reac, int nr, int64_t n, uint64_t seed,
                                   float* X, double* Y) {
  const int nv = NSPEC + dim + 1;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = (int64_t)(splitmix64(seed + (uint64_t)j) % (uint64_t)(K * np));
    int64_t k;
    int node;
    split_node(i, np, k, node);
    const T* uu = u + k * nv * np + node;
    chem_features<T>(uu, np, Tc[i], nullptr, X + j * 7);
    chem_node<T>(uu, np, Tc[i], sp_raw, reac, nr, Y + j * 10, Y + j * 10 + 5);
  }
}

unsigned grid_of(int64_t n) {
  int64_t g = (n + 127) / 128;
  if (g > 152 * 64) g = 152 * 64;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t dg_chem_init(DgThermo* th, const double* species_host, const double* reac_host, int nr) {
  if (nr < 1 || nr > 64) return cudaErrorInvalidValue;
  double* rows = (double*)calloc((size_t)RX_W * nr + SP_W * NSPEC, sizeof(double));
  if (!rows) return cudaErrorMemoryAllocation;
  for (int r = 0; r < nr; ++r) {
    const double* in = reac_host + 19 * r;  // [nu'(5), nu''(5), tb, eff(5), A, beta, theta]
    double* o = rows + RX_W * r;
    for (int q = 0; q < 16; ++q) o[q] = in[q];
    o[16] = log(in[16]);
    o[17] = in[17];
    o[18] = in[18];
    double dn = 0.0;
    long long meta = 0;
    for (int s = 0; s < NSPEC; ++s) {
      o[20 + s] = in[5 + s] - in[s];
      dn += o[20 + s];
      const double a = in[s], b = in[5 + s];
      if (!(a == 0.0 || a == 1.0 || a == 2.0 || a == 3.0) || !(b == 0.0 || b == 1.0 || b == 2.0 || b == 3.0)) {
        free(rows);  // the integer form holds nu in {0, 1, 2, 3}
        return cudaErrorInvalidValue;
      }
      meta |= (long long)a << (2 * s);
      meta |= (long long)b << (10 + 2 * s);
      if (o[20 + s] != 0.0) meta |= 1ll << (21 + s);
    }
    if (in[10] != 0.0) meta |= 1ll << 20;
    int sabs = 0, dnt = 0;
    for (int s = 0; s < NSPEC; ++s) {
      const int ds = (int)in[5 + s] - (int)in[s];
      sabs += ds < 0 ? -ds : ds;
      dnt += ds;
    }
    if (sabs <= 15 && dnt >= -3 && dnt <= 3) meta |= ((long long)sabs << 26) | (1ll << 30);
    o[19] = dn;
    memcpy(&o[RX_META], &meta, sizeof(meta));
    for (int s = 0; s < NSPEC; ++s) o[26 + s] = o[20 + s] * in[11 + s];  // dnu_s eff_s
  }
  double* sp = rows + (size_t)RX_W * nr;
  for (int s = 0; s < NSPEC; ++s) {
    const double* in = species_host + 8 * s;  // [W, a1..a7]
    double* o = sp + SP_W * s;
    // g/(RT) = h/(RT) - s/R = (a1 - a7) + T (a2/2 - a2) + T^2 (a3/3 - a3/2) + T^3 (a4/4 - a4/3)
    //         + T^4 (a5/5 - a5/4) + a6 / T - a1 ln T
    o[0] = 1e-6 / in[0];
    o[1] = 1e6 * in[0];
    o[2] = in[1] - in[7];
    o[3] = in[2] / 2.0 - in[2];
    o[4] = in[3] / 3.0 - in[3] / 2.0;
    o[5] = in[4] / 4.0 - in[4] / 3.0;
    o[6] = in[5] / 5.0 - in[5] / 4.0;
    o[7] = in[6];
    o[8] = in[1];
    o[9] = 1e-6 * DG_P0 / DG_RU;  // P = o[9] / T
    o[10] = DG_RU / (1e-6 * DG_P0);  // 1/P = o[10] T
    o[14] = log(1e-6 * DG_P0 / DG_RU);
  }
  // the same rows as pairs for the mixed form
  ChemTab32* t32 = (ChemTab32*)calloc(1, sizeof(ChemTab32));
  if (!t32) {
    free(rows);
    return cudaErrorMemoryAllocation;
  }
  dgdd::dd e2[dgdd::EXP_TAB];
  for (int j = 0; j < dgdd::EXP_TAB; ++j) e2[j] = dgdd::from_double(exp2(j / (double)dgdd::EXP_TAB));
  for (int s = 0; s < NSPEC; ++s) {
    const double* o = sp + SP_W * s;
    t32->cw[s] = dgdd::from_double(o[0]);
    t32->ow[s] = dgdd::from_double(ldexp(o[1], -SCALE2));
  }
  for (int r = 0; r < nr; ++r) {
    const double* o = rows + RX_W * r;
    if (reac_host[19 * r + 16] == 0.0) continue;  // ln A has no pair, and both rates are zero
    ChemRow32& w = t32->row[t32->n++];
    w.lnA = dgdd::from_double(o[16]);
    w.beta = dgdd::from_double(o[17]);
    w.mtheta = dgdd::from_double(-o[18]);
    for (int s = 0; s < NSPEC; ++s) {
      const float a = (float)o[s], b = (float)o[5 + s];
      w.eff[s] = dgdd::from_double(o[11 + s]);
      w.nf[s] = a;
      w.dn[s] = b - a;
      w.dn64[s] = (double)(b - a);
      w.jf[s] = a * (b - a);
      w.jb[s] = -b * (b - a);
      w.mask |= (w.nf[s] != 0.f) << s | (w.dn[s] != 0.f) << (5 + s) | (w.jf[s] != 0.f) << (10 + s) |
                (w.jb[s] != 0.f) << (15 + s);
      const int ia = (int)a, ib = (int)b;
      w.mask2 |= (ib > 0) << s | (ia & 1) << (5 + s) | (ib & 1) << (10 + s) | (ia == 1) << (15 + s) | (ib == 1) << (20 + s);
    }
    if (o[10] != 0.0) w.mask |= 1 << 20;
  }
  th->chem_tab32 = t32;  // host memory, freed with the context
  const size_t rs = th->f32 ? sizeof(float) : sizeof(double);
  cudaError_t e = cudaMalloc(&th->chem_exp2, sizeof(e2));
  if (e == cudaSuccess) e = cudaMemcpy(th->chem_exp2, e2, sizeof(e2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc((void**)&th->reac, sizeof(double) * RX_W * nr);
  if (e == cudaSuccess) e = cudaMemcpy(th->reac, rows, sizeof(double) * RX_W * nr, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc((void**)&th->species_raw, sizeof(double) * SP_W * NSPEC);
  if (e == cudaSuccess) e = cudaMemcpy(th->species_raw, sp, sizeof(double) * SP_W * NSPEC, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&th->src, rs * NSPEC * th->K * th->np);
  free(rows);
  th->nr = nr;
  return e;
}

template <typename T>
static cudaError_t chem_learned(DgThermo* th, const T* u, const double* dt_dev, int refresh, cudaStream_t s) {
  const int64_t total = th->K * th->np, ntiles = (total + 31) / 32;
  const DgChemMlp* m = (const DgChemMlp*)th->chem_mlp;
  const ChemArgs<T>& tab = *(const ChemArgs<T>*)th->chem_tab32;  // (the FP64 form's is empty)
  const dgdd::dd* e2 = (const dgdd::dd*)th->chem_exp2;
  const size_t smem = sizeof(dgtc5::Smem<10, CHEM_NR>);
  auto k1 = chem_mlp_tc5_kernel<T>;
  cudaError_t e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // persistent CTAs over tensor-core tiles of 128 nodes
  const int64_t rows = CHEM_NR * dgtc5::ROWS, tiles = (total + rows - 1) / rows;
  const unsigned g1 = (unsigned)(tiles < 152 * 5 ? tiles : 152 * 5);
  if (refresh) {
    if (!th->chem_corr || !th->chem_trust) return cudaErrorInvalidValue;
    e = launch_pdl(th->apart, k1, g1, dgtc5::THREADS, smem, s, u, th->T, th->K, th->np, th->dim, th->species_raw, th->reac, th->nr,
                   tab, e2, m, dt_dev, (T*)th->src, th->chem_flags, th->chem_corr, th->chem_trust, 2, 0, (T*)NULL, 0,
                   (unsigned long long*)NULL);
    if (e != cudaSuccess) return e;
    e = launch_pdl(th->apart, chem_refresh_kernel<T>, grid_of(ntiles * 32), 128, 0, s, u, th->T, th->K, th->np, th->dim,
                   th->species_raw, th->reac, th->nr, tab, e2, m, dt_dev, (T*)th->src, th->chem_corr, th->chem_flags,
                   th->chem_trust);
    if (e == cudaSuccess) th->corr_valid = 1;
    return e;
  }
  const int cmode = th->chem_corr && th->chem_trust && th->corr_valid ? 1 : 0;
  const unsigned per_tile = (unsigned)((ntiles + 127) / 128), checks = sizeof(T) == 4 ? per_tile : 0;
  static_assert(dgtc5::THREADS == 128, "one thread per tile");
  const uint64_t call = th->chem_calls++;
  e = launch_pdl(th->apart, k1, checks + g1, dgtc5::THREADS, smem, s, u, th->T, th->K, th->np, th->dim, th->species_raw, th->reac,
                 th->nr, tab, e2, m, dt_dev, (T*)th->src, th->chem_flags, th->chem_corr, th->chem_trust, cmode,
                 (int)checks, (T*)th->chem_sampled, call, th->chem_stats);
  if (e != cudaSuccess) return e;
  if constexpr (sizeof(T) == 8) {
    e = launch_pdl(th->apart, chem_sampled_kernel, per_tile, 128, 0, s, u, th->T, th->K, th->np, th->dim, th->species_raw, th->reac,
                   th->nr, dt_dev, th->chem_flags, (double*)th->chem_sampled, call);
    if (e != cudaSuccess) return e;
  }
  int64_t g3 = (ntiles + 3) / 4;
  if (g3 > 152 * 5) g3 = 152 * 5;
  return launch_pdl(th->apart, chem_fallback_kernel<T>, (unsigned)g3, 128, 0, s, u, th->T, th->K, th->np, th->dim, th->species_raw,
                    th->reac, th->nr, tab, e2, m, dt_dev, (T*)th->src, th->chem_flags, (const T*)th->chem_sampled, call,
                    th->chem_stats);
}

cudaError_t dg_chem_source(DgThermo* th, const void* u, int f32, const double* dt_dev, int refresh,
                           cudaStream_t s) {
  if (th->chem_mlp)
    return f32 ? chem_learned<float>(th, (const float*)u, dt_dev, refresh, s)
               : chem_learned<double>(th, (const double*)u, dt_dev, refresh, s);
  const unsigned grid = grid_of(th->K * th->np);
  const dgdd::dd* e2 = (const dgdd::dd*)th->chem_exp2;
  if (f32)
    return launch_pdl(th->apart, chem_kernel<float>, grid, 128, 0, s, (const float*)u, th->T, th->K, th->np, th->dim, th->species_raw,
                      th->reac, th->nr, *(const ChemTab32*)th->chem_tab32, e2, dt_dev, (float*)th->src);
  return launch_pdl(th->apart, chem_kernel<double>, grid, 128, 0, s, (const double*)u, th->T, th->K, th->np, th->dim,
                    th->species_raw, th->reac, th->nr, Chem64::Args(), e2, dt_dev, (double*)th->src);
}

cudaError_t dg_chem_mlp_set(DgThermo* th, const float* params_host, const double* st) {
  th->corr_valid = 0;
  if (!params_host) {
    if (th->chem_mlp) cudaFree(th->chem_mlp);
    th->chem_mlp = NULL;
    return cudaSuccess;
  }
  DgChemMlp* h = (DgChemMlp*)calloc(1, sizeof(DgChemMlp));
  if (!h) return cudaErrorMemoryAllocation;
  dg_mlp_pack<10>(params_host, &h->w);
  for (int q = 0; q < 7; ++q) {
    h->st.mean[q] = (float)st[DG_SRC_X_MEAN + q];
    h->st.inv_std[q] = (float)(1.0 / st[DG_SRC_X_STD + q]);
    h->st.lo[q] = (float)st[DG_SRC_BOX_LO + q];
    h->st.hi[q] = (float)st[DG_SRC_BOX_HI + q];
  }
  for (int q = 0; q < 10; ++q) {
    h->st.muY[q] = (float)st[DG_SRC_Y_MEAN + q];
    h->st.sdY[q] = (float)st[DG_SRC_Y_STD + q];
  }
  h->st.w_ref = (float)st[DG_SRC_OMEGA_REF];
  h->st.j_ref = (float)st[DG_SRC_JPI_REF];
  h->st.tol_mass = (float)st[DG_SRC_TOL_MASS];
  h->tol_check = st[DG_SRC_TOL_CHECK];
  h->floor = st[DG_SRC_FLOOR];
  h->st.floor32 = (float)st[DG_SRC_FLOOR];
  const int64_t ntiles = (th->K * th->np + 31) / 32;
  cudaError_t e = cudaSuccess;
  if (!th->chem_mlp) e = cudaMalloc(&th->chem_mlp, sizeof(DgChemMlp));
  if (e == cudaSuccess && !th->chem_stats) e = cudaMalloc((void**)&th->chem_stats, 3 * sizeof(unsigned long long));
  if (e == cudaSuccess && !th->chem_flags) e = cudaMalloc((void**)&th->chem_flags, (size_t)ntiles);
  if (e == cudaSuccess && !th->chem_sampled) e = cudaMalloc(&th->chem_sampled, sizeof(double) * NSPEC * ntiles);
  if (e == cudaSuccess) e = cudaMemset(th->chem_stats, 0, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMemcpy(th->chem_mlp, h, sizeof(DgChemMlp), cudaMemcpyHostToDevice);
  free(h);
  return e;
}

cudaError_t dg_chem_sample_dev(DgThermo* th, const void* u, int f32, int64_t n, uint64_t seed, float* X,
                           double* targets, cudaStream_t s) {
  if (f32)
    chem_sample_kernel<float><<<grid_of(n), 128, 0, s>>>((const float*)u, th->T, th->K, th->np, th->dim,
                                                         th->species_raw, th->reac, th->nr, n, seed, X, targets);
  else
    chem_sample_kernel<double><<<grid_of(n), 128, 0, s>>>((const double*)u, th->T, th->K, th->np, th->dim,
                                                          th->species_raw, th->reac, th->nr, n, seed, X, targets);
  return cudaGetLastError();
}
