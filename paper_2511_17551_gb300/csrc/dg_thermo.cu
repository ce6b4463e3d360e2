// Mixture thermodynamics on the device: temperature from internal energy by Newton
// iteration, Dalton pressure and frozen sound speed, per node.
//
// Thermally perfect species (stand-in for the RRHO database of the appendix,
// Eq. Internal_energy): cp_s/R_s = a1 + a2 T + a3 T^2 + a4 T^3 + a5 T^4 and
//   e_s(T) = R_s (a1 T + a2 T^2/2 + a3 T^3/3 + a4 T^4/4 + a5 T^5/5 + a6 - T),
// e = sum Y_s e_s (Eq. internal_energies), p = sum rho_s R_s T (Eq. eos).
// At set-up every species becomes one row of a coefficient table
//   [R_s a6, R_s (a1-1), R_s a2/2, R_s a3/3, R_s a4/4, R_s a5/5, R_s, 0],
// so a node folds its mixture into e(T) = b0 + b1 T + ... + b5 T^5 with 30 multiply-adds
// (no divisions) and evaluates e and cv = de/dT by Horner's rule.  Newton
// T <- T - (e(T) - e)/cv(T) is warm-started from the node's previous temperature and
// stops at |dT| <= 1e-12 T (at most 50 steps, T kept in [200, 1e4] K); failure latches
// DG_ENEWTON.  Mixed form: FP32 Newton on e(T) - b0 = e - b0 (the constant b0 is
// removed so FP32 resolves the residual) to |dT| <= 1e-6 T, then one Newton step on the
// residual in double-FP32 pairs.
#include <cuda_runtime.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include "dg_dd.cuh"
#include "dg_cvt.cuh"
#include "dg_internal.h"
#include "dg_launch.cuh"
#include "dg_thermo.h"

#define DG_RU 8.314462618
#define NSPEC 5

namespace {

__device__ __forceinline__ void latch(unsigned long long* st, unsigned long long code, int64_t e) {
  atomicCAS(st, 0ull, (code << 56) | (unsigned long long)(e & 0x00ffffffffffffffll));
}

template <typename R>
struct Poly {
  R b[6];  // e(T) = sum b_k T^k
  R Rmix;
  __device__ __forceinline__ R e(R T) const {
    return b[0] + T * (b[1] + T * (b[2] + T * (b[3] + T * (b[4] + T * b[5]))));
  }
  __device__ __forceinline__ R e_noconst(R T) const {
    return T * (b[1] + T * (b[2] + T * (b[3] + T * (b[4] + T * b[5]))));
  }
  __device__ __forceinline__ R cv(R T) const {
    return b[1] + T * (R(2) * b[2] + T * (R(3) * b[3] + T * (R(4) * b[4] + T * (R(5) * b[5]))));
  }
};

template <typename R>
__device__ __forceinline__ void build_poly(const R* cf, const R* Y, Poly<R>& P) {
#pragma unroll
  for (int k = 0; k < 6; ++k) P.b[k] = R(0);
  P.Rmix = R(0);
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
#pragma unroll
    for (int k = 0; k < 6; ++k) P.b[k] += Y[s] * cf[8 * s + k];
    P.Rmix += Y[s] * cf[8 * s + 6];
  }
}

__device__ __forceinline__ double clampT(double T) { return T < 200.0 ? 200.0 : (T > 1e4 ? 1e4 : T); }
// 200 <= T <= 1e4, false for NaN: positive doubles order as their bits do (200.0 is 0x40690000 00000000,
// 1e4 0x40c38800 00000000)
__device__ __forceinline__ bool in_fit_range(double T) {
  const unsigned h = (unsigned)__double2hiint(T);
  return h >= 0x40690000u && (h < 0x40c38800u || (h == 0x40c38800u && __double2loint(T) == 0));
}
__device__ __forceinline__ float clampTf(float T) { return T < 200.f ? 200.f : (T > 1e4f ? 1e4f : T); }

// FP64 Newton from T; returns true on convergence
__device__ __forceinline__ bool newton64(const Poly<double>& P, double e, double& T) {
  for (int it = 0; it < 50; ++it) {
    const double Tn = clampT(T - (P.e(T) - e) / P.cv(T));
    const double step = fabs(Tn - T);
    T = Tn;
    if (step <= 1e-12 * T) return true;
  }
  return false;
}

// FP64 form: the full FP64 Newton iteration, one thread per node
__global__ void thermo_update_kernel(const double* u, int64_t K, int np, int dim, const double* cf, double* Tc,
                                     double* pc, unsigned long long* status) {
  pdl_wait();
  const int nv = NSPEC + dim + 1;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < K * np;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = i / np;
    const int node = (int)(i % np);
    const double* uu = u + k * nv * np + node;
    double Y[NSPEC], rho = 0.0, ke = 0.0;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      Y[s] = uu[s * np];
      rho += Y[s];
    }
    for (int d = 0; d < dim; ++d) {
      const double m = uu[(NSPEC + d) * np];
      ke += m * m;
    }
    const double ir = 1.0 / rho;
    const double e = uu[(NSPEC + dim) * np] * ir - 0.5 * ke * ir * ir;
    double Tk = Tc[k * np + node];
    if (!(Tk >= 200.0 && Tk <= 1e4)) Tk = 1000.0;
    Poly<double> P;
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) Y[s] *= ir;
    build_poly<double>(cf, Y, P);
    const bool ok = rho > 0.0 && newton64(P, e, Tk);
    if (!ok) latch(status, DG_ST_NEWTON, k);
    Tc[k * np + node] = Tk;
    const double p = rho * P.Rmix * Tk;
    const double cv = P.cv(Tk);
    pc[(k * 2 + 0) * np + node] = p;
    pc[(k * 2 + 1) * np + node] = sqrt((cv + P.Rmix) / cv * p * ir);
  }
}

// the full FP64 iteration of a mixed-form node whose FP32 iteration did not converge, from T
__device__ __noinline__ bool newton64_node(const float* uu, int np, int dim, const double* cf, double& T) {
  double Y[NSPEC], rho = 0.0, ke = 0.0;
  for (int s = 0; s < NSPEC; ++s) {
    Y[s] = (double)uu[s * np];
    rho += Y[s];
  }
  for (int d = 0; d < dim; ++d) {
    const double m = (double)uu[(NSPEC + d) * np];
    ke += m * m;
  }
  const double ir = 1.0 / rho;
  for (int s = 0; s < NSPEC; ++s) Y[s] *= ir;
  Poly<double> P;
  build_poly<double>(cf, Y, P);
  return newton64(P, (double)uu[(NSPEC + dim) * np] * ir - 0.5 * ke * ir * ir, T);
}

// Mixed form: FP32 Newton on e(T) - b0 = e - b0, then one Newton correction on a residual in
// double-FP32 pairs (dg_dd.cuh): the FP32 state is exact in them, e - b0 keeps 46 bits through
// the cancellation of the formation energies, and the polynomial takes the FP32-rounded
// temperature coefficients (their rounding moves e by ~1e-7 relative, i.e. T by ~1e-4 K, as it
// did with the residual in FP64).  Nothing in the common path touches the FP64 pipe but one
// addition; 68 FP64 instructions a node bound the kernel before.
// Bytes per node: 36 of state, 16 of T, 8 of (p, c).  1.73 M nodes: 193 -> 45 us (2.3 TB/s), 4.6 M:
// 500 -> 101 us (2.7 TB/s); the same distance to the FP64 solution (1.6e-7, the coefficients').
template <int NP, int DIM>
__global__ void __launch_bounds__(256, 3) thermo_mixed_kernel(const float* u, int64_t K, const double* cf,
                                                           const float* cf32, double* Tc, float* pc,
                                                           unsigned long long* status) {
  using namespace dgdd;
  constexpr int NV = NSPEC + DIM + 1;
  __shared__ __align__(16) float c32[8 * NSPEC];
  __shared__ dd b0s[NSPEC];
  if (threadIdx.x < 8 * NSPEC) c32[threadIdx.x] = cf32[threadIdx.x];
  if (threadIdx.x < NSPEC) b0s[threadIdx.x] = from_double(cf[8 * threadIdx.x]);
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  for (int64_t base = blockIdx.x * (int64_t)256; base < K * NP; base += gridDim.x * (int64_t)256) {
    // element and node of base + threadIdx.x: the 64-bit division is the same in all threads
    const int64_t k0 = base / NP;
    const int off = (int)(base - k0 * NP) + (int)threadIdx.x;
    const int64_t k = k0 + off / NP;
    const int node = off % NP;
    if (k >= K) continue;
    const float* uu = u + k * NV * NP + node;
    float r[NSPEC], m[DIM];
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) r[s] = uu[s * NP];
#pragma unroll
    for (int d = 0; d < DIM; ++d) m[d] = uu[(NSPEC + d) * NP];
    const float E = uu[(NSPEC + DIM) * NP];
    double Tk = Tc[k * NP + node];
    dd rho = make(r[0], 0.f), ke = make(0.f, 0.f), b0 = mul(b0s[0], r[0]);
#pragma unroll
    for (int s = 1; s < NSPEC; ++s) {
      acc(rho, make(r[s], 0.f));
      acc_mul(b0, b0s[s], r[s]);
    }
    rho = norm(rho);
#pragma unroll
    for (int d = 0; d < DIM; ++d) acc(ke, two_prod(m[d], m[d]));
    const dd ir = rcp(rho);
    // rho (e - b0) = E - |m|^2 / (2 rho) - sum rho_s b0_s
    dd er = mul(mul(norm(ke), ir), -0.5f);
    acc(er, make(E, 0.f));
    acc(er, neg(b0));
    er = mul(norm(er), ir);
    Poly<float> P;
    float Y[NSPEC];
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) Y[s] = r[s] * ir.h;
    build_poly<float>(c32, Y, P);
    if (!in_fit_range(Tk)) Tk = 1000.0;
    float Tf = dgdd::narrow(Tk);
    bool conv = false;
    // (below 1e-12 kg/m^3 the products' low parts leave FP32's range: FP64)
    for (int it = 0; it < 12 && rho.h > 1e-12f; ++it) {
      const float Tn = clampTf(Tf - (P.e_noconst(Tf) - er.h) / P.cv(Tf));
      const float step = fabsf(Tn - Tf);
      Tf = Tn;
      if (step <= 1e-6f * Tf) {
        conv = true;
        break;
      }
    }
    // residual at Tf (exact in FP32) and the correction; cv in FP32 only scales it
    dd q = add(two_prod(P.b[5], Tf), P.b[4]);
    q = add(mul(q, Tf), P.b[3]);
    q = add(mul(q, Tf), P.b[2]);
    q = add(mul(q, Tf), P.b[1]);
    q = add(mul(q, Tf), neg(er));
    dd T = two_sum(Tf, -(q.h * (1.0f / P.cv(Tf))));
    if (T.h < 200.f || (T.h == 200.f && T.l < 0.f)) T = make(200.f, 0.f);
    if (T.h > 1e4f || (T.h == 1e4f && T.l > 0.f)) T = make(1e4f, 0.f);
    double T64 = to_double(T);
    bool ok = rho.h > 0.f;
    if (ok && !conv) ok = newton64_node(uu, NP, DIM, cf, T64);
    if (!ok) latch(status, DG_ST_NEWTON, k);
    Tc[k * NP + node] = T64;
    const float Tq = (ok && !conv) ? dgdd::narrow(T64) : T.h;
    const float pf = rho.h * P.Rmix * Tq, cvf = P.cv(Tq);
    pc[(k * 2 + 0) * NP + node] = pf;
    pc[(k * 2 + 1) * NP + node] = sqrtf((cvf + P.Rmix) / cvf * pf / rho.h);
  }
}

// (rho_s, v, T) -> conserved; seeds the temperature cache Tc, or (boundary states) gives (p, c).  The
// energy is summed over the species as rho e = sum_k T^k sum_s rho_s c_sk: 46 FP64 operations a node
// (the pipe bounds the kernel) instead of about 150 with mass fractions and (p, c), which the
// temperature solve of every later evaluation forms anew: 1.73 M nodes 457 -> 189 us a call.
template <typename T>
__global__ void __launch_bounds__(256) thermo_prim2cons_kernel(const double* w, T* u, int64_t K, int np, int dim,
                                                               const double* cf, double* Tc, T* pc) {
  const int nv = NSPEC + dim + 1;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x; base < K * np; base += gridDim.x * (int64_t)blockDim.x) {
    const int64_t k0 = base / np;  // the 64-bit division is the same in all threads
    const unsigned off = (unsigned)(base - k0 * np) + threadIdx.x, dk = off / (unsigned)np;
    const int64_t k = k0 + dk;
    if (k >= K) continue;
    const int node = (int)(off - dk * (unsigned)np);
    const double* ww = w + k * nv * np + node;
    T* uu = u + k * nv * np + node;
    double rho = 0.0;
    Poly<double> P;  // of rho_s instead of Y_s: rho e(T), rho R
    double r[NSPEC];
#pragma unroll
    for (int s = 0; s < NSPEC; ++s) {
      r[s] = ww[s * np];
      rho += r[s];
      uu[s * np] = narrow<T>(r[s]);
    }
    double ke = 0.0;
    for (int d = 0; d < dim; ++d) {
      const double v = ww[(NSPEC + d) * np];
      uu[(NSPEC + d) * np] = narrow<T>(rho * v);
      ke += v * v;
    }
    const double Tk = ww[(NSPEC + dim) * np];
    build_poly<double>(cf, r, P);
    uu[(NSPEC + dim) * np] = narrow<T>(P.e(Tk) + 0.5 * rho * ke);
    if (Tc) Tc[k * np + node] = Tk;
    if (pc) {
      const double p = P.Rmix * Tk, cv = P.cv(Tk);
      pc[(k * 2 + 0) * np + node] = (T)p;
      pc[(k * 2 + 1) * np + node] = (T)sqrt((cv + P.Rmix) / cv * p / rho);
    }
  }
}

__global__ void fill_kernel(double* a, int64_t n, double v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] = v;
}

unsigned grid_of(int64_t n) {
  int64_t g = (n + 255) / 256;
  if (g > 152 * 32) g = 152 * 32;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t dg_thermo_upload_basis() { return cudaSuccess; }

cudaError_t dg_thermo_init(DgThermo* th, int64_t K, int np, int dim, const double* species_host,
                           int mode, int f32, unsigned long long* status) {
  memset(th, 0, sizeof(*th));
  th->K = K;
  th->np = np;
  th->dim = dim;
  th->ns = NSPEC;
  th->mode = mode;
  th->f32 = f32;
  th->status = status;
  // per-species coefficient rows (see the header comment)
  double cf[8 * NSPEC];
  float cf32[8 * NSPEC];
  for (int s = 0; s < NSPEC; ++s) {
    const double* sp = species_host + 8 * s;
    const double Rs = DG_RU / sp[0];
    const double* a = sp + 1;
    const double row[8] = {Rs * a[5], Rs * (a[0] - 1.0), Rs * a[1] / 2.0, Rs * a[2] / 3.0,
                           Rs * a[3] / 4.0, Rs * a[4] / 5.0, Rs, 0.0};
    for (int k = 0; k < 8; ++k) {
      cf[8 * s + k] = row[k];
      cf32[8 * s + k] = (float)row[k];
    }
  }
  const size_t rs = f32 ? sizeof(float) : sizeof(double);
  cudaError_t e = cudaMalloc((void**)&th->species, sizeof(cf));
  if (e == cudaSuccess) e = cudaMemcpy(th->species, cf, sizeof(cf), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc((void**)&th->coef32, sizeof(cf32));
  if (e == cudaSuccess) e = cudaMemcpy(th->coef32, cf32, sizeof(cf32), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc((void**)&th->T, sizeof(double) * K * np);
  if (e == cudaSuccess) e = cudaMalloc(&th->pc, rs * 2 * K * np);
  if (e == cudaSuccess) e = cudaMalloc(&th->bc_pc, rs * 2 * 64);
  if (e == cudaSuccess) {
    fill_kernel<<<grid_of(K * np), 256>>>(th->T, K * np, 1000.0);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e;
}

void dg_thermo_free(DgThermo* th) {
  if (th->mlp) cudaFree(th->mlp);
  if (th->mlp_stats) cudaFree(th->mlp_stats);
  if (th->chem_mlp) cudaFree(th->chem_mlp);
  if (th->chem_stats) cudaFree(th->chem_stats);
  if (th->chem_flags) cudaFree(th->chem_flags);
  if (th->chem_sampled) cudaFree(th->chem_sampled);
  if (th->chem_corr) cudaFree(th->chem_corr);
  if (th->chem_trust) cudaFree(th->chem_trust);
  if (th->species) cudaFree(th->species);
  if (th->coef32) cudaFree(th->coef32);
  if (th->species_raw) cudaFree(th->species_raw);
  if (th->reac) cudaFree(th->reac);
  free(th->chem_tab32);
  if (th->chem_exp2) cudaFree(th->chem_exp2);
  if (th->src) cudaFree(th->src);
  if (th->T) cudaFree(th->T);
  if (th->pc) cudaFree(th->pc);
  if (th->bc_pc) cudaFree(th->bc_pc);
  memset(th, 0, sizeof(*th));
}

// cold start: every node's Newton iteration restarts from 1000 K
cudaError_t dg_thermo_reset(DgThermo* th, cudaStream_t s) {
  fill_kernel<<<grid_of(th->K * th->np), 256, 0, s>>>(th->T, th->K * th->np, 1000.0);
  return cudaGetLastError();
}

cudaError_t dg_thermo_update(DgThermo* th, const void* u, int f32, cudaStream_t s) {
  if (th->mode == 1 && th->mlp) return dg_mlp_thermo_update(th, u, f32, s);
  const unsigned grid = grid_of(th->K * th->np);
  if (!f32)
    return launch_pdl(th->apart, thermo_update_kernel, grid, 256, 0, s, (const double*)u, th->K, th->np, th->dim, th->species, th->T,
                      (double*)th->pc, th->status);
  if (th->dim == 3 && th->np == 64)
    return launch_pdl(th->apart, thermo_mixed_kernel<64, 3>, grid, 256, 0, s, (const float*)u, th->K, th->species, th->coef32, th->T,
                      (float*)th->pc, th->status);
  if (th->dim == 3 && th->np == 125)
    return launch_pdl(th->apart, thermo_mixed_kernel<125, 3>, grid, 256, 0, s, (const float*)u, th->K, th->species, th->coef32, th->T,
                      (float*)th->pc, th->status);
  return cudaErrorInvalidValue;  // mixtures are 3D with N = 3 or 4
}

cudaError_t dg_thermo_boundary(DgThermo* th, const double* bw, int n_bc, void* bc_u, cudaStream_t s) {
  if (n_bc > 64) return cudaErrorInvalidValue;
  if (th->f32)
    thermo_prim2cons_kernel<float><<<1, 64, 0, s>>>(bw, (float*)bc_u, n_bc, 1, th->dim, th->species,
                                                     NULL, (float*)th->bc_pc);
  else
    thermo_prim2cons_kernel<double><<<1, 64, 0, s>>>(bw, (double*)bc_u, n_bc, 1, th->dim, th->species,
                                                      NULL, (double*)th->bc_pc);
  return cudaGetLastError();
}

cudaError_t dg_thermo_prim2cons(DgThermo* th, const double* w, void* u, cudaStream_t s) {
  if (th->f32)
    thermo_prim2cons_kernel<float><<<grid_of(th->K * th->np), 256, 0, s>>>(
        w, (float*)u, th->K, th->np, th->dim, th->species, th->T, (float*)NULL);
  else
    thermo_prim2cons_kernel<double><<<grid_of(th->K * th->np), 256, 0, s>>>(
        w, (double*)u, th->K, th->np, th->dim, th->species, th->T, (double*)NULL);
  return cudaGetLastError();
}
