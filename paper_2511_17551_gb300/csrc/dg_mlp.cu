// Learned surrogates: training kernels (FP32, any number of outputs up to 16) and the
// temperature surrogate's BF16 tensor-core inference fused with the per-node FP64
// Newton polish and the Newton fallback.
//
// Temperature surrogate: x in R^7 -> 64 -> 64 -> 1, x = standardised (Y_1..Y_5, ln rho,
// e), output = standardised T.  Inference (dg_thermo_update in surrogate mode): 128-node
// tiles on the tcgen05 tensor cores (dg_mlp_tc5.cuh), then per node: one Newton step from
// the prediction, accept when the next correction would be <= 1e-6 T, otherwise run the
// plain Newton iteration (fallback, counted).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include "../../include/dg.h"
#include "dg_internal.h"
#include "dg_launch.cuh"
#include "dg_mlp.cuh"
#include "dg_mlp_tc5.cuh"
#include "dg_thermo.h"

#define NI DG_MLP_NI
#define NH DG_MLP_NH
#define NO_MAX DG_MLP_NO_MAX
#define DG_RU 8.314462618
#define NSPEC 5

// temperature surrogate: weights and input / output standardisation
struct __align__(16) DgMlpDev {
  DgMlpW<1> w;
  float mean[NI], inv_std[NI];
  float muT, sigT;
};

namespace {
using namespace dgmlp;

struct PolyD {
  double b[6], Rmix;
  __device__ __forceinline__ double e(double T) const {
    return b[0] + T * (b[1] + T * (b[2] + T * (b[3] + T * (b[4] + T * b[5]))));
  }
  __device__ __forceinline__ double cv(double T) const {
    return b[1] + T * (2.0 * b[2] + T * (3.0 * b[3] + T * (4.0 * b[4] + T * (5.0 * b[5]))));
  }
};

// mixture polynomial from the per-species coefficient rows of the context
// ([R a6, R (a1-1), R a2/2, R a3/3, R a4/4, R a5/5, R, 0] per species)
__device__ __forceinline__ void poly_d(const double* cf, const double* Y, PolyD& P) {
#pragma unroll
  for (int k = 0; k < 6; ++k) P.b[k] = 0.0;
  P.Rmix = 0.0;
#pragma unroll
  for (int s = 0; s < NSPEC; ++s) {
#pragma unroll
    for (int k = 0; k < 6; ++k) P.b[k] += Y[s] * cf[8 * s + k];
    P.Rmix += Y[s] * cf[8 * s + 6];
  }
}

__device__ __forceinline__ double clampT(double T) { return T < 200.0 ? 200.0 : (T > 1e4 ? 1e4 : T); }

#define MLP_WARPS 4

// Temperature surrogate on the fifth-generation tensor cores: CTAs of 128 threads take
// 128-node tiles through the tcgen05 tile engine (dg_mlp_tc5.cuh).  Each thread forms its
// node's features before the two tensor-core layers and, after them, polishes the
// predicted temperature by one Newton step with the residual check, or runs the plain
// Newton iteration (fallback, counted; also when the engine's waits ran out).
template <typename T>
__global__ void __launch_bounds__(dgtc5::THREADS, 4)
thermo_mlp_kernel(const T* u, int64_t K, int np, int dim, const double* sp, const float* sp32, double* Tc,
                  T* pc, unsigned long long* status, const DgMlpDev* mlp, unsigned long long* stats) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  dgtc5::Smem<1, 1>& sm = *reinterpret_cast<dgtc5::Smem<1, 1>*>(smem_raw);
  dgtc5::alloc_tmem<1, 1>(sm);
  __shared__ DgMlpDev m;
  copy_to_smem(m, mlp);
  __syncthreads();
  dgtc5::load_weights<1, 1>(sm, m.w);
  const int nv = NSPEC + dim + 1;
  const int64_t total = K * np;
  unsigned long long n_ok = 0, n_fb = 0;
  double Y[NSPEC], rho = 1.0, e = 0.0;  // this thread's node, carried from features to polish
  auto prod = [&](int64_t i, float* x, int) {
    if (i < total) {
      const T* uu = u + (i / np) * nv * np + (i % np);
      rho = 0.0;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) {
        Y[q] = (double)uu[q * np];
        rho += Y[q];
      }
      double ke = 0.0;
      for (int d = 0; d < dim; ++d) {
        const double mm = (double)uu[(NSPEC + d) * np];
        ke += mm * mm;
      }
      const double ir = 1.0 / rho;
      e = (double)uu[(NSPEC + dim) * np] * ir - 0.5 * ke * ir * ir;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) Y[q] *= ir;
    } else {
      rho = 1.0;
      e = 0.0;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) Y[q] = 0.2;
    }
    float f[NI];
#pragma unroll
    for (int q = 0; q < NSPEC; ++q) f[q] = (float)Y[q];
    f[5] = logf((float)rho);
    f[6] = (float)e;
#pragma unroll
    for (int q = 0; q < NI; ++q) x[q] = (f[q] - m.mean[q]) * m.inv_std[q];
    x[7] = 0.f;
    return true;
  };
  // the plain FP64 Newton iteration from T1 (fallback); false when it did not converge
  auto newton = [&](const PolyD& P, double& T1) {
    for (int it = 0; it < 50; ++it) {
      const double Tn = clampT(T1 - (P.e(T1) - e) / P.cv(T1));
      const double step = fabs(Tn - T1);
      T1 = Tn;
      if (step <= 1e-12 * T1) return true;
    }
    return false;
  };
  auto cons = [&](int64_t i, const float* y, bool, bool valid, int) {
    if (i >= total) return;
    const int64_t k = i / np;
    const int node = (int)(i % np);
    if (sizeof(T) == 4) {
      // mixed form: the same equation as its plain solve -- FP64 formation-energy constant
      // b0, FP32-rounded temperature coefficients, FP64 residual -- so accepted nodes and
      // the plain path agree to the acceptance tolerance
      float c32[6], R32 = 0.f;
      double b0 = 0.0;
#pragma unroll
      for (int q = 0; q < 6; ++q) c32[q] = 0.f;
#pragma unroll
      for (int q = 0; q < NSPEC; ++q) {
        b0 += Y[q] * sp[8 * q];
        const float yf = (float)Y[q];
#pragma unroll
        for (int r = 1; r < 6; ++r) c32[r] += yf * sp32[8 * q + r];
        R32 += yf * sp32[8 * q + 6];
      }
      auto e64 = [&](double t) {
        return b0 + t * ((double)c32[1] + t * ((double)c32[2] + t * ((double)c32[3] +
                         t * ((double)c32[4] + t * (double)c32[5]))));
      };
      auto cv32 = [&](float t) {
        return c32[1] + t * (2.f * c32[2] + t * (3.f * c32[3] + t * (4.f * c32[4] + t * 5.f * c32[5])));
      };
      double T1 = 1000.0;
      bool acc = false;
      if (valid) {
        const double T0 = clampT((double)(m.muT + m.sigT * y[0]));
        const float cv0 = cv32((float)T0);
        T1 = clampT(T0 - (e64(T0) - e) * (double)(1.0f / cv0));
        acc = fabs(e64(T1) - e) <= 1e-6 * (double)cv0 * T1;
      }
      if (acc) {
        ++n_ok;
      } else {
        ++n_fb;
        PolyD P;
        poly_d(sp, Y, P);
        if (!newton(P, T1)) atomicCAS(status, 0ull, (DG_ST_NEWTON << 56) | (unsigned long long)k);
      }
      Tc[k * np + node] = T1;
      const float Tq = (float)T1, rhof = (float)rho;
      const float pf = rhof * R32 * Tq, cvf = cv32(Tq);
      pc[(k * 2 + 0) * np + node] = (T)pf;
      pc[(k * 2 + 1) * np + node] = (T)sqrtf((cvf + R32) / cvf * pf / rhof);
    } else {
      PolyD P;
      poly_d(sp, Y, P);
      double T1 = 1000.0;
      bool acc = false;
      if (valid) {
        const double T0 = clampT((double)(m.muT + m.sigT * y[0]));
        // FP64 residuals; cv only scales the correction, FP32 is enough for it
        const float cv0 = (float)P.b[1] + (float)T0 * (2.f * (float)P.b[2] + (float)T0 *
                          (3.f * (float)P.b[3] + (float)T0 * (4.f * (float)P.b[4] + (float)T0 * 5.f * (float)P.b[5])));
        T1 = clampT(T0 - (P.e(T0) - e) / (double)cv0);
        acc = fabs(P.e(T1) - e) <= 1e-6 * (double)cv0 * T1;
      }
      if (acc) {
        ++n_ok;
      } else {
        ++n_fb;
        if (!newton(P, T1)) atomicCAS(status, 0ull, (DG_ST_NEWTON << 56) | (unsigned long long)k);
      }
      Tc[k * np + node] = T1;
      const double p = rho * P.Rmix * T1, cv = P.cv(T1);
      pc[(k * 2 + 0) * np + node] = (T)p;
      pc[(k * 2 + 1) * np + node] = (T)sqrt((cv + P.Rmix) / cv * p / rho);
    }
  };
  dgtc5::run_tiles<1, 1>(sm, total, prod, cons);
  if (stats) {
    for (int o = 16; o > 0; o >>= 1) {
      n_ok += __shfl_xor_sync(0xffffffffu, n_ok, o);
      n_fb += __shfl_xor_sync(0xffffffffu, n_fb, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&stats[0], n_ok);
      atomicAdd(&stats[1], n_fb);
    }
  }
}

// plain tensor-core forward for standardised inputs X[n][7] -> y[n][NO] (checks)
template <int NO>
__global__ void __launch_bounds__(32 * MLP_WARPS)
mlp_forward_tc_kernel(const DgMlpW<NO>* mlp, const float* X, float* y, int64_t n) {
  __shared__ DgMlpW<NO> m;
  __shared__ float feat[MLP_WARPS][16][17];
  __shared__ float yv[MLP_WARPS][NO][16];
  copy_to_smem(m, mlp);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t base = ((int64_t)blockIdx.x * MLP_WARPS + w) * 16; base < n;
       base += (int64_t)gridDim.x * MLP_WARPS * 16) {
    if (lane < 16) {
      const int64_t i = base + lane;
#pragma unroll
      for (int q = 0; q < 17; ++q) feat[w][lane][q] = (i < n && q < NI) ? X[i * NI + q] : 0.f;
    }
    __syncwarp();
    mlp16<NO>(m, feat[w], yv[w]);
    __syncwarp();
    if (lane < 16 && base + lane < n)
      for (int o = 0; o < NO; ++o) y[(base + lane) * NO + o] = yv[w][o][lane];
    __syncwarp();
  }
}

// FP32 SIMT forward of one sample per thread (reference path of the device code)
__global__ void mlp_forward_f32_kernel(const float* P, int no, const float* X, float* y, int64_t n) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    float h1[NH], h2[NH];
    for (int j = 0; j < NH; ++j) {
      float a = P[NH * NI + j];
      for (int k = 0; k < NI; ++k) a += P[j * NI + k] * X[s * NI + k];
      h1[j] = gelu_f(a);
    }
    for (int j = 0; j < NH; ++j) {
      float a = P[NH * NI + NH + NH * NH + j];
      for (int i = 0; i < NH; ++i) a += P[NH * NI + NH + j * NH + i] * h1[i];
      h2[j] = gelu_f(a);
    }
    for (int o = 0; o < no; ++o) {
      float out = P[dg_mlp_off_b3(no) + o];
      for (int j = 0; j < NH; ++j) out += P[dg_mlp_off_w3() + o * NH + j] * h2[j];
      y[s * no + o] = out;
    }
  }
}

// ------------------------------------------------------------------ training (FP32)
#define TS 32  // samples per tile
#define OFF_W1 0
#define OFF_B1 (NH * NI)
#define OFF_W2 (OFF_B1 + NH)
#define OFF_B2 (OFF_W2 + NH * NH)
constexpr int TT = 256;        // threads of a training CTA
constexpr int HP = NH + 4;     // padded row of a [sample][unit] array: float4 rows on distinct banks
constexpr int XP = NI + 1;     // features and a constant 1 (the bias column of layer 1's gradient)
struct __align__(16) TrainSmem {
  float W2[NH][NH], W2T[NH][HP];  // [j][i], [i][j]
  float W3[NO_MAX][HP];
  float h1[TS][HP], e1[TS][HP], h2[TS][HP], e2[TS][HP];  // activations, and GELU's derivative (e2: delta 2)
  float W1[NH][XP], b2[NH], b3[NO_MAX], X[TS][XP];
  float dy[TS][NO_MAX], r2[TS][NO_MAX];
};

// GELU and its derivative from one tanh
__device__ __forceinline__ void gelu_and_d(float x, float& g, float& d) {
  const float k = 0.7978845608028654f;
  const float t = tanhf(k * (x + 0.044715f * x * x * x));
  g = 0.5f * x * (1.0f + t);
  d = 0.5f * (1.0f + t) + 0.5f * x * (1.0f - t * t) * k * (1.0f + 3.0f * 0.044715f * x * x);
}

// acc[r][c] += sum over q of a[row r][q] b[q][col c] for this thread's 2 rows and 4 columns
// (a [.][HP], b [NH][LD])
template <int LD>
__device__ __forceinline__ void tile_2x4(const float* a0, const float* a1, const float* b, float (*acc)[4]) {
#pragma unroll 4
  for (int q = 0; q < NH; q += 4) {
    const float4 u = *reinterpret_cast<const float4*>(a0 + q), v = *reinterpret_cast<const float4*>(a1 + q);
    const float x0[4] = {u.x, u.y, u.z, u.w}, x1[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const float4 w = *reinterpret_cast<const float4*>(b + (q + r) * LD);
      acc[0][0] += x0[r] * w.x; acc[0][1] += x0[r] * w.y; acc[0][2] += x0[r] * w.z; acc[0][3] += x0[r] * w.w;
      acc[1][0] += x1[r] * w.x; acc[1][1] += x1[r] * w.y; acc[1][2] += x1[r] * w.z; acc[1][3] += x1[r] * w.w;
    }
  }
}

// per-CTA partial gradients of loss = (1/(B no)) sum_s sum_o (y_so - t_so)^2 over the
// CTA's tiles of TS samples, summed in a fixed order.  The three 64-wide products of a tile (layer 2,
// its transpose, its gradient) are 2 x 4 and 4 x 4 register tiles over 256 threads with 16-byte
// shared-memory reads; the gradient sums stay in registers over the tiles.  With 64 threads, one
// per unit, and every operand read 4 bytes at a time, a fitting iteration (two
// gathers, this, Adam) with a batch of 4,096 and ten outputs took 88 us, then 36, and 25 since the
// launches overlap (dg_launch.cuh); what is left is the chain of eight barriers of one tile per CTA
// (128 CTAs) and the launches.
__global__ void __launch_bounds__(TT) mlp_grad_kernel(const float* P, int no, const float* X, const float* t, int B,
                                                      float* partial) {
  extern __shared__ __align__(16) unsigned char raw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(raw);
  const int tid = threadIdx.x;
  const int OW3 = dg_mlp_off_w3(), OB3 = dg_mlp_off_b3(no), NPAR = dg_mlp_np(no);
  pdl_wait();
#pragma unroll 4
  for (int q = tid; q < NH * NH; q += TT) {
    const float w = P[OFF_W2 + q];
    S.W2[q / NH][q % NH] = w;
    S.W2T[q % NH][q / NH] = w;
  }
  for (int q = tid; q < NH * NI; q += TT) S.W1[q / NI][q % NI] = P[OFF_W1 + q];
  if (tid < NH) {
    S.W1[tid][NI] = P[OFF_B1 + tid];
    S.b2[tid] = P[OFF_B2 + tid];
  }
  for (int q = tid; q < no * NH; q += TT) S.W3[q / NH][q % NH] = P[OW3 + q];
  if (tid < no) S.b3[tid] = P[OB3 + tid];
  const float inv = 1.0f / ((float)B * (float)no);
  // thread roles: unit j of the one-unit passes with 8 samples from s8; columns 4 c4 of the tiled
  // passes with rows 2 r2 (samples) or 4 r2 (units)
  const int j = tid & (NH - 1), s8 = (tid >> 6) * 8, c4 = (tid & 15) * 4, rw = tid >> 4;
  float gW2[4][4] = {}, gW3[NO_MAX / 4] = {}, gW1[2] = {0.f, 0.f}, gb2 = 0.f, gb3 = 0.f, loss = 0.f;
  for (int s0 = blockIdx.x * TS; s0 < B; s0 += gridDim.x * TS) {
    const int ns = min(TS, B - s0);
    // samples past the batch: zero features, and zero dy below, add nothing
    for (int q = tid; q < TS * XP; q += TT) {
      const int s = q / XP, k = q % XP;
      S.X[s][k] = k == NI ? 1.0f : (s < ns ? X[(int64_t)(s0 + s) * NI + k] : 0.0f);
    }
    __syncthreads();
#pragma unroll 2
    for (int s = s8; s < s8 + 8; ++s) {
      float a = S.W1[j][NI];
#pragma unroll
      for (int k = 0; k < NI; ++k) a += S.W1[j][k] * S.X[s][k];
      gelu_and_d(a, S.h1[s][j], S.e1[s][j]);
    }
    __syncthreads();
    {
      float acc[2][4];
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[0][c] = acc[1][c] = S.b2[c4 + c];
      tile_2x4<HP>(S.h1[2 * rw], S.h1[2 * rw + 1], &S.W2T[0][c4], acc);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) gelu_and_d(acc[r][c], S.h2[2 * rw + r][c4 + c], S.e2[2 * rw + r][c4 + c]);
    }
    __syncthreads();
    for (int q = tid; q < TS * no; q += TT) {
      const int s = q / no, o = q % no;
      float y = S.b3[o];
#pragma unroll 4
      for (int i = 0; i < NH; i += 4) {
        const float4 w = *reinterpret_cast<const float4*>(&S.W3[o][i]);
        const float4 h = *reinterpret_cast<const float4*>(&S.h2[s][i]);
        y += w.x * h.x;
        y += w.y * h.y;
        y += w.z * h.z;
        y += w.w * h.w;
      }
      const float r = s < ns ? y - t[(int64_t)(s0 + s) * no + o] : 0.0f;
      S.dy[s][o] = 2.0f * r * inv;
      S.r2[s][o] = r * r * inv;
    }
    __syncthreads();
    // the output layer's gradients, then delta 2 in place of GELU's derivative
#pragma unroll
    for (int m = 0; m < NO_MAX / 4; ++m) {
      const int o = (tid >> 6) + 4 * m;
      if (o < no) {
        float g = 0.f;
#pragma unroll 8
        for (int s = 0; s < TS; ++s) g += S.dy[s][o] * S.h2[s][j];
        gW3[m] += g;
      }
    }
    if (tid < no) {
      float g = 0.f, l = 0.f;
      for (int s = 0; s < TS; ++s) {
        g += S.dy[s][tid];
        l += S.r2[s][tid];
      }
      gb3 += g;
      loss += l;
    }
#pragma unroll 2
    for (int s = s8; s < s8 + 8; ++s) {
      float back = 0.f;
      for (int o = 0; o < no; ++o) back += S.dy[s][o] * S.W3[o][j];
      S.e2[s][j] *= back;
    }
    __syncthreads();
    // layer 2's gradient (units 4 rw.. x inputs c4..)
    {
      float g[4][4] = {};
#pragma unroll 4
      for (int s = 0; s < TS; ++s) {
        const float4 d = *reinterpret_cast<const float4*>(&S.e2[s][4 * rw]);
        const float4 h = *reinterpret_cast<const float4*>(&S.h1[s][c4]);
        const float dd[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          g[r][0] += dd[r] * h.x;
          g[r][1] += dd[r] * h.y;
          g[r][2] += dd[r] * h.z;
          g[r][3] += dd[r] * h.w;
        }
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) gW2[r][c] += g[r][c];
    }
    if (tid < NH) {
      float g = 0.f;
#pragma unroll 8
      for (int s = 0; s < TS; ++s) g += S.e2[s][tid];
      gb2 += g;
    }
    // delta 1 = (delta 2 W2) gelu'(a1), in place of the derivative
    {
      float acc[2][4] = {};
      tile_2x4<NH>(S.e2[2 * rw], S.e2[2 * rw + 1], &S.W2[0][c4], acc);
#pragma unroll
      for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) S.e1[2 * rw + r][c4 + c] *= acc[r][c];
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 2; ++m) {  // layer 1: unit q / XP, feature q % XP (the last: the bias)
      const int q = tid + m * TT;
      float g = 0.f;
#pragma unroll 8
      for (int s = 0; s < TS; ++s) g += S.e1[s][q / XP] * S.X[s][q % XP];
      gW1[m] += g;
    }
    __syncthreads();
  }
  static_assert(NH * XP == 2 * TT, "two entries of layer 1's gradient per thread");
  float* out = partial + (int64_t)blockIdx.x * (NPAR + 1);
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) out[OFF_W2 + (4 * rw + r) * NH + c4 + c] = gW2[r][c];
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    const int q = tid + m * TT, u = q / XP, k = q % XP;
    out[k == NI ? OFF_B1 + u : OFF_W1 + u * NI + k] = gW1[m];
  }
#pragma unroll
  for (int m = 0; m < NO_MAX / 4; ++m) {
    const int o = (tid >> 6) + 4 * m;
    if (o < no) out[OW3 + o * NH + j] = gW3[m];
  }
  if (tid < NH) out[OFF_B2 + tid] = gb2;
  if (tid < no) {
    out[OB3 + tid] = gb3;
    S.r2[0][tid] = loss;
  }
  __syncthreads();
  if (tid == 0) {
    float l = 0.f;
    for (int o = 0; o < no; ++o) l += S.r2[0][o];
    out[NPAR] = l;
  }
}

// fixed-order sum of the partial gradients, then (optionally) one Adam step.  A CTA takes 32
// parameters, eight slices of the partials each, so that a parameter's sum is a chain of nb / 8
// loads instead of nb.
__global__ void __launch_bounds__(256) mlp_reduce_adam_kernel(const float* partial, int nb, int npar, float* grad,
                                                              float* P, float* mo, float* vo, int step, float lr,
                                                              float b1, float b2, float eps, double* loss) {
  __shared__ float part[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + lane;
  float s = 0.f;
  pdl_wait();
  if (q <= npar) {
#pragma unroll 8
    for (int b = w; b < nb; b += 8) s += partial[(int64_t)b * (npar + 1) + q];
  }
  part[w][lane] = s;
  __syncthreads();
  if (w != 0 || q > npar) return;
#pragma unroll
  for (int i = 1; i < 8; ++i) s += part[i][lane];
  if (q == npar) {
    if (loss) *loss = (double)s;
    return;
  }
  if (grad) grad[q] = s;
  if (P) {
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    const float m = b1 * mo[q] + (1.0f - b1) * s;
    const float v = b2 * vo[q] + (1.0f - b2) * s * s;
    mo[q] = m;
    vo[q] = v;
    P[q] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
  }
}

// counter-based sampling of node states (splitmix64 of seed + index)
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

template <typename T>
__global__ void sample_kernel(const T* u, const double* Tc, int64_t K, int np, int dim, int64_t n,
                              uint64_t seed, float* X, float* Tout) {
  const int nv = NSPEC + dim + 1;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = (int64_t)(splitmix64(seed + (uint64_t)j) % (uint64_t)(K * np));
    const int64_t k = i / np;
    const int node = (int)(i % np);
    const T* uu = u + k * nv * np + node;
    double rho = 0.0, ke = 0.0;
    for (int s = 0; s < NSPEC; ++s) rho += (double)uu[s * np];
    for (int d = 0; d < dim; ++d) {
      const double mm = (double)uu[(NSPEC + d) * np];
      ke += mm * mm;
    }
    for (int s = 0; s < NSPEC; ++s) X[j * NI + s] = (float)((double)uu[s * np] / rho);
    X[j * NI + 5] = (float)log(rho);
    X[j * NI + 6] = (float)((double)uu[(NSPEC + dim) * np] / rho - 0.5 * ke / (rho * rho));
    Tout[j] = (float)Tc[i];
  }
}

unsigned grid_of(int64_t n, int bs) {
  int64_t g = (n + bs - 1) / bs;
  if (g > 152 * 32) g = 152 * 32;
  return (unsigned)(g < 1 ? 1 : g);
}

void pack_host(const float* params, const double* stats, DgMlpDev* h) {
  memset(h, 0, sizeof(*h));
  dg_mlp_pack<1>(params, &h->w);
  for (int q = 0; q < NI; ++q) {
    h->mean[q] = (float)stats[q];
    h->inv_std[q] = (float)(1.0 / stats[NI + q]);
  }
  h->muT = (float)stats[2 * NI];
  h->sigT = (float)stats[2 * NI + 1];
}

}  // namespace

// ---------------------------------------------------------------- thermo hooks
cudaError_t dg_mlp_set(DgThermo* th, const float* params_host, const double* stats_host) {
  if (!params_host) {
    if (th->mlp) cudaFree(th->mlp);
    th->mlp = NULL;
    return cudaSuccess;
  }
  DgMlpDev h;
  pack_host(params_host, stats_host, &h);
  cudaError_t e = cudaSuccess;
  if (!th->mlp) e = cudaMalloc(&th->mlp, sizeof(DgMlpDev));
  if (e == cudaSuccess && !th->mlp_stats) e = cudaMalloc((void**)&th->mlp_stats, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMemset(th->mlp_stats, 0, 2 * sizeof(unsigned long long));
  if (e == cudaSuccess) e = cudaMemcpy(th->mlp, &h, sizeof(h), cudaMemcpyHostToDevice);
  return e;
}

cudaError_t dg_mlp_thermo_update(DgThermo* th, const void* u, int f32, cudaStream_t s) {
  const int64_t n = th->K * th->np;
  // persistent CTAs over tensor-core tiles of 128 nodes
  const size_t smem = sizeof(dgtc5::Smem<1, 1>);
  const int64_t t128 = (n + dgtc5::ROWS - 1) / dgtc5::ROWS;
  const unsigned grid = (unsigned)(t128 < 152 * 4 ? t128 : 152 * 4);
  cudaError_t e;
  if (f32) {
    auto k = thermo_mlp_kernel<float>;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, dgtc5::THREADS, smem, s>>>((const float*)u, th->K, th->np, th->dim, th->species, th->coef32, th->T,
                                         (float*)th->pc, th->status, (const DgMlpDev*)th->mlp, th->mlp_stats);
  } else {
    auto k = thermo_mlp_kernel<double>;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, dgtc5::THREADS, smem, s>>>((const double*)u, th->K, th->np, th->dim, th->species, th->coef32,
                                         th->T, (double*)th->pc, th->status, (const DgMlpDev*)th->mlp,
                                         th->mlp_stats);
  }
  return cudaGetLastError();
}

cudaError_t dg_mlp_sample(DgThermo* th, const void* u, int f32, int64_t n, uint64_t seed, float* X,
                          float* T, cudaStream_t s) {
  if (f32)
    sample_kernel<float><<<grid_of(n, 256), 256, 0, s>>>((const float*)u, th->T, th->K, th->np, th->dim,
                                                         n, seed, X, T);
  else
    sample_kernel<double><<<grid_of(n, 256), 256, 0, s>>>((const double*)u, th->T, th->K, th->np, th->dim,
                                                          n, seed, X, T);
  return cudaGetLastError();
}

// tcgen05 forward: persistent CTAs of 128 threads over 256-row tiles
__device__ unsigned g_tc5_err;
template <int NO>
static dg_status forward_tc5(const float* P, const float* X, float* y, int64_t n, cudaStream_t st) {
  const size_t smem = sizeof(dgtc5::Smem<NO, dgtc5::FWD_NR>);
  auto k = dgtc5::mlp_forward_tc5_kernel<NO>;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100) != cudaSuccess)
    return DG_ECUDA;
  unsigned* err = NULL;
  if (cudaGetSymbolAddress((void**)&err, g_tc5_err) != cudaSuccess) return DG_ECUDA;
  if (cudaMemsetAsync(err, 0, sizeof(unsigned), st) != cudaSuccess) return DG_ECUDA;
  const int64_t rows = dgtc5::FWD_NR * dgtc5::ROWS, tiles = (n + rows - 1) / rows;
  const int64_t ctas = 152 * 2 * dgtc5::FWD_CTAS;  // two waves of resident CTAs: 339 against 350 us at 4.6 M rows
  const unsigned grid = (unsigned)(tiles < ctas ? tiles : ctas);
  const int vec = (((uintptr_t)X | (uintptr_t)y) & 15) == 0;
  k<<<grid, dgtc5::THREADS, smem, st>>>(P, X, y, n, err, vec);
  if (cudaGetLastError() != cudaSuccess) return DG_ECUDA;
  unsigned h = 0;
  if (cudaMemcpyAsync(&h, err, sizeof(unsigned), cudaMemcpyDeviceToHost, st) != cudaSuccess) return DG_ECUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return DG_ECUDA;
  return h ? DG_ETIMEOUT : DG_OK;
}

template <int NO>
static dg_status forward_tc(const float* hp, const float* X, float* y, int64_t n, cudaStream_t st) {
  DgMlpW<NO> h;
  memset(&h, 0, sizeof(h));
  dg_mlp_pack<NO>(hp, &h);
  DgMlpW<NO>* d = NULL;
  if (cudaMalloc((void**)&d, sizeof(h)) != cudaSuccess) return DG_ENOMEM;
  cudaError_t e = cudaMemcpy(d, &h, sizeof(h), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    mlp_forward_tc_kernel<NO><<<grid_of((n + 15) / 16, MLP_WARPS), 32 * MLP_WARPS, 0, st>>>(d, X, y, n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d);
  return e == cudaSuccess ? DG_OK : DG_ECUDA;
}

// FP32 forward launch for the data-preparation module (dg_data.cu)
cudaError_t dg_mlp_forward_f32_launch(const float* P, int no, const float* X, float* y, int64_t n, cudaStream_t s) {
  mlp_forward_f32_kernel<<<grid_of(n, 128), 128, 0, s>>>(P, no, X, y, n);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- C ABI (training)
extern "C" {

int dg_mlp_nparams(int n_out) { return n_out >= 1 && n_out <= NO_MAX ? dg_mlp_np(n_out) : -1; }

size_t dg_mlp_workspace_bytes(int batch, int n_out) {
  if (batch < 1 || n_out < 1 || n_out > NO_MAX) return 0;
  int nb = (batch + TS - 1) / TS;
  if (nb > 152) nb = 152;
  return sizeof(float) * (size_t)nb * (dg_mlp_np(n_out) + 1);
}

static dg_status grad_common(const float* P, int no, const float* X, const float* t, int B, float* ws,
                             size_t ws_bytes, cudaStream_t st, int* nb_out) {
  if (!P || !X || !t || !ws || B < 1 || no < 1 || no > NO_MAX) return DG_EINVAL;
  if (ws_bytes < dg_mlp_workspace_bytes(B, no)) return DG_EINVAL;
  int nb = (B + TS - 1) / TS;
  if (nb > 152) nb = 152;
  const size_t smem = sizeof(TrainSmem);
  if (cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
      cudaSuccess)
    return DG_ECUDA;
  if (launch_pdl(false, mlp_grad_kernel, nb, TT, smem, st, P, no, X, t, B, ws) != cudaSuccess) return DG_ECUDA;
  *nb_out = nb;
  return DG_OK;
}

dg_status dg_mlp_grad(const float* params, int n_out, const float* X, const float* t, int batch, float* grad,
                      double* loss, float* workspace, size_t ws_bytes, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  int nb = 0;
  dg_status r = grad_common(params, n_out, X, t, batch, workspace, ws_bytes, st, &nb);
  if (r != DG_OK) return r;
  if (!grad) return DG_EINVAL;
  const int npar = dg_mlp_np(n_out);
  return launch_pdl(false, mlp_reduce_adam_kernel, (npar + 1 + 31) / 32, 256, 0, st, workspace, nb, npar, grad, (float*)NULL,
                    (float*)NULL, (float*)NULL, 0, 0.f, 0.f, 0.f, 0.f, loss) == cudaSuccess
             ? DG_OK
             : DG_ECUDA;
}

dg_status dg_mlp_train_step(float* params, int n_out, float* m, float* v, const float* X, const float* t,
                            int batch, int step, float lr, double* loss, float* workspace, size_t ws_bytes,
                            void* stream) {
  if (!m || !v || step < 1 || !(lr > 0.f)) return DG_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  int nb = 0;
  dg_status r = grad_common(params, n_out, X, t, batch, workspace, ws_bytes, st, &nb);
  if (r != DG_OK) return r;
  const int npar = dg_mlp_np(n_out);
  return launch_pdl(false, mlp_reduce_adam_kernel, (npar + 1 + 31) / 32, 256, 0, st, workspace, nb, npar, (float*)NULL, params,
                    m, v, step, lr, 0.9f, 0.999f, 1e-8f, loss) == cudaSuccess
             ? DG_OK
             : DG_ECUDA;
}

dg_status dg_mlp_forward(const float* params, int n_out, const float* X, float* y, int64_t n, int tensor_cores,
                         void* stream) {
  if (!params || !X || !y || n < 1 || n_out < 1 || n_out > NO_MAX) return DG_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  if (!tensor_cores) {
    mlp_forward_f32_kernel<<<grid_of(n, 128), 128, 0, st>>>(params, n_out, X, y, n);
    return cudaGetLastError() == cudaSuccess ? DG_OK : DG_ECUDA;
  }
  if (n_out != 1 && n_out != 10) return DG_EINVAL;  // the surrogates' output counts
  if (tensor_cores == 2) return n_out == 1 ? forward_tc5<1>(params, X, y, n, st) : forward_tc5<10>(params, X, y, n, st);
  if (tensor_cores != 1) return DG_EINVAL;
  const int npar = dg_mlp_np(n_out);
  float* hp = (float*)malloc(sizeof(float) * npar);
  if (!hp) return DG_ENOMEM;
  if (cudaMemcpy(hp, params, sizeof(float) * npar, cudaMemcpyDeviceToHost) != cudaSuccess) {
    free(hp);
    return DG_ECUDA;
  }
  dg_status r = n_out == 1 ? forward_tc<1>(hp, X, y, n, st) : forward_tc<10>(hp, X, y, n, st);
  free(hp);
  return r;
}

}  // extern "C"
