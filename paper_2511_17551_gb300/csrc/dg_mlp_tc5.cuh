// Fifth-generation tensor-core (tcgen05) forward of the 7 -> 64 -> 64 -> NO perceptron:
// one CTA of four warps evaluates tiles of NR x 128 rows, NR rows per thread.  Layers 1 and 2 are tcgen05.mma
// (kind::f16, BF16 operands from shared memory, FP32 accumulators in tensor memory);
// the epilogue of each reads its 32 rows per warp back with tcgen05.ld, adds the bias and
// applies GELU; the layer-2 epilogue also forms the NO outputs as FP32 dot products with
// W3 (as the warp-level path does), so the hidden units are rounded to BF16 only once.
//
// Shared-memory operands use the no-swizzle K-major canonical layout: core matrices of
// 8 rows x 16 bytes (8 BF16 of K), 128 bytes each; the two core matrices of a 16-wide K
// slice sit LBO = 128 bytes apart and consecutive 8-row groups SBO = (K/8) x 128 bytes
// apart, so element (row, k) of a [R][K] operand is at
//   (row/8) SBO + (k/8) 128 + (row%8) 16 + (k%8) 2 bytes.
// Tensor memory: 128 lanes (rows) x NR x 64 columns; layer 2 overwrites layer 1's accumulators,
// which every warp has read by then.  What bounds the engine: per row 128 tanh (MUFU) and about
// 1,100 other instructions, and the reads of the output layer's weights from shared memory
// (a 16-byte broadcast takes four cycles of its 128 bytes per cycle): with NR = 2 each weight
// serves two rows, and the two rows' chains fill each other's latencies.  Bias, GELU and output
// layer go two columns at a time through the packed FP32 operations.  4.6 M rows with ten outputs:
// 344 us a call (502 with one row per thread, 128 columns and scalar FP32; of it 30 us are the
// call's launch and wait).  Measured on copies: without the tanh the same time, without the
// output weights' loads 35 us less, with scalar FP32 26 us more; one row per thread 376 us at best.
// Every wait on an mbarrier
// is bounded; on a timeout the kernel records it, waits once more (bounded) for its MMAs in
// flight, frees its tensor memory and returns.
#pragma once
#include "dg_mlp.cuh"

namespace dgtc5 {

constexpr int ROWS = 128;     // rows per MMA (its M)
constexpr int THREADS = 128;  // four warps: one TMEM lane quarter each

template <int NO, int NR>
struct __align__(1024) Smem {
  __nv_bfloat16 X[NR * ROWS * 16];               // A of layer 1 [NR][128][16], features zero padded
  __nv_bfloat16 H[NR * ROWS * DG_MLP_NH];        // A of layer 2 [NR][128][64]
  __nv_bfloat16 W1[DG_MLP_NH * 16];              // B of layer 1 [64][16]
  __nv_bfloat16 W2[DG_MLP_NH * DG_MLP_NH];       // B of layer 2 [64][64]
  __align__(16) float b1[DG_MLP_NH], b2[DG_MLP_NH];
  __align__(16) float W3[NO][DG_MLP_NH];
  float b3[NO];
  unsigned long long bar;
  uint32_t tmem;
};

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// byte offset of element (row, k) in a K-major canonical operand with K columns
__device__ __forceinline__ uint32_t canon(int row, int k, int K) {
  return (uint32_t)((row >> 3) * (K / 8) * 128 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// shared-memory matrix descriptor: start address, LBO, SBO (all >> 4), descriptor
// version 1 (bits 46-47), base offset 0, no swizzle
__device__ __forceinline__ uint64_t sdesc(const void* p, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((su32(p) >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9 and
// 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, int acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(su32(bar))
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// generic-proxy writes to shared memory made visible to the tensor cores (async proxy)
__device__ __forceinline__ void fence_smem_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ bool wait_parity(unsigned long long* bar, uint32_t parity) {
  for (int it = 0; it < (1 << 16); ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(su32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// 16 consecutive FP32 columns of this thread's TMEM lane (as bits): valid after ld_wait, which
// takes the registers as in-out operands so that no use of them moves before the wait
__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void ld_wait(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ float2 pair_of(const uint32_t* r) {
  return make_float2(__uint_as_float(r[0]), __uint_as_float(r[1]));
}

// weights from the FP32 parameter vector (layout of dg_mlp_np) into the canonical
// BF16 operands, biases and the FP32 output layer
template <int NO, int NR>
__device__ __forceinline__ void load_weights(Smem<NO, NR>& s, const float* P) {
  constexpr int NI = DG_MLP_NI, NH = DG_MLP_NH;
  const int tid = threadIdx.x;
  for (int i = tid; i < NH * 16; i += THREADS) {
    const int j = i / 16, k = i % 16;
    *reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<unsigned char*>(s.W1) + canon(j, k, 16)) =
        __float2bfloat16(k < NI ? P[j * NI + k] : 0.0f);
  }
  // eight k at a time (one core-matrix row), all loads in flight
#pragma unroll
  for (int i = 0; i < NH * NH / 8 / THREADS; ++i) {
    const int q = tid + i * THREADS, j = q / (NH / 8), k = q % (NH / 8) * 8;
    const float* w = P + NH * NI + NH + j * NH + k;
    uint32_t pk[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) pk[c] = dgmlp::pack_bf16(w[2 * c], w[2 * c + 1]);
    *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.W2) + canon(j, k, NH)) =
        make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
  for (int j = tid; j < NH; j += THREADS) {
    s.b1[j] = P[NH * NI + j];
    s.b2[j] = P[NH * NI + NH + NH * NH + j];
  }
  for (int i = tid; i < NO * NH; i += THREADS) s.W3[i / NH][i % NH] = P[dg_mlp_off_w3() + i];
  if (tid < NO) s.b3[tid] = P[dg_mlp_off_b3(NO) + tid];
}

// the same from a packed BF16 weight image (dg_mlp_pack)
template <int NO, int NR>
__device__ __forceinline__ void load_weights(Smem<NO, NR>& s, const DgMlpW<NO>& w) {
  constexpr int NH = DG_MLP_NH;
  const int tid = threadIdx.x;
  // eight k at a time (one core-matrix row)
#pragma unroll
  for (int i = 0; i < NH * 16 / 8 / THREADS; ++i) {
    const int q = tid + i * THREADS;
    *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.W1) + canon(q / 2, q % 2 * 8, 16)) =
        reinterpret_cast<const uint4*>(w.W1)[q];
  }
#pragma unroll
  for (int i = 0; i < NH * NH / 8 / THREADS; ++i) {
    const int q = tid + i * THREADS;
    *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.W2) + canon(q / (NH / 8), q % (NH / 8) * 8, NH)) =
        reinterpret_cast<const uint4*>(w.W2)[q];
  }
  for (int j = tid; j < NH; j += THREADS) {
    s.b1[j] = w.b1[j];
    s.b2[j] = w.b2[j];
  }
  for (int i = tid; i < NO * NH; i += THREADS) s.W3[i / NH][i % NH] = w.W3[i / NH][i % NH];
  if (tid < NO) s.b3[tid] = w.b3[tid];
}

__device__ __forceinline__ float tanh_fast(float z) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(z));
  return t;
}
// dgmlp::gelu_fast on two values, bit for bit (the hidden activations are rounded to BF16
// afterwards: another rounding here would move some of them by a BF16 unit)
__device__ __forceinline__ float2 gelu2_exact(float2 x) {
  const float k = 0.7978845608028654f;
  float2 t = __fmul2_rn(make_float2(0.044715f, 0.044715f), x);
  t = __fmul2_rn(t, x);
  const float2 z = __fmul2_rn(make_float2(k, k), __ffma2_rn(t, x, x));
  const float2 h = __fmul2_rn(make_float2(0.5f, 0.5f), x);
  return __fmul2_rn(h, __fadd2_rn(make_float2(1.f, 1.f), make_float2(tanh_fast(z.x), tanh_fast(z.y))));
}
// the same function in fewer operations (FP32 rounding differs): for the output layer's inputs
__device__ __forceinline__ float2 gelu2(float2 x) {
  const float k = 0.7978845608028654f, k3 = 0.7978845608028654f * 0.044715f;
  const float2 z = __fmul2_rn(x, __ffma2_rn(make_float2(k3, k3), __fmul2_rn(x, x), make_float2(k, k)));
  const float2 h = __fmul2_rn(make_float2(0.5f, 0.5f), x);
  return __ffma2_rn(h, make_float2(tanh_fast(z.x), tanh_fast(z.y)), h);
}

// The tile engine (after alloc_tmem and load_weights): for each tile of NR x 128 rows of the CTA, thread t takes
// the rows tile NR 128 + 128 r + t.  prod(row, x, r) writes the row's 7 standardised features and
// returns a flag of its own; cons(row, out, flag, valid, r) gets the NO outputs, that flag and
// whether the launch's tensor-core waits all completed (when not, out is not valid).  Both are
// called by every thread of the CTA for every tile and r in turn (rows >= n included), so consumers
// may use warp votes.  The engine frees the tensor memory and returns false
// after a timeout (the remaining tiles still reach cons with valid = false, or with STOP are left out:
// for a prod that stages in the operands, which MMAs may then still be reading).  skip(row of
// thread t), called by every thread before a tile and returning the same in all, leaves the tile
// out.  The grid's CTAs from `first` on share the tiles.
// Tensor memory for the engine, first thing in a kernel (its latency then passes beside the loading
// of the weights)
template <int NO, int NR>
__device__ __forceinline__ void alloc_tmem(Smem<NO, NR>& s) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(&s.tmem)),
                 "r"((uint32_t)(64 * NR))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
}
struct NoSkip {
  __device__ __forceinline__ bool operator()(int64_t) const { return false; }
};
template <int NO, int NR, bool STOP = false, class Prod, class Cons, class Skip = NoSkip>
__device__ __forceinline__ bool run_tiles(Smem<NO, NR>& s, int64_t n, Prod prod, Cons cons, Skip skip = Skip(),
                                          int first = 0) {
  constexpr int NH = DG_MLP_NH;
  constexpr uint32_t TMEM_COLS = 64 * NR;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(su32(&s.bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  fence_smem_async();
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = s.tmem;
  const uint32_t lane_base = (uint32_t)(32 * warp) << 16;  // this warp's TMEM lane quarter
  constexpr uint32_t ID_L = idesc_bf16(ROWS, NH);
  uint32_t parity = 0;
  bool ok = true;
  const int64_t tiles = (n + NR * ROWS - 1) / (NR * ROWS);
  for (int64_t tile = blockIdx.x - first; tile < tiles; tile += gridDim.x - first) {
    const int64_t row0 = tile * (NR * ROWS) + tid;
    if (skip(row0)) continue;
    bool flag[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      float x[8];
      flag[r] = prod(row0 + r * ROWS, x, r);
      // features -> A of layer 1 (this thread's row: K 0-7 and the zero padding 8-15)
      uint4 lo;
      lo.x = dgmlp::pack_bf16(x[0], x[1]);
      lo.y = dgmlp::pack_bf16(x[2], x[3]);
      lo.z = dgmlp::pack_bf16(x[4], x[5]);
      lo.w = dgmlp::pack_bf16(x[6], x[7]);
      unsigned char* xb = reinterpret_cast<unsigned char*>(s.X + r * ROWS * 16);
      if (ok) {  // after a timeout MMAs may still be reading the operands (X, and H below)
        *reinterpret_cast<uint4*>(xb + canon(tid, 0, 16)) = lo;
        *reinterpret_cast<uint4*>(xb + canon(tid, 8, 16)) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    if (ok) {
      fence_smem_async();
      fence_before();
      __syncthreads();
      fence_after();
      if (tid == 0) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          mma(tmem + NH * r, sdesc(s.X + r * ROWS * 16, 128, 256), sdesc(s.W1, 128, 256), ID_L, 0);
        commit(&s.bar);
      }
      // the wait's outcome made uniform across the CTA; the phase flips only on completion
      ok = __syncthreads_and(wait_parity(&s.bar, parity)) != 0;
      if (ok) parity ^= 1u;
      fence_after();
    }
    if (ok) {
      // layer-1 epilogue: bias, GELU, BF16 -> A of layer 2 (this thread's rows)
#pragma unroll
      for (int c = 0; c < NH / 16; ++c) {
        uint32_t v[NR][16];
#pragma unroll
        for (int r = 0; r < NR; ++r) ld16(tmem + lane_base + NH * r + 16 * c, v[r]);
#pragma unroll
        for (int r = 0; r < NR; ++r) ld_wait(v[r]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pk[NR][4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float2 b = *reinterpret_cast<const float2*>(&s.b1[16 * c + 8 * h + 2 * q]);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              const float2 g = gelu2_exact(__fadd2_rn(pair_of(v[r] + 8 * h + 2 * q), b));
              pk[r][q] = dgmlp::pack_bf16(g.x, g.y);
            }
          }
#pragma unroll
          for (int r = 0; r < NR; ++r)
            *reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(s.H + r * ROWS * NH) +
                                      canon(tid, 16 * c + 8 * h, NH)) =
                make_uint4(pk[r][0], pk[r][1], pk[r][2], pk[r][3]);
        }
      }
      fence_smem_async();
      fence_before();
      __syncthreads();
      fence_after();
      if (tid == 0) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
#pragma unroll
          for (int kb = 0; kb < NH / 16; ++kb)
            mma(tmem + NH * r, sdesc(reinterpret_cast<unsigned char*>(s.H + r * ROWS * NH) + 256 * kb, 128, 1024),
                sdesc(reinterpret_cast<unsigned char*>(s.W2) + 256 * kb, 128, 1024), ID_L, kb > 0);
        commit(&s.bar);
      }
      ok = __syncthreads_and(wait_parity(&s.bar, parity)) != 0;
      if (ok) parity ^= 1u;
      fence_after();
    }
    // layer-2 epilogue: bias, GELU, then the NO outputs as FP32 dot products with W3, even and
    // odd columns apart
    float2 acc[NR][NO];
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int o = 0; o < NO; ++o) acc[r][o] = make_float2(s.b3[o], 0.f);
    if (ok) {
#pragma unroll
      for (int c = 0; c < NH / 16; ++c) {
        uint32_t v[NR][16];
#pragma unroll
        for (int r = 0; r < NR; ++r) ld16(tmem + lane_base + NH * r + 16 * c, v[r]);
#pragma unroll
        for (int r = 0; r < NR; ++r) ld_wait(v[r]);
#pragma unroll
        for (int q = 0; q < 16; q += 4) {
          const float4 b = *reinterpret_cast<const float4*>(&s.b2[16 * c + q]);
          float2 g0[NR], g1[NR];
#pragma unroll
          for (int r = 0; r < NR; ++r) {
            g0[r] = gelu2(__fadd2_rn(pair_of(v[r] + q), make_float2(b.x, b.y)));
            g1[r] = gelu2(__fadd2_rn(pair_of(v[r] + q + 2), make_float2(b.z, b.w)));
          }
#pragma unroll
          for (int o = 0; o < NO; ++o) {
            const float4 w = *reinterpret_cast<const float4*>(&s.W3[o][16 * c + q]);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
              acc[r][o] = __ffma2_rn(make_float2(w.x, w.y), g0[r], acc[r][o]);
              acc[r][o] = __ffma2_rn(make_float2(w.z, w.w), g1[r], acc[r][o]);
            }
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      float out[NO];
#pragma unroll
      for (int o = 0; o < NO; ++o) out[o] = acc[r][o].x + acc[r][o].y;
      cons(row0 + r * ROWS, out, flag[r], ok, r);
    }
    if (STOP && !ok) break;
    fence_before();
    __syncthreads();  // the next tile rewrites X, H and the accumulators
    fence_after();
  }
  if (!ok)  // uniform: the MMAs of the phase that timed out may still run; one more bounded wait
    wait_parity(&s.bar, parity);
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  return ok;
}

// y[n][NO] = network(X[n][7]) for standardised X.  *err is set to 1 when a bounded wait ran
// out (the outputs of that launch are then not valid).  Launch with THREADS threads and
// dynamic shared memory of sizeof(Smem<NO, FWD_NR>).  A tile's rows are contiguous in X and y: both go
// through shared memory in 16-byte accesses where the pointers allow (vec), the next tile's
// X requested while this one is computed; a thread's own row at a time would touch each
// 32-byte sector up to eight times.
constexpr int FWD_NR = 2, FWD_CTAS = 4;
template <int NO>
__global__ void __launch_bounds__(THREADS, FWD_CTAS)
    mlp_forward_tc5_kernel(const float* P, const float* X, float* y, int64_t n, unsigned* err, int vec) {
  constexpr int NR = FWD_NR, NI = DG_MLP_NI, XW = NR * ROWS * NI, V4 = XW / 4, PER = (V4 + THREADS - 1) / THREADS;
  constexpr int YW = NR * ROWS * NO;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Smem<NO, NR>& s = *reinterpret_cast<Smem<NO, NR>*>(smem_raw);
  // the hidden layer's operand is free from layer 2's MMAs to the next layer-1 epilogue: it stages
  // the outputs, then the next tile's inputs
  float *ys = reinterpret_cast<float*>(s.H), *xs = ys;
  static_assert(sizeof(s.H) >= sizeof(float) * YW && sizeof(s.H) >= sizeof(float) * XW, "staging");
  alloc_tmem<NO, NR>(s);
  load_weights<NO, NR>(s, P);
  const int tid = threadIdx.x;
  float4 next[PER];
  auto fetch = [&](int64_t tile) {
    const bool full = vec && (tile + 1) * (NR * ROWS) <= n;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int i = tid + j * THREADS;
      if (full && i < V4) next[j] = __ldg(reinterpret_cast<const float4*>(X + tile * XW) + i);
    }
  };
  fetch(blockIdx.x);
  auto prod = [&](int64_t row, float* x, int r) {
    const int64_t tile = row / (NR * ROWS);
    if (vec && (tile + 1) * (NR * ROWS) <= n) {  // the same in all threads
      if (r == 0) {
#pragma unroll
        for (int j = 0; j < PER; ++j) {
          const int i = tid + j * THREADS;
          if (i < V4) reinterpret_cast<float4*>(xs)[i] = next[j];
        }
        fetch(tile + gridDim.x);
        __syncthreads();
      }
#pragma unroll
      for (int k = 0; k < NI; ++k) x[k] = xs[(r * ROWS + tid) * NI + k];
    } else {
#pragma unroll
      for (int k = 0; k < NI; ++k) x[k] = row < n ? X[row * NI + k] : 0.0f;
    }
    x[7] = 0.f;
    return true;
  };
  auto cons = [&](int64_t row, const float* out, bool, bool valid, int r) {
    const int64_t tile = row / (NR * ROWS);
    if (NO > 1 && vec && (tile + 1) * (NR * ROWS) <= n) {  // the same in all threads
      if (!valid) return;
#pragma unroll
      for (int o = 0; o < NO; ++o) ys[(r * ROWS + tid) * NO + o] = out[o];
      if (r < NR - 1) return;
      __syncthreads();
      float4* d = reinterpret_cast<float4*>(y + tile * YW);
      for (int i = tid; i < YW / 4; i += THREADS) d[i] = reinterpret_cast<const float4*>(ys)[i];
    } else if (row < n && valid) {
#pragma unroll
      for (int o = 0; o < NO; ++o) y[row * NO + o] = out[o];
    }
  };
  if (!run_tiles<NO, NR, true>(s, n, prod, cons) && threadIdx.x == 0) atomicExch(err, 1u);
}

}  // namespace dgtc5
