// BF16 GEMM of the learned correction's MLP on the fifth-generation tensor cores (tcgen05, sm_100
// family): C = opA(A) opB(B) (+ bias) (ReLU), BF16 operands, FP32 accumulation in tensor memory.
//
// One CTA of 128 threads computes a 128 x 128 tile of C.  For each K chunk of 64 the threads stage
// the A tile (128 rows x 64) and the B tile (128 columns x 64) in shared memory in the canonical
// K-major layout without swizzle: 8-row x 16-byte core matrices, K-adjacent core matrices 128 bytes
// apart, 8-row groups 1024 bytes apart; out-of-range rows, columns and K entries are zero.  One
// thread then issues four tcgen05.mma (M = 128, N = 128, K = 16 each) that accumulate into a
// 128 x 128 FP32 tile in tensor memory, and commits them to the stage's mbarrier.  Two stages
// alternate, so the threads stage chunk i + 1 while the tensor core works on chunk i; a stage is
// overwritten only after its commit arrived (at most kAsyncSpin polls per wait; a wait that runs out
// records the failure in a device flag, lets the MMAs in flight land and skips the epilogue).
// Finally each warp reads its 32 rows of the accumulator with tcgen05.ld and applies bias and ReLU.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "ops.h"

namespace sbm {
namespace {

#include "tc_core.cuh"

constexpr int TBM = 128, TBN = 128, TBK = 64;
constexpr int kTcThreads = 128;

__device__ int g_tc_fault = 0;

// Byte offset of element (row r, k) of a 128 x 64 K-major no-swizzle tile.
__device__ __forceinline__ uint32_t tile_off(int r, int k) {
  return (uint32_t)(((r >> 3) * 8 + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// Stages the K chunk k0 .. k0+63 of rows r0 .. r0+127 of the operand X (op(X)(r, k) = X[r*ld + k] when
// KMAJ, else X[k*ld + r]) into the 128 x 64 K-major tile T.  16-byte pieces (8 consecutive k of one
// row, one row of a core matrix) are loaded with 16-byte loads where the piece lies inside the
// matrix and is 16-byte aligned (KMAJ); otherwise (MN-major storage: 8 consecutive r of one k, or the
// ragged edges) element by element.  Entries outside R x K are zero.
template <bool KMAJ>
__device__ __forceinline__ void stage_tile(unsigned char* T, const __nv_bfloat16* __restrict__ X, int ld, int R,
                                           int K, int r0, int k0, bool vec_ok) {
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  if (KMAJ) {
    for (int q = threadIdx.x; q < 128 * 8; q += kTcThreads) {   // piece q: row q / 8, k chunk q % 8
      const int r = q >> 3, c = q & 7;
      const int gr = r0 + r, gk = k0 + 8 * c;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (gr < R) {
        const __nv_bfloat16* src = X + (size_t)gr * ld + gk;
        if (vec_ok && gk + 8 <= K) {
          v = *reinterpret_cast<const uint4*>(src);
        } else {
          __nv_bfloat16 t[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) t[j] = gk + j < K ? src[j] : zero;
          v = *reinterpret_cast<const uint4*>(t);
        }
      }
      *reinterpret_cast<uint4*>(T + tile_off(r, 8 * c)) = v;
    }
  } else {
    for (int q = threadIdx.x; q < 64 * 16; q += kTcThreads) {   // piece q: k = q / 16, rows 8 (q % 16) ..
      const int kk = q >> 4, rc = (q & 15) * 8;
      const int gk = k0 + kk, gr = r0 + rc;
      __nv_bfloat16 t[8];
      if (gk < K) {
        const __nv_bfloat16* src = X + (size_t)gk * ld + gr;
        if (vec_ok && gr + 8 <= R) {
          *reinterpret_cast<uint4*>(t) = *reinterpret_cast<const uint4*>(src);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) t[j] = gr + j < R ? src[j] : zero;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] = zero;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) *reinterpret_cast<__nv_bfloat16*>(T + tile_off(rc + j, kk)) = t[j];
    }
  }
}

template <int TA, int TB>
__global__ void __launch_bounds__(kTcThreads) k_gemm_tc(int M, int N, int K, const __nv_bfloat16* __restrict__ A,
                                                        int lda, const __nv_bfloat16* __restrict__ B, int ldb,
                                                        const float* __restrict__ bias, int relu,
                                                        float* __restrict__ Cf, __nv_bfloat16* __restrict__ Cb,
                                                        int ldc) {
  // two stages of (A tile, B tile), 32 KB each, in dynamic shared memory (1024-byte aligned)
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  __shared__ __align__(8) unsigned long long bar[2];
  __shared__ uint32_t tmem_base;
  __shared__ int stop;
  const int m0 = blockIdx.y * TBM, n0 = blockIdx.x * TBN;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0) {                                   // 128 FP32 columns of tensor memory
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_addr(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
    stop = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint32_t idesc = idesc_bf16(TBM, TBN);
  // 16-byte loads need 16-byte aligned rows
  const bool va = (reinterpret_cast<uintptr_t>(A) & 15) == 0 && ((size_t)lda * 2) % 16 == 0;
  const bool vb = (reinterpret_cast<uintptr_t>(B) & 15) == 0 && ((size_t)ldb * 2) % 16 == 0;
  unsigned phase[2] = {0u, 0u};
  int it = 0;
  bool failed = false;
  for (int k0 = 0; k0 < K; k0 += TBK, ++it) {
    const int b = it & 1;
    unsigned char* As = tc_smem + b * 2 * (TBM * TBK * 2);
    unsigned char* Bs = As + TBM * TBK * 2;
    if (it >= 2) {                                   // the MMAs of chunk it - 2 read this stage
      const bool ok = stop ? true : mbar_wait(&bar[b], phase[b]);
      phase[b] ^= 1u;
      if (!__syncthreads_and(ok)) {
        failed = true;
        break;
      }
    }
    stage_tile<TA == 0>(As, A, lda, M, K, m0, k0, va);
    stage_tile<TB == 1>(Bs, B, ldb, N, K, n0, k0, vb);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic writes -> tensor core
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int ks = 0; ks < TBK / 16; ++ks) {        // K = 16 per instruction: two core matrices
        const uint64_t ad = smem_desc(smem_addr(As + ks * 256), 128, 1024);
        const uint64_t bd = smem_desc(smem_addr(Bs + ks * 256), 128, 1024);
        const uint32_t acc = (it > 0 || ks > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_addr(&bar[b]))
                   : "memory");
    }
  }
  // wait for the commits still outstanding (the last one or two chunks), bounded
  if (!failed) {
    bool ok = true;
    for (int j = (it >= 2 ? it - 2 : 0); j < it; ++j) {
      const int b = j & 1;
      ok = ok && mbar_wait(&bar[b], phase[b]);
      phase[b] ^= 1u;
    }
    failed = !__syncthreads_and(ok);
  }
  if (failed && threadIdx.x == 0) {                  // record it and let the MMAs in flight land
    atomicExch(&g_tc_fault, 1);
    mbar_wait(&bar[0], phase[0]);
    mbar_wait(&bar[1], phase[1]);
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  // epilogue: warp w owns accumulator rows (TMEM lanes) 32 w .. 32 w + 31
  const int m = m0 + warp * 32 + lane;
  if (!failed && K > 0) {
#pragma unroll 1
    for (int c0 = 0; c0 < TBN; c0 += 32) {
      uint32_t r[32];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
          "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
            "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
            "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
            "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (m < M) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int n = n0 + c0 + j;
          if (n < N) {
            float v = __uint_as_float(r[j]);
            if (bias) v += bias[n];
            if (relu) v = fmaxf(v, 0.f);
            if (Cf) Cf[(size_t)m * ldc + n] = v;
            if (Cb) Cb[(size_t)m * ldc + n] = __float2bfloat16_rn(v);
          }
        }
      }
    }
  } else if (K == 0 && m < M) {                      // empty contraction: C = bias (ReLU)
    for (int n = n0; n < n0 + TBN && n < N; ++n) {
      float v = bias ? bias[n] : 0.f;
      if (relu) v = fmaxf(v, 0.f);
      if (Cf) Cf[(size_t)m * ldc + n] = v;
      if (Cb) Cb[(size_t)m * ldc + n] = __float2bfloat16_rn(v);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem) : "memory");
}

// ----------------------------------------------------------------------------------------------
// The learned correction's MLP, F -> H -> H -> O, as one kernel on the tcgen05 tensor cores.
//
// A CTA takes a tile of 128 rows through all layers: the first layer streams the features and W1 in
// chunks of 64 features, the accumulator (128 x H FP32) stays in tensor memory, the activations
// go through registers (bias, ReLU, BF16) into a shared-memory tile that is the next layer's A
// operand, and only the outputs reach global memory.  Three roles run apart from one another,
// joined by mbarriers (in one loop of all threads, the feature loads, the weight copies and the
// tensor core's latency added up: 55 us against 40 at 16,384 x 2023 -> 128 -> 128 -> 64; four launches,
// the rounding of X among them, took 432):
//   - 16 warps bring the features of the first layer into a ring of A tiles and carry out the
//     epilogues;
//   - one thread copies the weight chunks of all layers, one after the other, into a ring of B
//     tiles; the weights are stored as core matrices, so a chunk is one contiguous bulk copy, and
//     the next layer's weights are in flight while a layer ends;
//   - one thread issues the MMAs.
// FP32 features are rounded to BF16 on the way in: a thread loads eight rows of one feature (each
// load instruction of a warp reads 32 consecutive features of a row, whatever the row's alignment)
// and writes them as one 16-byte piece of an MN-major operand, three chunks ahead in registers.
//
// What bounds it: with FP32 features the read of X (16,384 x 2023: 133 MB, 19.5 us at the measured
// copy bandwidth; 128 of the 152 SMs have a tile, each with three chunks of 32 KB in flight); with few
// rows the chain of layers (260 rows x 192: three GEMM launches took 97 us of a V-cycle, now 17).
constexpr int kTileRows = 128;
constexpr int kFeedWarps = 16;                     // feature loads and epilogues
constexpr int kFusedThreads = (kFeedWarps + 2) * 32;

// SA, SB: stages of the A and B rings.  F32IN: X is FP32 [rows][F], else BF16 [rows][Fpad].
template <int SA, int SB, bool F32IN>
__global__ void __launch_bounds__(kFusedThreads, 1) k_mlp_fused(const __grid_constant__ MlpTile P) {
  extern __shared__ __align__(1024) unsigned char fused_smem[];
  __shared__ __align__(8) unsigned long long full_a[SA], empty_a[SA], full_b[SB], empty_b[SB], acc_full, act_full;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  const int Hp = P.Hp, Op = P.Op, wmax = max(Hp, Op);
  constexpr uint32_t kABytes = kTileRows * kChunkK * 2;
  const uint32_t b_bytes = (uint32_t)wmax * kChunkK * 2;
  const uint32_t ring_a = smem_addr(fused_smem), ring_b = ring_a + SA * kABytes, act = ring_b + SB * b_bytes;
  const uint32_t act_sbo = (uint32_t)wmax * 16;      // bytes between the 8-row groups of the activation tile
  const int ntile = (P.rows + kTileRows - 1) / kTileRows;
  // chunks of the layers, in order
  const int n1 = (P.Fpad + kChunkK - 1) / kChunkK, n2 = (Hp + kChunkK - 1) / kChunkK;
  const int total = n1 + 2 * n2;
  uint32_t ncols = 32;
  while ((int)ncols < wmax) ncols <<= 1;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < SA; ++s) {
      mbar_init(&full_a[s], kFeedWarps);
      mbar_init(&empty_a[s], 1);
    }
    for (int s = 0; s < SB; ++s) {
      mbar_init(&full_b[s], 1);
      mbar_init(&empty_b[s], 1);
    }
    mbar_init(&acc_full, 1);
    mbar_init(&act_full, kFeedWarps);
    mbar_fence_init();
    failed = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  volatile int* stop = &failed;
  // a bounded wait; once one has run out, every role leaves its loop
  auto wait = [&](unsigned long long* bar, unsigned parity) {
    if (!mbar_wait(bar, parity)) *stop = 1;
    return *stop == 0;
  };

  if (warp == kFeedWarps) {                          // the weights
    if (lane == 0) {
      if (!P.early) pdl_wait();                      // early: written two or more launches back
      int g = 0;                                     // chunks of the ring so far
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x)
        for (int i = 0; i < total && ok; ++i, ++g) {
          if (g >= SB) ok = wait(&empty_b[g % SB], (unsigned)((g / SB - 1) & 1));
          if (!ok) break;
          const int at = i < n1 ? i : (i < n1 + n2 ? i - n1 : i - n1 - n2);
          const int K = i < n1 ? P.Fpad : Hp, np = i < n1 + n2 ? Hp : Op;
          const __nv_bfloat16* W = i < n1 ? P.W1 : (i < n1 + n2 ? P.W2 : P.W3);
          const unsigned bytes = (unsigned)(min(kChunkK, K - at * kChunkK) * np * 2);
          mbar_arrive_tx(&full_b[g % SB], bytes);
          bulk_load(fused_smem + SA * kABytes + (g % SB) * b_bytes, W + (size_t)at * kChunkK * np, bytes, &full_b[g % SB]);
        }
    }
  } else if (warp == kFeedWarps + 1) {               // the tensor core
    if (lane == 0) {
      int ga = 0, gb = 0, layers = 0;                // A and B chunks, layers with an activation tile so far
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x)
        for (int i = 0; i < total && ok; ++i, ++gb) {
          const int layer = i < n1 ? 0 : (i < n1 + n2 ? 1 : 2);
          const int at = i - (layer == 0 ? 0 : (layer == 1 ? n1 : n1 + n2));
          const int K = layer == 0 ? P.Fpad : Hp, np = layer == 2 ? Op : Hp;
          if (layer == 0) ok = wait(&full_a[ga % SA], (unsigned)((ga / SA) & 1));
          else if (at == 0) ok = wait(&act_full, (unsigned)(layers++ & 1));
          if (layer == 0 && at == 0 && tile != (int)blockIdx.x) ok = wait(&act_full, (unsigned)(layers++ & 1)) && ok;
          ok = ok && wait(&full_b[gb % SB], (unsigned)((gb / SB) & 1));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a = layer == 0 ? ring_a + (ga % SA) * kABytes : act + (uint32_t)at * (kChunkK / 8) * 128;
          const uint32_t b = ring_b + (gb % SB) * b_bytes;
          const uint32_t id = idesc_bf16(kTileRows, np, F32IN && layer == 0, true);
          for (int ks = 0; ks < min(kChunkK, K - at * kChunkK) / 16; ++ks)
            mma_bf16(tmem, smem_desc(a + ks * 256, 128, layer == 0 ? 1024 : act_sbo),
                     smem_desc(b + ks * (uint32_t)np * 32, (uint32_t)np * 16, 128), id, at > 0 || ks > 0);
          if (layer == 0) mma_commit(&empty_a[ga++ % SA]);
          mma_commit(&empty_b[gb % SB]);
          if (i == n1 - 1 || i == n1 + n2 - 1 || i == total - 1) mma_commit(&acc_full);
        }
    }
  } else {                                           // features and epilogues
    pdl_wait();
    pdl_trigger();
    int ga = 0, layers = 0;
    bool ok = true;
    auto arrive = [&](unsigned long long* bar) {     // this warp's writes to shared memory, then one arrival
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0)
        asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
                     : "memory");
    };
    auto stage_free = [&](int g) { return g < SA || wait(&empty_a[g % SA], (unsigned)((g / SA - 1) & 1)); };
    for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x) {
      const int row0 = tile * kTileRows;
      if constexpr (F32IN) {
        // FP32 features of chunk i: features lane and lane + 32 of the warp's 8 rows
        auto load_x = [&](int i, float (&v)[16]) {
          const int k = i * kChunkK + lane;
          const float* src = P.Xf + (size_t)(row0 + 8 * warp) * P.F + k;
          if (row0 + 8 * warp + 8 <= P.rows && (i + 1) * kChunkK <= P.F) {
#pragma unroll
            for (int r = 0; r < 8; ++r, src += P.F) {
              v[r] = __ldcs(src);
              v[8 + r] = __ldcs(src + 32);
            }
          } else {
#pragma unroll
            for (int r = 0; r < 8; ++r, src += P.F) {
              const bool in = row0 + 8 * warp + r < P.rows;
              v[r] = in && k < P.F ? __ldcs(src) : 0.f;
              v[8 + r] = in && k + 32 < P.F ? __ldcs(src + 32) : 0.f;
            }
          }
        };
        auto put = [&](int i, float (&v)[16]) {      // chunk i into its stage, chunk i + 3 into the registers
          if (i >= n1 || !ok) return;
          ok = stage_free(ga);
          if (!ok) return;
#pragma unroll
          for (int h = 0; h < 2; ++h) {              // one 16-byte piece (8 rows) per feature
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const __nv_bfloat162 b = __floats2bfloat162_rn(v[8 * h + 2 * q], v[8 * h + 2 * q + 1]);
              w[q] = *reinterpret_cast<const uint32_t*>(&b);
            }
            const int k = lane + 32 * h;
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(ring_a + (ga % SA) * kABytes + warp * 1024 +
                                                                       (k >> 3) * 128 + (k & 7) * 16),
                         "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                         : "memory");
          }
          if (i + 3 < n1) load_x(i + 3, v);
          arrive(&full_a[ga % SA]);
          ++ga;
        };
        float va[16], vb[16], vc[16];
        load_x(0, va);
        if (n1 > 1) load_x(1, vb);
        if (n1 > 2) load_x(2, vc);
        for (int i = 0; i < n1 && ok; i += 3) {
          put(i, va);
          put(i + 1, vb);
          put(i + 2, vc);
        }
      } else {                                       // BF16 rows, copied asynchronously, two chunks in flight
        for (int i = 0; i < n1 + 2 && ok; ++i) {
          if (i < n1) {
            ok = stage_free(ga + i);
            if (ok)
              stage_async<true>(ring_a + ((ga + i) % SA) * kABytes, P.Xb, P.Fpad, P.rows, P.Fpad, row0, kTileRows,
                                i * kChunkK, (int)threadIdx.x, kFeedWarps * 32);
          }
          cp_async_commit();
          cp_async_wait<2>();
          if (i >= 2) arrive(&full_a[(ga + i - 2) % SA]);
        }
        ga += n1;
      }
      // The end of a layer: the accumulator through bias and ReLU into the activation tile, or to
      // the output.  Four warps share a row quarter and take a quarter of the columns each.
      for (int layer = 0; layer < 3 && ok; ++layer) {
        ok = wait(&acc_full, (unsigned)(layers++ & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int r = 32 * (warp & 3) + lane, row = row0 + r;
        const int np = layer == 2 ? Op : Hp, n = layer == 2 ? P.O : P.H;
        const float* bias = layer == 0 ? P.b1 : (layer == 1 ? P.b2 : P.b3);
        for (int c0 = (warp >> 2) * (np / 4); c0 < ((warp >> 2) + 1) * (np / 4); c0 += 8) {
          float v[8];
          tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = c0 + j < n ? v[j] + bias[c0 + j] : 0.f;
          if (layer < 2) {
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const __nv_bfloat162 b = __floats2bfloat162_rn(fmaxf(v[2 * q], 0.f), fmaxf(v[2 * q + 1], 0.f));
              w[q] = *reinterpret_cast<const uint32_t*>(&b);
            }
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(act + (uint32_t)(r >> 3) * act_sbo +
                                                                       (uint32_t)(c0 / 8) * 128 + (r & 7) * 16),
                         "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                         : "memory");
          } else if (row < P.rows) {
            float* y = P.Y + (size_t)row * P.O + c0;
            if ((P.O & 3) == 0 && c0 + 8 <= P.O && P.y_vec) {
              reinterpret_cast<float4*>(y)[0] = make_float4(v[0], v[1], v[2], v[3]);
              reinterpret_cast<float4*>(y)[1] = make_float4(v[4], v[5], v[6], v[7]);
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j)
                if (c0 + j < P.O) y[j] = v[j];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        arrive(&act_full);                           // the tile is written and the accumulator read
      }
    }
    cp_async_wait<0>();
  }
  __syncthreads();
  if (failed && threadIdx.x == 0) {                  // record it; copies and MMAs in flight get time to land
    atomicExch(&g_tc_fault, 1);
    for (int s = 0; s < SB; ++s)
      for (unsigned p = 0; p < 2; ++p) mbar_wait(&full_b[s], p, 1u << 16);
    for (unsigned p = 0; p < 2; ++p) mbar_wait(&acc_full, p, 1u << 16);
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

template <int SA, int SB, bool F32IN>
cudaError_t launch_fused(const MlpTile& P, size_t smem, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_mlp_fused<SA, SB, F32IN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
  if (e != cudaSuccess) return e;
  const int ntile = (P.rows + kTileRows - 1) / kTileRows;
  SBM_PDL((k_mlp_fused<SA, SB, F32IN>), (unsigned)std::min(ntile, 152), kFusedThreads, smem, s, P);
  return cudaSuccess;
}

}  // namespace

// Two stages of 32 KB: at most 3 CTAs per SM, so the CTAs of an SM never ask for more than 3 x 128
// of its 512 tensor-memory columns (tcgen05.alloc would wait).
constexpr size_t kTcSmem = 2 * 2 * (size_t)TBM * TBK * 2;

template <int TA, int TB>
cudaError_t launch_tc(dim3 grid, int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B,
                      int ldb, const float* bias, int relu, float* Cf, __nv_bfloat16* Cb, int ldc, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_gemm_tc<TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kTcSmem);
  if (e != cudaSuccess) return e;
  k_gemm_tc<TA, TB><<<grid, kTcThreads, kTcSmem, s>>>(M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc);
  return cudaSuccess;
}

cudaError_t launch_gemm_tc(int M, int N, int K, int ta, int tb, const __nv_bfloat16* A, int lda,
                           const __nv_bfloat16* B, int ldb, const float* bias, int relu, float* Cf,
                           __nv_bfloat16* Cb, int ldc, cudaStream_t s) {
  if (M == 0 || N == 0) return cudaSuccess;
  const dim3 grid((N + TBN - 1) / TBN, (M + TBM - 1) / TBM);
  cudaError_t e;
  if (!ta && !tb) e = launch_tc<0, 0>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, s);
  else if (!ta && tb) e = launch_tc<0, 1>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, s);
  else if (ta && !tb) e = launch_tc<1, 0>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, s);
  else e = launch_tc<1, 1>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, s);
  if (e != cudaSuccess) return e;
  count_launches();
  return cudaGetLastError();
}

// Hidden widths up to 256: four A stages, three B stages of 64 x 256 BF16 and the 128 x 256 activation
// tile (224 KB) still fit an SM; wider networks run layer by layer.
bool mlp_fused_fits(int Hp, int Op) { return std::max(Hp, Op) <= 256; }

cudaError_t launch_mlp_fused(const MlpTile& P, cudaStream_t s) {
  if (P.rows == 0) return cudaSuccess;
  const size_t w = (size_t)std::max(P.Hp, P.Op);
  const size_t a = kTileRows * kChunkK * 2, b = w * kChunkK * 2, act = kTileRows * w * 2;
  cudaError_t e;
  if (w <= 128)
    e = P.Xf ? launch_fused<5, 5, true>(P, 5 * a + 5 * b + act, s) : launch_fused<5, 5, false>(P, 5 * a + 5 * b + act, s);
  else
    e = P.Xf ? launch_fused<4, 3, true>(P, 4 * a + 3 * b + act, s) : launch_fused<4, 3, false>(P, 4 * a + 3 * b + act, s);
  if (e != cudaSuccess) return e;
  count_launches();
  return cudaGetLastError();
}

int tc_fault_take() {
  int f = 0;
  if (cudaMemcpyFromSymbol(&f, g_tc_fault, sizeof(int)) != cudaSuccess) return -1;
  if (f) {
    const int zero = 0;
    if (cudaMemcpyToSymbol(g_tc_fault, &zero, sizeof(int)) != cudaSuccess) return -1;
  }
  return f;
}

}  // namespace sbm
