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
                                                        int ldc, int* fault) {
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
    atomicExch(fault, 1);
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
  } else if (m < M) {                                // empty contraction: C = bias (ReLU); a failed wait: zero
    for (int n = n0; n < n0 + TBN && n < N; ++n) {
      float v = bias && !failed ? bias[n] : 0.f;
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
// BWD: a training pass.  The same tile goes on through the loss gradient dY = 2 (Y - T) / count, dZ2 =
// (dY W3^T) o [H2 > 0] and dZ1 = (dZ2 W2^T) o [H1 > 0], the masks kept in registers; the BF16 features,
// activations and gradients go to memory for the weight gradients (k_wgrad), the FP32 column sums of
// dY, dZ2 and dZ1 (the bias gradients) and the loss to one partial sum per CTA.  With k_wgrad and
// k_grad_reduce a training pass of 4096 rows (2023 -> 128 -> 128 -> 64) takes 3 launches instead of 16; a call
// of sbm_mlp_gradients, with the gradient's copy to the host, 177 us instead of 1763.
//
// What bounds it: with FP32 features the read of X (16,384 x 2023: 133 MB, 19.5 us at the measured
// copy bandwidth; 128 of the 152 SMs have a tile, each with three chunks of 32 KB in flight); with few
// rows the chain of layers (260 rows x 192: three GEMM launches took 97 us of a V-cycle, now 17).
constexpr int kTileRows = 128;
constexpr int kFeedWarps = 16;                     // feature loads and epilogues
constexpr int kFusedThreads = (kFeedWarps + 2) * 32;

// SA, SB: stages of the A and B rings.  F32IN: X is FP32 [rows][F], else BF16 [rows][Fpad].
template <int SA, int SB, bool F32IN, bool BWD>
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
  const int n4 = BWD ? (Op + kChunkK - 1) / kChunkK : 0;
  const int total = n1 + 2 * n2 + (BWD ? n4 + n2 : 0);
  constexpr int kLayers = BWD ? 5 : 3;
  // layer of chunk i, the chunk's number in it, its contraction length and its output width
  auto layer_of = [&](int i, int& at, int& K, int& np) {
    const int start[6] = {0, n1, n1 + n2, n1 + 2 * n2, n1 + 2 * n2 + n4, total};
    int l = 0, first = 0;
#pragma unroll
    for (int q = 1; q < kLayers; ++q)
      if (i >= start[q]) l = q, first = start[q];
    at = i - first;
    K = l == 0 ? P.Fpad : (l == 3 ? Op : Hp);
    np = l == 2 ? Op : Hp;
    return l;
  };
  // BWD: column sums of dZ1, dZ2, dY by row quarter, and the loss
  const int nsum = 2 * Hp + Op;
  float* csum = reinterpret_cast<float*>(fused_smem + SA * kABytes + SB * b_bytes + kTileRows * wmax * 2);
  __shared__ float loss_w[kFeedWarps];
  if (BWD)
    for (int q = threadIdx.x; q < 4 * nsum; q += kFusedThreads) csum[q] = 0.f;
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
    if (!mbar_wait(bar, parity, P.spin)) *stop = 1;
    return *stop == 0;
  };
  int issued = 0;                                    // weight chunks copied, or handed to the tensor core, by this thread
  // (No role starts its bounded polls before the dependency wait: the kernels before this one would count
  // against the limit.)

  if (warp == kFeedWarps) {                          // the weights
    if (lane == 0) {
      if (!P.early) pdl_wait();                      // early: written two or more launches back
      int g = 0;                                     // chunks of the ring so far
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x)
        for (int i = 0; i < total && ok; ++i, ++g) {
          if (g == SB && P.early) pdl_wait();        // the ring is full
          if (g >= SB) ok = wait(&empty_b[g % SB], (unsigned)((g / SB - 1) & 1));
          if (!ok) break;
          int at, K, np;
          const int layer = layer_of(i, at, K, np);
          const int kn = min(kChunkK, K - at * kChunkK);
          const unsigned bytes = (unsigned)(kn * np * 2);
          unsigned char* dst = fused_smem + SA * kABytes + (g % SB) * b_bytes;
          unsigned long long* bar = &full_b[g % SB];
          mbar_arrive_tx(bar, bytes);
          if (layer < 3) {                           // k = inputs: one run of core matrices
            const __nv_bfloat16* W = layer == 0 ? P.W1 : (layer == 1 ? P.W2 : P.W3);
            bulk_load(dst, W + (size_t)at * kChunkK * np, bytes, bar);
          } else {                                   // k = outputs: a run for each group of 8 inputs
            const __nv_bfloat16* W = (layer == 3 ? P.W3 : P.W2) + (size_t)at * kChunkK * 8;
            for (int a = 0; a < Hp / 8; ++a) bulk_load(dst + a * kn * 16, W + (size_t)a * K * 8, (unsigned)kn * 16, bar);
          }
          issued = g + 1;
        }
    }
  } else if (warp == kFeedWarps + 1) {               // the tensor core
    if (lane == 0) {
      pdl_wait();
      int ga = 0, gb = 0, layers = 0;                // A and B chunks, layers with an activation tile so far
      bool ok = true;
      for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x)
        for (int i = 0; i < total && ok; ++i, ++gb) {
          int at, K, np;
          const int layer = layer_of(i, at, K, np);
          if (layer == 0) ok = wait(&full_a[ga % SA], (unsigned)((ga / SA) & 1));
          else if (at == 0) ok = wait(&act_full, (unsigned)(layers++ & 1));
          if (layer == 0 && at == 0 && tile != (int)blockIdx.x) ok = wait(&act_full, (unsigned)(layers++ & 1)) && ok;
          ok = ok && wait(&full_b[gb % SB], (unsigned)((gb / SB) & 1));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a = layer == 0 ? ring_a + (ga % SA) * kABytes : act + (uint32_t)at * (kChunkK / 8) * 128;
          const uint32_t b = ring_b + (gb % SB) * b_bytes;
          const int kn = min(kChunkK, K - at * kChunkK);
          const uint32_t id = idesc_bf16(kTileRows, np, F32IN && layer == 0, layer < 3);
          // B core matrices, k step of 8 / columns step of 8: forward W's rows, backward W's columns
          const uint32_t b_lbo = layer < 3 ? (uint32_t)np * 16 : 128, b_sbo = layer < 3 ? 128 : (uint32_t)kn * 16;
          for (int ks = 0; ks < kn / 16; ++ks)
            mma_bf16(tmem, smem_desc(a + ks * 256, 128, layer == 0 ? 1024 : act_sbo),
                     smem_desc(b + ks * 2 * b_lbo, b_lbo, b_sbo), id, at > 0 || ks > 0);
          if (layer == 0) mma_commit(&empty_a[ga++ % SA]);
          mma_commit(&empty_b[gb % SB]);
          issued = gb + 1;
          if ((at + 1) * kChunkK >= K) mma_commit(&acc_full);
        }
    }
  } else {                                           // features and epilogues
    pdl_wait();
    pdl_trigger();
    int ga = 0, layers = 0;
    float loss = 0.f;
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
            if (BWD && i * kChunkK + k < P.Fpad) {   // the BF16 features for the weight gradient
              unsigned short* xs = reinterpret_cast<unsigned short*>(P.Xs) + (size_t)(row0 + 8 * warp) * P.Fpad + i * kChunkK + k;
#pragma unroll
              for (int r = 0; r < 8; ++r, xs += P.Fpad)
                if (row0 + 8 * warp + r < P.rows) *xs = (unsigned short)(w[r >> 1] >> (16 * (r & 1)));
            }
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
      // The end of a layer: the accumulator through bias and ReLU (backward: the ReLU mask) into the
      // activation tile, or to the output.  Four warps share a row quarter and take a quarter of the
      // columns each.
      unsigned long long mask1 = 0, mask2 = 0;       // BWD: H1 > 0, H2 > 0 at this thread's columns
      for (int layer = 0; layer < kLayers && ok; ++layer) {
        ok = wait(&acc_full, (unsigned)(layers++ & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int r = 32 * (warp & 3) + lane, row = row0 + r;
        const int np = layer == 2 ? Op : Hp, n = layer == 2 ? P.O : P.H;
        const float* bias = layer == 0 ? P.b1 : (layer == 1 ? P.b2 : P.b3);
        const int cbeg = (warp >> 2) * (np / 4);
        for (int c0 = cbeg; c0 < cbeg + np / 4; c0 += 8) {
          float v[8];
          tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
          if (layer < 3) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = c0 + j < n ? v[j] + bias[c0 + j] : 0.f;
          }
          if (layer < 2) {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = fmaxf(v[j], 0.f);
          }
          if (layer == 2 && !BWD) {
            if (row < P.rows) {
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
            continue;
          }
          if constexpr (BWD) {
            if (layer == 2) {                        // the loss and its gradient
              const float* t = P.T + (size_t)row * P.O + c0;
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float d = row < P.rows && c0 + j < P.O ? v[j] - t[j] : 0.f;
                loss += d * d;
                v[j] = 2.f * d * P.inv_count;
              }
            } else if (layer > 2) {
              const unsigned m = (unsigned)((layer == 3 ? mask2 : mask1) >> (c0 - cbeg)) & 0xffu;
#pragma unroll
              for (int j = 0; j < 8; ++j) v[j] = (m >> j) & 1u ? v[j] : 0.f;
            }
          }
          uint32_t w[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
            w[q] = *reinterpret_cast<const uint32_t*>(&b);
          }
          if (layer < 4)
            asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(act + (uint32_t)(r >> 3) * act_sbo +
                                                                       (uint32_t)(c0 / 8) * 128 + (r & 7) * 16),
                         "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                         : "memory");
          if constexpr (BWD) {
            if (layer < 2) {                         // rounded activations above zero (sign clear, value set)
              unsigned long long m = 0;
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const unsigned h = (w[j >> 1] >> (16 * (j & 1))) & 0xffffu;
                m |= (unsigned long long)(h != 0u && h < 0x8000u && h <= 0x7f80u) << j;
              }
              (layer == 0 ? mask1 : mask2) |= m << (c0 - cbeg);
            }
            __nv_bfloat16* g = layer == 0 ? P.H1 : (layer == 1 ? P.H2 : (layer == 2 ? P.dY : (layer == 3 ? P.dZ2 : P.dZ1)));
            if (row < P.rows)
              *reinterpret_cast<uint4*>(g + (size_t)row * np + c0) = make_uint4(w[0], w[1], w[2], w[3]);
            if (layer >= 2) {
              // column sums over the warp's 32 rows: lanes exchange halves of the columns until the four
              // lanes 4 j .. 4 j + 3 hold column j, then add among themselves
#pragma unroll
              for (int half = 4; half >= 1; half >>= 1) {
                const bool upper = (lane & (4 * half)) != 0;
#pragma unroll
                for (int j = 0; j < half; ++j) {
                  const float send = upper ? v[j] : v[j + half], keep = upper ? v[j + half] : v[j];
                  v[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * half);
                }
              }
              v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
              v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
              if ((lane & 3) == 0)
                csum[(warp & 3) * nsum + (layer == 4 ? 0 : (layer == 3 ? Hp : 2 * Hp)) + c0 + (lane >> 2)] += v[0];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        arrive(&act_full);                           // the tile is written and the accumulator read
      }
    }
    if constexpr (BWD) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
      if (lane == 0) loss_w[warp] = loss;
    }
    cp_async_wait<0>();
  }
  __syncthreads();
  if constexpr (BWD) {                               // this CTA's partial sums, in a fixed order
    for (int q = threadIdx.x; q < nsum; q += kFusedThreads)
      P.bias_part[(size_t)blockIdx.x * nsum + q] = (csum[q] + csum[nsum + q]) + (csum[2 * nsum + q] + csum[3 * nsum + q]);
    if (threadIdx.x == 0) {
      float t = 0.f;
      for (int w = 0; w < kFeedWarps; ++w) t += loss_w[w];
      P.loss_part[blockIdx.x] = t;
      if (blockIdx.x == 0)
        for (int b = gridDim.x; b < kLossParts; ++b) P.loss_part[b] = 0.f;
    }
  }
  if (failed) {                                      // record it; copies and MMAs in flight get time to land
    if (threadIdx.x == 0) atomicExch(P.fault, 1);
    const bool mma = warp == kFeedWarps + 1;         // (warps 16 and 17 alone have issued any)
    for (int q = mma ? max(0, issued - 1) : max(0, issued - SB); q < issued; ++q)
      mbar_wait(mma ? &empty_b[q % SB] : &full_b[q % SB], (unsigned)((q / SB) & 1), 1u << 16);
  }
  __syncthreads();
  if (!BWD && failed)                                // a defined result: zero outputs for all of this CTA's rows
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
      const size_t beg = (size_t)tile * kTileRows, end = min(beg + kTileRows, (size_t)P.rows);
      for (size_t q = beg * P.O + threadIdx.x; q < end * P.O; q += kFusedThreads) P.Y[q] = 0.f;
    }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

template <int SA, int SB, bool F32IN, bool BWD>
cudaError_t launch_fused(const MlpTile& P, cudaStream_t s) {
  const size_t w = (size_t)std::max(P.Hp, P.Op);
  const size_t smem = SA * (size_t)kTileRows * kChunkK * 2 + SB * w * kChunkK * 2 + kTileRows * w * 2 +
                      (BWD ? 4 * (size_t)(2 * P.Hp + P.Op) * sizeof(float) : 0);
  const cudaError_t e = cudaFuncSetAttribute(k_mlp_fused<SA, SB, F32IN, BWD>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  SBM_PDL((k_mlp_fused<SA, SB, F32IN, BWD>), (unsigned)mlp_fused_ctas(P.rows), kFusedThreads, smem, s, P);
  return cudaSuccess;
}

// ----------------------------------------------------------------------------------------------
// The weight gradients of a training pass, dW1 = X^T dZ1, dW2 = H1^T dZ2, dW3 = H2^T dY, in one launch.
//
// Their contraction runs over the batch (thousands of rows) and their outputs are few tiles (18 of
// 128 x 128 for 2048 -> 128 -> 128 -> 64), so each tile's rows are split over as many CTAs as fill the SMs;
// every CTA writes an FP32 partial tile, which k_grad_reduce sums in a fixed order.  Both operands are
// contiguous along M and N and are read as they lie (MN-major), eight warps copying asynchronously and
// one thread issuing the MMAs.  At 4096 rows
// 19 us; with one CTA per tile each of the three products took 650 us.
constexpr int kWgradStages = 4;
constexpr int kWgradFeed = 8;
constexpr int kWgradThreads = (kWgradFeed + 1) * 32;

__global__ void __launch_bounds__(kWgradThreads, 1) k_wgrad(const __grid_constant__ WgradArgs P) {
  extern __shared__ __align__(1024) unsigned char wgrad_smem[];
  __shared__ __align__(8) unsigned long long full[kWgradStages], empty[kWgradStages], done;
  __shared__ uint32_t tmem_base;
  __shared__ int failed;
  constexpr int S = kWgradStages;
  constexpr uint32_t kTile = 128 * kChunkK * 2;
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  const int split = (int)blockIdx.x % P.splits;
  int t = (int)blockIdx.x / P.splits, q = 0;
  while (q < 2 && t >= P.g[q].tiles_m * P.g[q].tiles_n) t -= P.g[q].tiles_m * P.g[q].tiles_n, ++q;
  const WgradArgs::Gemm& g = P.g[q];
  const int m0 = (t % g.tiles_m) * 128, n0 = (t / g.tiles_m) * 128;
  const int nt = min(128, (g.N - n0 + 31) / 32 * 32);
  const int k_beg = split * P.split_rows, k_end = min(P.rows, k_beg + P.split_rows);
  const int nchunk = k_end > k_beg ? (k_end - k_beg + kChunkK - 1) / kChunkK : 0;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(smem_addr(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], kWgradFeed);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&done, 1);
    mbar_fence_init();
    failed = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base, ring = smem_addr(wgrad_smem);
  volatile int* stop = &failed;
  auto wait = [&](unsigned long long* bar, unsigned parity) {
    if (!mbar_wait(bar, parity)) *stop = 1;
    return *stop == 0;
  };
  pdl_wait();
  pdl_trigger();
  if (warp == kWgradFeed) {
    if (lane == 0) {
      bool ok = true;
      const uint32_t id = idesc_bf16(128, nt, true, true);
      for (int i = 0; i < nchunk && ok; ++i) {
        ok = wait(&full[i % S], (unsigned)((i / S) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a = ring + (i % S) * 2 * kTile, b = a + kTile;
#pragma unroll
        for (int ks = 0; ks < kChunkK / 16; ++ks)    // rows past the range are zero
          mma_bf16(tmem, smem_desc(a + ks * 256, 128, 1024), smem_desc(b + ks * 256, 128, 1024), id, i > 0 || ks > 0);
        mma_commit(&empty[i % S]);
      }
      if (ok && nchunk > 0) mma_commit(&done);
    }
  } else {
    bool ok = true;
    for (int i = 0; i < nchunk + 2 && ok; ++i) {     // two chunks in flight beyond the one handed over
      if (i < nchunk) {
        ok = i < S || wait(&empty[i % S], (unsigned)((i / S - 1) & 1));
        if (ok) {
          const uint32_t a = ring + (i % S) * 2 * kTile;
          stage_async<false>(a, g.A, g.lda, g.M, k_end, m0, 128, k_beg + i * kChunkK, (int)threadIdx.x, kWgradFeed * 32);
          stage_async<false>(a + kTile, g.B, g.ldb, g.N, k_end, n0, nt, k_beg + i * kChunkK, (int)threadIdx.x, kWgradFeed * 32);
        }
      }
      cp_async_commit();
      cp_async_wait<2>();
      if (i >= 2) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0)
          asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(
                           smem_addr(&full[(i - 2) % S]))
                       : "memory");
      }
    }
    cp_async_wait<0>();
    if (ok && nchunk > 0) ok = wait(&done, 0);
    if (ok) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int m = m0 + 32 * (warp & 3) + lane;
      float* out = P.part + (size_t)split * P.part_stride + g.out + (size_t)m * g.N + n0;
      for (int c0 = (warp >> 2) * (nt / 2); c0 < ((warp >> 2) + 1) * (nt / 2); c0 += 8) {
        float v[8];
        tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
        if (nchunk == 0) {
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = 0.f;
        }
        if (m < g.M) {
          if ((g.N & 3) == 0 && (P.part_stride & 3) == 0 && (g.out & 3) == 0 && n0 + c0 + 8 <= g.N) {
            reinterpret_cast<float4*>(out + c0)[0] = make_float4(v[0], v[1], v[2], v[3]);
            reinterpret_cast<float4*>(out + c0)[1] = make_float4(v[4], v[5], v[6], v[7]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (n0 + c0 + j < g.N) out[c0 + j] = v[j];
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (failed && threadIdx.x == 0) {
    atomicExch(P.fault, 1);
    for (int s = 0; s < S; ++s)
      for (unsigned p = 0; p < 2; ++p) mbar_wait(&empty[s], p, 1u << 16);
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem) : "memory");
}

// The packed gradient: weights from the partial tiles, biases from the column sums, both in a fixed order.
__global__ void __launch_bounds__(256) k_grad_reduce(int n, int splits, size_t part_stride, const float* __restrict__ part,
                                                     int ctas, const float* __restrict__ bias_part,
                                                     const __grid_constant__ MlpWeights M, float* __restrict__ G) {
  pdl_entry();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n) return;
  int col = -1;
  if (e >= M.ob1 && e < M.oW2) col = e - M.ob1;
  else if (e >= M.ob2 && e < M.oW3) col = M.Hp + e - M.ob2;
  else if (e >= M.ob3) col = 2 * M.Hp + e - M.ob3;
  float s = 0.f;
  if (col >= 0) {
    for (int b = 0; b < ctas; ++b) s += bias_part[(size_t)b * (2 * M.Hp + M.Op) + col];
  } else {
#pragma unroll 4
    for (int k = 0; k < splits; ++k) s += part[(size_t)k * part_stride + e];
  }
  G[e] = s;
}

}  // namespace

// Two stages of 32 KB: at most 3 CTAs per SM, so the CTAs of an SM never ask for more than 3 x 128
// of its 512 tensor-memory columns (tcgen05.alloc would wait).
constexpr size_t kTcSmem = 2 * 2 * (size_t)TBM * TBK * 2;

template <int TA, int TB>
cudaError_t launch_tc(dim3 grid, int M, int N, int K, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B,
                      int ldb, const float* bias, int relu, float* Cf, __nv_bfloat16* Cb, int ldc, int* fault,
                      cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(k_gemm_tc<TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kTcSmem);
  if (e != cudaSuccess) return e;
  k_gemm_tc<TA, TB><<<grid, kTcThreads, kTcSmem, s>>>(M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, fault);
  return cudaSuccess;
}

cudaError_t launch_gemm_tc(int M, int N, int K, int ta, int tb, const __nv_bfloat16* A, int lda,
                           const __nv_bfloat16* B, int ldb, const float* bias, int relu, float* Cf,
                           __nv_bfloat16* Cb, int ldc, int* fault, cudaStream_t s) {
  if (M == 0 || N == 0) return cudaSuccess;
  const dim3 grid((N + TBN - 1) / TBN, (M + TBM - 1) / TBM);
  cudaError_t e;
  if (!ta && !tb) e = launch_tc<0, 0>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, fault, s);
  else if (!ta && tb) e = launch_tc<0, 1>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, fault, s);
  else if (ta && !tb) e = launch_tc<1, 0>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, fault, s);
  else e = launch_tc<1, 1>(grid, M, N, K, A, lda, B, ldb, bias, relu, Cf, Cb, ldc, fault, s);
  if (e != cudaSuccess) return e;
  count_launches();
  return cudaGetLastError();
}

// Hidden widths up to 256: four A stages, three B stages of 64 x 256 BF16 and the 128 x 256 activation
// tile (224 KB) still fit an SM; wider networks run layer by layer.
bool mlp_fused_fits(int Hp, int Op) { return std::max(Hp, Op) <= 256; }

int mlp_fused_ctas(int rows) { return std::min((rows + kTileRows - 1) / kTileRows, kLossParts); }

cudaError_t launch_mlp_fused(const MlpTile& P, cudaStream_t s) {
  if (P.rows == 0) return cudaSuccess;
  const bool wide = std::max(P.Hp, P.Op) > 128;
  cudaError_t e;
  if (P.T) {                                         // training pass (the column sums take up to 9 KB)
    if (!wide) e = P.Xf ? launch_fused<5, 5, true, true>(P, s) : launch_fused<5, 5, false, true>(P, s);
    else e = P.Xf ? launch_fused<3, 3, true, true>(P, s) : launch_fused<3, 3, false, true>(P, s);
  } else {
    if (!wide) e = P.Xf ? launch_fused<5, 5, true, false>(P, s) : launch_fused<5, 5, false, false>(P, s);
    else e = P.Xf ? launch_fused<4, 3, true, false>(P, s) : launch_fused<4, 3, false, false>(P, s);
  }
  if (e != cudaSuccess) return e;
  count_launches();
  return cudaGetLastError();
}

cudaError_t launch_wgrad(const WgradArgs& P, int n, int ctas, const float* bias_part, const MlpWeights& M, float* G,
                         cudaStream_t s) {
  constexpr size_t smem = kWgradStages * 2 * 128 * kChunkK * 2;
  const cudaError_t e = cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int tiles = 0;
  for (const auto& g : P.g) tiles += g.tiles_m * g.tiles_n;
  SBM_PDL(k_wgrad, (unsigned)(tiles * P.splits), kWgradThreads, smem, s, P);
  SBM_PDL(k_grad_reduce, (unsigned)((n + 255) / 256), 256, 0, s, n, P.splits, P.part_stride, P.part, ctas, bias_part, M, G);
  count_launches(2);
  return cudaGetLastError();
}

int tc_fault_take(int* fault) {
  int f = 0;
  if (cudaMemcpy(&f, fault, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
  if (f) {
    const int zero = 0;
    if (cudaMemcpy(fault, &zero, sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return -1;
  }
  return f;
}

}  // namespace sbm
