// Device helpers shared by the tcgen05 kernels (tc_gemm.cu): shared-memory operand
// tiles without swizzle, their asynchronous staging, instruction descriptors and accumulator loads.
// Included inside namespace sbm { namespace { ... } }.
//
// An operand chunk holds `nr` rows or columns of the product (the M or N index, here mn) times 64
// entries of the contraction (k) as core matrices of 128 bytes, (mn / 8) * 1024 + (k / 8) * 128 bytes
// apart.  A core matrix is 8 mn x 16 bytes of k (K-major: k contiguous in memory) or 8 k x 16 bytes
// of mn (MN-major: mn contiguous); tcgen05 reads either form, chosen by a bit of the instruction
// descriptor, so neither storage order of a matrix needs a transposition on the way in.
#pragma once

constexpr int kChunkK = 64;                        // contraction entries of one staged chunk

// Shared-memory matrix descriptor (tcgen05): start address, leading (k direction) and stride
// (8 mn) byte offsets, all >> 4; bits 46-48 hold the fixed value 1; no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  const uint64_t a = (uint64_t)(addr >> 4) & 0x3FFFu;
  return a | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) | ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator, BF16 A and B, N >> 3 and
// M >> 4; a_mn / b_mn: the operand is MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn = false, bool b_mn = false) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate ? 1u : 0u)
      : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

// 8 consecutive FP32 accumulator columns of the calling thread's row (TMEM lane).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Asynchronous 16-byte copy to shared memory; only the first `bytes` (0..16) come from src, the rest
// is filled with zeros.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Starts the copies of one operand chunk, op(X)(mn, k) for mn0 <= mn < mn0 + nr, k0 <= k < k0 + 64, into
// the tile at `dst`; X(mn, k) = X[mn * ld + k] (KMAJ) or X[k * ld + mn].  Entries outside MN x K are
// zero.  X is 16-byte aligned and ld, mn0, k0 are multiples of 8; nr is a multiple of 32.  Eight
// consecutive lanes write one 128-byte core matrix (no bank conflict) and a warp reads runs of 64 bytes.
template <bool KMAJ>
__device__ __forceinline__ void stage_async(uint32_t dst, const __nv_bfloat16* __restrict__ X, int ld, int MN, int K,
                                            int mn0, int nr, int k0, int tid, int nthreads) {
  for (int q = tid; q < nr * 8; q += nthreads) {
    int off, bytes;
    const __nv_bfloat16* src;
    if (KMAJ) {                                      // row q's low bits, then the k piece, then 8-row groups
      const int r = mn0 + ((q & 7) | ((q >> 6) << 3)), k = k0 + 8 * ((q >> 3) & 7);
      off = q * 16;
      bytes = r < MN ? min(16, max(0, 2 * (K - k))) : 0;
      src = X + (size_t)r * ld + k;
    } else {                                         // k low bits, mn piece (2 bits), k group, mn piece
      const int g = ((q >> 3) & 3) | ((q >> 8) << 2), c = (q >> 5) & 7, kk = (q & 7) | (c << 3);
      const int mn = mn0 + 8 * g, k = k0 + kk;
      off = g * 1024 + c * 128 + (q & 7) * 16;
      bytes = k < K ? min(16, max(0, 2 * (MN - mn))) : 0;
      src = X + (size_t)k * ld + mn;
    }
    cp_async16(dst + off, bytes > 0 ? (const void*)src : (const void*)X, bytes);
  }
}
