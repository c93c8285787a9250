// Thread-per-cell CUDA kernels for small cells ((p+1)^d <= 16: 2D p = 1..3 and 3D p = 1; the FP32
// operator and residual + restriction also for 3D p = 2).
//
// One thread owns one cell: its (p+1)^d values, the interior-face couplings to its 2d
// neighbours, its surrogate-face terms and its block inverse live in registers.  Every loop
// over nodes, lines and directions is unrolled, so each 1D-matrix coefficient is a uniform,
// immediate-offset read of the kernel parameter block (constant cache broadcast).  The per-DoF
// kernels of level_ops.cu issue about 175 instructions per DoF, mostly shared-memory traffic;
// here the arithmetic is the same (Eqs. 7, 10, 11, 14, 16, 18) but the instruction stream is a
// fraction of that.  Cells of an odd number of values are read through their 16-byte-aligned
// window and stored through shared memory (cell_core.cuh); launches over a whole level take the
// colours interleaved (interleaved_warp).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "ops.h"

namespace sbm {
namespace {

#include "cell_core.cuh"

// Launches over all cells of a level interleave the colours: block b takes chunk b / 2^D (of
// blockDim.x consecutive cells) of colour b mod 2^D.  The face neighbours of a cell all have
// other colours, so with the colours taken one after another every colour's values would be read
// from DRAM once for its own pass and again in the passes of the colours next to it; interleaved,
// the blocks in flight cover the same stretch of the mesh in every colour and the neighbours'
// values are found in L2.  Sets the first cell of the calling thread's warp and the end of its
// colour (the warp holds min(32, end - a0w) cells, none if that is <= 0).
template <int D, typename R>
__device__ __forceinline__ void interleaved_warp(const LevelParams<R>& P, int& a0w, int& end) {
  constexpr int NCOL = 1 << D;
  const int c = (int)blockIdx.x % NCOL;
  a0w = P.colour_start[c] + ((int)blockIdx.x / NCOL) * (int)blockDim.x + ((int)threadIdx.x & ~31);
  end = P.colour_start[c + 1];
}

// y = A x (MODE 0) or y = f - A x (MODE 1), one thread per cell, colours interleaved.
template <int D, int N1, typename TI, typename R, int MODE>
__device__ __forceinline__ void apply_cell_body(const LevelParams<R>& P, const TI* __restrict__ x,
                                                const R* __restrict__ f, R* __restrict__ y) {
  constexpr int NP = CD<D, N1>::NP;
  int a0w, end;
  interleaved_warp<D, R>(P, a0w, end);
  const int a = a0w + ((int)threadIdx.x & 31);
  const bool valid = a < end;
  int nb[2 * D];
  if (valid) load_nbr<D, R>(P, a, nb);             // set-up data: read before the wait
  pdl_wait();
  pdl_trigger();
  R r[NP];
  if (valid) {
    cell_apply<D, N1, TI, R>(P, x, a, nb, r);
    if (MODE == 1) {
      R fv[NP];
      load_cell<D, N1, R, R>(f, a, P.n_act, fv);
#pragma unroll
      for (int i = 0; i < NP; ++i) r[i] = fv[i] - r[i];
    }
  }
  if constexpr (cell_vec16<NP, R>()) {
    if (valid) store_cell<D, N1, R>(y, a, r);
  } else {
    __shared__ WarpStage<NP, R> stage;
    if (a0w < end) warp_store_cells<NP, R>(y, a0w, min(32, end - a0w), r, stage.v[threadIdx.x >> 5]);
  }
}

template <int D, int N1, typename TI, typename R, int MODE>
__global__ void __launch_bounds__(kCellThreads) k_apply_cell(const __grid_constant__ LevelParams<R> P,
                                                             const TI* __restrict__ x, const R* __restrict__ f,
                                                             R* __restrict__ y) {
  apply_cell_body<D, N1, TI, R, MODE>(P, x, f, y);
}

// The same, compiled for 24 resident warps per SM (80 registers).  Used for the double-float
// operator of 2D p = 2: at its natural 96 registers an SM holds 20 warps, and the 512^2 p = 2 grid
// of 3164 warps then runs as 1.04 waves whose last warps run alone; at 80 every warp is resident
// at once.  (2D p = 3 spills heavily at 80; p = 1 needs fewer than 80.)
template <int D, int N1, typename TI, typename R, int MODE>
__global__ void __launch_bounds__(kCellThreads, 6) k_apply_cell_occ(const __grid_constant__ LevelParams<R> P,
                                                                    const TI* __restrict__ x,
                                                                    const R* __restrict__ f, R* __restrict__ y) {
  apply_cell_body<D, N1, TI, R, MODE>(P, x, f, y);
}


// The NN entries of boundary cell b's block stored by entry (LevelParams::binvS, aselfS); nothing if b < 0.
template <int NN, typename R>
__device__ __forceinline__ void load_block(const R* __restrict__ S, int ld, int b, R (&B)[NN]) {
  if (b < 0) return;
#pragma unroll
  for (int q = 0; q < NN; ++q) B[q] = __ldg(S + (size_t)q * ld + b);
}
// y = B t, B by columns (never called with NN != NP * NP).
template <int NP, int NN, typename R>
__device__ __forceinline__ void dense_apply(const R (&B)[NN], const R (&t)[NP], R (&y)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) y[i] = 0;
#pragma unroll
  for (int j = 0; j < NP; ++j)
#pragma unroll
    for (int i = 0; i < NP; ++i) y[i] += B[NN > 1 ? j * NP + i : 0] * t[j];
}

// One colour group of the block Gauss-Seidel sweep, one thread per cell: block b updates cells of
// the segment whose block range holds b.
//
// A launch of a small level is bound by the longest chain of dependent reads, that of the boundary
// cells: the neighbours, then the dense inverse.  PRE: the inverse (set-up data) is read into registers
// before the dependency wait.  It is read by entry (binvS), 128 contiguous bytes per warp and entry; from
// the cells' own blocks every one of the (p+1)^(2d) loads touched 32 lines.  V-cycle of the 512^2 p = 2 star
// 107 -> 96 us, of the 64^3 p = 1 sphere 29 us less (89 now).  PRE is for launches of up to 32 warps per SM (32-thread
// blocks) and (p+1)^d <= 9 FP32 values; larger launches hide the reads behind other warps.
template <int D, int N1, typename R, bool PRE>
__global__ void __launch_bounds__(PRE ? 32 : kCellThreads) k_smooth_cell(const __grid_constant__ LevelParams<R> P,
                                                              const __grid_constant__ SmoothSegs G, int zero_start,
                                                              const R* __restrict__ f, R* __restrict__ u, int early) {
  constexpr int NP = CD<D, N1>::NP;
  int sg = 0;
#pragma unroll
  for (int k = 1; k < SmoothSegs::kMax; ++k)
    if (k < G.n && (int)blockIdx.x >= G.blk[k]) sg = k;
  const int a0w = G.first[sg] + ((int)blockIdx.x - G.blk[sg]) * (int)blockDim.x + ((int)threadIdx.x & ~31);
  const int end = G.last[sg];
  const int a = a0w + ((int)threadIdx.x & 31);
  const bool valid = a < end;
  const int off = a - G.cs[sg], bidx = off < G.nbnd[sg] ? G.b0[sg] + off : -1;
  int nb[2 * D];
  R t[NP];
  R B[PRE ? NP * NP : 1];
  if (valid) {
    load_nbr<D, R>(P, a, nb);                        // set-up data: read before the wait
    if (early) load_cell_l2<D, N1, R, R>(f, a, P.n_act, t);   // f written two or more launches back
    if constexpr (PRE) load_block(P.binvS, P.bnd_ld, bidx, B);
  }
  pdl_wait();
  pdl_trigger();
  R y[NP];
  if (valid) {
    if (!early) load_cell<D, N1, R, R>(f, a, P.n_act, t);
    smooth_rhs<D, N1, R>(P, G.col[sg], zero_start, nb, t, u);
    if (PRE && bidx >= 0) dense_apply(B, t, y);
    else block_solve<D, N1, R>(P, bidx, t, y);
    smooth_relax<D, N1, R>(P, zero_start, a, u, y);
  }
  if constexpr (cell_vec16<NP, R>()) {
    if (valid) store_cell<D, N1, R>(u, a, y);
  } else {
    __shared__ WarpStage<NP, R> stage;
    if (a0w < end) warp_store_cells<NP, R>(u, a0w, min(32, end - a0w), y, stage.v[threadIdx.x >> 5]);
  }
}

// Residual and p-restriction fused, one thread per cell (Eqs. 11, 18).
// SM0: also the first colour group (colour 0) of the coarse level's first pre-smoothing sweep from
// zero, zc_K = omega A_KK^-1 rc_K for coarse cells K of colour 0 (their neighbours, of later
// colours, are still zero), with the coarse level's parameters Pc; that sweep then starts at group 1.
template <int D, int N1, int NC, typename R, bool SM0>
__global__ void __launch_bounds__(kCellThreads) k_resid_restrict_p_cell(const __grid_constant__ LevelParams<R> P,
                                                                        const __grid_constant__ TransferParams<R> T,
                                                                        const R* __restrict__ u,
                                                                        const R* __restrict__ f, R* __restrict__ rc,
                                                                        int early,
                                                                        const __grid_constant__ LevelParams<R> Pc,
                                                                        R* __restrict__ zc) {
  constexpr int NP = CD<D, N1>::NP;
  constexpr int NPC = D == 2 ? NC * NC : NC * NC * NC;
  int a0w, end;
  interleaved_warp<D, R>(P, a0w, end);               // colours interleaved
  const int a = a0w + ((int)threadIdx.x & 31);
  int nb[2 * D];
  R fa[NP];
  if (a < end) {
    load_nbr<D, R>(P, a, nb);                        // set-up data: read before the wait
    if (early) load_cell_l2<D, N1, R, R>(f, a, P.n_act, fa);  // f written two or more launches back
  }
  pdl_wait();
  pdl_trigger();
  if (a >= end) return;
  if (!early) load_cell<D, N1, R, R>(f, a, P.n_act, fa);
  R r[NP];
  cell_apply<D, N1, R, R>(P, u, a, nb, r);
#pragma unroll
  for (int i = 0; i < NP; ++i) r[i] = fa[i] - r[i];
  R out[NPC];
#pragma unroll
  for (int j = 0; j < NPC; ++j) {
    const int j0 = j % NC, j1 = (j / NC) % NC, j2 = D == 3 ? j / (NC * NC) : 0;
    R acc = 0;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const int i0 = i % N1, i1 = (i / N1) % N1, i2 = D == 3 ? i / (N1 * N1) : 0;
      R wgt = T.Pp[i0 * NC + j0] * T.Pp[i1 * NC + j1];
      if (D == 3) wgt *= T.Pp[i2 * NC + j2];
      acc += wgt * r[i];
    }
    out[j] = acc;
    rc[(size_t)a * NPC + j] = acc;
  }
  if constexpr (SM0) {
    if (a < Pc.colour_start[1]) {                    // same mesh: the coarse cell has index a
      R y[NPC];
      block_solve<D, NC, R>(Pc, a < Pc.colour_nbnd[0] ? Pc.bstart[0] + a : -1, out, y);
#pragma unroll
      for (int j = 0; j < NPC; ++j) y[j] = Pc.omega == R(1) ? y[j] : Pc.omega * y[j];
      store_cell<D, NC, R>(zc, a, y);
    }
  }
}

// h-transfer weight of fine node i (child o of its parent) and coarse node j, p = 1 on both
// meshes (Eqs. 17, 18): the tensor product of the 1D child matrices.
template <int D, typename R>
__device__ __forceinline__ R h_weight(const TransferParams<R>& T, int o, int i, int j) {
  R wgt = T.Ph[o & 1][(i & 1) * 2 + (j & 1)] * T.Ph[(o >> 1) & 1][((i >> 1) & 1) * 2 + ((j >> 1) & 1)];
  if (D == 3) wgt *= T.Ph[(o >> 2) & 1][((i >> 2) & 1) * 2 + ((j >> 2) & 1)];
  return wgt;
}

// One group of 2^D adjacent lanes per coarse cell, lane o of the group handling child o: the
// child's residual in registers, its restriction, then a fixed butterfly sum over the group.
// SM0: also the first colour group of the coarse level's first pre-smoothing sweep from zero (see
// k_resid_restrict_p_cell), computed by lane 0 of each coarse cell's group.
//
// PRE (as in k_smooth_cell): with SM0 the coarse cells' inverses, and in 2D the children's self blocks instead
// of their surrogate-face terms, are read before the dependency wait: V-cycle of the 512^2 p = 2 star 95.7 ->
// 94.1 us.  (3D keeps the order of its operations, see k_vcycle_tail_cta.  Not at 2D p = 2,
// k_resid_restrict_p_cell: 81 registers of block made that V-cycle 1.8 us longer; nor after the wait in the
// operator: 44 -> 46 us at 2048^2 p = 2.)
template <int D, typename R, bool SM0, bool PRE>
__global__ void __launch_bounds__(PRE ? 32 : kCellThreads) k_resid_restrict_h_cell(const __grid_constant__ LevelParams<R> P,
                                                                        const __grid_constant__ TransferParams<R> T,
                                                                        const R* __restrict__ u,
                                                                        const R* __restrict__ f, R* __restrict__ rc,
                                                                        int early,
                                                                        const __grid_constant__ LevelParams<R> Pc,
                                                                        R* __restrict__ zc) {
  constexpr int NCOL = 1 << D, NP = CD<D, 2>::NP;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int cc = t / NCOL, o = t % NCOL;
  R out[NP];
#pragma unroll
  for (int j = 0; j < NP; ++j) out[j] = 0;
  // the child and its neighbours are set-up data: read before the wait
  const int a = cc < T.n_act_c ? T.children[(size_t)o * T.n_act_c + cc] : -1;
  int nb[2 * D];
  R fa[NP];
  constexpr int NPRE = PRE && D == 2 ? NP * NP : 1, NPRC = PRE && SM0 ? NP * NP : 1;
  R A[NPRE], B[NPRC];
  if (a >= 0) {
    load_nbr<D, R>(P, a, nb);
    if (early) load_cell_l2<D, 2, R, R>(f, a, P.n_act, fa);   // f written two or more launches back
    if constexpr (PRE && D == 2) load_block<NPRE>(P.aselfS, P.bnd_ld, boundary_index(P, a, 1 << D), A);
  }
  if constexpr (PRE && SM0)
    load_block<NPRC>(Pc.binvS, Pc.bnd_ld, o == 0 && cc < T.n_act_c && cc < Pc.colour_nbnd[0] ? Pc.bstart[0] + cc : -1, B);
  pdl_wait();
  pdl_trigger();
  if (a >= 0) {
    R r[NP];
    if (!early) load_cell<D, 2, R, R>(f, a, P.n_act, fa);
    cell_apply<D, 2, R, R, NPRE>(P, u, a, nb, r, &A);
#pragma unroll
    for (int i = 0; i < NP; ++i) r[i] = fa[i] - r[i];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      R acc = 0;
#pragma unroll
      for (int i = 0; i < NP; ++i) acc += h_weight<D, R>(T, o, i, j) * r[i];
      out[j] = acc;
    }
  }
#pragma unroll
  for (int off = 1; off < NCOL; off <<= 1)
#pragma unroll
    for (int j = 0; j < NP; ++j) out[j] += __shfl_xor_sync(0xffffffffu, out[j], off);
  if (o == 0 && cc < T.n_act_c) {
#pragma unroll
    for (int j = 0; j < NP; ++j) rc[(size_t)cc * NP + j] = out[j];
    if constexpr (SM0) {
      if (cc < Pc.colour_start[1]) {
        R y[NP];
        const int bc = cc < Pc.colour_nbnd[0] ? Pc.bstart[0] + cc : -1;
        if (PRE && bc >= 0) dense_apply<NP, NPRC>(B, out, y);
        else block_solve<D, 2, R>(Pc, bc, out, y);
#pragma unroll
        for (int j = 0; j < NP; ++j) y[j] = Pc.omega == R(1) ? y[j] : Pc.omega * y[j];
        store_cell<D, 2, R>(zc, cc, y);
      }
    }
  }
}


// ----------------------------------------------------------------------------------------------
// The V-cycle below and including level `top` (all of them p = 1 h-levels) in one launch of a
// thread-block cluster, with every level vector held in the cluster's shared memory.
//
// Layout: colour c of a level (cells [cs_c, ce_c) of the colour-major order) is cut into
// chunks of m[c] consecutive cells, chunk k living on CTA k of the cluster; a CTA stores its
// chunks of all colours back to back (colour c from cell slot off[c]) once for z (element
// offset zoff) and once for the right-hand side (roff).  A CTA updates only the cells it
// stores; neighbour, child and parent values of other CTAs are read through distributed shared
// memory.  Every phase (one colour of a sweep, the fused residual/restriction, the coarse solve,
// a prolongation) ends with a cluster barrier, whose release/acquire semantics order the shared
// memory writes of the phase before the reads of the next.
// ----------------------------------------------------------------------------------------------
template <typename R>
__device__ __forceinline__ int colour_of(const TailLevel<R>& L, int a, int ncol) {
  int c = 0;
#pragma unroll
  for (int k = 1; k < 8; ++k)
    if (k < ncol && a >= L.P.colour_start[k]) c = k;
  return c;
}

// Generic address of the NP values of cell a (colour col) of vector `vo` (zoff or roff) of L.
template <int NP, typename R>
__device__ __forceinline__ R* tail_cell(const cooperative_groups::cluster_group& cl, R* sm, const TailLevel<R>& L,
                                        int vo, int a, int col) {
  const int rel = a - L.P.colour_start[col];
  const int rk = rel / L.m[col];
  R* p = sm + vo + (size_t)(L.off[col] + rel - rk * L.m[col]) * NP;
  return cl.map_shared_rank(p, (unsigned)rk);
}

template <int D, typename R>
__global__ void __launch_bounds__(kTailThreads, 1) k_vcycle_tail(const TailLevel<R>* __restrict__ TL, int top,
                                                                 const R* __restrict__ r_top, R* __restrict__ z_top,
                                                                 const double* __restrict__ coarse_inv, int pre,
                                                                 int post, int ssor, int gather_off) {
  namespace cg = cooperative_groups;
  const cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char tail_smem[];
  R* sm = reinterpret_cast<R*>(tail_smem);
  const int rank = (int)cl.block_rank();
  constexpr int NCOL = 1 << D, NP = CD<D, 2>::NP;

  // this CTA's cells of colour col of L: fn(cell, slot)
  auto for_own = [&](const TailLevel<R>& L, int col, auto&& fn) {
    const int cs = L.P.colour_start[col], ce = L.P.colour_start[col + 1], m = L.m[col];
    const int first = cs + rank * m;
    const int cnt = min(m, ce - first);
    for (int j = threadIdx.x; j < cnt; j += kTailThreads) fn(first + j, L.off[col] + j);
  };
  auto loader = [&cl, sm](const TailLevel<R>& L, int vo) {
    const TailLevel<R>* Lp = &L;
    return [&cl, sm, Lp, vo](int n, int ncol, R(&un)[NP]) {
      load_np_vec<NP, R>(tail_cell<NP>(cl, sm, *Lp, vo, n, ncol), un);
    };
  };
  auto smooth = [&](const TailLevel<R>& L, int col, bool zs) {
    for_own(L, col, [&](int a, int slot) {
      const LevelParams<R>& P = L.P;
      int nb[2 * D];
      load_nbr<D, R>(P, a, nb);
      R c[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) c[i] = 0;
      add_couplings_f<D, 2, R>(P.k, col, zs, nb, loader(L, L.zoff), c);
      R t[NP];
      load_np_vec<NP, R>(sm + L.roff + (size_t)slot * NP, t);
#pragma unroll
      for (int i = 0; i < NP; ++i) t[i] -= P.hscale * c[i];
      const int off = a - P.colour_start[col];
      R y[NP];
      block_solve<D, 2, R>(P, off < P.colour_nbnd[col] ? P.bstart[col] + off : -1, t, y);
      R* zu = sm + L.zoff + (size_t)slot * NP;
      if (P.omega != R(1)) {
        R uo[NP];
        if (zs) {
#pragma unroll
          for (int i = 0; i < NP; ++i) uo[i] = 0;
        } else {
          load_np_vec<NP, R>(zu, uo);
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) y[i] = (R(1) - P.omega) * uo[i] + P.omega * y[i];
      }
      store_np_vec<NP, R>(zu, y);
    });
  };

  {                                                // right-hand side of the top level
    const TailLevel<R>& L = TL[top];
    for (int col = 0; col < NCOL; ++col)
      for_own(L, col, [&](int a, int slot) {
#pragma unroll
        for (int i = 0; i < NP; ++i) sm[L.roff + (size_t)slot * NP + i] = r_top[(size_t)a * NP + i];
      });
    cl.sync();
  }
  for (int l = top; l >= 1; --l) {                 // down: pre-smooth, residual, restrict
    const TailLevel<R>& L = TL[l];
    if (pre == 0) {
      for (int q = threadIdx.x; q < L.ncell * NP; q += kTailThreads) sm[L.zoff + q] = R(0);
      cl.sync();
    }
    for (int k = 0; k < pre; ++k) {
      for (int col = 0; col < NCOL; ++col) {
        smooth(L, col, k == 0);
        cl.sync();
      }
      if (ssor)
        for (int q = 0; q < NCOL; ++q) {
          smooth(L, NCOL - 1 - q, false);
          cl.sync();
        }
    }
    const TailLevel<R>& Lc = TL[l - 1];
    for (int ccol = 0; ccol < NCOL; ++ccol)
      for_own(Lc, ccol, [&](int cc, int slot) {
        R out[NP];
#pragma unroll
        for (int j = 0; j < NP; ++j) out[j] = 0;
#pragma unroll 1
        for (int o = 0; o < NCOL; ++o) {
          const int a = L.T.children[(size_t)o * L.T.n_act_c + cc];
          if (a < 0) continue;
          const int ca = colour_of(L, a, NCOL);
          int nb[2 * D];
          load_nbr<D, R>(L.P, a, nb);
          R v[NP], y[NP], f[NP];
          load_np_vec<NP, R>(tail_cell<NP>(cl, sm, L, L.zoff, a, ca), v);
          load_np_vec<NP, R>(tail_cell<NP>(cl, sm, L, L.roff, a, ca), f);
#pragma unroll
          for (int i = 0; i < NP; ++i) y[i] = 0;
          const int off = a - L.P.colour_start[ca];
          add_self<D, 2, R>(L.P, nb, off < L.P.colour_nbnd[ca] ? L.P.bstart[ca] + off : -1, v, y);
          add_couplings_f<D, 2, R>(L.P.k, ca, false, nb, loader(L, L.zoff), y);
#pragma unroll
          for (int i = 0; i < NP; ++i) y[i] = f[i] - L.P.hscale * y[i];
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            R acc = 0;
#pragma unroll
            for (int i = 0; i < NP; ++i) acc += h_weight<D, R>(L.T, o, i, j) * y[i];
            out[j] += acc;
          }
        }
        store_np_vec<NP, R>(sm + Lc.roff + (size_t)slot * NP, out);
      });
    cl.sync();
  }
  {                                                // coarse solve in FP64, one warp per row
    const TailLevel<R>& L0 = TL[0];
    const int n0 = L0.P.n_act * NP;
    R* g = sm + gather_off;                        // this CTA's copy of the whole coarse rhs
    for (int a = threadIdx.x; a < L0.P.n_act; a += kTailThreads) {
      R v[NP];
      load_np_vec<NP, R>(tail_cell<NP>(cl, sm, L0, L0.roff, a, colour_of(L0, a, NCOL)), v);
      store_np_vec<NP, R>(g + (size_t)a * NP, v);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int nwarp = (int)cl.num_blocks() * (kTailThreads / 32);
    for (int row = rank * (kTailThreads / 32) + (threadIdx.x >> 5); row < n0; row += nwarp) {
      double acc = 0;
      for (int c = lane; c < n0; c += 32) acc += coarse_inv[(size_t)row * n0 + c] * (double)g[c];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
      if (lane == 0) {
        const int cell = row / NP;
        tail_cell<NP>(cl, sm, L0, L0.zoff, cell, colour_of(L0, cell, NCOL))[row - cell * NP] = (R)acc;
      }
    }
    cl.sync();
  }
  for (int l = 1; l <= top; ++l) {                 // up: prolongate, post-smooth
    const TailLevel<R>& L = TL[l];
    const TailLevel<R>& Lc = TL[l - 1];
    for (int col = 0; col < NCOL; ++col)
      for_own(L, col, [&](int a, int slot) {
        const int code = L.T.parent_code[a];
        if (code < 0) return;
        const int par = code >> 3, o = code & 7;
        R e[NP], u[NP];
        load_np_vec<NP, R>(tail_cell<NP>(cl, sm, Lc, Lc.zoff, par, colour_of(Lc, par, NCOL)), e);
        R* zu = sm + L.zoff + (size_t)slot * NP;
        load_np_vec<NP, R>(zu, u);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          R acc = 0;
#pragma unroll
          for (int j = 0; j < NP; ++j) acc += h_weight<D, R>(L.T, o, i, j) * e[j];
          u[i] += acc;
        }
        store_np_vec<NP, R>(zu, u);
      });
    cl.sync();
    for (int k = 0; k < post; ++k) {
      if (ssor)
        for (int col = 0; col < NCOL; ++col) {
          smooth(L, col, false);
          cl.sync();
        }
      for (int q = 0; q < NCOL; ++q) {
        smooth(L, NCOL - 1 - q, false);
        cl.sync();
      }
    }
  }
  {                                                // correction of the top level out
    const TailLevel<R>& L = TL[top];
    for (int col = 0; col < NCOL; ++col)
      for_own(L, col, [&](int a, int slot) {
#pragma unroll
        for (int i = 0; i < NP; ++i) z_top[(size_t)a * NP + i] = sm[L.zoff + (size_t)slot * NP + i];
      });
  }
}

// ----------------------------------------------------------------------------------------------
// The V-cycle of levels 0..top (p = 1 h-levels) in one CTA: all data of those levels in shared
// memory, phases separated by __syncthreads(); see TailCta.
// ----------------------------------------------------------------------------------------------
// Threads of the one-CTA tail.  (With 1024 in 2D every phase was 50 to 100 cycles longer, the barrier and
// the idle warps' share of it.)
constexpr int kTailCtaThreads = 512;

// Set when the tail's staging copies did not complete within kAsyncSpin polls (the tail then
// copied the data itself); tail_fault_take() reads and clears it.
__device__ int g_tail_fault;

// What bounds it: the latency of some 25 dependent phases.  So:
//   - the tables arrive as one bulk copy, before the dependency wait;
//   - the level descriptors are in shared memory (indexed reads of the parameter block missed the
//     constant cache in every phase);
//   - every phase's code appears once, in one loop over the levels down and up again, so the instructions
//     of a phase are in the cache from its first use on;
//   - a cell's neighbours, boundary index and parent are one 16-byte record; a missing neighbour is a
//     zero cell, so no load waits for a branch;
//   - 2D: an interior cell applies a dense inverse like a boundary cell, so a warp of both takes one path,
//     and boundary residuals use stored self blocks.  (Against fast diagonalisation the V-cycle's
//     error against 64 bits moves by -8 to +13% with the geometry family and size, +1.6% in the mean over p = 1
//     disks and stars of 32^2 to 1024^2; with the inverse in two parts by -9 to +7%, the same mean.)
//   - 3D keeps the operations of the tail's first form in their order, to the same bits (the tests pin them): the
//     long 3D p = 3 solves (96^3 to 1e-12) end after another number of steps when the rounding of their V-cycle
//     changes.  (The per-level kernels round otherwise; they differ in most values by a unit or so.)
//   - vectors and blocks are laid out free of bank conflicts (TailCta).
// What is left in 2D is bound by the shared-memory reads of the largest level's phases (the 64^2 level: 850 to
// 1500 cycles a colour group, 4200 the restriction) and by each thread's chain on the smaller ones (500 to
// 600 cycles): a V-cycle of the 512^2 p = 2 star (tail: 64^2 .. 8^2) went 127 -> 107 us. In 3D the restriction
// of the largest level, with the surrogate-face terms of its boundary cells, is the longest phase: a V-cycle
// of a 64^3 p = 1 sphere (16^3 .. 4^3) takes 89 us with this order of operations and 76 with the 2D form.
template <int D, typename R>
__global__ void __launch_bounds__(kTailCtaThreads, 1) k_vcycle_tail_cta(const __grid_constant__ TailCta<R> TP,
                                                                        const R* __restrict__ r_top,
                                                                        R* __restrict__ z_top,
                                                                        const double* __restrict__ coarse_inv) {
  extern __shared__ __align__(16) unsigned char tcta_smem[];
  constexpr int NCOL = 1 << D, NP = CD<D, 2>::NP, NT = kTailCtaThreads;
  constexpr int W = NP * (int)sizeof(R) / 16, PW = NP / W;      // 16-byte words of a cell, values of a word
  constexpr unsigned BLK = NP * NP * sizeof(R) + 16;            // a padded boundary block
  static_assert(NP == NCOL, "one value per child in the restriction's exchange");
  const int top = TP.top, tid = threadIdx.x;
  const TailLevelDesc* lev = reinterpret_cast<const TailLevelDesc*>(tcta_smem);
  __shared__ __align__(8) unsigned long long tbar;
  if (tid == 0) {
    mbar_init(&tbar, 1);
    mbar_fence_init();
    mbar_arrive_tx(&tbar, TP.image_bytes);
    bulk_load(tcta_smem, TP.image, TP.image_bytes, &tbar);
  }
  for (unsigned q = tid; q < TP.vec_bytes / 8; q += NT)         // z and f: zero
    reinterpret_cast<uint4*>(tcta_smem + TP.image_bytes)[q] = make_uint4(0u, 0u, 0u, 0u);
  R P0[4], P1[4];                                    // 1D transfer matrices of the two children
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    P0[q] = TP.T.Ph[0][q];
    P1[q] = TP.T.Ph[1][q];
  }
  __syncthreads();                                   // the barrier is initialised before anyone polls it
  if (!__syncthreads_and(mbar_wait(&tbar, 0))) {     // record, let the copy land, copy by hand
    if (tid == 0) {
      atomicExch(&g_tail_fault, 1);
      mbar_wait(&tbar, 0);
    }
    __syncthreads();
    for (unsigned q = tid; q < TP.image_bytes / 16; q += NT)
      reinterpret_cast<uint4*>(tcta_smem)[q] = static_cast<const uint4*>(TP.image)[q];
    __syncthreads();
  }

  // the NP values of cell a of the vector at byte offset v of a level of n cells
  auto load = [&](unsigned v, int n, unsigned a, R(&x)[NP]) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      R t[PW];
      load_np_vec<PW, R>(reinterpret_cast<const R*>(tcta_smem + v + (unsigned)(w * (n + 1) + (int)a) * 16u), t);
#pragma unroll
      for (int i = 0; i < PW; ++i) x[w * PW + i] = t[i];
    }
  };
  auto store = [&](unsigned v, int n, unsigned a, const R(&x)[NP]) {
#pragma unroll
    for (int w = 0; w < W; ++w) {
      R t[PW];
#pragma unroll
      for (int i = 0; i < PW; ++i) t[i] = x[w * PW + i];
      store_np_vec<PW, R>(reinterpret_cast<R*>(tcta_smem + v + (unsigned)(w * (n + 1) + (int)a) * 16u), t);
    }
  };
  // 3D: c += the couplings to the neighbours of the record q, unscaled
  auto couple3 = [&](const uint4& q, unsigned z, int n, const R(&b)[8], R wt, R(&c)[NP]) {
    const unsigned w[3] = {q.x, q.y, q.z};
#pragma unroll
    for (int s = 0; s < 2 * D; ++s) {
      R u[NP];
      load(z, n, (s & 1) ? w[s >> 1] >> 16 : w[s >> 1] & 0xffffu, u);
#pragma unroll
      for (int tl = 0; tl < NP / 2; ++tl)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          // explicit: the compiler is free to fuse either product of a sum of two
          R acc = fma(b[4 * (s & 1) + 2 * i], u[dof<D, 2>(s >> 1, 0, tl)], R(0));
          acc = fma(b[4 * (s & 1) + 2 * i + 1], u[dof<D, 2>(s >> 1, 1, tl)], acc);
          c[dof<D, 2>(s >> 1, i, tl)] += wt * acc;
        }
    }
  };
  // 2D: t -= the couplings to the neighbours of the record q (Eq. 10)
  auto couple = [&](const uint4& q, unsigned z, int n, const R(&b)[8], R(&t)[NP]) {
    const unsigned w[3] = {q.x, q.y, q.z};
#pragma unroll
    for (int s = 0; s < 2 * D; ++s) {
      R u[NP];
      load(z, n, (s & 1) ? w[s >> 1] >> 16 : w[s >> 1] & 0xffffu, u);
#pragma unroll
      for (int tl = 0; tl < NP / 2; ++tl)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int k = dof<D, 2>(s >> 1, i, tl);
          t[k] -= b[4 * (s & 1) + 2 * i] * u[dof<D, 2>(s >> 1, 0, tl)];
          t[k] -= b[4 * (s & 1) + 2 * i + 1] * u[dof<D, 2>(s >> 1, 1, tl)];
        }
    }
  };
  // y += sign * T^T t for a transposed NP x NP block T
  auto block = [&](const R* T, const R(&t)[NP], R sign, R(&y)[NP]) {
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      R c[NP];
      load_np_vec<NP, R>(T + j * NP, c);
      const R tj = sign * t[j];
#pragma unroll
      for (int i = 0; i < NP; ++i) y[i] += c[i] * tj;
    }
  };
  pdl_wait();
  pdl_trigger();
  {                                                  // the top level's right-hand side
    const int n = lev[top].n_act;
    const unsigned f = lev[top].f;
    if (reinterpret_cast<uintptr_t>(r_top) % 16 == 0) {
      for (int q0 = tid; q0 < n * W; q0 += 4 * NT) { // four words in flight per thread
        uint4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (q0 + k * NT < n * W) v[k] = reinterpret_cast<const uint4*>(r_top)[q0 + k * NT];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int q = q0 + k * NT;
          if (q < n * W) *reinterpret_cast<uint4*>(tcta_smem + f + (unsigned)((q % W) * (n + 1) + q / W) * 16u) = v[k];
        }
      }
    } else {
      for (int q = tid; q < n * NP; q += NT)
        reinterpret_cast<R*>(tcta_smem + f)[((q % NP) / PW * (n + 1) + q / NP) * PW + q % PW] = r_top[q];
    }
    __syncthreads();
  }
  for (int step = 0; step <= 2 * top; ++step) {      // down: top .. 1, the coarse solve, up: 1 .. top
    const bool down = step < top;
    const int l = down ? top - step : step - top;
    if (step == top) {                               // coarse solve: 8 lanes per row
      const int n0 = TP.n0, na = lev[0].n_act;
      auto at = [&](unsigned v, int c) -> R& {       // unknown c of level 0
        return reinterpret_cast<R*>(tcta_smem + v)[((c % NP) / PW * (na + 1) + c / NP) * PW + c % PW];
      };
      const unsigned r0 = lev[0].f, z0 = lev[0].z;
      if (TP.cinv) {
        // the transpose staged in shared memory.  FP32 tail: the inverse is stored as double-float
        // and every product is exact (two_prod) and summed in double-float on the FP32 pipes (about
        // 48 bits; the input and the result are FP32), since one SM's FP64 pipe made this the tail's
        // longest phase.  FP64 tail: FP64 throughout.
        for (int base = 0; base < n0; base += NT / 8) {
          const int row = base + tid / 8, c0 = tid & 7;
          if constexpr (sizeof(R) == 4) {
            const dfl* aT = reinterpret_cast<const dfl*>(tcta_smem + TP.cinv);
            dfl acc(0.f);
            if (row < n0)
              for (int c = c0; c < n0; c += 8) acc += aT[(size_t)c * n0 + row] * (float)at(r0, c);
#pragma unroll
            for (int off = 4; off > 0; off >>= 1)
              acc += dfl(__shfl_xor_sync(0xffffffffu, acc.hi, off), __shfl_xor_sync(0xffffffffu, acc.lo, off));
            if (row < n0 && c0 == 0) at(z0, row) = (R)__fadd_rn(acc.hi, acc.lo);
          } else {
            const double* aT = reinterpret_cast<const double*>(tcta_smem + TP.cinv);
            double acc = 0.0;
            if (row < n0)
              for (int c = c0; c < n0; c += 8) acc += aT[(size_t)c * n0 + row] * (double)at(r0, c);
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
            if (row < n0 && c0 == 0) at(z0, row) = (R)acc;
          }
        }
      } else {                                       // from global memory, one warp per row
        const int lane = tid & 31;
        for (int row = tid >> 5; row < n0; row += NT / 32) {
          double acc = 0;
          for (int c = lane; c < n0; c += 32) acc += coarse_inv[(size_t)row * n0 + c] * (double)at(r0, c);
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
          if (lane == 0) at(z0, row) = (R)acc;
        }
      }
      __syncthreads();
      continue;
    }
    const TailLevelDesc& L = lev[l];
    const int n = L.n_act;
    const unsigned z = L.z, f = L.f;
    const R* M = reinterpret_cast<const R*>(tcta_smem + L.mats);
    const uint4* rec = reinterpret_cast<const uint4*>(tcta_smem + L.rec);
    R bc[8];                                         // the level's couplings
#pragma unroll
    for (int i = 0; i < 8; ++i) bc[i] = M[i];
    if (!down) {                                     // prolongation (Eq. 17)
      const int nc = lev[l - 1].n_act;
      const unsigned zc = lev[l - 1].z;
      for (int a = tid; a < n; a += NT) {
        const unsigned code = rec[a].w >> 16;
        if (code == 0xffffu) continue;
        R e[NP], u[NP];
        load(zc, nc, code >> 3, e);
        load(z, n, a, u);
        if constexpr (D == 3) {
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            R acc = 0;
#pragma unroll
            for (int j = 0; j < NP; ++j) acc += h_weight<D, R>(TP.T, (int)(code & 7u), i, j) * e[j];
            u[i] += acc;
          }
        } else {
#pragma unroll
          for (int dir = 0; dir < D; ++dir) {
            const bool hi = (code >> dir) & 1u;
#pragma unroll
            for (int tl = 0; tl < NP / 2; ++tl) {
              const int i0 = dof<D, 2>(dir, 0, tl), i1 = dof<D, 2>(dir, 1, tl);
              const R e0 = e[i0], e1 = e[i1];
              e[i0] = (hi ? P1[0] : P0[0]) * e0 + (hi ? P1[1] : P0[1]) * e1;
              e[i1] = (hi ? P1[2] : P0[2]) * e0 + (hi ? P1[3] : P0[3]) * e1;
            }
          }
#pragma unroll
          for (int i = 0; i < NP; ++i) u[i] += e[i];
        }
        store(z, n, a, u);
      }
      __syncthreads();
    }
    // smoothing: forward sweeps down, reverse sweeps up; ssor: each step forward, then reverse
    const int sweeps = (down ? TP.pre : TP.post) << (TP.ssor ? 1 : 0);
    const R om = TP.omega[l];
    const unsigned binv = L.binv;
    for (int sw = 0; sw < sweeps; ++sw) {
      const bool fwd = TP.ssor ? (sw & 1) == 0 : down;
      for (int gi = 0; gi <= D; ++gi) {              // one colour group (its cells share no face)
        const TailLevelDesc::Group& G = L.grp[fwd ? gi : D - gi];
        const int end2 = G.end2;
        for (int idx = tid; idx < end2; idx += NT) {
          const int a = idx + (idx < G.end0 ? G.first0 : (idx < G.end1 ? G.first1 : G.first2));
          const uint4 q = rec[a];
          R t[NP], y[NP];
          load(f, n, a, t);
          const unsigned b = q.w & 0xffffu;
#pragma unroll
          for (int i = 0; i < NP; ++i) y[i] = R(0);
          if constexpr (D == 3) {
            const LevelParams<R>& LP = TP.P[l];
            couple3(q, z, n, bc, LP.k.w[0] * LP.k.w[0], y);
#pragma unroll
            for (int i = 0; i < NP; ++i) t[i] -= LP.hscale * y[i];
            block_solve_at<D, 2, R>(LP, b == 0xffffu ? nullptr : reinterpret_cast<const R*>(tcta_smem + binv + b * BLK), t, y);
          } else {
            couple(q, z, n, bc, t);
            block(b == 0xffffu ? M + 8 : reinterpret_cast<const R*>(tcta_smem + binv + b * BLK), t, R(1), y);
          }
          if (om != R(1)) {
            R uo[NP];
            load(z, n, a, uo);
#pragma unroll
            for (int i = 0; i < NP; ++i) y[i] = (R(1) - om) * uo[i] + om * y[i];
          }
          store(z, n, a, y);
        }
        __syncthreads();
      }
    }
    if (down) {
      // residual and restriction (Eq. 18): a warp takes 32 / 2^d coarse cells, lanes o * (32 / 2^d) + i child o
      // of coarse cell i, so that the lanes of one child read neighbouring cells
      const unsigned short* ch = reinterpret_cast<const unsigned short*>(tcta_smem + L.ch);
      const int nc = lev[l - 1].n_act, nl = nc * NCOL;
      R* rc = reinterpret_cast<R*>(tcta_smem + lev[l - 1].f);
      const unsigned aself = L.aself;
      for (int base = 0; base < nl; base += NT) {    // (the same passes for the whole block: exchanges)
        constexpr int CPW = 32 / NCOL;
        const int o = (tid & 31) / CPW, cc = (base + (tid & ~31)) / NCOL + (tid & (CPW - 1));
        const unsigned a = cc < nc ? ch[cc * NCOL + o] : 0xffffu;
        R r[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) r[i] = R(0);
        if (a != 0xffffu) {
          const uint4 q = rec[a];
          const unsigned b = q.w & 0xffffu;
          R u[NP];
          load(z, n, a, u);
          load(f, n, a, r);
          if constexpr (D == 3) {
            const LevelParams<R>& LP = TP.P[l];
            const unsigned w[3] = {q.x, q.y, q.z};
            int nb[2 * D];
#pragma unroll
            for (int s = 0; s < 2 * D; ++s) {
              const int m = (int)((s & 1) ? w[s >> 1] >> 16 : w[s >> 1] & 0xffffu);
              nb[s] = m == n ? -1 : m;
            }
            R y[NP], out[NP];
#pragma unroll
            for (int i = 0; i < NP; ++i) y[i] = 0;
            add_self<D, 2, R>(LP, nb, b == 0xffffu ? -1 : (int)b, u, y);
            couple3(q, z, n, bc, LP.k.w[0] * LP.k.w[0], y);
#pragma unroll
            for (int i = 0; i < NP; ++i) r[i] = r[i] - LP.hscale * y[i];
#pragma unroll
            for (int j = 0; j < NP; ++j) {
              R acc = 0;
#pragma unroll
              for (int i = 0; i < NP; ++i) acc += h_weight<D, R>(TP.T, o, i, j) * r[i];
              out[j] = acc;
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) r[j] = out[j];
          } else {
            if (aself) block(b == 0xffffu ? M + 8 + NP * NP : reinterpret_cast<const R*>(tcta_smem + aself + b * BLK), u, R(-1), r);
            else block(b == 0xffffu ? M + 8 + NP * NP : TP.aselfT[l] + b * (NP * NP), u, R(-1), r);
            couple(q, z, n, bc, r);
#pragma unroll
            for (int dir = 0; dir < D; ++dir) {
              const bool hi = (o >> dir) & 1;
#pragma unroll
              for (int tl = 0; tl < NP / 2; ++tl) {
                const int i0 = dof<D, 2>(dir, 0, tl), i1 = dof<D, 2>(dir, 1, tl);
                const R e0 = r[i0], e1 = r[i1];
                r[i0] = (hi ? P1[0] : P0[0]) * e0 + (hi ? P1[2] : P0[2]) * e1;
                r[i1] = (hi ? P1[1] : P0[1]) * e0 + (hi ? P1[3] : P0[3]) * e1;
              }
            }
          }
        }
        // the sum over the children: at each exchange a lane keeps half of the values
        int j = 0;
#pragma unroll
        for (int half = NP / 2, off = CPW; half >= 1; half >>= 1, off <<= 1) {
          const bool upper = (tid & off) != 0;
          if (upper) j += half;
#pragma unroll
          for (int i = 0; i < half; ++i) {
            const R send = upper ? r[i] : r[i + half], keep = upper ? r[i + half] : r[i];
            r[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        }
        if (cc < nc) rc[(j / PW * (nc + 1) + cc) * PW + j % PW] = r[0];
      }
      __syncthreads();
    }
  }
  const int n = lev[top].n_act;
  const unsigned z = lev[top].z;
  if (reinterpret_cast<uintptr_t>(z_top) % 16 == 0) {
    for (int q = tid; q < n * W; q += NT)
      reinterpret_cast<uint4*>(z_top)[q] =
          *reinterpret_cast<const uint4*>(tcta_smem + z + (unsigned)((q % W) * (n + 1) + q / W) * 16u);
  } else {
    for (int q = tid; q < n * NP; q += NT)
      z_top[q] = reinterpret_cast<const R*>(tcta_smem + z)[((q % NP) / PW * (n + 1) + q / NP) * PW + q % PW];
  }
}

inline unsigned cdiv(size_t a, size_t b) { return (unsigned)((a + b - 1) / b); }

// Grid of an interleaved launch (interleaved_warp) over all cells of a level: 2^dim blocks per
// chunk, as many chunks as the largest colour needs.
template <typename R>
unsigned interleaved_grid(const LevelParams<R>& P, int dim, unsigned bs) {
  const int ncol = 1 << dim;
  int longest = 0;
  for (int c = 0; c < ncol; ++c) longest = std::max(longest, P.colour_start[c + 1] - P.colour_start[c]);
  return (unsigned)ncol * cdiv((size_t)longest, bs);
}

}  // namespace

bool cell_kernels(int dim, int p) { return dim == 2 || (dim == 3 && p <= 2); }
bool cell_smoother(int dim, int p) { return dim == 2 || (dim == 3 && p == 1); }

// (p+1)^d <= 16: every thread-per-cell kernel; SBM_CELL_DISPATCH3 adds 3D p = 2 (FP32 operator).
#define SBM_CELL_DISPATCH(dim, p, MACRO)            \
  do {                                              \
    if (dim == 2 && p == 1) { MACRO(2, 2); }        \
    else if (dim == 2 && p == 2) { MACRO(2, 3); }   \
    else if (dim == 2 && p == 3) { MACRO(2, 4); }   \
    else if (dim == 3 && p == 1) { MACRO(3, 2); }   \
    else return cudaErrorInvalidValue;              \
  } while (0)
#define SBM_CELL_DISPATCH3(dim, p, MACRO)           \
  do {                                              \
    if (dim == 3 && p == 2) { MACRO(3, 3); }        \
    else SBM_CELL_DISPATCH(dim, p, MACRO);          \
  } while (0)

template <typename TI, typename R>
cudaError_t launch_apply_cell(int dim, int p, const LevelParams<R>& P, const TI* x, const R* f, R* y, int mode,
                              cudaStream_t s) {
  if (P.n_act == 0) return cudaSuccess;
#define SBM_AC(D, N1)                                                                           \
  {                                                                                             \
    const unsigned bs = cell_block(P.n_act), g = interleaved_grid(P, dim, bs);                 \
    if constexpr (std::is_same<R, dfl>::value && D == 2 && N1 == 3) {                           \
      if (mode == 0) SBM_PDL((k_apply_cell_occ<D, N1, TI, R, 0>), g, bs, 0, s, P, x, f, y);    \
      else SBM_PDL((k_apply_cell_occ<D, N1, TI, R, 1>), g, bs, 0, s, P, x, f, y);              \
    } else {                                                                                    \
      if (mode == 0) SBM_PDL((k_apply_cell<D, N1, TI, R, 0>), g, bs, 0, s, P, x, f, y);        \
      else SBM_PDL((k_apply_cell<D, N1, TI, R, 1>), g, bs, 0, s, P, x, f, y);                  \
    }                                                                                           \
  }
  if constexpr (std::is_same<TI, float>::value && std::is_same<R, float>::value) SBM_CELL_DISPATCH3(dim, p, SBM_AC);
  else SBM_CELL_DISPATCH(dim, p, SBM_AC);
#undef SBM_AC
  count_launches();
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_smooth_cell(int dim, int p, const LevelParams<R>& P, int reverse, int zero_start, const R* f,
                               R* u, cudaStream_t s, int early, int first_group) {
  if (reverse) zero_start = 0;
  int launched = 0;
  const int ng = n_colour_groups(P, dim);
  for (int q = first_group; q < ng; ++q) {   // (the launcher in level_ops.cu chose this path for the level)
    const int g = reverse ? ng - 1 - q : q;
    const int zm = group_zero_mode(P, zero_start, q);
    const unsigned bs = cell_block(group_cells(P, dim, g));
    const SmoothSegs G = smooth_segs(P, dim, g, (int)bs);
    if (G.n == 0 || G.blk[G.n] == 0) continue;
    const int fe = launched > 0 || early;            // after the sweep's first launch f is two back
#define SBM_SC(D, N1)                                                                                   \
  {                                                                                                     \
    constexpr bool kPre = CD<D, N1>::NP <= 9 && sizeof(R) == 4;                                         \
    if (kPre && bs == 32 && P.binvS) SBM_PDL((k_smooth_cell<D, N1, R, kPre>), G.blk[G.n], bs, 0, s, P, G, zm, f, u, fe); \
    else SBM_PDL((k_smooth_cell<D, N1, R, false>), G.blk[G.n], bs, 0, s, P, G, zm, f, u, fe);           \
  }
    SBM_CELL_DISPATCH(dim, p, SBM_SC);
#undef SBM_SC
    count_launches();
    ++launched;
  }
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_resid_restrict_p_cell(int dim, int pf, const LevelParams<R>& P, const TransferParams<R>& T,
                                        const R* u, const R* f, R* rc, cudaStream_t s, int early,
                                        const LevelParams<R>* Pc, R* zc) {
  if (P.n_act == 0) return cudaSuccess;
  const unsigned bs = cell_block(P.n_act), g = interleaved_grid(P, dim, bs);
  const bool sm0 = Pc != nullptr && zc != nullptr;
  const LevelParams<R>& Q = sm0 ? *Pc : P;           // unused without the fused first group
#define SBM_RRPC(D, N1, NC)                                                                                \
  {                                                                                                        \
    if (sm0) SBM_PDL((k_resid_restrict_p_cell<D, N1, NC, R, true>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc); \
    else SBM_PDL((k_resid_restrict_p_cell<D, N1, NC, R, false>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc);    \
  }
  if (dim == 2 && pf == 2) SBM_RRPC(2, 3, 2)
  else if (dim == 2 && pf == 3) SBM_RRPC(2, 4, 3)
  else if (dim == 3 && pf == 2) SBM_RRPC(3, 3, 2)
  else return cudaErrorInvalidValue;
#undef SBM_RRPC
  count_launches();
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_resid_restrict_h_cell(int dim, const LevelParams<R>& P, const TransferParams<R>& T, const R* u,
                                        const R* f, R* rc, cudaStream_t s, int early, const LevelParams<R>* Pc,
                                        R* zc) {
  if (T.n_act_c == 0) return cudaSuccess;
  const unsigned bs = cell_block((size_t)T.n_act_c << dim), g = cdiv((size_t)T.n_act_c << dim, bs);
  const bool sm0 = Pc != nullptr && zc != nullptr;
  const LevelParams<R>& Q = sm0 ? *Pc : P;
  constexpr bool kPre = sizeof(R) == 4;
  const bool pre = kPre && bs == 32 && (dim == 3 ? sm0 : P.aselfS != nullptr) && (!sm0 || Q.binvS);
#define SBM_RRHC(D)                                                                                               \
  {                                                                                                               \
    if (sm0 && pre) SBM_PDL((k_resid_restrict_h_cell<D, R, true, kPre>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc); \
    else if (sm0) SBM_PDL((k_resid_restrict_h_cell<D, R, true, false>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc);  \
    else if (pre) SBM_PDL((k_resid_restrict_h_cell<D, R, false, kPre && D == 2>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc); \
    else SBM_PDL((k_resid_restrict_h_cell<D, R, false, false>), g, bs, 0, s, P, T, u, f, rc, early, Q, zc);          \
  }
  if (dim == 2) SBM_RRHC(2)
  else if (dim == 3) SBM_RRHC(3)
  else return cudaErrorInvalidValue;
#undef SBM_RRHC
  count_launches();
  return cudaGetLastError();
}

size_t tail_smem_limit() {
  static size_t limit = 0;
  if (limit == 0) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    limit = optin > 1024 ? (size_t)optin - 1024 : 0;   // room for the kernels' static shared memory
  }
  return limit;
}

template <int D, typename R>
bool tail_fits_kernel(int size, size_t smem) {
  auto kern = k_vcycle_tail<D, R>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tail_smem_limit()) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(size);
  cfg.blockDim = dim3(kTailThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int nclusters = 0;
  const cudaError_t e = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg);
  if (e != cudaSuccess) cudaGetLastError();          // clear a refused query
  return e == cudaSuccess && nclusters >= 1;
}

bool tail_cluster_fits(int dim, int prec, int size, size_t smem) {
  if (smem > tail_smem_limit()) return false;
  if (dim == 2) return prec == 0 ? tail_fits_kernel<2, double>(size, smem) : tail_fits_kernel<2, float>(size, smem);
  return prec == 0 ? tail_fits_kernel<3, double>(size, smem) : tail_fits_kernel<3, float>(size, smem);
}

template <typename R>
cudaError_t launch_vcycle_tail(int dim, const TailLevel<R>* TL, int top, const R* r, R* z, const double* coarse_inv,
                               int pre, int post, int ssor, const TailPlan& plan, cudaStream_t s) {
  if (plan.cluster < 1) return cudaErrorNotSupported;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.cluster);
  cfg.blockDim = dim3(kTailThreads);
  cfg.dynamicSmemBytes = plan.smem_bytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e;
  if (dim == 2) e = cudaLaunchKernelEx(&cfg, k_vcycle_tail<2, R>, TL, top, r, z, coarse_inv, pre, post, ssor, plan.gather_off);
  else e = cudaLaunchKernelEx(&cfg, k_vcycle_tail<3, R>, TL, top, r, z, coarse_inv, pre, post, ssor, plan.gather_off);
  count_launches();
  return e;
}

template <typename K>
bool tail_cta_fits_kernel(K kern, size_t smem) {
  cudaFuncAttributes fa{};
  int dev = 0, optin = 0;
  if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const size_t room = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
  if (smem > room) return false;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

bool tail_cta_fits(int dim, int prec, size_t smem) {
  if (dim == 2) return prec == 0 ? tail_cta_fits_kernel(k_vcycle_tail_cta<2, double>, smem)
                                 : tail_cta_fits_kernel(k_vcycle_tail_cta<2, float>, smem);
  return prec == 0 ? tail_cta_fits_kernel(k_vcycle_tail_cta<3, double>, smem)
                   : tail_cta_fits_kernel(k_vcycle_tail_cta<3, float>, smem);
}

int tail_fault_take() {
  int f = 0;
  if (cudaMemcpyFromSymbol(&f, g_tail_fault, sizeof(int)) != cudaSuccess) return -1;
  if (f) {
    const int zero = 0;
    if (cudaMemcpyToSymbol(g_tail_fault, &zero, sizeof(int)) != cudaSuccess) return -1;
  }
  return f;
}

template <typename R>
cudaError_t launch_vcycle_tail_cta(int dim, const TailCta<R>& TP, const R* r, R* z, const double* coarse_inv,
                                   size_t smem, cudaStream_t s) {
  if (dim == 2)
    SBM_PDL((k_vcycle_tail_cta<2, R>), 1, kTailCtaThreads, smem, s, TP, r, z, coarse_inv);
  else
    SBM_PDL((k_vcycle_tail_cta<3, R>), 1, kTailCtaThreads, smem, s, TP, r, z, coarse_inv);
  count_launches();
  return cudaGetLastError();
}
template cudaError_t launch_vcycle_tail_cta<double>(int, const TailCta<double>&, const double*, double*,
                                                    const double*, size_t, cudaStream_t);
template cudaError_t launch_vcycle_tail_cta<float>(int, const TailCta<float>&, const float*, float*, const double*,
                                                   size_t, cudaStream_t);

template cudaError_t launch_vcycle_tail<double>(int, const TailLevel<double>*, int, const double*, double*,
                                                const double*, int, int, int, const TailPlan&, cudaStream_t);
template cudaError_t launch_vcycle_tail<float>(int, const TailLevel<float>*, int, const float*, float*, const double*,
                                               int, int, int, const TailPlan&, cudaStream_t);
template cudaError_t launch_apply_cell<double, double>(int, int, const LevelParams<double>&, const double*,
                                                       const double*, double*, int, cudaStream_t);
template cudaError_t launch_apply_cell<float, float>(int, int, const LevelParams<float>&, const float*, const float*,
                                                     float*, int, cudaStream_t);
template cudaError_t launch_apply_cell<float, double>(int, int, const LevelParams<double>&, const float*,
                                                      const double*, double*, int, cudaStream_t);
template cudaError_t launch_apply_cell<float, dfl>(int, int, const LevelParams<dfl>&, const float*, const dfl*,
                                                   dfl*, int, cudaStream_t);
template cudaError_t launch_smooth_cell<double>(int, int, const LevelParams<double>&, int, int, const double*,
                                                double*, cudaStream_t, int, int);
template cudaError_t launch_smooth_cell<float>(int, int, const LevelParams<float>&, int, int, const float*, float*,
                                               cudaStream_t, int, int);
template cudaError_t launch_resid_restrict_p_cell<double>(int, int, const LevelParams<double>&,
                                                          const TransferParams<double>&, const double*, const double*,
                                                          double*, cudaStream_t, int, const LevelParams<double>*,
                                                          double*);
template cudaError_t launch_resid_restrict_p_cell<float>(int, int, const LevelParams<float>&,
                                                         const TransferParams<float>&, const float*, const float*,
                                                         float*, cudaStream_t, int, const LevelParams<float>*, float*);
template cudaError_t launch_resid_restrict_h_cell<double>(int, const LevelParams<double>&,
                                                          const TransferParams<double>&, const double*, const double*,
                                                          double*, cudaStream_t, int, const LevelParams<double>*,
                                                          double*);
template cudaError_t launch_resid_restrict_h_cell<float>(int, const LevelParams<float>&, const TransferParams<float>&,
                                                         const float*, const float*, float*, cudaStream_t, int,
                                                         const LevelParams<float>*, float*);

}  // namespace sbm
