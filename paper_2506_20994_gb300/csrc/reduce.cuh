// Deterministic block reductions and the fixed launch shape of the solver's
// vector kernels.
//
// Every reduction runs in two passes with a fixed grid: pass one writes one
// partial per block (grid-stride loop in a fixed order, a fixed warp-shuffle
// tree inside the block), pass two sums the partials in index order in one
// block.  The result is therefore bitwise reproducible run to run, which the
// solvers' checkpoint/resume relies on.
#pragma once

#include "common.cuh"

namespace ax {

constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 152 * 4;  // 4 blocks per SM of the 152-SM part

// Sum of v over the block (kRedThreads threads); valid in thread 0.
// Deterministic order: lane l of quantity q's warp adds threads l, l + 32, ...
// in order, then a fixed shuffle tree.  Through shared memory, because the
// fp64 pipe takes about 19 cycles an SM for each warp-wide addition whatever
// lanes are active: 13 of them a block and quantity, where a shuffle tree in
// each of the eight warps and a serial sum need 48 (at 608 blocks 3 us of the
// update kernel's time per quantity).
template <int NV>
AX_D void block_sum(double (&v)[NV]) {
  __shared__ double buf[NV][kRedThreads];
  __shared__ double tot[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) buf[q][threadIdx.x] = v[q];
  __syncthreads();
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < NV) {
    double s = buf[q][lane];
#pragma unroll
    for (int k = 1; k < kRedThreads / 32; ++k) s += buf[q][lane + 32 * k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) tot[q] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = tot[k];
  }
}

// Sums partials[q * nblk + b] over b for q < NV: one warp per quantity,
// lane l adding b = l, l+32, ... in order, then a fixed shuffle tree.
template <int NV>
AX_D void warp_sum_partials(const double *__restrict__ partials, int nblk, double *out) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= NV) return;
  double s = 0.0;
  for (int b = lane; b < nblk; b += 32) s += partials[(size_t)q * nblk + b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) out[q] = s;
}

// The second pass inside the first one's kernel: every block stores its NV
// sums (v, valid in thread 0) as partials[q * gridDim.x + blockIdx.x]; the
// block that arrives last adds them in index order (one warp per quantity, as
// warp_sum_partials) and its thread 0 calls f(sums).  `ticket` is zero before
// the launch and left zero.  A launch of its own for one block costs a kernel
// boundary and 2 us, in the loops of the solvers once or twice an iteration.
template <int NV, class F>
AX_D void finish_sums(double (&v)[NV], double *partials, unsigned *ticket, F f) {
  __shared__ double t[NV];
  __shared__ bool last;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < NV; ++q) partials[(size_t)q * gridDim.x + blockIdx.x] = v[q];
    __threadfence();  // the partials before the ticket
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;  // block-uniform
  __threadfence();  // the ticket before the other blocks' partials
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < NV) {
    double s = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(partials + (size_t)q * gridDim.x + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) t[q] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    *ticket = 0u;
    f(t);
  }
}

}  // namespace ax
