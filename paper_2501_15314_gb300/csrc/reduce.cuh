// Reductions of several values at once over the threads of a block, in a fixed
// order (bitwise reproducible).
//
// The Gram-Schmidt kernels reduce up to kMaxRestart + 1 sums per thread.  A
// butterfly over the warp for each of them takes 5 additions and shuffles per
// value; in FP64 (64 cycles of latency, 16 cycles of an SM's pipe per warp) that
// was 30 us per launch for 12 values and 8 blocks per SM, whatever the
// vectors' length.  Here the first steps of the butterfly halve the number of
// values: a lane keeps one half and sends the other, so N values take N - 1
// additions and shuffles (N a power of two) and leave one total per lane.
// Measured on GB300: FP64 dots with 12 vectors at 32^3 42 -> 7 us, FP32 ones with
// 8 vectors at 128^3 25 -> 16 us; with fewer, fuller blocks (red_blocks) the FP64
// step at 32^3 2.12 -> 1.71 ms.
#pragma once

#include <cstdint>

#include "ibm_internal.cuh"

namespace ibm {

// Blocks of kRedThreads threads for a reduction over n items (values, or groups
// of four): whole rounds of one block per SM with about eight items per thread,
// at most kRedBlocks (the partial sums' place); where that is less than one
// round, two items per thread.
inline int red_blocks(int64_t n) {
  const int64_t round = 152 * kRedThreads;
  const int64_t rounds = (n + 8 * round - 1) / (8 * round);
  const int64_t few = (n + 2 * kRedThreads - 1) / (2 * kRedThreads);
  const int64_t b = few < 152 ? few : 152 * rounds;
  return (int)(b < 1 ? 1 : (b < kRedBlocks ? b : kRedBlocks));
}

__host__ __device__ constexpr int pow2_ceil(int n) {
  int p = 1;
  while (p < n) p *= 2;
  return p;
}

// Totals of acc[0..NQ) over the warp, NQ <= 32: lane L returns that of value
// L / (32 / P), P the power of two from NQ up (0 where there is none).
template <int NQ, typename T, typename Add, typename Xor>
__device__ __forceinline__ T warp_totals(T (&acc)[NQ], Add add, Xor shfl_xor) {
  constexpr int P = pow2_ceil(NQ);
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int h = P / 2; h >= 1; h >>= 1, o >>= 1) {
    const int n = h == P / 2 ? NQ : 2 * h;   // values left
    const bool up = lane & o;
#pragma unroll
    for (int q = 0; q < h; ++q) {
      const T lo = acc[q], hi = q + h < n ? acc[q + h < NQ ? q + h : 0] : T{};
      acc[q] = add(up ? hi : lo, shfl_xor(up ? lo : hi, o));
    }
  }
  T v = acc[0];
#pragma unroll
  for (int k = 16 / P; k > 0; k >>= 1) v = add(v, shfl_xor(v, k));
  return v;
}

// Sums over the block of acc[0..nq), nq <= NQ, written as FP64 to out[q] (one
// thread per value adds the warps' totals in order).
template <int NQ, int WARPS, typename T, typename Add, typename Xor, typename Wide>
__device__ __forceinline__ void block_totals(T (&acc)[NQ], int nq, double* out, Add add,
                                             Xor shfl_xor, Wide wide) {
  constexpr int C = NQ < 32 ? NQ : 32;   // values per pass
  __shared__ T sh[WARPS][NQ];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int b = 0; b < NQ; b += C) {
    T part[C];
#pragma unroll
    for (int q = 0; q < C; ++q) part[q] = b + q < NQ ? acc[b + q < NQ ? b + q : 0] : T{};
    const T v = warp_totals<C>(part, add, shfl_xor);
    constexpr int per = 32 / pow2_ceil(C);
    if (lane % per == 0 && lane / per < C && b + lane / per < NQ) sh[wid][b + lane / per] = v;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nq; q += WARPS * 32) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) s += wide(sh[w][q]);
    out[q] = s;
  }
}

}  // namespace ibm
