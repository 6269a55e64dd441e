// The greedy walk of step (4) over one sequence's scores, shared by the pair kernel and
// the cluster network kernel's fused tail (Sec. 3.5: c_s = argmax_k phi(s-1, c_{s-1}, k),
// left to right, ties to the lower index).
//
// A walk that looks for each step's best candidate as it comes to it waits for a row of scores
// and a butterfly over the candidates' lanes 16 times in a row. Which candidate is best after a
// given predecessor does not depend on the walk, so the CTA finds it for every row of scores
// first, a thread per row, and the walk then only follows the table. Selection of one request 95.2
// -> 91.6 us, of 32 133.2 -> 128.7 (with the cluster kernel's records summed four at a time), of 64
// at 16 candidates 317.7 -> 313.6.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace lilicorr {
namespace walk {

// best[row] = the best candidate of a row of scores, ties to the lower index; a NaN never wins
// over an earlier candidate, so the result is always a candidate. Row 0 is the anchor's (A [K]),
// row 1 + s*K + k that of predecessor k at slot pair s (P [(L-1)][K][K]); A and P in any memory,
// best [1 + (L-1)*K] in shared memory. Called by `threads` threads numbered `tid`, which
// meet at a barrier of the caller's before the table is read. Rows of 16 or 32 scores in shared
// memory share banks 16 or 32 at a time, so there the threads of a warp start at different
// candidates (walks of 2048 sequences of 8 slots x 32: 58 us from candidate 0 in every row, 17 so;
// of 8 x 8, where they share eight at a time, 6.0 from candidate 0 and 7.9 so).
__device__ __forceinline__ void best_of_rows(const float* A, const float* P, int L, int K,
                                             uint8_t* best, int tid, int threads) {
  const bool turned = (K & 15) == 0;
  for (int row = tid; row < 1 + (L - 1) * K; row += threads) {
    const float* r = row == 0 ? A : P + (size_t)(row - 1) * K;
    float v = r[0];
    int c = 0;
    if (turned && v == v) {                      // (a NaN in front stays the choice)
      const int k0 = row * K / 32;
      v = -INFINITY;
      c = K;
#pragma unroll 4
      for (int j = 0; j < K; ++j) {
        const int k = (k0 + j) & (K - 1);
        const float x = r[k];
        if (x > v || (x == v && k < c)) { v = x; c = k; }
      }
    } else {
#pragma unroll 4
      for (int k = 1; k < K; ++k) {
        const float x = r[k];
        if (x > v) { v = x; c = k; }
      }
    }
    best[row] = (uint8_t)c;
  }
}

// The walk without a table, by one full warp: a butterfly over the candidates' lanes per step, the
// same choices. Bounded by the chain of L steps, where the table is by its 1 + (L-1)*K rows.
__device__ __forceinline__ void walk_steps(const float* A, const float* P, int L, int K,
                                           uint8_t* path) {
  const int lane = threadIdx.x & 31;
  int width = 1;                                 // lanes that hold candidates, rounded up
  while (width < K) width <<= 1;
  int c = 0;
  for (int s = 0; s < L; ++s) {
    const float* r = s == 0 ? A : P + ((size_t)(s - 1) * K + c) * K;
    float v = lane < K ? r[lane] : -INFINITY;
    const bool front_nan = __shfl_sync(0xffffffffu, v != v, 0);
    c = v == v && lane < K ? lane : 32;          // a NaN never wins
    if (v != v) v = -INFINITY;
    for (int o = width >> 1; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, v, o);
      const int oc = __shfl_xor_sync(0xffffffffu, c, o);
      if (ov > v || (ov == v && oc < c)) { v = ov; c = oc; }
    }
    c = front_nan ? 0 : __shfl_sync(0xffffffffu, c, 0);    // but in front it stays the choice
    if (lane == 0) path[s] = (uint8_t)c;
  }
}

// The walk along the table, by one full warp: the choices go to path[L] in shared memory.
__device__ __forceinline__ void follow(const uint8_t* best, int L, int K, uint8_t* path) {
  int c = best[0];
  if ((threadIdx.x & 31) == 0) path[0] = (uint8_t)c;
  for (int s = 1; s < L; ++s) {
    c = best[1 + (s - 1) * K + c];
    if ((threadIdx.x & 31) == 0) path[s] = (uint8_t)c;
  }
  __syncwarp();
}

}  // namespace walk
}  // namespace lilicorr
