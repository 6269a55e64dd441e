// Diagnostics of a selected block: the local next-candidate distributions of Eq.
// "localar", the decision gaps of Eq. "margin" along a path, and coverage / oracle prefix
// / prefix acceptance against ground-truth tokens (Sec. 3.3 "Oracle-prefix supervision";
// Sec. 3.1 prefix acceptance).
//
// Every kernel here is latency bound (a few MB at most), so each row, step and slot gets its
// own lanes instead of a place in a loop:
// local_softmax_kernel: a power-of-two group of lanes per score row (the anchor row of a
//   sequence, or the row of one predecessor at one slot pair); lane k holds sigma * score[k],
//   group max and sum.
// path_probs_kernel: a CTA per sequence, a warp per step: the path is given, so every step knows
//   its predecessor; the same softmax over the row of the predecessor, the chosen candidate's
//   probability and its gap to the best other candidate; the logarithms are summed in step order
//   at the end. 200 sequences of 15 steps: 19 us (a warp walking the steps) -> 5.9 us cold. Many
//   sequences of few steps are a warp's each.
// acceptance_kernel: a warp per sequence (four lanes where many are short), a lane per slot; runs
//   end at the first zero of the group's ballot. 14 us (a thread per sequence) -> 3.9 us cold.
#include "internal.cuh"

namespace lilicorr {

namespace {

constexpr int DG_THREADS = 256;

// softmax over the K values z of a group of G lanes (G a power of two, lanes >= K hold -inf):
// this lane's probability and the row maximum
template <int G>
__device__ __forceinline__ float group_softmax(float z, int lane, int K, float& zmax) {
  float m = lane < K ? z : -INFINITY;
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const float e = lane < K ? expf(z - m) : 0.f;
  float sum = e;
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  zmax = m;
  return e / sum;
}

template <int G>
__global__ void __launch_bounds__(DG_THREADS)
local_softmax_kernel(int B, int L, int K, const float* __restrict__ A, const float* __restrict__ P,
                     float sigma, float* __restrict__ pa, float* __restrict__ pp) {
  pdl_wait();
  const int rows_per_seq = 1 + (L - 1) * K;
  const long long row = (long long)blockIdx.x * (DG_THREADS / G) + threadIdx.x / G;
  const int lane = threadIdx.x % G;
  // every lane takes part in the shuffles, but a whole warp may leave: the rows of 32 lanes then
  // need no guards (1024 sequences of 8 slots x 32, 33.6 -> 30.6 us)
  const bool live = row < (long long)B * rows_per_seq;
  if (G == 32 && !live) return;
  const int b = live ? (int)(row / rows_per_seq) : 0, r = live ? (int)(row % rows_per_seq) : 0;
  const size_t o = ((size_t)b * (L - 1) * K + (r - 1)) * K;
  const float* src = r == 0 ? A + (size_t)b * K : P + o;
  const float z = live && lane < K ? sigma * src[lane] : -INFINITY;
  float m;
  const float p = group_softmax<G>(z, lane, K, m);
  if (live && lane < K) (r == 0 ? pa + (size_t)b * K : pp + o)[lane] = p;
}

// W (1 or 8) warps per sequence
template <int W>
__global__ void __launch_bounds__(DG_THREADS)
path_probs_kernel(int B, int L, int K, const float* __restrict__ A,
                  const float* __restrict__ P, const int32_t* __restrict__ choice, float sigma,
                  float* __restrict__ prob, float* __restrict__ gap, float* __restrict__ log_prob) {
  pdl_wait();
  static_assert(W == 1 || W == DG_THREADS / 32, "a warp or a CTA per sequence");
  __shared__ float s_log[LILICORR_MAX_L];          // (W = 1 sums as it goes)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = W == 1 ? blockIdx.x * (DG_THREADS / 32) + warp : blockIdx.x;
  if (b >= B) return;
  float lp = 0.f;
  int prev = 0;
  for (int s = W == 1 ? 0 : warp; s < L; s += W) {
    const int c = choice[(size_t)b * L + s];
    if (W > 1) prev = s > 0 ? choice[(size_t)b * L + s - 1] : 0;
    const bool valid = c >= 0 && c < K && prev >= 0 && prev < K;
    const float* row = s == 0 ? A + (size_t)b * K
                              : P + (((size_t)b * (L - 1) + (s - 1)) * K + (valid ? prev : 0)) * K;
    const float z = lane < K ? sigma * row[lane] : -INFINITY;
    float m;
    const float p = group_softmax<32>(z, lane, K, m);
    const float pc = __shfl_sync(0xffffffffu, p, valid ? c : 0);
    const float zc = __shfl_sync(0xffffffffu, z, valid ? c : 0);
    const float other = warp_max((lane < K && lane != c) ? z : -INFINITY);
    if (lane == 0) {
      const size_t o = (size_t)b * L + s;
      const float ps = valid ? pc : NAN;               // a choice outside [0, K) has no probability
      if (prob) prob[o] = ps;
      if (gap) gap[o] = valid ? (K > 1 ? zc - other : INFINITY) : NAN;
      if (W == 1) lp += logf(ps);
      else s_log[s] = logf(ps);
    }
    prev = c;
  }
  if (!log_prob) return;
  if (W > 1) {
    __syncthreads();
    if (threadIdx.x == 0)
      for (int s = 0; s < L; ++s) lp += s_log[s];
  }
  if (W == 1 ? lane == 0 : threadIdx.x == 0) log_prob[b] = lp;
}

// length of the run of ones that starts at the first lane of this lane's group of G
template <int G>
__device__ __forceinline__ int run_length(bool one) {
  const uint32_t zeros = ~__ballot_sync(0xffffffffu, one) >> (threadIdx.x & 31 & ~(G - 1));
  return min(zeros ? __ffs(zeros) - 1 : 32, G);
}

// G (4 or 32) lanes per sequence, which take its slots G at a time
template <int G>
__global__ void __launch_bounds__(DG_THREADS)
acceptance_kernel(int B, int L, int K, const int32_t* __restrict__ ids,
                  const int32_t* __restrict__ tokens, const int32_t* __restrict__ truth,
                  int32_t* __restrict__ covered, int32_t* __restrict__ oracle_prefix,
                  int32_t* __restrict__ accepted) {
  pdl_wait();
  const int b = blockIdx.x * (DG_THREADS / G) + threadIdx.x / G;
  const int lane = threadIdx.x & (G - 1);
  int prefix = 0, acc = 0;
  for (int s0 = 0; s0 < L; s0 += G) {              // (the same rounds in every lane of a warp)
    const int s = s0 + lane;
    bool cov = false, same = false;
    if (b < B && s < L) {
      const size_t o = (size_t)b * L + s;
      const int32_t g = truth[o];
#pragma unroll 8
      for (int k = 0; k < K; ++k) cov |= ids[o * K + k] == g;
      same = tokens[o] == g;
      if (covered) covered[o] = cov ? 1 : 0;
    }
    // a run goes on into the next slots only if it filled the ones before
    const int more = run_length<G>(cov), more_acc = run_length<G>(same);
    if (prefix == s0) prefix += more;
    if (acc == s0) acc += more_acc;
  }
  if (lane != 0 || b >= B) return;
  if (oracle_prefix) oracle_prefix[b] = prefix;
  if (accepted) accepted[b] = acc;
}

bool shape_ok(int B, int L, int K) {
  return B >= 0 && L > 0 && L <= LILICORR_MAX_L && K > 0 && K <= LILICORR_MAX_K;
}

}  // namespace

}  // namespace lilicorr

using namespace lilicorr;

extern "C" lilicorr_status_t lilicorr_local_softmax(int B, int L, int K, const float* anchor_scores,
                                                    const float* pair_scores, float sigma,
                                                    float* anchor_probs, float* pair_probs,
                                                    cudaStream_t stream) {
  if (!shape_ok(B, L, K)) return LILICORR_ERR_SHAPE;
  if (!(sigma > 0.f) || !isfinite(sigma)) return LILICORR_ERR_ARG;
  if (B == 0) return LILICORR_OK;
  if (!anchor_scores || !anchor_probs || (L > 1 && (!pair_scores || !pair_probs)))
    return LILICORR_ERR_ARG;
  const long long rows = (long long)B * (1 + (L - 1) * K);
  // the fewest lanes that hold a row
  const int group = K <= 8 ? 8 : K <= 16 ? 16 : 32;
  const int grid = ceil_div(rows, DG_THREADS / group);
  auto* kernel = K <= 8 ? local_softmax_kernel<8> : K <= 16 ? local_softmax_kernel<16>
                                                            : local_softmax_kernel<32>;
  return launch_k(kernel, grid, DG_THREADS, 0, stream, B, L, K, anchor_scores, pair_scores, sigma,
                  anchor_probs, pair_probs);
}

extern "C" lilicorr_status_t lilicorr_path_probs(int B, int L, int K, const float* anchor_scores,
                                                 const float* pair_scores, const int32_t* choice,
                                                 float sigma, float* prob, float* gap,
                                                 float* log_prob, cudaStream_t stream) {
  if (!shape_ok(B, L, K)) return LILICORR_ERR_SHAPE;
  if (!(sigma > 0.f) || !isfinite(sigma)) return LILICORR_ERR_ARG;
  if (B == 0) return LILICORR_OK;
  if (!anchor_scores || (L > 1 && !pair_scores) || !choice) return LILICORR_ERR_ARG;
  // a CTA per sequence, or a warp each where sequences are many for their steps (K = 8, us, CTA /
  // warp: 2048 of 1 slot 4.3 / 2.6, of 4 4.3 / 4.6, of 16 9.2 / 13.9; 4096 of 4 7.2 / 5.4, of 8
  // 9.4 / 8.9; 16,384 of 1 20.8 / 5.1, of 16 55 / 49, of 64 192 / 183)
  const bool warps = L == 1 || (B >= 8 * num_sms() && B >= 3LL * num_sms() * L);
  return launch_k(warps ? path_probs_kernel<1> : path_probs_kernel<DG_THREADS / 32>,
                  warps ? ceil_div(B, DG_THREADS / 32) : B, DG_THREADS, 0, stream, B, L, K,
                  anchor_scores, pair_scores, choice, sigma, prob, gap, log_prob);
}

extern "C" lilicorr_status_t lilicorr_block_acceptance(int B, int L, int K, const int32_t* ids,
                                                       const int32_t* tokens, const int32_t* truth,
                                                       int32_t* covered, int32_t* oracle_prefix,
                                                       int32_t* accepted, cudaStream_t stream) {
  if (!shape_ok(B, L, K)) return LILICORR_ERR_SHAPE;
  if (B == 0) return LILICORR_OK;
  if (!ids || !tokens || !truth) return LILICORR_ERR_ARG;
  // a warp per sequence, but four lanes where many short ones would leave most of its lanes idle
  // (us, warp / four lanes: 16,384 of one slot x 4 3.8 / 2.0, of 8 x 8 4.1 / 3.0, of 16 x 2 3.7 /
  // 3.4; 4096 of 8 x 32 5.8 / 9.7)
  const bool few = L <= 8 && B >= 32 * num_sms();
  return launch_k(few ? acceptance_kernel<4> : acceptance_kernel<32>,
                  ceil_div((long long)B * (few ? 4 : 32), DG_THREADS), DG_THREADS, 0, stream, B, L, K,
                  ids, tokens, truth, covered, oracle_prefix, accepted);
}
