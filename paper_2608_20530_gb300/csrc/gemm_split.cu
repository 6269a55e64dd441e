// Tensor-core linear layer for few output tiles: C[M, N] = epilogue(A W^T), bf16 A and W, with
// Kd split over a thread-block cluster.
//
// A head of width 1024 with one request multiplies 120 node rows by [1024 .. 3072, 1024 .. 2048]
// weights: 16 to 48 tiles of 128 x 64, so a kernel with one CTA per tile leaves two thirds of
// the SMs idle while the others stream Kd / 64 chunks one after the other. Here S = 1, 2, 4 or 8
// CTAs, one cluster, share a tile: each multiplies its part of Kd into its own tensor memory,
// parks the 128 x BN partial sums in its shared memory, and after a cluster barrier every CTA
// adds up the S partials of the rows r, r + S, r + 2S, ... (distributed shared memory, in rank
// order, so the result is the same on every call) and runs the epilogue on them.
// gemm_split_ways says how S follows from the sizes.
//
// Roles: warp 0 (one lane) streams 128 x 64 tiles of A and BN x 64 tiles of W by TMA (128-byte
// swizzle, four stages), warp 1 issues tcgen05.mma (M = 128, N = BN), warps 4-7 drain the
// accumulator, all eight warps reduce. The weights are constant while a head lives, so their
// first four chunks are requested before the wait on the preceding launch: only A's copy,
// the products and the reduction are left on the chain. What bounds it is that latency, not a
// pipe: with these products, the RMSNorms folded into them and the target chain beside the
// body, the network of width 1024 went from 170 to 115 us for one request and from 352 to 309
// for 24 (its prologue's 15- and 24-row products; 103 and 280 with what followed); serving_b32's
// drafter-state product (512 rows, 16 tiles, Kd = 4096) beside the top-K pass 136.7 -> 131.7 us a
// call. The same epilogues as the persistent kernel (gemm_tc.cu): bias, per-sequence bias, SiLU,
// residual, and the RMSNorm folded into the products around it. Every mbarrier wait is bounded;
// on timeout the kernel records LILICORR_ERR_TIMEOUT, keeps every thread on its barriers, lets
// copies in flight land, frees its tensor memory and returns.
#include "tc_ptx.cuh"

namespace lilicorr {

namespace {
using namespace tc;

constexpr int SP_THREADS = 256;
constexpr int SP_STAGES = 4;
constexpr int SP_BK = 64;
constexpr int SP_FEW = 64;               // rows up to which sums leave the tensor core early
constexpr uint32_t SP_A_BYTES = 128 * SP_BK * 2;
constexpr long long SP_WAIT = 4000000000ll;   // SM cycles, where the arguments give no limit
constexpr float SP_RMS_EPS = 1e-6f;

struct SplitArgs {
  GemmArgs g;
  int S;             // CTAs per tile (cluster size)
  int w_const;       // W is constant: its copies may start before the preceding launch ends
};

template <int BN, bool FEW>
struct SpCfg {
  // two CTAs fit an SM by shared memory: their columns must too, or clusters could hold one
  // another up at the allocation
  static constexpr uint32_t TMEM_COLS = FEW ? 4 * BN : BN;
  static_assert(2 * TMEM_COLS <= 512, "two CTAs an SM");
  static constexpr uint32_t B_BYTES = BN * SP_BK * 2;
  static constexpr size_t RING = (size_t)SP_STAGES * (SP_A_BYTES + B_BYTES);
  static constexpr int PLD = BN + 4;                       // row stride of the partial sums
  static_assert((size_t)128 * PLD * 4 <= RING, "partials alias the ring");
  static constexpr size_t SMEM = 1024 + RING;
};

// v += x, and e += what that rounded off (Knuth's two-sum).
__device__ __forceinline__ void two_sum(float& v, float& e, float x) {
  const float s = __fadd_rn(v, x), b = __fsub_rn(s, v);
  e = __fadd_rn(e, __fadd_rn(__fsub_rn(v, __fsub_rn(s, b)), __fsub_rn(x, b)));
  v = s;
}

// FEW (M <= 64): the sums of a product of few rows are held to what the few-row CUDA-core kernel,
// which had these sizes, gives. The tensor core truncates each time it adds 16 products to an
// accumulator, always towards zero, so a chain of n adds is about n * 1.2e-8 of the result
// short (measured: 2.4e-8 after two, 9.5e-8 after eight, 4.0e-7 after 32). Here an accumulator takes
// two adds, two accumulators a 64-wide chunk, two chunks in flight, and a thread per row adds
// them up in fp32 registers. Relative error against 64 bits, few-row kernel / one chain / this, at
// Kd = 512, 1024, 2048 and 4096:
// 6.2e-8 / 1.2e-7 / 6.1e-8, 6.9e-8 / 2.3e-7 / 6.8e-8, 7.9e-8 / 4.7e-7 / 7.8e-8, 8.4e-8 / 4.7e-7 / 7.8e-8
// (the ranks' parts are added with their rounding errors carried). It costs a product 0.4 to 2.3 us
// (64 x 1024 x 1024: 4.5 -> 5.1 us, the few-row kernel 25.7; 16 x 1024 x 4096: 5.5 -> 7.7, 11.9), a
// whole network of up to 64 nodes about a tenth (width 512, 48 nodes: 70 -> 77 us; 230 with the
// few-row kernel).
template <int BN, bool FEW>
__global__ void __launch_bounds__(SP_THREADS, FEW ? 2 : 1)
    gemm_split_kernel(const __grid_constant__ CUtensorMap mapA,
                      const __grid_constant__ CUtensorMap mapW, const SplitArgs sa) {
  using Cfg = SpCfg<BN, FEW>;
  constexpr int PLD = Cfg::PLD;
  const GemmArgs& g = sa.g;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + SP_STAGES * SP_A_BYTES;
  float* part = reinterpret_cast<float*>(smem);            // once the products are done
  constexpr int NACC = FEW ? 2 : 1;
  __shared__ __align__(8) uint64_t full[SP_STAGES], empty[SP_STAGES], acc_full[NACC], acc_empty[NACC];
  __shared__ uint32_t tmem_base;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = sa.S, rank = blockIdx.x;                   // gridDim.x = cluster size = S
  const int n0 = blockIdx.y * BN, m0 = blockIdx.z * 128;
  const int nk = (g.Kd + SP_BK - 1) / SP_BK;
  const long long wait = g.wait_limit > 0 ? g.wait_limit : SP_WAIT;
  const int kc0 = nk * rank / S, kcn = nk * (rank + 1) / S - kc0;   // this CTA's chunks (>= 1)

  if (threadIdx.x == 0) {
    for (int s = 0; s < SP_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NACC; ++b) {
      mbar_init(&acc_full[b], 1);
      if (FEW) mbar_init(&acc_empty[b], (g.M + 31) / 32);      // the warps that drain
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&tmem_base, Cfg::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  const int pre = min(kcn, SP_STAGES);
  auto load_w = [&](int i) {
    const int s = i % SP_STAGES;
    mbar_expect_tx(&full[s], SP_A_BYTES + Cfg::B_BYTES);
    tma_load_2d(sB + (size_t)s * Cfg::B_BYTES, &mapW, &full[s], (kc0 + i) * SP_BK, n0);
  };
  auto load_a = [&](int i) {
    const int s = i % SP_STAGES;
    tma_load_2d(sA + (size_t)s * SP_A_BYTES, &mapA, &full[s], (kc0 + i) * SP_BK, m0);
  };
  // (a test's starved producer issues no copies: 1 in every CTA, 2 in the cluster's first)
  const bool starved = g.test_starve == 1 || (g.test_starve == 2 && rank == 0);
  const bool producer = warp == 0 && lane == 0 && !starved;
  if (producer) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&mapA)) : "memory");
    if (sa.w_const)
      for (int i = 0; i < pre; ++i) load_w(i);
  }
  // this thread's columns in the reduction, and what it adds to them
  constexpr int TPR = BN / 4;                       // threads per row
  const int c = (threadIdx.x % TPR) * 4, n = n0 + c;
  const int rows = min(128, g.M - m0);
  const bool col_ok = n < g.N;                      // N is a multiple of 8
  float4 bias = make_float4(0.f, 0.f, 0.f, 0.f), gain = bias;
  auto load_vectors = [&] {
    if (g.bias && col_ok)
      bias = make_float4(g.bias[n], g.bias[n + 1], g.bias[n + 2], g.bias[n + 3]);
    if (g.c2 && col_ok)
      gain = make_float4(g.c2_gain[n], g.c2_gain[n + 1], g.c2_gain[n + 2], g.c2_gain[n + 3]);
  };
  if (sa.w_const) load_vectors();                   // constant with the weights
  pdl_wait();

  if (producer)
    for (int i = 0; i < pre; ++i) {
      if (!sa.w_const) load_w(i);
      load_a(i);
    }
  if (!sa.w_const) load_vectors();
  // the residual of this thread's first rows, asked for before the products
  constexpr int RP = 4;                             // rounds of the reduction at S = 2
  float4 res[RP];
  auto row_of = [&](int i) { return rank + S * (threadIdx.x / TPR) + i * S * (SP_THREADS / TPR); };
#pragma unroll
  for (int i = 0; i < RP; ++i)
    res[i] = g.residual && col_ok && row_of(i) < rows
                 ? *reinterpret_cast<const float4*>(g.residual + (size_t)(m0 + row_of(i)) * g.ldr + n)
                 : make_float4(0.f, 0.f, 0.f, 0.f);

  if (warp == 0) {
    if (producer) {
      for (int i = pre; i < kcn; ++i) {
        if (!mbar_wait(&empty[i % SP_STAGES], ((i / SP_STAGES) & 1) ^ 1, wait)) {
          abort_flag = 1;
          break;
        }
        load_w(i);
        load_a(i);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc(128, BN);
      for (int i = 0; i < kcn; ++i) {
        const int s = i % SP_STAGES;
        if (!mbar_wait(&full[s], (i / SP_STAGES) & 1, wait)) {
          abort_flag = 1;
          break;
        }
        tc_fence_after();
        const uint64_t ad = smem_desc(sA + (size_t)s * SP_A_BYTES);
        const uint64_t bd = smem_desc(sB + (size_t)s * Cfg::B_BYTES);
        if constexpr (FEW) {
          const int b = i & 1;
          if (!mbar_wait(&acc_empty[b], ((i >> 1) & 1) ^ 1, wait)) {
            abort_flag = 1;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < SP_BK / 16; ++k)
            mma_bf16(tmem + (2 * b + (k >> 1)) * BN, ad + 2ull * k, bd + 2ull * k, idesc, k & 1);
          mma_commit(&empty[s]);
          mma_commit(&acc_full[b]);
        } else {
#pragma unroll
          for (int k = 0; k < SP_BK / 16; ++k)
            mma_bf16(tmem, ad + 2ull * k, bd + 2ull * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
          mma_commit(&empty[s]);
        }
      }
      if (!FEW) mma_commit(&acc_full[0]);
    }
  } else if (warp >= 4) {
    // ---- partial sums of this CTA's part of Kd: thread = row. Every copy has landed and been
    //      multiplied once the accumulator is complete, so they may overwrite the ring.
    const int q = warp & 3, row = q * 32 + lane;
    const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16);
    if constexpr (FEW) {
      if (q * 32 < rows) {
        float sum[BN];
#pragma unroll
        for (int j = 0; j < BN; ++j) sum[j] = 0.f;
        bool ok = true;
        for (int i = 0; i < kcn; ++i) {
          const int b = i & 1;
          ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (i >> 1) & 1, wait));
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < BN; c += 16) {
            uint32_t r0[16], r1[16];
            tmem_ld16_nowait(lanes + 2 * b * BN + c, r0);
            tmem_ld16_nowait(lanes + (2 * b + 1) * BN + c, r1);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[c + j] += __uint_as_float(r0[j]) + __uint_as_float(r1[j]);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
        if (!ok) {
          abort_flag = 1;
        } else {
#pragma unroll
          for (int j = 0; j < BN; j += 4)
            *reinterpret_cast<float4*>(part + row * PLD + j) =
                make_float4(sum[j], sum[j + 1], sum[j + 2], sum[j + 3]);
        }
      }
    } else {
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[0], 0, wait));
      tc_fence_after();
      if (!ok) {
        abort_flag = 1;
      } else {
#pragma unroll
        for (int c = 0; c < BN; c += 32) {
          uint32_t r[32];
          tmem_ld32(lanes + c, r);
#pragma unroll
          for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<float4*>(part + row * PLD + c + j) =
                make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                            __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
        }
      }
    }
    tc_fence_before();
  }
  __syncwarp();
  cluster_sync();                      // every CTA's partials are in place

  // ---- reduction and epilogue: rows rank, rank + S, ...
  const float ss_scale = 1.0f / (float)(g.ss_dim > 0 ? g.ss_dim : g.Kd);
  // the threads of a row stay together: all run the same number of rounds
  const int rounds = max(1, (FEW ? SP_FEW : 128) / (S * (SP_THREADS / TPR)));
  auto sum_row = [&](int i) {                       // the S partials of a row, in rank order
    // threads past the last row sum it too: left out by a branch, a partial row tile took up to 0.7 us
    // longer (96 x 512 x 512: 4.1 to 4.8 us by how it was compiled, so 4.2)
    const int r = min(row_of(i), rows - 1);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (S == 1) return *reinterpret_cast<const float4*>(part + r * PLD + c);
    const uint32_t local = smem_u32(part + r * PLD + c);
    float4 t[8];                                    // every partial in flight, then the sum
#pragma unroll
    for (int p = 0; p < 8; ++p)
      if (p < S) t[p] = ld_cluster_f4(local, p);
    if constexpr (FEW) {
      float4 e = make_float4(0.f, 0.f, 0.f, 0.f);   // what the adds round off
#pragma unroll
      for (int p = 0; p < 8; ++p)
        if (p < S) {
          two_sum(v.x, e.x, t[p].x);
          two_sum(v.y, e.y, t[p].y);
          two_sum(v.z, e.z, t[p].z);
          two_sum(v.w, e.w, t[p].w);
        }
      v.x += e.x; v.y += e.y; v.z += e.z; v.w += e.w;
    } else {
#pragma unroll
      for (int p = 0; p < 8; ++p)
        if (p < S) { v.x += t[p].x; v.y += t[p].y; v.z += t[p].z; v.w += t[p].w; }
    }
    return v;
  };
  auto finish_row = [&](int i, const float4& v, const float4& rr) {
    const int r = row_of(i);
    const bool live = r < rows;
    const int m = m0 + r;
    float rs = 1.f;
    if (g.ss_in) {                                  // folded RMSNorm of the input rows
      float s = 0.f;
      if (live)
        for (int i = threadIdx.x % TPR; i < g.ss_slots; i += TPR) s += g.ss_in[(size_t)m * SS_LD + i];
#pragma unroll
      for (int o = TPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      rs = rsqrtf(s * ss_scale + SP_RMS_EPS);
    }
    const bool out = live && col_ok;
    float4 x = make_float4(fmaf(v.x, rs, bias.x), fmaf(v.y, rs, bias.y), fmaf(v.z, rs, bias.z),
                           fmaf(v.w, rs, bias.w));
    if (g.bias_rows && out) {
      const float4 br = *reinterpret_cast<const float4*>(
          g.bias_rows + (size_t)(m / g.rows_per_bias) * g.N + n);
      x.x += br.x; x.y += br.y; x.z += br.z; x.w += br.w;
    }
    if (g.act == ACT_SILU) {
      if (!FEW && g.c_dt == LILICORR_BF16) {          // (few rows: exp, as the few-row kernel)
        x.x = silu_tanh(x.x); x.y = silu_tanh(x.y); x.z = silu_tanh(x.z); x.w = silu_tanh(x.w);
      } else {
        x.x = silu_f(x.x); x.y = silu_f(x.y); x.z = silu_f(x.z); x.w = silu_f(x.w);
      }
    }
    if (g.residual) { x.x += rr.x; x.y += rr.y; x.z += rr.z; x.w += rr.w; }
    if (out && g.C) {
      if (g.c_dt == LILICORR_BF16)
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(g.C) + (size_t)m * g.ldc + n) =
            make_uint2(pack_bf16x2(x.x, x.y), pack_bf16x2(x.z, x.w));
      else
        *reinterpret_cast<float4*>(static_cast<float*>(g.C) + (size_t)m * g.ldc + n) = x;
    }
    if (g.c2) {                                     // the next RMSNorm's input, and its sums
      float s = 0.f;
      if (out) {
        s = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, x.w * x.w)));
        const float4 y = make_float4(x.x * gain.x, x.y * gain.y, x.z * gain.z, x.w * gain.w);
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(g.c2) + (size_t)m * g.ldc2 + n) =
            make_uint2(pack_bf16x2(y.x, y.y), pack_bf16x2(y.z, y.w));
        if (g.c3) {
          const float4 t = *reinterpret_cast<const float4*>(
              g.c3_t + (size_t)(m / g.c3_rows_per) * g.N + n);
          *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(g.c3) + (size_t)m * g.ldc2 + n) =
              make_uint2(pack_bf16x2(y.x * t.x, y.y * t.y), pack_bf16x2(y.z * t.z, y.w * t.w));
        }
      }
#pragma unroll
      for (int o = TPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (live && threadIdx.x % TPR == 0) g.ss_out[(size_t)m * SS_LD + blockIdx.y] = s;
    }
  };
  float4 sum[RP];
#pragma unroll
  for (int i = 0; i < RP; ++i)
    if (i < rounds) sum[i] = sum_row(i);
  // the peers' partials are read: the barrier that lets them leave is met behind the stores
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < RP; ++i)
    if (i < rounds) finish_row(i, sum[i], res[i]);
  for (int i = RP; i < rounds; ++i)                 // S = 1: the other rounds read theirs now
    finish_row(i, sum_row(i),
               g.residual && col_ok && row_of(i) < rows
                   ? *reinterpret_cast<const float4*>(g.residual + (size_t)(m0 + row_of(i)) * g.ldr + n)
                   : make_float4(0.f, 0.f, 0.f, 0.f));

  // ---- teardown: no CTA leaves while a peer may still read its partials
  if (abort_flag) {
    if (threadIdx.x == 0) {
      set_status(g.status, LILICORR_ERR_TIMEOUT);
      const long long t0 = clock64();               // let copies in flight land
      while (clock64() - t0 < wait / 10) {
      }
    }
    __syncthreads();
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, Cfg::TMEM_COLS);
  }
}

template <int BN, bool FEW>
lilicorr_status_t launch_split(const GemmArgs& g, int S, cudaStream_t st) {
  static bool configured[64] = {false};
  LL_TRY(allow_max_dynamic_smem(gemm_split_kernel<BN, FEW>, configured));
  CUtensorMap ma, mw;
  const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if (!make_map(&ma, g.A, bf, 2, g.M, g.Kd, g.lda, 128, SP_BK)) return LILICORR_ERR_CUDA;
  if (!make_map(&mw, g.W, bf, 2, g.N, g.Kd, g.ldw, BN, SP_BK)) return LILICORR_ERR_CUDA;
  SplitArgs sa;
  sa.g = g;
  sa.S = S;
  sa.w_const = g.w_const;
  return launch_cluster_k(gemm_split_kernel<BN, FEW>,
                          dim3(S, ceil_div(g.N, BN), ceil_div(g.M, 128)), SP_THREADS,
                          SpCfg<BN, FEW>::SMEM, S, st, ma, mw, sa);
}

int split_tiles(const GemmArgs& g, int bn) { return ceil_div(g.M, 128) * ceil_div(g.N, bn); }

}  // namespace

int gemm_split_ss_slots(int N) { return ceil_div(N, 64); }

// CTAs per tile (0: too many tiles, the persistent kernel's case). Measured back to back, us for
// S = 1 / 2 / 4 / 8 and the persistent kernel:
//   120 x 1024 x 1024   8.6  6.4  4.9  5.6   7.7        64 x 256 x 4096   20.8 11.8  7.2  5.5  20.4
//   120 x 3072 x 1024   8.7  6.5  6.2 11.8   7.8       360 x 1024 x 2560  15.0  9.6  8.1 13.8  14.3
//   480 x 1024 x 1024   8.8  6.5  6.6 13.4   7.9       480 x 1024 x 2048  13.0  8.7  7.8 14.3  12.2
//   960 x 1024 x 1024   8.7  7.6 12.6 25.1   8.0      1024 x 512 x 512     6.7  5.5  6.0 13.0   5.7
// So S doubles while the CTAs fit one an SM and keep two chunks of Kd each, or two an SM and keep
// four; eight ways, whose clusters are harder to place, only where Kd is long.
// Of few rows one chunk each will do: the shorter a CTA's sum, the closer (64 x 1024 x 256: S = 4 4.0 us
// and an error of 5.4e-8, S = 1 4.8 and 6.1e-8; the few-row kernel 24.4 and 5.5e-8).
int gemm_split_ways(const GemmArgs& g) {
  const int tiles = split_tiles(g, 64), nk = ceil_div(g.Kd, SP_BK), sms = num_sms();
  const int least = g.M <= SP_FEW ? 2 : 4;
  int S = 1;
  while (S < 4 && ((2 * S * tiles <= sms && nk >= least * S) || (S * tiles <= sms && nk >= 8 * S)))
    S *= 2;
  if (S == 4 && 8 * tiles <= sms && nk >= 40) S = 8;
  return S > 1 || 2 * tiles <= sms ? S : 0;
}

bool gemm_split_supported(const GemmArgs& g) {
  if (!gemm_tc_operands_ok(g)) return false;
  if (g.c2 && (!g.c2_gain || !g.ss_out || g.c_dt != LILICORR_F32 || !aligned16(g.c2) ||
               (g.ldc2 % 8) || gemm_split_ss_slots(g.N) > SS_LD))
    return false;
  if (g.bias_rows && !aligned16(g.bias_rows)) return false;
  if (ceil_div(g.M, 128) > 65535 || ceil_div(g.N, 64) > 65535) return false;
  return gemm_split_ways(g) > 0;
}

// Whether the network gives a product to this kernel. Measured back to back, us, this kernel (S ways)
// against what else takes the product:
//   65-128 rows, Kd = 64 or 256: 5.3-6.1 / 4.7-5.4 (S = 1 / 2), whole-K copies (gemm_small.cu)
//     3.0-3.8 / 3.5-4.3; Kd = 512, fp32 out: 3.9-4.5 (S = 4) against 4.2-5.3, bf16 out 4.1-4.9 against
//     4.3-4.5, 48 tiles (S = 2) 5.7-6.0 against 4.5-5.3
//   more rows, fp32 / bf16 out, persistent kernel: Kd = 64 or 256, 6.0 / 5.9 and 5.1-5.4 / 5.2-5.6 against
//     4.1 / 3.6 and 4.7-5.0 / 4.2-4.5; Kd = 512, S = 4, 4.3-4.6 / 4.3-4.8 against 5.9 / 5.4, S = 2 with a CTA
//     an SM 5.8-6.1 / 5.9-6.1 against 5.9-6.1 / 5.4, with two 6.6-7.2 / 6.5-7.2 against 6.0 / 5.5; Kd = 1024, S = 4,
//     4.8-6.9 / 4.8-7.0 against 8.0 / 7.5, S = 2 with two CTAs an SM 7.4-8.3 / 7.6-8.3 against 8.1 / 7.7;
//     Kd = 2048, S = 2, 9.5-10.5 against 12.1 / 11.7
//   5-64 rows, few-row kernel: 3.6-4.4 (Kd = 256 or 384) and 4.1-5.2 (512 or 1024) against 2.7-4.3 while
//     that is one wave of CTAs, against 4.9-72 beyond; Kd = 4096, one wave: 6.1-6.7 against 6.1-6.4 (5.4 against 5.0 at 8 rows), but on
//     a quarter of the SMs (beside the top-K pass, selection of 32 requests: 127.5 -> 126.1).
// Where every product folds an RMSNorm, the kernels that the fold saves decide up to 128 rows: on heads
// of width 64 and 128 this kernel's networks took 1.3 to 1.5 times as long as the unfolded ones with
// whole-K copies (two requests of 64 nodes at width 128: 99.9 against 66.8 us), on width 320 0.83.
// Up to 64 rows only where its error is no larger than the few-row kernel's: Kd over at
// least four CTAs (2560 columns x Kd 328, two CTAs 6.3e-8 against 5.7e-8), 16 chunks each at most. On
// networks of width 320 or 384 it takes 64 to 73 us where the few-row kernel takes 77 to 203. Up to
// four rows the few-row kernel has no second wave, and its unfolded networks are ahead (one sequence
// of four nodes, width 512: 55.1 against 64.3 us, 1024: 73.1 against 81.7).
bool gemm_split_takes(const GemmArgs& g) {
  if (!gemm_split_supported(g)) return false;
  const int S = gemm_split_ways(g), nk = ceil_div(g.Kd, SP_BK);
  const bool fold = g.c2 || g.ss_in;
  if (g.M <= SP_FEW)
    return g.M > 4 && S >= 4 && nk <= 16 * S &&
           (fold || ceil_div(g.N, 4) * ceil_div(g.M, 16) > num_sms() || (nk >= 40 && g.M > 8));
  if (fold && g.M <= 128) return nk >= 5;
  const bool bf16 = g.c_dt == LILICORR_BF16;
  if (gemm_small_supported(g)) return S >= 4 && !bf16;
  if (S == 2) {
    const bool one = 2 * split_tiles(g, 64) <= num_sms();
    return nk >= (bf16 ? (one ? 14 : 24) : (one ? 8 : 16));
  }
  return S >= 4;
}

lilicorr_status_t launch_gemm_split(const GemmArgs& g, cudaStream_t st) {
  if (g.M == 0 || g.N == 0) return LILICORR_OK;
  const int S = gemm_split_ways(g);
  return g.M <= SP_FEW ? launch_split<64, true>(g, S, st) : launch_split<64, false>(g, S, st);
}

}  // namespace lilicorr
