// Step (2): the scoring network's fp32 CUDA-core kernels (Sec. 3.2; App. A "Architecture").
//
// Node construction, RMSNorm, target state, bidirectional attention with the two
// learned bias tables, the fusion input and row normalisation, plus a tiled
// fp32 linear layer with fused bias / per-sequence bias / SiLU / residual
// epilogue. The fp32 head runs every matrix product here; the bf16 head runs its
// large products on the tensor cores (gemm_tc.cu) and the rest here.
#include <type_traits>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace lilicorr {

namespace {

constexpr float RMS_EPS = 1e-6f;
constexpr float UNIT_EPS = 1e-12f;

// ----------------------------------------------------------------------------- linear
// fp32 CUDA-core linear layer. A CTA of 256 threads owns a 64 x 64 output tile; its four
// groups of 64 threads (8 x 8 outputs each thread) take a quarter each of every 32-wide step of
// Kd and add their sums up at the end. What bounds it: one wave of CTAs (2048 rows x 256
// columns are 128 tiles), so the chain of Kd steps within a CTA, and shared-memory reads (a
// 16-byte read takes four cycles of the SM: 8 x 8 outputs read 16 values for 64 products, 8 x 4
// outputs 12 for 32). One group with all of Kd had one warp per scheduler, each read of shared
// memory exposed: 31 us for 2048 x 256 x 256. Pairs of columns are one f32x2 multiply-add; the
// next step's operands are loaded (16 bytes a thread where rows allow) while this one is
// multiplied.
// 2048 x 256 x 256: 31 -> 15.5 us; 2048 x 256 x 512: 55 -> 23.6 us (cold).
// Few tiles leave SMs idle and the chain of steps as long: there a cluster of 2, 4 or 8 CTAs
// splits Kd (warm, in a graph; the 16 x 32 blocks that had these sizes / split): 128 x 256 x 256
// 5.1 / 4.4 us, 512 x 256 x 512 13.3 / 7.6, 1024 x 256 x 256 15.8 / 7.3, 512 x 256 x 4096
// 91 / 33; its error against 64 bits is a third of theirs (9e-8 to 2e-7; 3e-7 to 1e-6).
// Whole fp32 networks of 4 and 8 sequences of 128 nodes, D 256: 224 -> 145 and 293 -> 195 us.
constexpr int GB_M = 64, GB_N = 64, GB_K = 32, G_THREADS = 256, G_GROUPS = 4;

__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  return ((uint64_t)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// four consecutive elements of row r starting at column k (zeros outside [0, rows) x [0, cols))
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p, int r, int rows, int k, int cols, int ld) {
  if (r >= rows) return make_float4(0.f, 0.f, 0.f, 0.f);
  p += (size_t)r * ld + k;
  if (VEC) return k < cols ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
  return make_float4(k < cols ? p[0] : 0.f, k + 1 < cols ? p[1] : 0.f, k + 2 < cols ? p[2] : 0.f,
                     k + 3 < cols ? p[3] : 0.f);
}
template <bool VEC>
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p, int r, int rows, int k, int cols,
                                        int ld) {
  if (r >= rows) return make_float4(0.f, 0.f, 0.f, 0.f);
  p += (size_t)r * ld + k;
  if (VEC) {
    if (k >= cols) return make_float4(0.f, 0.f, 0.f, 0.f);
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
  }
  return make_float4(k < cols ? __bfloat162float(p[0]) : 0.f,
                     k + 1 < cols ? __bfloat162float(p[1]) : 0.f,
                     k + 2 < cols ? __bfloat162float(p[2]) : 0.f,
                     k + 3 < cols ? __bfloat162float(p[3]) : 0.f);
}

// VEC: rows of both operands in whole aligned groups of four elements
// SPLIT: the CTAs of a cluster take a part of Kd's steps each (at least one) and then a part of
// the tile's rows each, whose sums they read from one another
// PER_SM: CTAs an SM holds. Two (128 registers) from two tiles an SM on, so that one's first loads and
// last sums run beside the other's products: with one such products of short Kd took longer than 4 x 4
// outputs a thread at four CTAs an SM had (65,536 x 256 x 64: 100 us, one 170, two 106;
// 32,768 x 512 x 32: 70, 143, 89), and long ones gain too (8192 x 512 x 512: 121, two 111). In one wave
// one is ahead (2048 x 256 x 256: 11.0, two 11.9); in less than two the first SMs to come free would
// take two each (network of width 512, four sequences of 100 nodes, 168 tiles: 267 us, with two 283).
template <typename TA, typename TW, typename TC, bool VEC, bool SPLIT, int PER_SM = 1>
__global__ void __launch_bounds__(G_THREADS, PER_SM) gemm_simt_kernel(GemmArgs g, int ways) {
  pdl_wait();
  constexpr int LDT = GB_M + 4, KG = GB_K / G_GROUPS;
  static_assert(GB_M == GB_N && GB_M * GB_K == 8 * G_THREADS, "two groups of four a thread");
  // [buffer][A or W][k][row]; after the products two groups' sums at a time
  __shared__ __align__(16) float sm[2][2][GB_K][LDT];
  static_assert(sizeof(sm) >= 2 * GB_M * LDT * sizeof(float), "two groups' sums fit");
  const TA* A = static_cast<const TA*>(g.A);
  const TW* W = static_cast<const TW*>(g.W);
  const int tid = threadIdx.x, grp = tid >> 6;
  const int rank = SPLIT ? blockIdx.x % ways : 0;
  const int m0 = blockIdx.y * GB_M, n0 = (SPLIT ? blockIdx.x / ways : blockIdx.x) * GB_N;
  const int steps = (g.Kd + GB_K - 1) / GB_K;
  const int kbeg = SPLIT ? steps * rank / ways * GB_K : 0;
  const int kend = SPLIT ? min(g.Kd, steps * (rank + 1) / ways * GB_K) : g.Kd;
  const int tx = tid & 7, ty = (tid >> 3) & 7;
  const int lr = tid >> 3, lk = (tid & 7) * 4;        // rows lr and lr + 32, columns lk..lk + 3
  uint64_t acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  float4 ra[2], rw[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      ra[h] = load4<VEC>(A, m0 + lr + 32 * h, g.M, k0 + lk, g.Kd, g.lda);
      rw[h] = load4<VEC>(W, n0 + lr + 32 * h, g.N, k0 + lk, g.Kd, g.ldw);
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = lr + 32 * h;
      sm[b][0][lk][r] = ra[h].x; sm[b][0][lk + 1][r] = ra[h].y;
      sm[b][0][lk + 2][r] = ra[h].z; sm[b][0][lk + 3][r] = ra[h].w;
      sm[b][1][lk][r] = rw[h].x; sm[b][1][lk + 1][r] = rw[h].y;
      sm[b][1][lk + 2][r] = rw[h].z; sm[b][1][lk + 3][r] = rw[h].w;
    }
  };
  fetch(kbeg);
  stash(0);
  __syncthreads();
  int b = 0;
  for (int k0 = kbeg; k0 < kend; k0 += GB_K, b ^= 1) {
    const bool more = k0 + GB_K < kend;
    if (more) fetch(k0 + GB_K);
#pragma unroll
    for (int kk = 0; kk < KG; ++kk) {
      // rows ty*4.. and 32 + ty*4.., columns tx*4.. and 32 + tx*4..
      const float* as = sm[b][0][grp * KG + kk];
      const float* ws = sm[b][1][grp * KG + kk];
      const float4 a0 = *reinterpret_cast<const float4*>(as + ty * 4);
      const float4 a1 = *reinterpret_cast<const float4*>(as + 32 + ty * 4);
      const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(ws + tx * 4);
      const ulonglong2 w1 = *reinterpret_cast<const ulonglong2*>(ws + 32 + tx * 4);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint64_t aa = pack_f32x2(a[i], a[i]);
        acc[i][0] = fma_f32x2(aa, w0.x, acc[i][0]);
        acc[i][1] = fma_f32x2(aa, w0.y, acc[i][1]);
        acc[i][2] = fma_f32x2(aa, w1.x, acc[i][2]);
        acc[i][3] = fma_f32x2(aa, w1.y, acc[i][3]);
      }
    }
    if (more) stash(b ^ 1);           // its last readers are behind the previous barrier
    __syncthreads();
  }
  // ---- the groups' sums: 2 into 0 and 3 into 1, then both for the epilogue
  float* red = &sm[0][0][0][0];
  auto at = [&](int q, int i, int j) {              // thread's rows i, column quads j
    return reinterpret_cast<ulonglong2*>(red + (size_t)q * GB_M * LDT +
                                         ((i >> 2) * 32 + ty * 4 + (i & 3)) * LDT + j * 32 + tx * 4);
  };
  auto put = [&](int q) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) *at(q, i, j) = make_ulonglong2(acc[i][2 * j], acc[i][2 * j + 1]);
  };
  if (grp >= 2) put(grp - 2);
  __syncthreads();
  if (grp < 2) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const ulonglong2 o = *at(grp, i, j);
        acc[i][2 * j] = add_f32x2(acc[i][2 * j], o.x);
        acc[i][2 * j + 1] = add_f32x2(acc[i][2 * j + 1], o.y);
      }
    // each thread overwrites only what it has just read itself
    put(grp);
  }
  if (SPLIT) tc::cluster_sync();             // every CTA's sums are in place
  else __syncthreads();
  // ---- epilogue: 16 threads a row, four columns each
  TC* C = static_cast<TC*>(g.C);
  const int c = (tid & 15) * 4, n = n0 + c;
  const int rows = SPLIT ? GB_M / ways : GB_M;
#pragma unroll
  for (int r1 = tid >> 4; r1 < rows; r1 += G_THREADS / 16) {
    const int r = rank * rows + r1, m = m0 + r;
    if (m >= g.M) break;
    float s[4];
    if (SPLIT) {                             // in the order of Kd
#pragma unroll
      for (int j = 0; j < 4; ++j) s[j] = 0.f;
#pragma unroll 4
      for (int q = 0; q < ways; ++q) {
        const float4 s0 = tc::ld_cluster_f4(tc::smem_u32(red + r * LDT + c), q);
        const float4 s1 = tc::ld_cluster_f4(tc::smem_u32(red + (GB_M + r) * LDT + c), q);
        s[0] += s0.x + s1.x; s[1] += s0.y + s1.y; s[2] += s0.z + s1.z; s[3] += s0.w + s1.w;
      }
    } else {
      const float4 s0 = *reinterpret_cast<const float4*>(red + r * LDT + c);
      const float4 s1 = *reinterpret_cast<const float4*>(red + (GB_M + r) * LDT + c);
      s[0] = s0.x + s1.x; s[1] = s0.y + s1.y; s[2] = s0.z + s1.z; s[3] = s0.w + s1.w;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (n + j >= g.N) break;
      float v = s[j];
      if (g.bias) v += g.bias[n + j];
      if (g.bias_rows) v += g.bias_rows[(size_t)(m / g.rows_per_bias) * g.N + n + j];
      if (g.act == ACT_SILU) v = silu_f(v);
      if (g.residual) v += g.residual[(size_t)m * g.ldr + n + j];
      st_elem(C, (size_t)m * g.ldc + n + j, v);
    }
  }
  if (SPLIT) {
    __syncwarp();
    tc::cluster_sync();                      // no CTA leaves while a peer reads its sums
  }
}

template <typename TA, typename TW, bool VEC>
lilicorr_status_t gemm_dispatch_c(const GemmArgs& g, dim3 grid, cudaStream_t st) {
  if (VEC && (long long)grid.x * grid.y > 2 * num_sms()) {
    if (g.c_dt == LILICORR_F32)
      return launch_k(gemm_simt_kernel<TA, TW, float, VEC, false, 2>, grid, G_THREADS, 0, st, g, 1);
    return launch_k(gemm_simt_kernel<TA, TW, __nv_bfloat16, VEC, false, 2>, grid, G_THREADS, 0, st, g, 1);
  }
  if (g.c_dt == LILICORR_F32)
    return launch_k(gemm_simt_kernel<TA, TW, float, VEC, false>, grid, G_THREADS, 0, st, g, 1);
  return launch_k(gemm_simt_kernel<TA, TW, __nv_bfloat16, VEC, false>, grid, G_THREADS, 0, st, g, 1);
}
// (bf16 weights: through the testing header's path 7 only; the network gives fp32 activations and bf16
// weights to the 16 x 32 blocks, which are as fast there)
template <typename TW>
lilicorr_status_t gemm_split_dispatch_c(const GemmArgs& g, dim3 grid, int ways, cudaStream_t st) {
  grid.x *= ways;
  if (g.c_dt == LILICORR_F32)
    return launch_cluster_k(gemm_simt_kernel<float, TW, float, true, true>, grid, G_THREADS, 0,
                            ways, st, g, ways);
  return launch_cluster_k(gemm_simt_kernel<float, TW, __nv_bfloat16, true, true>, grid, G_THREADS,
                          0, ways, st, g, ways);
}

// groups of four elements: Kd and the row strides multiples of 4, bases on 16 (fp32) or 8
// (bf16) bytes; other operands are read element by element
bool gemm_simt_vec(const GemmArgs& g) {
  const uintptr_t am = g.a_dt == LILICORR_F32 ? 15 : 7, wm = g.w_dt == LILICORR_F32 ? 15 : 7;
  return g.Kd % 4 == 0 && g.lda % 4 == 0 && g.ldw % 4 == 0 &&
         !(reinterpret_cast<uintptr_t>(g.A) & am) && !(reinterpret_cast<uintptr_t>(g.W) & wm);
}

template <typename TA>
lilicorr_status_t gemm_dispatch_w(const GemmArgs& g, dim3 grid, cudaStream_t st) {
  const bool vec = gemm_simt_vec(g);
  if (g.w_dt == LILICORR_F32)
    return vec ? gemm_dispatch_c<TA, float, true>(g, grid, st)
               : gemm_dispatch_c<TA, float, false>(g, grid, st);
  return vec ? gemm_dispatch_c<TA, __nv_bfloat16, true>(g, grid, st)
             : gemm_dispatch_c<TA, __nv_bfloat16, false>(g, grid, st);
}

// ----------------------------------------------------------------------------- skinny linear
// Few rows (one per slot or per sequence) against long rows (Kd up to H).
// CTA (column block of SK_NB, row block of SK_MB): its 256 threads split Kd in
// 8-element vectors, each accumulating SK_MB x SK_NB partial dot products, reduced by
// warp shuffles and shared memory. Many CTAs stream disjoint weight rows.
constexpr int SK_NB = 4, SK_MB = 16, SK_THREADS = 256;

__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  const float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 a = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
  }
}

// TWO: the launch holds two products, the second at blockIdx.z = 1. A kernel of its own: the choice and
// the narrower product's early exit cost one-product launches too (bf16, 173 -> 255 registers: 16 x
// 256 x 4096 6.3 -> 9.7 us, 4 x 1536 x 256 2.8 -> 4.5).
template <typename TA, typename TW, typename TC, int MB, bool TWO>
__global__ void __launch_bounds__(SK_THREADS) gemm_skinny_kernel(const GemmArgs g0, const GemmArgs g1) {
  pdl_wait();
  const GemmArgs& g = TWO && blockIdx.z ? g1 : g0;
  __shared__ float red[SK_THREADS / 32][MB * SK_NB];
  const TA* A = static_cast<const TA*>(g.A);
  const TW* W = static_cast<const TW*>(g.W);
  const int n0 = blockIdx.x * SK_NB, m0 = blockIdx.y * MB;
  if (TWO && n0 >= g.N) return;
  const int nb = min(SK_NB, g.N - n0), mb = min(MB, g.M - m0);
  float acc[MB][SK_NB];
#pragma unroll
  for (int i = 0; i < MB; ++i)
#pragma unroll
    for (int j = 0; j < SK_NB; ++j) acc[i][j] = 0.f;
  for (int k = threadIdx.x * 8; k < g.Kd; k += SK_THREADS * 8) {
    float w[SK_NB][8];
#pragma unroll
    for (int j = 0; j < SK_NB; ++j) {
      if (j < nb) load8(W + (size_t)(n0 + j) * g.ldw + k, w[j]);
      else
#pragma unroll
        for (int e = 0; e < 8; ++e) w[j][e] = 0.f;
    }
    // all row loads first (predicated, no early exit) so they are in flight together
    float a[MB][8];
#pragma unroll
    for (int i = 0; i < MB; ++i) {
      if (i < mb) load8(A + (size_t)(m0 + i) * g.lda + k, a[i]);
      else
#pragma unroll
        for (int e = 0; e < 8; ++e) a[i][e] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < MB; ++i)
#pragma unroll
      for (int j = 0; j < SK_NB; ++j)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[i][j] = fmaf(a[i][e], w[j][e], acc[i][j]);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < MB; ++i) {
    if (i >= mb) break;                            // rows past M: nothing to reduce
#pragma unroll
    for (int j = 0; j < SK_NB; ++j) {
      const float v = warp_sum(acc[i][j]);
      if (lane == 0) red[warp][i * SK_NB + j] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x < MB * SK_NB) {
    const int i = threadIdx.x / SK_NB, j = threadIdx.x % SK_NB;
    if (i < mb && j < nb) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < SK_THREADS / 32; ++w) v += red[w][threadIdx.x];
      const int m = m0 + i, n = n0 + j;
      if (g.bias) v += g.bias[n];
      if (g.bias_rows) v += g.bias_rows[(size_t)(m / g.rows_per_bias) * g.N + n];
      if (g.act == ACT_SILU) v = silu_f(v);
      if (g.residual) v += g.residual[(size_t)m * g.ldr + n];
      st_elem(static_cast<TC*>(g.C), (size_t)m * g.ldc + n, v);
    }
  }
}

// ----------------------------------------------------------------------------- row-block linear
// Per-sequence products with fp32 activations and more rows than the few-row kernel takes
// (the target state t of a batch against W_a and the fusion layer's t block: M = B up to
// 1024, Kd = D). CTA = 16 rows x 32 columns: lane = output column, warp = two rows. Per
// chunk of Kd, the 16 activation rows and the 32 weight rows are staged in shared memory by
// one round of asynchronous 16-byte copies (all in flight at once, coalesced); each lane
// then reads its weight row and the warp's two activation rows (broadcasts). No
// cross-lane reduction.
constexpr int GR_M = 16, GR_N = 32, GR_THREADS = 256;
__device__ __forceinline__ void cp16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
               ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <typename TW>
struct GrCfg {
  static constexpr int KC = sizeof(TW) == 2 ? 256 : 128;      // Kd chunk staged at a time
  static constexpr int AS = KC + 4;                           // row strides (elements), padded
  static constexpr int WS = KC + 16 / (int)sizeof(TW);        // so 8 lanes' 16-byte reads differ in bank
};
template <typename TW, typename TC, bool TWO>                   // TWO: as the few-row kernel's
__global__ void __launch_bounds__(GR_THREADS) gemm_rows_kernel(const GemmArgs g0, const GemmArgs g1) {
  pdl_wait();
  const GemmArgs& g = TWO && blockIdx.z ? g1 : g0;
  using Cfg = GrCfg<TW>;
  constexpr int KC = Cfg::KC, AS = Cfg::AS, WS = Cfg::WS;
  constexpr int WV = 16 / (int)sizeof(TW);                    // weights per 16-byte piece
  __shared__ __align__(16) float As[GR_M * AS];
  __shared__ __align__(16) TW Ws[GR_N * WS];
  const float* A = static_cast<const float*>(g.A);
  const TW* W = static_cast<const TW*>(g.W);
  const int m0 = blockIdx.y * GR_M, n0 = blockIdx.x * GR_N;
  if (TWO && n0 >= g.N) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = n0 + lane, r0 = 2 * warp;
  float acc0 = 0.f, acc1 = 0.f;
  for (int k0 = 0; k0 < g.Kd; k0 += KC) {
    const int kc = min(KC, g.Kd - k0);                          // a multiple of 8
    __syncthreads();                                            // the previous chunk is consumed
    for (int i = threadIdx.x; i < GR_M * (kc / 4); i += GR_THREADS) {
      const int r = i / (kc / 4), c = 4 * (i % (kc / 4));
      float* dst = &As[r * AS + c];
      if (m0 + r < g.M) cp16(dst, A + (size_t)(m0 + r) * g.lda + k0 + c);
      else *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int i = threadIdx.x; i < GR_N * (kc / WV); i += GR_THREADS) {
      const int r = i / (kc / WV), c = WV * (i % (kc / WV));
      TW* dst = &Ws[r * WS + c];
      if (n0 + r < g.N) cp16(dst, W + (size_t)(n0 + r) * g.ldw + k0 + c);
      else *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const TW* wr = &Ws[lane * WS];
    const float* a0p = &As[r0 * AS];
    const float* a1p = a0p + AS;
#pragma unroll 4
    for (int k = 0; k < kc; k += 8) {
      float w[8];
      load8(wr + k, w);
      const float4 a0 = *reinterpret_cast<const float4*>(a0p + k);
      const float4 a1 = *reinterpret_cast<const float4*>(a0p + k + 4);
      const float4 b0 = *reinterpret_cast<const float4*>(a1p + k);
      const float4 b1 = *reinterpret_cast<const float4*>(a1p + k + 4);
      acc0 = fmaf(a0.x, w[0], fmaf(a0.y, w[1], fmaf(a0.z, w[2], fmaf(a0.w, w[3], acc0))));
      acc0 = fmaf(a1.x, w[4], fmaf(a1.y, w[5], fmaf(a1.z, w[6], fmaf(a1.w, w[7], acc0))));
      acc1 = fmaf(b0.x, w[0], fmaf(b0.y, w[1], fmaf(b0.z, w[2], fmaf(b0.w, w[3], acc1))));
      acc1 = fmaf(b1.x, w[4], fmaf(b1.y, w[5], fmaf(b1.z, w[6], fmaf(b1.w, w[7], acc1))));
    }
  }
  if (n >= g.N) return;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = m0 + r0 + i;
    if (m >= g.M) continue;
    float v = i ? acc1 : acc0;
    if (g.bias) v += g.bias[n];
    if (g.bias_rows) v += g.bias_rows[(size_t)(m / g.rows_per_bias) * g.N + n];
    if (g.act == ACT_SILU) v = silu_f(v);
    if (g.residual) v += g.residual[(size_t)m * g.ldr + n];
    st_elem(static_cast<TC*>(g.C), (size_t)m * g.ldc + n, v);
  }
}

template <typename TA, typename TW, int MB>
lilicorr_status_t skinny_dispatch_m(const GemmArgs& g, const GemmArgs* g1, cudaStream_t st) {
  const dim3 grid(ceil_div(g1 ? max(g.N, g1->N) : g.N, SK_NB), ceil_div(g.M, MB), g1 ? 2 : 1);
  if constexpr (std::is_same<TA, float>::value)
    if (g1)                                        // fp32 in and out (launch_gemm_skinny)
      return launch_k(gemm_skinny_kernel<TA, TW, float, MB, true>, grid, SK_THREADS, 0, st, g, *g1);
  if (g.c_dt == LILICORR_F32)
    return launch_k(gemm_skinny_kernel<TA, TW, float, MB, false>, grid, SK_THREADS, 0, st, g, g);
  return launch_k(gemm_skinny_kernel<TA, TW, __nv_bfloat16, MB, false>, grid, SK_THREADS, 0, st, g, g);
}
// rows per CTA: one per sequence-level row (M = 1), four for a few, else sixteen
template <typename TA, typename TW>
lilicorr_status_t skinny_dispatch_c(const GemmArgs& g, const GemmArgs* g1, cudaStream_t st) {
  if (g.M == 1) return skinny_dispatch_m<TA, TW, 1>(g, g1, st);
  if (g.M <= 4) return skinny_dispatch_m<TA, TW, 4>(g, g1, st);
  return skinny_dispatch_m<TA, TW, SK_MB>(g, g1, st);
}
template <typename TA>
lilicorr_status_t skinny_dispatch_w(const GemmArgs& g, const GemmArgs* g1, cudaStream_t st) {
  if (g.w_dt == LILICORR_F32) return skinny_dispatch_c<TA, float>(g, g1, st);
  return skinny_dispatch_c<TA, __nv_bfloat16>(g, g1, st);
}

// ----------------------------------------------------------------------------- target state
// tn[b] = RMSNorm_H(mean over the n_tgt captured layers of T[b]) * gain (App. A).
// One CTA per sequence; each thread owns 8-element vectors of the row (H % 8 == 0),
// keeps its means in registers between the two passes (up to TN_VPT vectors).
constexpr int TN_THREADS = 512, TN_VPT = 4;

template <typename T, typename TO>
__global__ void __launch_bounds__(TN_THREADS)
target_norm_kernel(const T* __restrict__ Tin, int n_tgt, int H, const float* __restrict__ gain,
                   TO* __restrict__ tn) {
  pdl_wait();
  __shared__ float red[TN_THREADS / 32];
  __shared__ float s_total;
  const int b = blockIdx.x;
  const T* tb = Tin + (size_t)b * n_tgt * H;
  const int nv = H / 8;
  float mean[TN_VPT][8];
  float ss = 0.f;
  const float inv_p = 1.0f / (float)n_tgt;
#pragma unroll
  for (int q = 0; q < TN_VPT; ++q) {
    const int v = threadIdx.x + q * TN_THREADS;
#pragma unroll
    for (int e = 0; e < 8; ++e) mean[q][e] = 0.f;
    if (v >= nv) continue;
    for (int l = 0; l < n_tgt; ++l) {
      float x[8];
      load8(tb + (size_t)l * H + v * 8, x);
#pragma unroll
      for (int e = 0; e < 8; ++e) mean[q][e] += x[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      mean[q][e] *= inv_p;
      ss += mean[q][e] * mean[q][e];
    }
  }
  // rows longer than TN_VPT * TN_THREADS * 8 are handled by a second strided pass
  for (int v = threadIdx.x + TN_VPT * TN_THREADS; v < nv; v += TN_THREADS) {
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int l = 0; l < n_tgt; ++l) {
      float x[8];
      load8(tb + (size_t)l * H + v * 8, x);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] += x[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      acc[e] *= inv_p;
      ss += acc[e] * acc[e];
      st_elem(tn, (size_t)b * H + v * 8 + e, acc[e]);
    }
  }
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < TN_THREADS / 32 ? red[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) s_total = v;
  }
  __syncthreads();
  const float r = rsqrtf(s_total / (float)H + RMS_EPS);
#pragma unroll
  for (int q = 0; q < TN_VPT; ++q) {
    const int v = threadIdx.x + q * TN_THREADS;
    if (v >= nv) continue;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      st_elem(tn, (size_t)b * H + v * 8 + e, mean[q][e] * r * gain[v * 8 + e]);
  }
  for (int v = threadIdx.x + TN_VPT * TN_THREADS; v < nv; v += TN_THREADS)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const size_t o = (size_t)b * H + v * 8 + e;
      st_elem(tn, o, ld_elem(tn, o) * r * gain[v * 8 + e]);
    }
}

// ----------------------------------------------------------------------------- nodes
// CTA (r, part): slot row r = b*L + s, one part of the columns. For candidate k (Sec. 3.2; App. A):
//   c1 = SiLU(W_c1 f_k + b_c1)   (first layer of the confidence network; the second
//                                 layer is a linear launch that adds into x)
//   x  = fold[id_k] + hproj[r] + slot[s] + rank[k]
// with f_k = [logp_k, exp(logp_k), logp_0 - logp_k, k / (K-1), 1{k = 0}].
constexpr int NODE_COLS_MAX = 1984;
static_assert(NODE_COLS_MAX * (LILICORR_N_CONF + 1) * sizeof(float) +
              LILICORR_MAX_K * (LILICORR_N_CONF + 1) * sizeof(float) <= 48 * 1024,
              "staged weights and the static arrays");
template <typename TC1>
__global__ void node_build_kernel(int L, int K, int D, int cols, int V,
                                  const int32_t* __restrict__ ids,
                                  const float* __restrict__ logp, const float* __restrict__ fold,
                                  const float* __restrict__ hproj, const float* __restrict__ slot,
                                  const float* __restrict__ rank, const float* __restrict__ w1,
                                  const float* __restrict__ b1, TC1* __restrict__ c1,
                                  float* __restrict__ x, uint32_t* status) {
  pdl_wait();
  __shared__ float f[LILICORR_MAX_K][LILICORR_N_CONF];
  __shared__ int sid[LILICORR_MAX_K];
  extern __shared__ __align__(16) float s_w[];     // [N_CONF][cols] = W_c1^T, then b_c1 [cols]
  const int r = blockIdx.x;
  const int s = r % L;
  const int c0 = blockIdx.y * cols, nc = min(cols, D - c0);    // this CTA's columns
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
#pragma unroll
    for (int j = 0; j < LILICORR_N_CONF; ++j)
      s_w[j * cols + i] = w1[(c0 + i) * LILICORR_N_CONF + j];
    s_w[LILICORR_N_CONF * cols + i] = b1[c0 + i];
  }
  if (threadIdx.x < K) {
    const int k = threadIdx.x;
    const float lp = logp[(size_t)r * K + k];
    const float lp0 = logp[(size_t)r * K];
    f[k][0] = lp;
    f[k][1] = expf(lp);
    f[k][2] = lp0 - lp;
    f[k][3] = K > 1 ? (float)k / (float)(K - 1) : 0.f;
    f[k][4] = k == 0 ? 1.f : 0.f;
    int id = ids[(size_t)r * K + k];
    if (id < 0 || id >= V) {          // an id outside the vocabulary: flag it, read row 0
      set_status(status, LILICORR_ERR_ARG);
      id = 0;
    }
    sid[k] = id;
  }
  __syncthreads();
  const int nc4 = nc / 4;
#pragma unroll 2
  for (int i = threadIdx.x; i < K * nc4; i += blockDim.x) {
    const int k = i / nc4, nl = (i % nc4) * 4, n = c0 + nl;
    const size_t node = (size_t)r * K + k;
    const float4 fo = *reinterpret_cast<const float4*>(fold + (size_t)sid[k] * D + n);
    const float4 hp = *reinterpret_cast<const float4*>(hproj + (size_t)r * D + n);
    const float4 sl = *reinterpret_cast<const float4*>(slot + (size_t)s * D + n);
    const float4 rk = *reinterpret_cast<const float4*>(rank + (size_t)k * D + n);
    float4 o;
    o.x = fo.x + hp.x + sl.x + rk.x;
    o.y = fo.y + hp.y + sl.y + rk.y;
    o.z = fo.z + hp.z + sl.z + rk.z;
    o.w = fo.w + hp.w + sl.w + rk.w;
    *reinterpret_cast<float4*>(x + node * D + n) = o;
    float4 z = *reinterpret_cast<const float4*>(s_w + LILICORR_N_CONF * cols + nl);
#pragma unroll
    for (int j = 0; j < LILICORR_N_CONF; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(s_w + j * cols + nl);
      const float fj = f[k][j];
      z.x = fmaf(w.x, fj, z.x);
      z.y = fmaf(w.y, fj, z.y);
      z.z = fmaf(w.z, fj, z.z);
      z.w = fmaf(w.w, fj, z.w);
    }
    if constexpr (sizeof(TC1) == 2) {          // bf16 operand: tanh-based SiLU, 8-byte store
      uint2 u;
      u.x = bf16_pack2(silu_tanh(z.x), silu_tanh(z.y));
      u.y = bf16_pack2(silu_tanh(z.z), silu_tanh(z.w));
      *reinterpret_cast<uint2*>(c1 + node * D + n) = u;
    } else {
      *reinterpret_cast<float4*>(c1 + node * D + n) =
          make_float4(silu_f(z.x), silu_f(z.y), silu_f(z.z), silu_f(z.w));
    }
  }
}

// ----------------------------------------------------------------------------- RMSNorm
template <typename TY>
__global__ void rmsnorm_kernel(const float* __restrict__ x, int M, int D,
                               const float* __restrict__ gain, TY* __restrict__ y) {
  pdl_wait();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const float* xr = x + (size_t)row * D;
  float ss = 0.f;
  for (int i = lane; i < D; i += 32) ss += xr[i] * xr[i];
  ss = warp_sum(ss);
  const float r = rsqrtf(ss / (float)D + RMS_EPS);
  for (int i = lane; i < D; i += 32) st_elem(y, (size_t)row * D + i, xr[i] * r * gain[i]);
}

// fin[row] = [xf, xf * t_b] with xf = RMSNorm(x[row]) * gain: the x and x*t blocks of
// the fusion layer's input [x; t; x*t] (App. A); the t block is a per-sequence bias.
template <typename TY>
__global__ void fusion_input_kernel(const float* __restrict__ x, int M, int LK, int D,
                                    const float* __restrict__ gain, const float* __restrict__ t,
                                    TY* __restrict__ fin) {
  pdl_wait();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  const float* xr = x + (size_t)row * D;
  const float* tb = t + (size_t)(row / LK) * D;
  float ss = 0.f;
  for (int i = lane; i < D; i += 32) ss += xr[i] * xr[i];
  ss = warp_sum(ss);
  const float r = rsqrtf(ss / (float)D + RMS_EPS);
  for (int i = lane; i < D; i += 32) {
    const float xf = xr[i] * r * gain[i];
    st_elem(fin, (size_t)row * 2 * D + i, xf);
    st_elem(fin, (size_t)row * 2 * D + D + i, xf * tb[i]);
  }
}

// The unit out, in and anchor vectors, a warp per row: v / max(||v||, 1e-12). oi [N, 2d] holds a
// node's out and in vectors side by side (rows 2i and 2i + 1 here), anc [B, d] the anchors. Three
// launches that read their rows twice, word by word, before: 5 us each at one request, where
// this one takes 3.7 (cold); at 65,536 nodes of 512 the bytes bound both (80 us).
template <bool VEC>
__global__ void unit_vectors_kernel(const float* __restrict__ oi, const float* __restrict__ anc,
                                    int N, int B, int d, float* __restrict__ out,
                                    float* __restrict__ in, float* __restrict__ anchor) {
  pdl_wait();
  const long long row = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= 2ll * N + B) return;
  const float* src;
  float* dst;
  if (row < 2ll * N) {
    src = oi + (size_t)row * d;
    dst = (row & 1 ? in : out) + (size_t)(row >> 1) * d;
  } else {
    src = anc + (size_t)(row - 2ll * N) * d;
    dst = anchor + (size_t)(row - 2ll * N) * d;
  }
  float ss = 0.f;
  if (VEC && d <= 1024) {                     // the row stays in registers
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 4 * (lane + 32 * u);
      v[u] = i < d ? *reinterpret_cast<const float4*>(src + i) : make_float4(0.f, 0.f, 0.f, 0.f);
      ss = fmaf(v[u].x, v[u].x, fmaf(v[u].y, v[u].y, fmaf(v[u].z, v[u].z, fmaf(v[u].w, v[u].w, ss))));
    }
    const float inv = 1.0f / fmaxf(sqrtf(warp_sum(ss)), UNIT_EPS);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = 4 * (lane + 32 * u);
      if (i < d)
        *reinterpret_cast<float4*>(dst + i) =
            make_float4(v[u].x * inv, v[u].y * inv, v[u].z * inv, v[u].w * inv);
    }
    return;
  }
  for (int i = lane; i < d; i += 32) ss += src[i] * src[i];
  const float inv = 1.0f / fmaxf(sqrtf(warp_sum(ss)), UNIT_EPS);
  for (int i = lane; i < d; i += 32) dst[i] = src[i] * inv;
}

// ----------------------------------------------------------------------------- attention
// A CTA takes a block of queries of one (sequence, head): all L*K nodes attend to all L*K
// nodes (no mask), logits q.k / sqrt(hd) + dist[h, s_j - s_i + L - 1] + same[h] * 1{s_i == s_j}.
// qkv rows hold [q | k | v], each D wide, head h in columns [h*hd, (h+1)*hd).
//
// Bound by shared-memory reads, so a warp takes AQ = 4 queries at once and everything moves in
// 16-byte pieces: scores with a lane per key, four keys and four queries a lane (8 reads per 64
// products); P V with a lane per four columns (and, below 128-wide heads, per part of the
// keys), the four queries' probabilities of a key one piece (2 reads per 16 products). One
// query a warp and single words read twice per product: 128 nodes x 128 (sequence, head)
// pairs of 32, 45 us -> 22 us (cold).
// While all queries fit the GPU's warps at one each (few short sequences), a warp takes AQ = 1:
// the same sums, a quarter of the chain. Whole networks at D 256: two sequences of 8 nodes
// 85.1 -> 82.1 us, of 32 nodes 102.9 -> 99.6; one of 32 at D 64 59.4 -> 55.3. At two waves of
// CTAs AQ = 4 is ahead (one sequence of 256 nodes: 164, AQ = 1 172).

__device__ __forceinline__ void fma4(float& acc, const float4& a, const float4& b) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  acc = fmaf(a.w, b.w, acc);
}

template <typename TO, int AQ>
__global__ void __launch_bounds__(256)
attention_kernel(const float* __restrict__ qkv, int L, int K, int D, int n_heads, int q_per_cta,
                 const float* __restrict__ dist, const float* __restrict__ same,
                 TO* __restrict__ out) {
  pdl_wait();
  extern __shared__ __align__(16) float sm[];
  const int LK = L * K, hd = D / n_heads;
  const int b = blockIdx.x / n_heads, h = blockIdx.x % n_heads;
  const int q0 = blockIdx.y * q_per_cta, q1 = min(LK, q0 + q_per_cta);
  const int nw = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kld = hd + 4;                      // K rows a piece apart in banks
  float* Ks = sm;                              // [LK][hd + 4]
  float* Vs = Ks + (size_t)LK * kld;           // [LK][hd]
  float* Qw = Vs + (size_t)LK * hd;            // [nw][AQ][hd]
  float* Pw = Qw + (size_t)nw * AQ * hd;       // [nw][LK][AQ]
  float* s_dist = Pw + (size_t)nw * LK * AQ;   // [2L - 1]
  const size_t ld = 3 * (size_t)D;
  const float* base = qkv + (size_t)b * LK * ld + h * hd;
  const int hv = hd / 4;                       // 16-byte pieces per head row
#pragma unroll 4
  for (int i = threadIdx.x; i < LK * hv; i += blockDim.x) {
    const int j = i / hv, c = (i % hv) * 4;
    *reinterpret_cast<float4*>(Ks + j * kld + c) =
        *reinterpret_cast<const float4*>(base + j * ld + D + c);
    *reinterpret_cast<float4*>(Vs + j * hd + c) =
        *reinterpret_cast<const float4*>(base + j * ld + 2 * D + c);
  }
  for (int i = threadIdx.x; i < 2 * L - 1; i += blockDim.x)
    s_dist[i] = dist[(size_t)h * (2 * L - 1) + i];
  __syncthreads();
  const float scale = rsqrtf((float)hd);
  const float sh = same[h];
  float* q = Qw + (size_t)warp * AQ * hd;
  float* p = Pw + (size_t)warp * LK * AQ;
  auto load_p = [&](int j, float (&e)[AQ]) {
    if constexpr (AQ == 4) {
      const float4 v = *reinterpret_cast<const float4*>(p + 4 * j);
      e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
    } else {
      e[0] = p[j];
    }
  };
  auto store_p = [&](int j, const float (&e)[AQ]) {
    if constexpr (AQ == 4)
      *reinterpret_cast<float4*>(p + 4 * j) = make_float4(e[0], e[1], e[2], e[3]);
    else
      p[j] = e[0];
  };
  // P V: lane = columns 4 cg.., keys ks, ks + nks, ...
  const int cg = lane % hv, ks = lane / hv, nks = 32 / hv;
  for (int i0 = q0 + AQ * warp; i0 < q1; i0 += AQ * nw) {
    const int nq = min(AQ, q1 - i0);           // a short last group repeats its last query
    for (int i = lane; i < AQ * hv; i += 32)
      *reinterpret_cast<float4*>(q + 4 * i) = *reinterpret_cast<const float4*>(
          base + (size_t)(i0 + min(i / hv, nq - 1)) * ld + 4 * (i % hv));
    __syncwarp();
    int si[AQ];
    float mx[AQ];
#pragma unroll
    for (int a = 0; a < AQ; ++a) {
      si[a] = (i0 + min(a, nq - 1)) / K;
      mx[a] = -INFINITY;
    }
    for (int j0 = 0; j0 < LK; j0 += 128) {
      float s[4][AQ];
      const float* kr[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        kr[t] = Ks + min(j0 + lane + 32 * t, LK - 1) * kld;
#pragma unroll
        for (int a = 0; a < AQ; ++a) s[t][a] = 0.f;
      }
      for (int c = 0; c < hd; c += 4) {
        float4 qv[AQ];
#pragma unroll
        for (int a = 0; a < AQ; ++a) qv[a] = *reinterpret_cast<const float4*>(q + a * hd + c);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (AQ == 1 && j0 + 32 * t >= LK) break;      // no lane has a key there
          const float4 kv = *reinterpret_cast<const float4*>(kr[t] + c);
#pragma unroll
          for (int a = 0; a < AQ; ++a) fma4(s[t][a], qv[a], kv);
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int j = j0 + lane + 32 * t;
        if (j >= LK) continue;
        const int sj = j / K;
#pragma unroll
        for (int a = 0; a < AQ; ++a) {
          s[t][a] = s[t][a] * scale + s_dist[sj - si[a] + L - 1] + (si[a] == sj ? sh : 0.f);
          mx[a] = fmaxf(mx[a], s[t][a]);
        }
        store_p(j, s[t]);
      }
    }
    float sum[AQ];
#pragma unroll
    for (int a = 0; a < AQ; ++a) {
      mx[a] = warp_max(mx[a]);
      sum[a] = 0.f;
    }
    for (int j = lane; j < LK; j += 32) {      // each lane the keys it scored
      float e[AQ];
      load_p(j, e);
#pragma unroll
      for (int a = 0; a < AQ; ++a) {
        e[a] = __expf(e[a] - mx[a]);
        sum[a] += e[a];
      }
      store_p(j, e);
    }
    __syncwarp();
    float4 o[AQ];
#pragma unroll
    for (int a = 0; a < AQ; ++a) {
      sum[a] = 1.0f / warp_sum(sum[a]);
      o[a] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (ks < nks)
#pragma unroll 4
      for (int j = ks; j < LK; j += nks) {
        const float4 v = *reinterpret_cast<const float4*>(Vs + j * hd + 4 * cg);
        float w[AQ];
        load_p(j, w);
#pragma unroll
        for (int a = 0; a < AQ; ++a) {
          o[a].x = fmaf(w[a], v.x, o[a].x);
          o[a].y = fmaf(w[a], v.y, o[a].y);
          o[a].z = fmaf(w[a], v.z, o[a].z);
          o[a].w = fmaf(w[a], v.w, o[a].w);
        }
      }
#pragma unroll
    for (int a = 0; a < AQ; ++a) {
      float4 r = o[a];
      for (int k = 1; k < nks; ++k) {          // the parts of the keys, in order
        const int src = cg + k * hv;
        r.x += __shfl_sync(0xffffffffu, o[a].x, src);
        r.y += __shfl_sync(0xffffffffu, o[a].y, src);
        r.z += __shfl_sync(0xffffffffu, o[a].z, src);
        r.w += __shfl_sync(0xffffffffu, o[a].w, src);
      }
      if (ks == 0 && a < nq) {
        TO* dst = out + ((size_t)b * LK + i0 + a) * D + h * hd + 4 * cg;
        st_elem(dst, 0, r.x * sum[a]);
        st_elem(dst, 1, r.y * sum[a]);
        st_elem(dst, 2, r.z * sum[a]);
        st_elem(dst, 3, r.w * sum[a]);
      }
    }
    __syncwarp();
  }
}

// floats of shared memory beside s_dist, for `warps` warps
size_t attention_floats(int LK, int hd, int warps) {
  return (size_t)LK * (2 * hd + 4) + (size_t)warps * 4 * (hd + LK);     // AQ <= 4
}

}  // namespace

// What the CUDA-core attention core may take of shared memory decides which heads exist (the
// limit lies at 200 KB of this); launch_attention takes as many warps as then fit.
size_t attention_smem_bytes(int LK, int hd, int warps) {
  return sizeof(float) * ((size_t)LK * (hd + 1) + (size_t)LK * hd + (size_t)warps * hd +
                          (size_t)warps * LK);
}

bool gemm_rows_supported(const GemmArgs& g) {
  return g.a_dt == LILICORR_F32 && g.M > 0 && g.N > 0 && g.Kd % 8 == 0 && g.lda % 4 == 0 &&
         g.ldw % 8 == 0 && (reinterpret_cast<uintptr_t>(g.A) & 15) == 0 &&
         (reinterpret_cast<uintptr_t>(g.W) & 15) == 0;
}

lilicorr_status_t launch_gemm_rows(const GemmArgs& g, cudaStream_t st, const GemmArgs* g1) {
  if (!gemm_rows_supported(g) || (g1 && !gemm_rows_supported(*g1))) return LILICORR_ERR_SHAPE;
  if (g1 && (g.c_dt != LILICORR_F32 || g1->c_dt != LILICORR_F32)) {
    LL_TRY(launch_gemm_rows(g, st));
    return launch_gemm_rows(*g1, st);
  }
  const dim3 grid(ceil_div(g1 ? max(g.N, g1->N) : g.N, GR_N), ceil_div(g.M, GR_M), g1 ? 2 : 1);
  if (g1)
    return g.w_dt == LILICORR_F32
               ? launch_k(gemm_rows_kernel<float, float, true>, grid, GR_THREADS, 0, st, g, *g1)
               : launch_k(gemm_rows_kernel<__nv_bfloat16, float, true>, grid, GR_THREADS, 0, st, g, *g1);
  if (g.w_dt == LILICORR_F32) {
    if (g.c_dt == LILICORR_F32)
      return launch_k(gemm_rows_kernel<float, float, false>, grid, GR_THREADS, 0, st, g, g);
    return launch_k(gemm_rows_kernel<float, __nv_bfloat16, false>, grid, GR_THREADS, 0, st, g, g);
  }
  if (g.c_dt == LILICORR_F32)
    return launch_k(gemm_rows_kernel<__nv_bfloat16, float, false>, grid, GR_THREADS, 0, st, g, g);
  return launch_k(gemm_rows_kernel<__nv_bfloat16, __nv_bfloat16, false>, grid, GR_THREADS, 0, st, g, g);
}

lilicorr_status_t launch_gemm_skinny(const GemmArgs& g, cudaStream_t st, const GemmArgs* g1) {
  if (g.M == 0 || g.N == 0) return LILICORR_OK;
  // two products in one launch: fp32 in and out, rows in whole groups of eight
  if (g1 && (g.a_dt != LILICORR_F32 || g.c_dt != LILICORR_F32 || g1->c_dt != LILICORR_F32 ||
             g.Kd % 8 || g.lda % 8 || g.ldw % 8 || g1->ldw % 8)) {
    LL_TRY(launch_gemm_skinny(g, st));
    return launch_gemm_skinny(*g1, st);
  }
  if ((g.Kd % 8) || (g.lda % 8) || (g.ldw % 8)) return launch_gemm_simt(g, st);
  if (g.a_dt == LILICORR_F32) return skinny_dispatch_w<float>(g, g1, st);
  return skinny_dispatch_w<__nv_bfloat16>(g, g1, st);
}

// CTAs per tile of the split kernel: as many as still are one wave with a step of Kd each; eight
// only for few tiles, since 16 clusters of eight did not run at once (256 x 256 x 512: 11.5 us,
// four ways 7.6).
int gemm_simt_ways(const GemmArgs& g) {
  if (g.a_dt != LILICORR_F32 || g.M <= 0 || g.N <= 0 || !gemm_simt_vec(g)) return 0;
  const long long tiles = (long long)ceil_div(g.N, GB_N) * ceil_div(g.M, GB_M);
  const int steps = ceil_div(g.Kd, GB_K);
  int ways = tiles <= 8 ? 8 : 4;
  while (ways > 1 && (tiles * ways > num_sms() || steps < ways)) ways /= 2;
  return ways > 1 ? ways : 0;
}

lilicorr_status_t launch_gemm_simt_split(const GemmArgs& g, cudaStream_t st) {
  const int ways = gemm_simt_ways(g);
  if (!ways) return LILICORR_ERR_SHAPE;
  const dim3 grid(ceil_div(g.N, GB_N), ceil_div(g.M, GB_M));
  return g.w_dt == LILICORR_F32 ? gemm_split_dispatch_c<float>(g, grid, ways, st)
                                : gemm_split_dispatch_c<__nv_bfloat16>(g, grid, ways, st);
}

lilicorr_status_t launch_gemm_simt(const GemmArgs& g, cudaStream_t st) {
  if (g.M == 0 || g.N == 0) return LILICORR_OK;
  dim3 grid(ceil_div(g.N, GB_N), ceil_div(g.M, GB_M));
  if (g.a_dt == LILICORR_F32) return gemm_dispatch_w<float>(g, grid, st);
  return gemm_dispatch_w<__nv_bfloat16>(g, grid, st);
}

lilicorr_status_t launch_target_norm(const void* T, lilicorr_dtype_t dt, int B, int n_tgt, int H,
                                     const float* gain, void* tn, lilicorr_dtype_t tn_dt,
                                     cudaStream_t st) {
  if (B == 0) return LILICORR_OK;
  if (dt == LILICORR_F32 && tn_dt == LILICORR_F32)
    LL_TRY(launch_k(target_norm_kernel<float, float>, B, TN_THREADS, 0, st, 
        static_cast<const float*>(T), n_tgt, H, gain, static_cast<float*>(tn)));
  else if (dt == LILICORR_BF16 && tn_dt == LILICORR_F32)
    LL_TRY(launch_k(target_norm_kernel<__nv_bfloat16, float>, B, TN_THREADS, 0, st, 
        static_cast<const __nv_bfloat16*>(T), n_tgt, H, gain, static_cast<float*>(tn)));
  else if (dt == LILICORR_BF16)
    LL_TRY(launch_k(target_norm_kernel<__nv_bfloat16, __nv_bfloat16>, B, TN_THREADS, 0, st, 
        static_cast<const __nv_bfloat16*>(T), n_tgt, H, gain, static_cast<__nv_bfloat16*>(tn)));
  else
    return LILICORR_ERR_DTYPE;
  return LILICORR_OK;
}

lilicorr_status_t launch_node_build(const lilicorr_head* h, int B, const int32_t* ids,
                                    const float* logp, const float* hproj, void* c1,
                                    lilicorr_dtype_t c1_dt, float* x, uint32_t* status,
                                    cudaStream_t st) {
  const lilicorr_head_desc& d = h->desc;
  if (B == 0) return LILICORR_OK;
  const float* fold = static_cast<const float*>(h->fold);
  // Few slot rows: their columns over several CTAs, at least 128 each, until two an SM (one
  // request of 15 slots x 8 candidates x 1024: 15 CTAs of eight rounds of gathers, 14.1 us cold,
  // to 120 of one, 5.8). Many rows keep one CTA each, which stages the confidence weights once.
  // Wide heads are split for any number of rows: a CTA stages 24 bytes a column in the 48 KB that a
  // launch may have unasked.
  const int parts = max(ceil_div(d.D, NODE_COLS_MAX),
                        min(ceil_div(2 * num_sms(), B * d.L), d.D / 128));
  const int cols = ceil_div(ceil_div(d.D, parts), 4) * 4;
  const dim3 grid(B * d.L, ceil_div(d.D, cols));
  const size_t smem = sizeof(float) * (LILICORR_N_CONF + 1) * cols;
  if (c1_dt == LILICORR_F32)
    return launch_k(node_build_kernel<float>, grid, 256, smem, st, d.L, d.K, d.D, cols, d.V, ids,
                    logp, fold, hproj, h->slot, h->rank, h->conf1_w, h->conf1_b,
                    static_cast<float*>(c1), x, status);
  return launch_k(node_build_kernel<__nv_bfloat16>, grid, 256, smem, st, d.L, d.K, d.D, cols, d.V,
                  ids, logp, fold, hproj, h->slot, h->rank, h->conf1_w, h->conf1_b,
                  static_cast<__nv_bfloat16*>(c1), x, status);
}

lilicorr_status_t launch_rmsnorm(const float* x, int M, int D, const float* gain, void* y,
                                 lilicorr_dtype_t y_dt, cudaStream_t st) {
  if (M == 0) return LILICORR_OK;
  const int grid = ceil_div(M, 8);
  if (y_dt == LILICORR_F32)
    LL_TRY(launch_k(rmsnorm_kernel<float>, grid, 256, 0, st, x, M, D, gain, static_cast<float*>(y)));
  else
    LL_TRY(launch_k(rmsnorm_kernel<__nv_bfloat16>, grid, 256, 0, st, x, M, D, gain,
                                                        static_cast<__nv_bfloat16*>(y)));
  return LILICORR_OK;
}

lilicorr_status_t launch_fusion_input(const float* x, int B, int LK, int D, const float* gain,
                                      const float* t, void* fin, lilicorr_dtype_t dt,
                                      cudaStream_t st) {
  const int M = B * LK;
  if (M == 0) return LILICORR_OK;
  const int grid = ceil_div(M, 8);
  if (dt == LILICORR_F32)
    LL_TRY(launch_k(fusion_input_kernel<float>, grid, 256, 0, st, x, M, LK, D, gain, t, static_cast<float*>(fin)));
  else
    LL_TRY(launch_k(fusion_input_kernel<__nv_bfloat16>, grid, 256, 0, st, x, M, LK, D, gain, t,
                                                             static_cast<__nv_bfloat16*>(fin)));
  return LILICORR_OK;
}

lilicorr_status_t launch_unit_vectors(const float* oi, const float* anc, int N, int B, int d,
                                      float* out, float* in, float* anchor, cudaStream_t st) {
  const long long rows = 2ll * N + B;
  if (rows == 0) return LILICORR_OK;
  // d is a multiple of 8 and oi and anc are the workspace's; the caller's vectors may lie anywhere
  const bool vec = aligned16(out) && aligned16(in) && aligned16(anchor);
  return launch_k(vec ? unit_vectors_kernel<true> : unit_vectors_kernel<false>, ceil_div(rows, 8),
                  256, 0, st, oi, anc, N, B, d, out, in, anchor);
}

lilicorr_status_t launch_attention(const float* qkv, int B, int L, int K, int D, int n_heads,
                                   const float* dist, const float* same, void* out,
                                   lilicorr_dtype_t out_dt, cudaStream_t st) {
  if (B == 0) return LILICORR_OK;
  const int LK = L * K, hd = D / n_heads;
  // the most warps whose queries and probabilities fit beside K and V (every head that
  // exists leaves room for two)
  const size_t most = SMEM_PER_BLOCK_MAX - 2 * LILICORR_MAX_L * sizeof(float);
  int warps = 8;
  while (warps > 2 && attention_floats(LK, hd, warps) * sizeof(float) > most) warps /= 2;
  // one query a warp while that is one wave of CTAs, else four
  const int aq = (long long)B * n_heads * ceil_div(LK, warps) <= num_sms() ? 1 : 4;
  // More (sequence, head) pairs than SMs: no warps without a query, so that more CTAs fit an SM
  // (whole networks of width 64 and 1024 sequences of 4, 8, 16, 32 nodes: 256 -> 155, 328 -> 233,
  // 442 -> 396, 721 -> 725 us; one query a warp as before AQ = 4: 168, 261, 458, 839). In one wave
  // the idle warps help to bring K and V (16 sequences of 12 nodes, width 256: 115, without 120).
  if ((long long)B * n_heads > num_sms()) warps = min(warps, ceil_div(LK, aq));
  const size_t smem = (attention_floats(LK, hd, warps) + 2 * L - 1) * sizeof(float);
  // split the queries of a (sequence, head) over CTAs until the grid covers the GPU; each warp
  // takes whole groups of AQ
  int qblocks = aq == 1 ? ceil_div(LK, warps) : ceil_div(4 * num_sms(), B * n_heads);
  qblocks = max(1, min(qblocks, ceil_div(LK, aq * warps)));
  const int q_per_cta = ceil_div(ceil_div(LK, qblocks), aq) * aq;
  qblocks = ceil_div(LK, q_per_cta);
  const dim3 grid(B * n_heads, qblocks);
  const auto launch = [&](auto q, auto* to) -> lilicorr_status_t {
    auto* kern = attention_kernel<std::remove_pointer_t<decltype(to)>, decltype(q)::value>;
    static bool cfg[64] = {false};             // one per kernel: q and to name it
    LL_TRY(allow_max_dynamic_smem(kern, cfg));
    return launch_k(kern, grid, warps * 32, smem, st, qkv, L, K, D, n_heads, q_per_cta, dist, same,
                    to);
  };
  const std::integral_constant<int, 1> q1;
  const std::integral_constant<int, 4> q4;
  if (out_dt == LILICORR_F32) {
    float* to = static_cast<float*>(out);
    return aq == 1 ? launch(q1, to) : launch(q4, to);
  }
  __nv_bfloat16* to = static_cast<__nv_bfloat16*>(out);
  return aq == 1 ? launch(q1, to) : launch(q4, to);
}

}  // namespace lilicorr
