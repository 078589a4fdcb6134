// fp32 GEMM D[M][N] = A[M][K] . W[N][K]^T of the fp32 model (exact-token
// parity mode), on packed FP32 FMAs (fma.rn.f32x2).
//
// What bounds it: a decode step of this mode has 8-64 rows, so each product
// is a stream of W with M FMAs per weight: at 64 rows the FMA pipes (about
// 37 TFMA/s) take as long as HBM, below that HBM and the launch chain do.
// Tile and split, and why:
//  - a CTA covers 16 RG rows x 64 columns, a warp 16 rows x 64 columns, a lane 8
//    rows x 4 columns (half a warp shares its rows): 12 16-byte shared-memory reads
//    per 64 FFMA2.  Each read takes four cycles of the 128 B/clk that shared memory
//    returns, broadcast or not: 16 rows x 2 columns per lane needed 18;
//  - FFMA2 pairs run along k (even and odd k in the two halves), the order in
//    which both operands lie in memory: no transpose, and two shorter sums;
//  - the KG warps that share a row group each take their part of every
//    64-wide K stage, and K is split over a cluster of up to 8 CTAs while every
//    cluster runs at once; partials meet in shared memory (DSMEM across the
//    cluster) in a fixed order: deterministic, no workspace, no atomics;
//  - four cp.async stages; the first stages' W rows are read before the
//    dependency wait (weights do not change during a step).
// Measured at 64 rows, per launch with its launch latency (about 5 us),
// before -> now (before: 32 x 128 tiles, one row per lane, no K split, 12 to
// 48 CTAs): 2304 x 768 170 -> 16 us, 768 x 768 159 -> 14, 3072 x 768 163 ->
// 21, 768 x 3072 613 -> 22, head 30,522 x 768 (32 rows) 195 -> 60; two decode calls
// of the 768-wide 12-layer model, 8 sequences at k = 4, and their logits 29.6
// -> 1.72 ms.  What is left is the first loads, the cluster barriers and the
// reduction.  Sixteen warps per CTA (twice the K groups) measured slower (1.92 ms:
// twice the partials to sum), plain FFMA as well (1.77 ms: issue slots).
#include <algorithm>

#include "kf_tc.cuh"

namespace kf {

namespace {
constexpr int kFN = 64;              // columns per CTA
constexpr int kFK = 64;              // K per stage
constexpr int kFLd = kFK + 4;        // floats per row: lanes 4 banks apart, conflict-free 16-byte reads
constexpr int kFStages = 4;

__host__ __device__ constexpr int f32_kg(int RG) { return RG == 1 ? 8 : RG == 2 ? 4 : 2; }
__host__ __device__ constexpr int f32_stage_floats(int RG) { return (16 * RG + kFN) * kFLd; }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool in) {
  const int n = in ? 16 : 0;         // 0: zero-fill, src not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
// acc += {a0 w0, a1 w1}
__device__ __forceinline__ void fma2(float2& acc, float a0, float a1, float w0, float w1) {
  acc = f2_split(fma_f2(f2(a0, a1), f2(w0, w1), f2(acc.x, acc.y)));
}
// four consecutive columns of one row
__device__ __forceinline__ void epi_f32_vec4(const Epi& e, int row, int col, float4 v, int N) {
  switch (e.kind) {
    case EPI_STORE: epi_vec4<float, EPI_STORE>(e, row, col, v, N); break;
    case EPI_BIAS_GELU: epi_vec4<float, EPI_BIAS_GELU>(e, row, col, v, N); break;
    case EPI_RESID: epi_vec4<float, EPI_RESID>(e, row, col, v, N); break;
    case EPI_NOISE_OUT: epi_vec4<float, EPI_NOISE_OUT>(e, row, col, v, N); break;
    case EPI_LOGITS: epi_vec4<float, EPI_LOGITS>(e, row, col, v, N); break;
    case EPI_STORE_F32: epi_vec4<float, EPI_STORE_F32>(e, row, col, v, N); break;
  }
}
}  // namespace

template <int RG>
__global__ void __launch_bounds__(RG * f32_kg(RG) * 32) k_gemm_f32(GemmDesc g, int kps, int splits) {
  constexpr int KG = f32_kg(RG), BM = 16 * RG, NT = RG * KG * 32;
  constexpr int KW = kFK / KG;                       // a warp's k per stage
  constexpr int SF = f32_stage_floats(RG);
  static_assert(KG * BM * kFLd <= kFStages * SF, "the partials reuse the stages");
  extern __shared__ __align__(16) float fsm[];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rg = warp % RG, kg = warp / RG;
  const int col0 = blockIdx.x * kFN, row0 = blockIdx.y * BM;
  const int k0 = blockIdx.z * kps, k1 = min(g.K, k0 + kps);
  const int nst = (k1 - k0 + kFK - 1) / kFK;
  const float* A = static_cast<const float*>(g.A);
  const float* W = static_cast<const float*>(g.W);
  const uint32_t sbase = smem_u32(fsm);

  // stage i: each thread copies the same 16-byte column of every NT / 16-th row
  constexpr int kC = kFK / 4, kStep = NT / kC;        // 16-byte columns, rows per pass
  const int lr = t / kC, lk = (t % kC) * 4;
  const uint32_t ldst = sbase + (uint32_t)(lr * kFLd + lk) * 4;
  auto load = [&](int i, const float* src, int ld, int rows, int limit, int at) {
    const uint32_t dst = ldst + (uint32_t)((i % kFStages) * SF + at * kFLd) * 4;
    const int k = i * kFK;
    const bool ink = k0 + lk + k < k1;
    src += k;
#pragma unroll
    for (int r = 0; r < rows; r += kStep) {
      if (rows % kStep && r + lr >= rows) break;
      const bool in = ink && r + lr < limit;
      cp_async16(dst + (uint32_t)(r * kFLd) * 4, in ? src : g.W, in);
      src += (size_t)kStep * ld;
    }
  };
  const float* wsrc = W + (size_t)(col0 + lr) * g.ldw + k0 + lk;    // (not read past N, M or k1)
  const float* asrc = A + (size_t)(row0 + lr) * g.lda + k0 + lk;
  auto load_w = [&](int i) { load(i, wsrc, g.ldw, kFN, g.N - col0, BM); };
  auto load_a = [&](int i) { load(i, asrc, g.lda, BM, g.M - row0, 0); };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

  // weights are constant during a step: read ahead of the dependency
  for (int i = 0; i < kFStages - 1; ++i)
    if (i < nst) load_w(i);
  pdl_wait();
  for (int i = 0; i < kFStages - 1; ++i) {
    if (i < nst) load_a(i);
    commit();                                        // the first group holds the W rows above too
  }

  // lanes 0..15 take the warp's first 8 rows, lanes 16..31 the other 8; a lane
  // has columns l, l + 16, l + 32, l + 48
  constexpr int R = 8, C = 4;
  const int half = lane >> 4, l16 = lane & 15;
  float2 acc[R][C];                                  // even k, odd k
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c) acc[r][c] = make_float2(0.f, 0.f);
  for (int i = 0; i < nst; ++i) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kFStages - 2) : "memory");
    __syncthreads();                                 // stage i is here; stage i - 1 has been read
    if (i + kFStages - 1 < nst) {
      load_w(i + kFStages - 1);
      load_a(i + kFStages - 1);
    }
    commit();
    const float* as = fsm + (i % kFStages) * SF + (rg * 16 + half * R) * kFLd + kg * KW;
    const float* ws = fsm + (i % kFStages) * SF + (BM + l16) * kFLd + kg * KW;
    auto ldw = [&](int k, float4* w) {
#pragma unroll
      for (int c = 0; c < C; ++c) w[c] = *reinterpret_cast<const float4*>(ws + 16 * c * kFLd + k);
    };
    // two rows' A reads run ahead of the FMAs of the two before them, and an
    // accumulator's two FMAs lie eight instructions apart
    float4 a[2][2], w[C], wn[C];
#pragma unroll
    for (int r = 0; r < 2; ++r) a[0][r] = *reinterpret_cast<const float4*>(as + r * kFLd);
    ldw(0, w);
#pragma unroll 1
    for (int k = 0; k < KW; k += 4) {
      const int kn = k + 4 < KW ? k + 4 : 0;         // (the last read is not used)
      ldw(kn, wn);
#pragma unroll
      for (int b = 0; b < R / 2; ++b) {
        const int rn = (b + 1) % (R / 2) * 2;
#pragma unroll
        for (int r = 0; r < 2; ++r)
          a[(b + 1) & 1][r] = *reinterpret_cast<const float4*>(as + (rn + r) * kFLd + (b == R / 2 - 1 ? kn : k));
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int c = 0; c < C; ++c) fma2(acc[2 * b + r][c], a[b & 1][r].x, a[b & 1][r].y, w[c].x, w[c].y);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int c = 0; c < C; ++c) fma2(acc[2 * b + r][c], a[b & 1][r].z, a[b & 1][r].w, w[c].z, w[c].w);
      }
#pragma unroll
      for (int c = 0; c < C; ++c) w[c] = wn[c];
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // partials [KG][BM][kFLd]: even + odd k
  float* P = fsm + (size_t)(kg * BM + rg * 16 + half * R) * kFLd + l16;
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c)
      P[r * kFLd + 16 * c] = acc[r][c].x + acc[r][c].y;
  if (splits > 1) cluster_sync();
  else __syncthreads();
  // CTA q of the cluster sums rows q, q + S, ...: splits in order, then warps
  const int S = splits, q = splits > 1 ? (int)cluster_rank() : 0;
  auto sum4 = [&](int rr, int c) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < S; ++s)
#pragma unroll
      for (int w = 0; w < KG; ++w) {
        const uint32_t at = sbase + (uint32_t)((w * BM + rr) * kFLd + c) * 4;
        v = add4(v, S > 1 ? ld_dsmem4(at, (uint32_t)s)
                          : *reinterpret_cast<const float4*>(fsm + (w * BM + rr) * kFLd + c));
      }
    return v;
  };
  const int mine = (BM - q + S - 1) / S;
  if (g.epi.kind == EPI_HEAD) {
    for (int i = t; i < mine * 2; i += NT) {         // one 32-id record each
      const int rr = q + S * (i >> 1), c = (i & 1) * 32;
      if (row0 + rr >= g.M || col0 + c >= g.N) continue;
      float v[32];
#pragma unroll
      for (int j = 0; j < 8; ++j) *reinterpret_cast<float4*>(v + 4 * j) = sum4(rr, c + 4 * j);
      epi_run32<float>(g.epi, row0 + rr, col0 + c, v, g.N);
    }
  } else {
    for (int i = t; i < mine * (kFN / 4); i += NT) {
      const int rr = q + S * (i / (kFN / 4)), c = (i % (kFN / 4)) * 4;
      if (row0 + rr >= g.M || col0 + c >= g.N) continue;
      epi_f32_vec4(g.epi, row0 + rr, col0 + c, sum4(rr, c), g.N);
    }
  }
  if (splits > 1) cluster_sync();                    // the partials stay until all have read them
}

template <int RG>
static int launch_rg(const GemmDesc& g, cudaStream_t s) {
  constexpr int KG = f32_kg(RG);
  const int n_tiles = ceil_div(g.N, kFN), m_tiles = ceil_div(g.M, 16 * RG);
  const int st = ceil_div(g.K, kFK);
  // K over a cluster of up to 8 CTAs, one stage each at least, while all
  // clusters run at once with an SM per CTA (a cluster lies within a GPC: 48 of 3
  // do not fit 152 SMs, and the last two doubled up on their SMs: 3072 x 768 at 64
  // rows 24 us at 3 splits, 16 at 2)
  int splits = std::min(8, st);
  while (splits > 1 && n_tiles * m_tiles > active_clusters(splits)) --splits;
  const int kps = ceil_div(st, splits) * kFK;
  splits = ceil_div(g.K, kps);                       // no empty splits
  // within a wave an SM per CTA (more than half of its shared memory): two on one
  // SM leave another idle, and dependent launch makes that common, the next
  // kernel's CTAs arriving while some SMs are still busy (a step 2.14 -> 1.79 ms
  // for two calls); past a wave two per SM hide each other's loads
  const size_t need = (size_t)kFStages * f32_stage_floats(RG) * 4;
  const bool alone = n_tiles * m_tiles * splits <= device_sms();
  const size_t smem = alone ? std::max(need, (size_t)116 * 1024) : need;
  static PerDevice attr;
  set_smem_attr(attr, k_gemm_f32<RG>, smem);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles, m_tiles, splits);
  cfg.blockDim = dim3(RG * KG * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (splits > 1) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = 1;
    at[na].val.clusterDim.y = 1;
    at[na].val.clusterDim.z = splits;
    ++na;
  }
  if (g_pdl) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = at;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, k_gemm_f32<RG>, g, kps, splits) == cudaSuccess ? 0 : -1;
}

int launch_gemm_f32(const GemmDesc& g, cudaStream_t s) {
  if (g.M == 0 || g.N == 0) return 0;
  // 16-byte rows and groups of four columns: every product of the fp32 model
  // (its widths are multiples of 32)
  if (g.K % 4 || g.N % 4 || g.lda % 4 || g.ldw % 4 || (reinterpret_cast<uintptr_t>(g.A) & 15) ||
      (reinterpret_cast<uintptr_t>(g.W) & 15))
    return -1;
  // rows of the tile: the fewest 16-row groups that hold M (64 at most)
  switch (std::min(4, ceil_div(g.M, 16))) {
    case 1: return launch_rg<1>(g, s);
    case 2: return launch_rg<2>(g, s);
    case 3: return launch_rg<3>(g, s);
  }
  return launch_rg<4>(g, s);
}

}  // namespace kf
