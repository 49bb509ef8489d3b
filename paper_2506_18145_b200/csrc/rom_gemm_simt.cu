// Plain fp32-FMA tiled GEMM, C[M,N] = A[M,Kd] * B[e][N,Kd]^T with fp32 accumulation.
// gemm_f32 is the projection path of the fp32 configuration (a tf32 tensor path would not hold the 1e-4 tolerance); gemm_simt, under
// ROM_FLAG_SIMT_GEMM, a bisecting aid for the bf16 tensor path.
#include "rom_internal.cuh"

namespace rom {
namespace {

constexpr int BM = 64, BN = 64, BK = 16;

__device__ __forceinline__ void load_vec(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 q = __ldg(reinterpret_cast<const uint4*>(p));
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void load_vec(const float* p, float (&v)[4]) {
  const float4 q = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}

template <typename T>
__device__ __forceinline__ void epi_store_scalar(const Epilogue& ep, int m, int n, float v) {
  switch (ep.mode) {
    case EPI_STORE:
      reinterpret_cast<T*>(ep.C)[(size_t)m * ep.ldc + n] = from_f32<T>(v);
      break;
    case EPI_INPROJ:
      reinterpret_cast<T*>(ep.C)[(size_t)m * ep.ldc + n] = from_f32<T>(n >= ep.R ? silu_f(v) : v);
      break;
    case EPI_XPROJ:
      if (n < ep.R) reinterpret_cast<T*>(ep.C)[(size_t)m * ep.R + n] = from_f32<T>(v);
      else if (n < ep.R + ep.N) ep.Bm[(size_t)m * ep.N + (n - ep.R)] = v;
      else ep.Cm[(size_t)m * ep.N + (n - ep.R - ep.N)] = v;
      break;
    case EPI_F32:
      reinterpret_cast<float*>(ep.C)[(size_t)m * ep.ldc + n] = v;
      break;
    default:
      reinterpret_cast<T*>(ep.C)[(size_t)m * ep.ldc + n] = from_f32<T>(softplus_f(v + (ep.bias ? ep.bias[n] : 0.0f)));
      break;
  }
}

template <typename T>
__global__ void __launch_bounds__(256)
gemm_simt(const T* __restrict__ A, int lda, const T* __restrict__ Bw, int ldb, int64_t b_expert_stride,
          int M_max, int N, int Kd, const int32_t* __restrict__ tile_expert, const int32_t* __restrict__ num_m_tiles_dev,
          Epilogue ep) {
  pdl_sync();
  __shared__ float As[BK][BM + 1];
  __shared__ float Bs[BK][BN + 1];
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  int M = M_max;
  if (num_m_tiles_dev) M = min(M_max, *num_m_tiles_dev * kTileM);
  if (m0 >= M) return;
  const T* Bp = Bw;
  if (tile_expert) {
    const int e = tile_expert[m0 / kTileM];
    if (e < 0) return;
    Bp = Bw + (size_t)e * b_expert_stride;
  }
  const int tid = threadIdx.x;
  const int ty = tid / 16, tx = tid % 16;
  float acc[4][4] = {};
  // each thread brings 4 elements of the A tile and 4 of the B tile per K block; the next block's elements are
  // requested before the current block is multiplied, so the global-memory latency overlaps the arithmetic
  float pa[4], pb[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = tid + 256 * j;
      const int r = i / BK, k = i % BK;
      const int m = m0 + r, n = n0 + r, kk = k0 + k;
      pa[j] = (m < M && kk < Kd) ? to_f32(A[(size_t)m * lda + kk]) : 0.0f;
      pb[j] = (n < N && kk < Kd) ? to_f32(Bp[(size_t)n * ldb + kk]) : 0.0f;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < Kd; k0 += BK) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = tid + 256 * j;
      As[i % BK][i / BK] = pa[j];
      Bs[i % BK][i / BK] = pb[j];
    }
    __syncthreads();
    if (k0 + BK < Kd) fetch(k0 + BK);
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[k][ty * 4 + i]; b[i] = Bs[k][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n < N) epi_store_scalar<T>(ep, m, n, acc[i][j]);
    }
  }
}

// fp32 storage: C[M,N] = A[M,Kd] * B[e][N,Kd]^T on cp.async stages.  Operand rows lie in shared memory as in global (contracted
// index innermost, pitch padded so that eight rows fall into different banks); a thread owns TM x TN outputs on rows and columns
// (BM / TM) and (BN / TN) apart and takes four contracted elements of each per step.
//   <128, 128, 8, 8, 1, 16>: shared-memory reads and FMAs in balance; for grids that fill the GPU.
//   <32, 32, 4, 4, 4, 64>: the contracted index of a stage is split over four thread groups, so that a small product has four
//     times the blocks' worth of threads in flight and a quarter of the serial steps (256 rows x 1024 columns x 256: the 64 x 64
//     register-staged kernel took 28 us, waiting for one 16-wide stage after another).  <32, 32, 4, 4, 8, 128>, <16, 16, 2, 4, 8, 128>: see
//     launch_gemm_simt.
// TO_TOKENS (EPI_OUTPROJ; top-1): a row leaves, times its gate, at its token's position (no pass for the combine: 256 tokens of 256 57.0 -> 54.9 us
// a layer).  An instance of its own, its rows' tokens and gates read ahead of the stores: as one more output op of the stores above it
// takes every product in 128 x 128 tiles a quarter longer (In Proj of 4000 tokens of 512: 288 -> 361 us; the layer 725 -> 804, now 711).
template <int BM, int BN, int TM, int TN, int KS, int BKF, bool TO_TOKENS>
__global__ void __launch_bounds__(BM / TM * (BN / TN) * KS)
gemm_f32(const float* __restrict__ A, int lda, const float* __restrict__ Bw, int ldb, int64_t b_expert_stride, int M_max, int N, int Kd,
         const int32_t* __restrict__ tile_expert, const int32_t* __restrict__ num_m_tiles_dev, const int32_t* __restrict__ assign_of_row, Epilogue ep) {
  pdl_sync();
  constexpr int TY = BM / TM, TX = BN / TN, GT = TY * TX, NT = GT * KS, PITCH = BKF + 4, STAGES = 3, KG = BKF / KS;
  extern __shared__ __align__(16) float smf[];
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  // (requested together: one after another they cost a small product three trips to the L2 before its first operand)
  const int nmt = num_m_tiles_dev ? __ldcg(num_m_tiles_dev) : 0, e = tile_expert ? __ldcg(tile_expert + m0 / kTileM) : 0;
  const int as = tile_expert && assign_of_row ? __ldcg(assign_of_row + m0) : 0;
  const int M = num_m_tiles_dev ? min(M_max, nmt * kTileM) : M_max;
  if (m0 >= M || e < 0 || as < 0) return;      // a segment's padding is at its end: nothing but padding here, nobody reads it
  const float* Bp = Bw + (size_t)e * b_expert_stride;
  const int tid = threadIdx.x, kg = tid / GT, tx = tid % GT % TX, ty = tid % GT / TX;
  auto fetch = [&](int k0, int stage) {
    float* sa = smf + stage * (BM + BN) * PITCH;
    float* sb = sa + BM * PITCH;
    constexpr int VR = BKF / 4;
#pragma unroll
    for (int i = tid; i < (BM + BN) * VR; i += NT) {
      const int r = i / VR, k = (i - r * VR) * 4;
      const bool isA = r < BM;
      const int row = isA ? m0 + r : n0 + r - BM;
      const bool ok = (isA ? row < M : row < N) && k0 + k < Kd;
      const float* src = ok ? (isA ? A + (size_t)row * lda : Bp + (size_t)row * ldb) + k0 + k : A;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared((isA ? sa + r * PITCH : sb + (r - BM) * PITCH) + k);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int n_k = (Kd + BKF - 1) / BKF;
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < n_k) fetch(s * BKF, s);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[TM][TN] = {};
  for (int kb = 0; kb < n_k; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();
    if (kb + STAGES - 1 < n_k) fetch((kb + STAGES - 1) * BKF, (kb + STAGES - 1) % STAGES);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    const float* sa = smf + (kb % STAGES) * (BM + BN) * PITCH + kg * KG;
    const float* sb = sa + BM * PITCH;
#pragma unroll
    for (int k = 0; k < KG; k += 4) {
      float4 a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(sa + (ty + i * TY) * PITCH + k);
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = *reinterpret_cast<const float4*>(sb + (tx + j * TX) * PITCH + k);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
  }
  if (KS > 1) {
    // the groups' partial sums, added in group order
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) smf[(kg * BM + ty + i * TY) * (BN + 1) + tx + j * TX] = acc[i][j];
    __syncthreads();
    for (int i = tid; i < BM * BN; i += NT) {
      const int r = i / BN, c = i % BN;
      float v = 0.0f;
#pragma unroll
      for (int g = 0; g < KS; ++g) v += smf[(g * BM + r) * (BN + 1) + c];
      if (m0 + r >= M || n0 + c >= N) continue;
      if constexpr (TO_TOKENS) {
        const int t = __ldg(ep.row_token + m0 + r);
        if (t >= 0) reinterpret_cast<float*>(ep.C)[(size_t)t * ep.ldc + n0 + c] = fmaf(__ldg(ep.row_scale + t), v, 0.0f);
      } else {
        epi_store_scalar<float>(ep, m0 + r, n0 + c, v);
      }
    }
    return;
  }
  if constexpr (TO_TOKENS) {
    int t[TM];
    float g[TM];
#pragma unroll
    for (int i = 0; i < TM; ++i) t[i] = m0 + ty + i * TY < M ? __ldg(ep.row_token + m0 + ty + i * TY) : -1;
#pragma unroll
    for (int i = 0; i < TM; ++i) g[i] = t[i] >= 0 ? __ldg(ep.row_scale + t[i]) : 0.0f;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      if (t[i] < 0) continue;
      float* row = reinterpret_cast<float*>(ep.C) + (size_t)t[i] * ep.ldc + n0 + tx;
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (n0 + tx + j * TX < N) row[j * TX] = fmaf(g[i], acc[i][j], 0.0f);
    }
  } else {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int m = m0 + ty + i * TY, n = n0 + tx + j * TX;
        if (m < M && n < N) epi_store_scalar<float>(ep, m, n, acc[i][j]);
      }
  }
}

// Few rows, long K (the x Proj of a single-token step): C[M,N] = A[M,Kd] * B[N,Kd]^T with the K dimension split over
// all 256 threads of a block.  A block owns 2 rows x 4 columns, so a handful of rows still spreads over
// (M/2) x (N/4) blocks and every thread has only Kd / (256 V) rounds of loads in flight behind one another
// (V = 16 bytes of T; Kd % (256 V) == 0).  Partial sums: lanes by shuffles, then the 8 warps in warp order.
template <typename T>
__global__ void __launch_bounds__(256)
gemm_skinny(const T* __restrict__ A, int lda, const T* __restrict__ Bw, int ldb, int M, int N, int Kd, Epilogue ep) {
  pdl_sync();
  constexpr int V = 16 / sizeof(T);
  __shared__ float part[8][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n0 = blockIdx.x * 4;
  const int r0 = blockIdx.y * 2;
  const bool row1 = r0 + 1 < M;
  float acc[2][4] = {};
  for (int k = threadIdx.x * V; k < Kd; k += 256 * V) {
    float a0[V], a1[V];
    load_vec(A + (size_t)r0 * lda + k, a0);
    if (row1) load_vec(A + (size_t)(r0 + 1) * lda + k, a1);
    else {
#pragma unroll
      for (int i = 0; i < V; ++i) a1[i] = 0.0f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float w[V];
      load_vec(Bw + (size_t)min(n0 + j, N - 1) * ldb + k, w);
#pragma unroll
      for (int i = 0; i < V; ++i) {
        acc[0][j] = fmaf(a0[i], w[i], acc[0][j]);
        acc[1][j] = fmaf(a1[i], w[i], acc[1][j]);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float v = acc[r][j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) part[warp][r * 4 + j] = v;
    }
  __syncthreads();
  if (threadIdx.x < 8) {
    const int r = threadIdx.x >> 2, j = threadIdx.x & 3;
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += part[w][threadIdx.x];
    if (r0 + r < M && n0 + j < N) epi_store_scalar<T>(ep, r0 + r, n0 + j, v);
  }
}

}  // namespace

template <int BM_, int BN_, int TM, int TN, int KS, int BKF>
static cudaError_t launch_f32(const float* A, int lda, const float* B, int ldb, int64_t stride, int M, int N, int Kd, const int32_t* te, const int32_t* nmt,
                              const int32_t* assign_of_row, const Epilogue& ep, cudaStream_t st) {
  constexpr int smem = 3 * (BM_ + BN_) * (BKF + 4) * (int)sizeof(float);
  static_assert(smem >= KS * BM_ * (BN_ + 1) * (int)sizeof(float) || KS == 1, "partial sums reuse the stages");
  auto kern = ep.mode == EPI_OUTPROJ ? gemm_f32<BM_, BN_, TM, TN, KS, BKF, true> : gemm_f32<BM_, BN_, TM, TN, KS, BKF, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  launch_k(kern, dim3((M + BM_ - 1) / BM_, (N + BN_ - 1) / BN_), BM_ / TM * (BN_ / TN) * KS, smem, st, A, lda, B, ldb, stride, M, N, Kd, te, nmt, assign_of_row, ep);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_gemm_simt(int dtype, const void* A, int lda, const void* Bw, int ldb, int64_t b_expert_stride,
                             int M_max, int N, int Kd, const int32_t* tile_expert, const int32_t* num_m_tiles_dev,
                             const Epilogue& epi, cudaStream_t st, const int32_t* assign_of_row, int n_rows) {
  if (dtype == ROM_F32) {
    const float* a = (const float*)A;
    const float* b = (const float*)Bw;
    // large tiles once they give every SM a block
    if ((long long)((M_max + 127) / 128) * ((N + 127) / 128) >= 148)
      return launch_f32<128, 128, 8, 8, 1, 16>(a, lda, b, ldb, b_expert_stride, M_max, N, Kd, tile_expert, num_m_tiles_dev, assign_of_row, epi, st);
    // Blocks of 32 x 32 that have work.  Grouped, M_max counts a row tile of padding for every expert; half of that is there on average,
    // and half a block of 32 rows an expert where blocks that are all padding leave at once.
    long long rows = M_max;
    if (tile_expert && n_rows > 0) {
      const int experts = (M_max - (int)align_up((size_t)n_rows, kTileM)) / kTileM;
      const int least = (experts < n_rows ? experts : n_rows) * kTileM, mean = n_rows + experts * kTileM / 2;
      rows = assign_of_row ? n_rows + experts * 16 : mean > least ? mean : least;
    }
    const long long blocks = (rows + 31) / 32 * ((N + 31) / 32);
    // Longer contractions whose last stage is not mostly empty in stages of 128 over eight groups, half as many serial steps, as long as all
    // blocks are resident at once (two an SM); in 16 x 16 tiles where 32 x 32 leave most SMs idle.  us, stages of 64 / 128 / 16 x 16 tiles:
    // 32 blocks, K = 512: 8.2 / 7.9 / 4.1; 64, 512: 8.2 / 8.0 / 7.7; 64, 320: 5.8 / 6.3 / 6.2; 256, 1024: 43.5 / 37.5 / 38; 512, 1024: 44 / 54 / 54;
    // 2048, 512: 76 / 102 / 112.  Grouped (whole calls): 96 blocks, K = 512: 67.8 / 59.2; 200, 512: 85.6 / 83.2; 288, 1024: 140.6 / 137.4; 320, 1024:
    // 177.3 / 185.4.  Between 150 and 220 blocks of one product, where some SMs have two and most one, stages of 64: 200, 1024: 1 / 1.2 / 1.08.
    const bool whole = Kd > 256 && 10 * Kd >= 9 * ((Kd + 127) / 128 * 128);
    if (!tile_expert && Kd >= 256 && (blocks <= 48 || (whole && blocks <= 74)))
      return launch_f32<16, 16, 2, 4, 8, 128>(a, lda, b, ldb, b_expert_stride, M_max, N, Kd, tile_expert, num_m_tiles_dev, assign_of_row, epi, st);
    if (whole && blocks <= 290 && (tile_expert || blocks <= 148 || blocks >= 225))
      return launch_f32<32, 32, 4, 4, 8, 128>(a, lda, b, ldb, b_expert_stride, M_max, N, Kd, tile_expert, num_m_tiles_dev, assign_of_row, epi, st);
    return launch_f32<32, 32, 4, 4, 4, 64>(a, lda, b, ldb, b_expert_stride, M_max, N, Kd, tile_expert, num_m_tiles_dev, assign_of_row, epi, st);
  }
  dim3 grid((M_max + BM - 1) / BM, (N + BN - 1) / BN);
  launch_k(gemm_simt<__nv_bfloat16>, grid, 256, 0, st, (const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)Bw, ldb, b_expert_stride,
                                                M_max, N, Kd, tile_expert, num_m_tiles_dev, epi);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_gemm_skinny(int dtype, const void* A, int lda, const void* Bw, int ldb, int M, int N, int Kd,
                               const Epilogue& epi, cudaStream_t st) {
  dim3 grid((N + 3) / 4, (M + 1) / 2);
  if (dtype == ROM_BF16)
    launch_k(gemm_skinny<__nv_bfloat16>, grid, 256, 0, st, (const __nv_bfloat16*)A, lda, (const __nv_bfloat16*)Bw, ldb, M, N, Kd, epi);
  else
    launch_k(gemm_skinny<float>, grid, 256, 0, st, (const float*)A, lda, (const float*)Bw, ldb, M, N, Kd, epi);
  count_launch();
  return cudaGetLastError();
}

}  // namespace rom
