// x Proj of the shared small projections on the tensor path for few tokens (Section 4.3): (delta | B | C) = U W_x^T, bf16 in, delta in
// bf16, B and C in fp32.
//
// What bounds it: the bytes one SM takes in (about 46 a clock of the tile loads).  The output is at most 160 wide, so that a tile is 128
// tokens and a short sequence has few of them: 24 tiles of 3051 tokens left 124 SMs idle while the others each read 1.5 MB.  Here a
// cluster of S CTAs shares a tile's contracted index, every CTA contracts its K blocks into its own tensor memory, the partial sums go to
// shared memory and each CTA adds the rows it writes over the cluster, in CTA order.  No load is multicast.
// 3051 tokens of 3072 channels: 18 -> 12 us (S = 4); 8192 of 2048: 13.4 -> 10.9 (S = 2).
#include "rom_tc_ptx.cuh"

namespace rom {
namespace {

constexpr int X_N = 160;                         // columns at most (one tile)
constexpr int X_STAGES = 5;
constexpr int X_STAGE = BLOCK_M * BLOCK_K * 2 + X_N * BLOCK_K * 2;
constexpr int X_PITCH = X_N + 4;                 // floats per row of the partial sums
constexpr int X_EPI = 8;                         // epilogue warps
constexpr int X_THREADS = 64 + 32 * X_EPI;
constexpr int X_SMEM = X_STAGES * X_STAGE + 256 + 1024;
static_assert(BLOCK_M * X_PITCH * 4 <= X_STAGES * X_STAGE, "the partial sums take the place of the operand stages");

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

template <int S>
__global__ void __launch_bounds__(X_THREADS, 1)
x_proj_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, int M, int N, int num_kb,
              int block_n, uint32_t idesc, Epilogue ep, int32_t* __restrict__ status, uint32_t wait_limit, uint32_t stall) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;      // 128B-swizzled tiles need 1024-byte alignment
  unsigned char* smem = smem_raw + (base - raw);
  const uint32_t bars = base + X_STAGES * X_STAGE;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (X_STAGES + s); };
  const uint32_t done_bar = bars + 8u * 2 * X_STAGES;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + X_STAGES * X_STAGE + 8 * (2 * X_STAGES + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_rank(), m0 = blockIdx.y * BLOCK_M;
  const int kb0 = num_kb * rank / S, kb1 = num_kb * (rank + 1) / S;
  if (tid == 0) {
    for (int s = 0; s < X_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(done_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(256) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the weights of the first stages: not written by the kernel before this one, and everything before that one is complete
  const int n_ahead = min(X_STAGES, kb1 - kb0);
  const uint32_t stage_tx = (uint32_t)(BLOCK_M + block_n) * BLOCK_K * 2;
  if (tid == 0) {
    for (int s = 0; s < n_ahead; ++s) {
      mbar_expect_tx(full_bar(s), stage_tx + (s == 0 ? stall : 0u));      // (fault injection: 16 bytes that never come)
      tma_load_2d(base + s * X_STAGE + BLOCK_M * BLOCK_K * 2, &tmap_b, full_bar(s), (kb0 + s) * BLOCK_K, 0);
    }
  }
  pdl_sync();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  bool ok = true;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0, issued = 0; uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        const uint32_t sa = base + stage * X_STAGE;
        if (kb - kb0 >= n_ahead) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, wait_limit)) { ok = false; break; }
          mbar_expect_tx(full_bar(stage), stage_tx);
          tma_load_2d(sa + BLOCK_M * BLOCK_K * 2, &tmap_b, full_bar(stage), kb * BLOCK_K, 0);
        }
        tma_load_2d(sa, &tmap_a, full_bar(stage), kb * BLOCK_K, m0);
        ++issued;
        if (++stage == X_STAGES) { stage = 0; phase ^= 1u; }
      }
      if (!ok) {
        if (!*abort_flag) latch_timeout(status, 41);
        *abort_flag = 1;
      }
      // the CTA does not go on before its copies have landed, or had a bounded time to (another role may give up after the last was issued)
      for (int i = 0; i < min(issued, X_STAGES); ++i) {
        if (--stage < 0) { stage = X_STAGES - 1; phase ^= 1u; }
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(full_bar(stage), phase)) break;
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(full_bar(stage), phase, abort_flag, wait_limit)) { ok = false; break; }
        tc_fence_after();
        const uint64_t ad = make_smem_desc(base + stage * X_STAGE), bd = make_smem_desc(base + stage * X_STAGE + BLOCK_M * BLOCK_K * 2);
#pragma unroll
        for (int k = 0; k < BLOCK_K / UMMA_K; ++k) umma_bf16(tmem, ad + 2u * k, bd + 2u * k, idesc, kb > kb0 || k > 0 ? 1u : 0u);
        umma_commit(empty_bar(stage));
        if (++stage == X_STAGES) { stage = 0; phase ^= 1u; }
      }
      if (!ok) {
        if (!*abort_flag) latch_timeout(status, 42);
        *abort_flag = 1;
      }
      umma_commit(done_bar);      // (after a wait that ran out too: what has been issued is waited for below)
    }
  }
  // every product of this CTA is complete: its operands have been read and its sums lie in tensor memory.  (No other wait in the
  // kernel needs the outcome: all threads go on to the barriers, and after a timeout write rows that the status disowns.)
  if (warp >= 2) {
    ok = __all_sync(0xffffffffu, mbar_wait(done_bar, 0, abort_flag, wait_limit));
    if (!ok && lane == 0) {
      if (!*abort_flag) latch_timeout(status, 43);
      *abort_flag = 1;
    }
    if (*abort_flag)              // give the products in flight a bounded time all the same: the stages are about to be written
      for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
        if (mbar_try_wait(done_bar, 0)) break;
    __syncwarp();
    tc_fence_after();
    const int quarter = warp & 3, row = quarter * 32 + lane;
    float* dst = reinterpret_cast<float*>(smem) + row * X_PITCH;
    for (int c = 32 * ((warp - 2) >> 2); c < block_n; c += 64) {
      uint32_t r[32];
      tmem_ld32_issue(tmem + ((uint32_t)(quarter * 32) << 16) + c, r);
      tmem_ld_wait(r);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<float4*>(dst + c + 4 * i) = make_float4(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]), __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  // rows rank, rank + S, ...: the partial sums of the cluster in CTA order, eight columns a thread
  const int nv = N / 8, items = BLOCK_M / S * nv;
  uint32_t peer[S];
#pragma unroll
  for (int c = 0; c < S; ++c) peer[c] = map_rank(base, c);
  constexpr int G = S <= 4 ? 8 / S : 1;      // pieces whose loads are in flight together
  for (int i0 = tid; i0 < items; i0 += X_THREADS * G) {
    float4 p[G][S][2];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int i = min(i0 + g * X_THREADS, items - 1), at = (i / nv * S + rank) * X_PITCH + i % nv * 8;
#pragma unroll
      for (int c = 0; c < S; ++c) { p[g][c][0] = ld_cluster4(peer[c] + 4 * at); p[g][c][1] = ld_cluster4(peer[c] + 4 * at + 16); }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int i = i0 + g * X_THREADS, n = i % nv * 8;
      const size_t m = (size_t)m0 + i / nv * S + rank;
      float v[8] = {};
#pragma unroll
      for (int c = 0; c < S; ++c) {
        const float q[8] = {p[g][c][0].x, p[g][c][0].y, p[g][c][0].z, p[g][c][0].w, p[g][c][1].x, p[g][c][1].y, p[g][c][1].z, p[g][c][1].w};
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += q[j];
      }
      if (i >= items || m >= (size_t)M) continue;
      if (n < ep.R) {
        V16<__nv_bfloat16>::store(reinterpret_cast<__nv_bfloat16*>(ep.C) + m * ep.R + n, v);
      } else {
        float* d = n < ep.R + ep.N ? ep.Bm + m * ep.N + (n - ep.R) : ep.Cm + m * ep.N + (n - ep.R - ep.N);
        *reinterpret_cast<float4*>(d) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(d + 4) = make_float4(v[4], v[5], v[6], v[7]);
      }
    }
  }
  cluster_sync();                      // nobody leaves while its sums may still be read
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
  }
}

// CTAs that share a tile: 8 up to 8 tiles, 4 up to 33, 2 up to 66, as long as each has four K blocks; 1: the general GEMM's kernel, whose tiles
// then have an SM each.  us of a layer of 1024 channels, 8 / 4 / 2 / 1 CTAs: 4 tiles 97.9 / 98.4 / 99.7 / 102.6, 8 113.7 / 113.4 / 114.7 / 117.4,
// 15 147.4 / 146.9 / 147.6 / 150.6, 16 (clusters of eight no longer all resident) 156.4 / 148.8 / 149.9 / 152.4, 33 - / 228.9 / 229.7 / 231.9,
// 34 (nor those of four) - / 237.4 / 230.7 / 233.5, 66 - / - / 352.2 / 355.1.
int x_proj_split(int M, int Kd) {
  const int tiles = (M + BLOCK_M - 1) / BLOCK_M, num_kb = (Kd + BLOCK_K - 1) / BLOCK_K;
  int S = 8;
  while (S > 1 && (tiles * S > (S == 8 ? 64 : 132) || num_kb < 4 * S)) S >>= 1;
  return S;
}

}  // namespace

bool x_proj_applicable(int M, int N, int Kd) { return N <= X_N && N % 8 == 0 && x_proj_split(M, Kd) > 1; }

cudaError_t launch_x_proj(const void* A, const void* Bw, int M, int N, int Kd, const Epilogue& epi, int32_t* status, cudaStream_t st, bool test_stall) {
  const int S = x_proj_split(M, Kd), block_n = (N + 31) / 32 * 32;
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, A, (uint64_t)M, (uint64_t)Kd, (uint64_t)Kd, BLOCK_M)) return cudaErrorInvalidValue;
  if (!make_tmap(&tb, Bw, (uint64_t)N, (uint64_t)Kd, (uint64_t)Kd, (uint32_t)block_n)) return cudaErrorInvalidValue;
  auto kern = S == 8 ? x_proj_kernel<8> : S == 4 ? x_proj_kernel<4> : x_proj_kernel<2>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, X_SMEM);
  if (e != cudaSuccess) return e;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(block_n >> 3) << 17) | ((uint32_t)(BLOCK_M >> 4) << 24);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(S, (M + BLOCK_M - 1) / BLOCK_M);
  cfg.blockDim = dim3(X_THREADS);
  cfg.dynamicSmemBytes = X_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = S; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, ta, tb, M, N, (Kd + BLOCK_K - 1) / BLOCK_K, block_n, idesc, epi, status, test_stall ? WAIT_LIMIT_TEST : WAIT_LIMIT,
                            test_stall ? 16u : 0u);
}

}  // namespace rom
