// dt Proj of the shared small projections on the tensor path (Section 4.3): Delta = softplus(delta W_dt^T + b_dt), bf16 in and out,
// for a dt rank of at most 128 (two K blocks).
//
// What bounds it: instruction issue, then the 2 bytes an output that leave.  The contraction is short, so that the time is the
// epilogue's: in the general GEMM an output cost 16 thread instructions (issue slots 70 % busy, fp32 pipe 38 %, special-function unit
// 35 %, DRAM nearly idle).  Here the sum with the bias and the polynomial run on packed pairs, the bias waits in shared memory, and a
// warp's 32 x 64 outputs leave through one tensor-map store from the swizzled staging rows (its range check replaces the row and column
// tests).  A CTA also keeps ONE block of 256 channels, whose weights it loads once, before the kernel that writes delta has ended, and
// streams 32 KB of delta a tile; alone that gave 55 -> 53 us at 16384 x 4096, with the shorter epilogue 35 (20 us at the copy
// bandwidth); 65536 x 3072: 198 -> 131; 8192 x 2048: 28 -> 23.
#include "rom_tc_ptx.cuh"

namespace rom {
namespace {

constexpr int DT_N = 256;                        // channels per CTA
constexpr int DT_EPI = 16;                       // epilogue warps
constexpr int DT_THREADS = 64 + 32 * DT_EPI;
constexpr int DT_ACC = 2;                        // accumulators in tensor memory
constexpr int DT_TMEM = DT_ACC * DT_N;
constexpr int A_KB = BLOCK_M * BLOCK_K * 2, B_KB = DT_N * BLOCK_K * 2;      // bytes of a K block
constexpr int DT_OUT = DT_EPI * 32 * 128;        // 32 rows x 64 channels per epilogue warp
__host__ __device__ constexpr int dt_stages(int nkb) { return nkb == 1 ? 4 : 3; }
__host__ __device__ constexpr int dt_smem(int nkb) { return nkb * B_KB + dt_stages(nkb) * nkb * A_KB + DT_OUT + DT_N * 4 + 256 + 1024; }

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(map), "r"(src), "r"(x), "r"(y) : "memory");
}
// softplus_bf16 of a pair: the same operations, two at a time where the fp32 pipe can
__device__ __forceinline__ float2 softplus2_bf16(float2 v) {
  const float2 t = __fmul2_rn(v, make_float2(1.4426950408889634f, 1.4426950408889634f));
  const float2 e = make_float2(ex2_ftz(-fabsf(t.x)), ex2_ftz(-fabsf(t.y)));
  auto two = [](float c) { return make_float2(c, c); };
  float2 q = __ffma2_rn(two(0.04066344f), e, two(-0.15602953f));
  q = __ffma2_rn(q, e, two(0.30539998f));
  q = __ffma2_rn(q, e, two(-0.49678875f));
  q = __ffma2_rn(q, e, two(0.99993682f));
  return __ffma2_rn(e, q, make_float2(fmaxf(v.x, 0.0f), fmaxf(v.y, 0.0f)));
}

template <int NKB>
__global__ void __launch_bounds__(DT_THREADS, 1)
dt_proj_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, const __grid_constant__ CUtensorMap tmap_c,
               const float* __restrict__ bias, int M, int N, int block_n, uint32_t idesc, int n_tiles, int32_t* __restrict__ status,
               uint32_t wait_limit, uint32_t stall) {
  constexpr int STAGES = dt_stages(NKB), SA = NKB * A_KB;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;      // 128B-swizzled tiles need 1024-byte alignment
  unsigned char* smem = smem_raw + (base - raw);
  const uint32_t sb = base, sa0 = base + NKB * B_KB;
  unsigned char* out_stage = smem + NKB * B_KB + STAGES * SA;
  float* bias_s = reinterpret_cast<float*>(out_stage + DT_OUT);
  const uint32_t bars = base + NKB * B_KB + STAGES * SA + DT_OUT + DT_N * 4;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bars + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bars + 8u * (2 * STAGES + DT_ACC + a); };
  const uint32_t w_bar = bars + 8u * (2 * STAGES + 2 * DT_ACC), drain_bar = w_bar + 8;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(out_stage + DT_OUT + DT_N * 4 + 8 * (2 * STAGES + 2 * DT_ACC + 2));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tile = blockIdx.x % n_tiles, m_first = blockIdx.x / n_tiles, m_step = gridDim.x / n_tiles;
  const int m_tiles = (M + BLOCK_M - 1) / BLOCK_M;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < DT_ACC; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), DT_EPI); }
    mbar_init(w_bar, 1);
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    // the weights: not written by the kernel before this one, and everything before that one is complete
    mbar_expect_tx(w_bar, (uint32_t)(NKB * block_n * BLOCK_K * 2) + stall);      // (fault injection: 16 bytes that never come)
#pragma unroll
    for (int kb = 0; kb < NKB; ++kb) tma_load_2d(sb + kb * B_KB, &tmap_b, w_bar, kb * BLOCK_K, n_tile * block_n);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(DT_TMEM) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  for (int i = threadIdx.x; i < DT_N; i += DT_THREADS) bias_s[i] = bias && n_tile * block_n + i < N ? __ldg(bias + n_tile * block_n + i) : 0.0f;
  pdl_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  bool ok = true;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0, issued = 0; uint32_t phase = 0;
      for (int m = m_first; m < m_tiles; m += m_step) {
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, wait_limit)) { ok = false; break; }
        mbar_expect_tx(full_bar(stage), (uint32_t)SA);
#pragma unroll
        for (int kb = 0; kb < NKB; ++kb) tma_load_2d(sa0 + stage * SA + kb * A_KB, &tmap_a, full_bar(stage), kb * BLOCK_K, m * BLOCK_M);
        ++issued;
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
      }
      if (!ok) {
        if (!*abort_flag) latch_timeout(status, 31);
        *abort_flag = 1;
      }
      // the CTA does not exit before its copies have landed, or had a bounded time to (another role may give up after the last was issued)
      for (int i = 0; i < min(issued, STAGES); ++i) {
        if (--stage < 0) { stage = STAGES - 1; phase ^= 1u; }
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(full_bar(stage), phase)) break;
      }
      for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
        if (mbar_try_wait(w_bar, 0)) break;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      int stage = 0, acc = 0; uint32_t phase = 0, acc_phase = 0;
      bool issued_any = false;
      ok = mbar_wait(w_bar, 0, abort_flag, wait_limit);
      for (int m = m_first; m < m_tiles && ok; m += m_step) {
        if (!mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, wait_limit) || !mbar_wait(full_bar(stage), phase, abort_flag, wait_limit)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int kb = 0; kb < NKB; ++kb) {
          const uint64_t ad = make_smem_desc(sa0 + stage * SA + kb * A_KB), bd = make_smem_desc(sb + kb * B_KB);
#pragma unroll
          for (int k = 0; k < BLOCK_K / UMMA_K; ++k) umma_bf16(tmem_base + acc * DT_N, ad + 2u * k, bd + 2u * k, idesc, (kb | k) != 0 ? 1u : 0u);
        }
        umma_commit(empty_bar(stage));
        umma_commit(tfull_bar(acc));
        issued_any = true;
        if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        if (++acc == DT_ACC) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) {
        if (!*abort_flag) latch_timeout(status, 32);
        *abort_flag = 1;
      }
      if (*abort_flag && issued_any) {
        umma_commit(drain_bar);
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(drain_bar, 0)) break;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..17)
    const int quarter = warp & 3, c0 = 2 * ((warp - 2) >> 2);      // this warp's lane quarter and 32-column chunks c0, c0 + 1
    uint4* stage = reinterpret_cast<uint4*>(out_stage + (warp - 2) * 32 * 128);
    const int n0 = n_tile * block_n + c0 * 32, n_chunks = max(0, min(2, (block_n >> 5) - c0));
    int acc = 0; uint32_t acc_phase = 0;
    for (int m = m_first; m < m_tiles; m += m_step) {
      // warp-uniform outcome: the tensor-memory loads below need the whole warp
      if (!__all_sync(0xffffffffu, mbar_wait(tfull_bar(acc), acc_phase, abort_flag, wait_limit))) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * DT_N;
      for (int cc = 0; cc < n_chunks; ++cc) {
        uint32_t r[32], o[16];
        tmem_ld32_issue(taddr + (c0 + cc) * 32, r);
        tmem_ld_wait(r);
        if (cc + 1 == n_chunks) {          // all of it is in registers: the accumulator may be written again
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty_bar(acc));
        }
        const float4* bq = reinterpret_cast<const float4*>(bias_s + (c0 + cc) * 32);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 b = bq[i];
          const float2 v0 = softplus2_bf16(__fadd2_rn(make_float2(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1])), make_float2(b.x, b.y)));
          const float2 v1 = softplus2_bf16(__fadd2_rn(make_float2(__uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])), make_float2(b.z, b.w)));
          const __nv_bfloat162 h0 = __float22bfloat162_rn(v0), h1 = __float22bfloat162_rn(v1);
          o[2 * i] = *reinterpret_cast<const uint32_t*>(&h0);
          o[2 * i + 1] = *reinterpret_cast<const uint32_t*>(&h1);
        }
        if (cc == 0) {                     // the store of the tile before has read the staging rows
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) stage[lane * 8 + ((4 * cc + i) ^ (lane & 7))] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
      }
      if (n_chunks == 0) {
        if (lane == 0) mbar_arrive(tempty_bar(acc));
      } else {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {                   // (rows and columns past the end are not written)
          tma_store_2d(&tmap_c, smem_u32(stage), n0, m * BLOCK_M + quarter * 32);
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
      }
      if (++acc == DT_ACC) { acc = 0; acc_phase ^= 1u; }
    }
    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok && lane == 0) {
      if (!*abort_flag) latch_timeout(status, 33);
      *abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(DT_TMEM) : "memory");
  }
}

}  // namespace

bool dt_proj_applicable(int N, int Kd) {
  int num_sms = 0;
  return Kd <= 2 * BLOCK_K && current_device_sm_count(&num_sms) == cudaSuccess && (N + DT_N - 1) / DT_N <= num_sms;
}

cudaError_t launch_dt_proj(const void* A, const void* Bw, int M, int N, int Kd, const Epilogue& epi, int32_t* status, cudaStream_t st, bool test_stall) {
  int num_sms = 0;
  cudaError_t e = current_device_sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  const int block_n = N >= DT_N ? DT_N : (N + 31) / 32 * 32;
  const int n_tiles = (N + block_n - 1) / block_n, m_tiles = (M + BLOCK_M - 1) / BLOCK_M;
  const int rows = num_sms / n_tiles;
  CUtensorMap ta, tb, tc;
  if (!make_tmap(&ta, A, (uint64_t)M, (uint64_t)Kd, (uint64_t)Kd, BLOCK_M)) return cudaErrorInvalidValue;
  if (!make_tmap(&tb, Bw, (uint64_t)N, (uint64_t)Kd, (uint64_t)Kd, (uint32_t)block_n)) return cudaErrorInvalidValue;
  if (!make_tmap(&tc, epi.C, (uint64_t)M, (uint64_t)N, (uint64_t)N, 32)) return cudaErrorInvalidValue;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(block_n >> 3) << 17) | ((uint32_t)(BLOCK_M >> 4) << 24);
  auto go = [&](auto kern, int smem) -> cudaError_t {
    const cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e2 != cudaSuccess) return e2;
    count_launch();
    return launch_k(kern, dim3((unsigned)(n_tiles * (m_tiles < rows ? m_tiles : rows))), DT_THREADS, smem, st, ta, tb, tc, epi.bias, M, N, block_n, idesc, n_tiles, status,
                    test_stall ? WAIT_LIMIT_TEST : WAIT_LIMIT, test_stall ? 16u : 0u);
  };
  return Kd <= BLOCK_K ? go(dt_proj_kernel<1>, dt_smem(1)) : go(dt_proj_kernel<2>, dt_smem(2));
}

}  // namespace rom
