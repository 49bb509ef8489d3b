// bf16 grouped GEMM on the 5th-generation tensor cores (tcgen05 + TMEM), operands staged by TMA.
//
//   C[M, N] = A[M, Kd] * B[e(m)][N, Kd]^T,  fp32 accumulation in tensor memory.
//
// A holds token rows grouped by expert, every expert segment padded to a multiple of the 128-row
// tile, so a row tile never straddles two experts and a device-built table gives the expert of each
// row tile; the number of row tiles is read from device memory (no host synchronisation).  This is
// the per-expert Conv/Gate projection and Out projection of Section 4.2 (dropless, Section 5.1); with
// one "expert" it also serves the shared x Proj / dt Proj.
//
// One persistent CTA per SM, 320 threads:
//   warp 0      TMA producer: A tile 128x64 and B tile block_n x 64 per stage, 128-byte swizzle
//   warp 1      allocates TMEM, issues tcgen05.mma (one thread), commits to mbarriers
//   warps 2..9  epilogue: tcgen05.ld of the 128 x block_n fp32 accumulator, fused output op, stores;
//               two warps share each 32-lane quarter of tensor memory and take alternate 32-column
//               chunks, and the load of the next chunk is in flight while one chunk is processed
// The accumulator is double-buffered in TMEM (2 x 256 columns) so the epilogue of tile i overlaps
// the MMAs of tile i+1.  Every mbarrier wait is bounded; on expiry the CTA latches an error code in
// the status word, waits (bounded) for its own copies and for the MMAs it already issued, frees its
// TMEM and returns.
//
// CG = 2: a cluster of two CTAs (cta_group::2) works on one 256 x 256 tile, each staging its own 128 rows of A and half of B; the copies
// of both count on the leader's barriers, the leader issues the MMAs, and each CTA drains its own half of the accumulator.  No load is
// multicast.  What bounds it: the tensor pipe at the clock the power limit leaves (1430 TFLOP/s at 16384 x 8192 x 2048 in a cool
// call, 0.86 of the measured cuBLAS burst; about the sustained cuBLAS rate in a loop), then the 3 to 12 % of padding rows.  One CTA
// per tile took 433 us there, pairs 385 (415 before the issuing thread's descriptor steps were compile-time constants: with four
// MMAs of 128 cycles a block it has 500 cycles for its wait, descriptors and commit).
#include "rom_tc_ptx.cuh"

namespace rom {
namespace {

constexpr int NUM_EPI_WARPS_C = 8;
constexpr int MAX_BLOCK_N = 256;
constexpr int MAX_STAGES = 4;
constexpr int A_STAGE_BYTES = BLOCK_M * BLOCK_K * 2;          // 16 KB
constexpr int B_STAGE_BYTES = MAX_BLOCK_N * BLOCK_K * 2;      // 32 KB
constexpr int STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
constexpr int ACC_STAGES = 2;
constexpr int TMEM_COLS = 512;
// The softplus output ops (per-expert dt Proj; the shared one where its rank exceeds 128, otherwise rom_dt_proj.cu) have few K blocks
// per tile: their time is their epilogue's, so they run sixteen epilogue warps instead of eight.
__host__ __device__ constexpr int epi_warps_of(int mode) { return (mode == EPI_SOFTPLUS || mode == EPI_SOFTPLUS_ROWS) ? 16 : NUM_EPI_WARPS_C; }
__host__ __device__ constexpr int threads_of(int mode) { return 64 + 32 * epi_warps_of(mode); }
// Operand stages and epilogue staging per output op.  The softplus epilogue gives up one operand stage for a 32 x 32 fp32 staging
// square per epilogue warp, through which its stores become whole 128-byte row segments.
__host__ __device__ constexpr bool f32_out(int mode) { return mode == EPI_SOFTPLUS || mode == EPI_F32 || mode == EPI_SOFTPLUS_ROWS; }
// The x Proj (a narrow B tile, one wave of row tiles, time set by how many bytes of A are in flight) runs six
// smaller stages: its B tile is at most XPROJ_BLOCK_N rows.
constexpr int XPROJ_BLOCK_N = 160;
// CG = 2 (CTA pairs): each CTA stages its own 128 rows of A and its half, 128 rows, of a 256-wide B tile.
__host__ __device__ constexpr int stage_bytes_of(int mode, int cg = 1) {
  if (cg == 2) return 2 * A_STAGE_BYTES;
  return mode == EPI_XPROJ ? A_STAGE_BYTES + XPROJ_BLOCK_N * BLOCK_K * 2 : STAGE_BYTES;
}
__host__ __device__ constexpr int stages_of(int mode, int cg = 1) {
  return cg == 2 ? (f32_out(mode) ? 5 : 6) : f32_out(mode) ? 3 : mode == EPI_XPROJ ? 6 : MAX_STAGES;
}
// bf16 rows of a grouped product leave through 32 rows x 64 columns a warp (row_out).
__host__ __device__ constexpr bool row_out(int mode) { return mode == EPI_STORE || mode == EPI_INPROJ || mode == EPI_OUTPROJ || mode == EPI_SWIGLU; }
__host__ __device__ constexpr int out_stage_bytes_of(int mode) { return f32_out(mode) || row_out(mode) ? epi_warps_of(mode) * 32 * 32 * 4 : 0; }
__host__ __device__ constexpr int smem_bytes_of(int mode, int cg = 1) {
  return stages_of(mode, cg) * stage_bytes_of(mode, cg) + 1024 /*alignment slack*/ + 256 /*barriers*/ + out_stage_bytes_of(mode);
}

// Bias of the 32 columns [n0, n0+32) (EPI_SOFTPLUS only), requested before the accumulator chunk is waited for.
template <int MODE>
__device__ __forceinline__ void load_bias(const Epilogue& ep, int n0, int N, float4 (&bq)[8]) {
  if constexpr (MODE == EPI_SOFTPLUS || MODE == EPI_SOFTPLUS_ROWS) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      bq[i] = (ep.bias && n0 + 4 * i < N) ? __ldg(reinterpret_cast<const float4*>(ep.bias + n0) + i) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
}

// x Proj output op on 32 consecutive accumulator columns [n0, n0+32) of row m (n0 % 32 == 0); columns at or beyond N are skipped in groups
// of 8 (N % 8 == 0).  m: output row; m_tok (with row_token): row of the B / C parts, the token of this expert-order row.
__device__ __forceinline__ void epi_xproj32(const Epilogue& ep, size_t m, size_t m_tok, int n0, int N, const uint32_t (&r)[32]) {
#pragma unroll
  for (int j = 0; j < 32; j += 8) {
    const int n = n0 + j;
    if (n >= N) break;
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[j + i]);
    if (n < ep.R) {
      uint4 q;
      uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        w[i] = *reinterpret_cast<uint32_t*>(&h);
      }
      *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(ep.C) + m * ep.R + n) = q;
    } else {
      float* dst = (n < ep.R + ep.N) ? ep.Bm + m_tok * ep.N + (n - ep.R) : ep.Cm + m_tok * ep.N + (n - ep.R - ep.N);
      *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
    }
  }
}

// Row-store output ops: a lane puts 32 columns of its row into the warp's staging rows (128 bytes each, 16-byte pieces swizzled), and the
// warp writes two adjacent chunks as whole 128-byte row segments, four rows a store instruction.  Straight from the accumulator's lanes a
// store touched 32 rows with 16 bytes each: 32 half-filled sectors, eight times the requests of the LSU and twice the write sectors of
// the L2, which together with the activation took longer than the 16 K blocks of a 1024-wide contraction (tensor pipe 53 %).
// 8192 x 4096 x 1024: 72 -> 63 us; 6102 x 6144 x 1536 106 -> 102; 16384 x 8192 x 2048 385 -> 378.
template <int MODE>
__device__ __forceinline__ void stage_rows32(uint4* stage, int cc, const uint32_t (&r)[32], const uint32_t (&up)[32], bool silu, float scale, int lane) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint4 q;
    uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float2 v = make_float2(__uint_as_float(r[8 * j + 2 * i]), __uint_as_float(r[8 * j + 2 * i + 1]));
      if (MODE == EPI_SWIGLU || (MODE == EPI_INPROJ && silu)) {      // SiLU, the operations of silu_fast two at a time
        const float2 t = __fmul2_rn(v, make_float2(-1.4426950408889634f, -1.4426950408889634f));
        const float2 d = __fadd2_rn(make_float2(ex2_ftz(t.x), ex2_ftz(t.y)), make_float2(1.0f, 1.0f));
        v = __fmul2_rn(v, make_float2(rcp_ftz(d.x), rcp_ftz(d.y)));
      }
      if (MODE == EPI_SWIGLU) v = __fmul2_rn(v, make_float2(__uint_as_float(up[8 * j + 2 * i]), __uint_as_float(up[8 * j + 2 * i + 1])));
      if (MODE == EPI_OUTPROJ) v = __fmul2_rn(v, make_float2(scale, scale));
      const __nv_bfloat162 h = __float22bfloat162_rn(v);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    stage[lane * 8 + ((4 * cc + j) ^ (lane & 7))] = q;
  }
}
// orow: output row of this lane's accumulator row, -1: not stored
__device__ __forceinline__ void flush_rows64(const Epilogue& ep, const uint4* stage, int orow, int n0, int N, int lane) {
  const int p = lane & 7, n = n0 + 8 * p;
#pragma unroll
  for (int r4 = 0; r4 < 8; ++r4) {
    const int R = r4 * 4 + (lane >> 3), to = __shfl_sync(0xffffffffu, orow, R);
    const uint4 q = stage[R * 8 + (p ^ (R & 7))];
    if (to >= 0 && n < N) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(ep.C) + (size_t)to * ep.ldc + n) = q;
  }
}

// Softplus output op on a 32 (rows of this warp) x 32 (columns) accumulator square: every lane activates its row,
// the square goes through a swizzled shared-memory staging area, and is written as whole 128-byte row segments
// (8 lanes per row, 4 rows per store instruction) instead of 32 scattered 16-byte pieces.
template <int MODE>
__device__ __forceinline__ void epi_softplus32(const Epilogue& ep, float* sw, int row0, int M_valid, int n0, int N,
                                               const uint32_t (&r)[32], const float4 (&bq)[8], int lane) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float4 o;
    if constexpr (MODE == EPI_F32) {      // plain fp32 rows, no bias, no activation
      o = make_float4(__uint_as_float(r[4 * c]), __uint_as_float(r[4 * c + 1]), __uint_as_float(r[4 * c + 2]), __uint_as_float(r[4 * c + 3]));
    } else {
      const float4 b = bq[c];
      o = make_float4(softplus_bf16(__uint_as_float(r[4 * c]) + b.x), softplus_bf16(__uint_as_float(r[4 * c + 1]) + b.y),
                      softplus_bf16(__uint_as_float(r[4 * c + 2]) + b.z), softplus_bf16(__uint_as_float(r[4 * c + 3]) + b.w));
    }
    *reinterpret_cast<float4*>(sw + lane * 32 + ((c ^ (lane & 7)) << 2)) = o;
  }
  __syncwarp();
  if constexpr (MODE == EPI_F32) {
    const int c = lane & 7;
    const int n = n0 + 4 * c;
#pragma unroll
    for (int r4 = 0; r4 < 8; ++r4) {
      const int R = r4 * 4 + (lane >> 3);
      const float4 v = *reinterpret_cast<const float4*>(sw + R * 32 + ((c ^ (R & 7)) << 2));
      if (row0 + R < M_valid && n < N) {
        float4* dst = reinterpret_cast<float4*>(reinterpret_cast<float*>(ep.C) + (size_t)(row0 + R) * ep.ldc + n);
        if (ep.accumulate) atomicAdd(dst, v);      // split K: the partial sums of a tile meet in C (zeroed by the launcher)
        else *dst = v;
      }
    }
  } else {
    // rounded to bf16: a lane takes 8 columns (two staged float4), 4 lanes one 64-byte row segment, 8 rows per store
    const int c8 = lane & 3;
    const int n = n0 + 8 * c8;
#pragma unroll
    for (int r8 = 0; r8 < 4; ++r8) {
      const int R = r8 * 8 + (lane >> 2);
      const float4 v0 = *reinterpret_cast<const float4*>(sw + R * 32 + (((2 * c8) ^ (R & 7)) << 2));
      const float4 v1 = *reinterpret_cast<const float4*>(sw + R * 32 + (((2 * c8 + 1) ^ (R & 7)) << 2));
      uint4 q;
      __nv_bfloat162 h0 = __floats2bfloat162_rn(v0.x, v0.y), h1 = __floats2bfloat162_rn(v0.z, v0.w);
      __nv_bfloat162 h2 = __floats2bfloat162_rn(v1.x, v1.y), h3 = __floats2bfloat162_rn(v1.z, v1.w);
      q.x = *reinterpret_cast<uint32_t*>(&h0); q.y = *reinterpret_cast<uint32_t*>(&h1);
      q.z = *reinterpret_cast<uint32_t*>(&h2); q.w = *reinterpret_cast<uint32_t*>(&h3);
      if (row0 + R < M_valid && n < N) {
        // per-expert dt Proj at top-1: the row goes to its token's position (padding rows are skipped)
        const int orow = MODE == EPI_SOFTPLUS_ROWS ? __ldg(ep.row_token + row0 + R) : row0 + R;
        if (orow >= 0) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(ep.C) + (size_t)orow * ep.ldc + n) = q;
      }
    }
  }
  __syncwarp();
}

// MN: which operands are MN-major tiles: MN_NONE, MN_B (data gradient on the weights as stored) or MN_BOTH (weight gradient).
enum : int { MN_NONE = 0, MN_B = 1, MN_BOTH = 2 };
template <int MODE, int CG, int MN>
__global__ void __launch_bounds__(threads_of(MODE), 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
               int M_max, int N, int Kd, int block_n, uint32_t idesc,
               const int32_t* __restrict__ tile_expert, const int32_t* __restrict__ num_m_tiles_dev,
               Epilogue ep, int32_t* __restrict__ status, uint32_t wait_limit, int withhold_kb,
               const int32_t* __restrict__ k_seg, int n_seg,
               const int32_t* __restrict__ pad_offsets, int n_experts) {
  constexpr bool a_mn = MN == MN_BOTH, b_mn = MN != MN_NONE;
  constexpr int STAGES = stages_of(MODE, CG);
  constexpr int SB = stage_bytes_of(MODE, CG);      // bytes per operand stage (multiple of 1024)
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;               // 128B-swizzled tiles need 1024-byte alignment
  unsigned char* smem = smem_raw + (base - raw);
  const uint32_t bars = base + STAGES * SB;                   // barrier block (8-byte aligned)
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
  auto tfull_bar = [&](int a) { return bars + 8u * (2 * STAGES + a); };
  auto tempty_bar = [&](int a) { return bars + 8u * (2 * STAGES + ACC_STAGES + a); };
  const uint32_t drain_bar = bars + 8u * (2 * STAGES + 2 * ACC_STAGES);      // abort path only: completion of the MMAs already issued
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + STAGES * SB + 8 * (2 * STAGES + 2 * ACC_STAGES + 1));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);
  float* out_stage = reinterpret_cast<float*>(smem + STAGES * SB + 256);        // [epilogue warps] staging of the rows that leave

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < ACC_STAGES; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), CG * epi_warps_of(MODE)); }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (CG == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  pdl_sync();                                       // (nothing above reads or writes memory of an earlier kernel)

  // CTA pairs: the pair shares one 256 x 256 tile; CTA r owns rows [128 r, 128 r + 128) of it and stages half of B.  An expert with
  // an odd number of 128-row tiles ends in a pair whose second CTA works on a copy of the first one's rows and stores nothing.
  const uint32_t rank = CG == 2 ? cluster_rank() : 0;
  const int worker = CG == 2 ? (int)blockIdx.x / 2 : (int)blockIdx.x, n_workers = CG == 2 ? (int)gridDim.x / 2 : (int)gridDim.x;
  __shared__ int pair_off[CG == 2 ? kMaxE + 1 : 1], tile_off[CG == 2 ? kMaxE + 1 : 1];      // pairs / 128-row tiles before each expert

  int num_m_tiles = (M_max + BLOCK_M - 1) / BLOCK_M;
  if (num_m_tiles_dev) num_m_tiles = min(num_m_tiles, *num_m_tiles_dev);
  const int M_valid = min(M_max, num_m_tiles * BLOCK_M);
  // EPI_SWIGLU: a tile holds 128 gate columns and the 128 up columns of the same hidden units
  const int n_tiles = MODE == EPI_SWIGLU ? N / 128 : (N + block_n - 1) / block_n;
  // Weight-gradient mode (k_seg != nullptr): n_seg independent problems share A and B; problem s contracts the K range
  // [k_seg[s], k_seg[s+1]) (multiples of BLOCK_K; an expert's padded row segment) and writes rows [s M_max, (s+1) M_max) of C.
  // Split-K mode (k_seg == nullptr, n_seg > 1): the K range is cut into n_seg equal pieces whose partial sums add up in C.
  if (CG == 2 && pad_offsets) {
    if (threadIdx.x == 0) {
      int o = 0;
      for (int e = 0; e <= n_experts; ++e) {
        tile_off[e] = pad_offsets[e] / BLOCK_M;
        pair_off[e] = o;
        if (e < n_experts) o += ((pad_offsets[e + 1] - pad_offsets[e]) / BLOCK_M + 1) / 2;
      }
    }
    __syncthreads();
  }
  const int m_units = CG == 1 ? num_m_tiles : pad_offsets ? pair_off[n_experts] : (num_m_tiles + 1) / 2;
  const int seg_tiles = m_units * n_tiles;
  const int total_tiles = n_seg * seg_tiles;
  const int num_kb = (Kd + BLOCK_K - 1) / BLOCK_K;
  const int split_kb = (num_kb + n_seg - 1) / n_seg;
  // m_tile: this CTA's 128-row tile; own: it exists (false: the missing half of a pair)
  auto decode = [&](int tile, int& m_tile, int& n_tile, int& seg, int& kb0, int& nkb, bool& own, int& e) {
    seg = 0; kb0 = 0; nkb = num_kb; own = true;
    int lt = tile;
    if (n_seg > 1 || k_seg) {
      seg = tile / seg_tiles;
      lt = tile - seg * seg_tiles;
      if (k_seg) {
        kb0 = k_seg[seg] / BLOCK_K;
        nkb = (k_seg[seg + 1] - k_seg[seg]) / BLOCK_K;
      } else {
        kb0 = seg * split_kb;
        nkb = min(split_kb, num_kb - kb0);
      }
    }
    m_tile = lt / n_tiles;
    n_tile = lt - m_tile * n_tiles;
    if (CG == 1) {
      e = tile_expert ? tile_expert[m_tile] : 0;
    } else if (pad_offsets) {
      const int u = m_tile;
      int lo = 0, hi = n_experts - 1;                // last expert with pair_off <= u
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pair_off[mid] <= u) lo = mid; else hi = mid - 1;
      }
      e = lo;
      m_tile = tile_off[e] + 2 * (u - pair_off[e]) + (int)rank;
      own = m_tile < tile_off[e + 1];
      if (!own) --m_tile;
    } else {
      e = 0;
      m_tile = 2 * m_tile + (int)rank;               // (rows past the end are filled with zeros and not stored)
    }
  };
  const int b_boxes = b_mn ? (block_n + 63) / 64 : 1;
  const uint32_t stage_tx = CG == 2 ? 2 * SB : A_STAGE_BYTES + (b_mn ? (uint32_t)b_boxes * MN_BOX_BYTES : (uint32_t)block_n * BLOCK_K * 2);

  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();                      // both CTAs' barriers and tensor memory exist before either is used
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      int issued = 0;
      bool ok = true;
      // CTA pairs under fault injection (tests only): from the second stage on 16 bytes are expected that never come (leaving its copies
      // out, as below, takes a test in this loop: 1 % of the whole kernel, out_proj 446 against 451 us at 16384 x 2048 x 8192)
      uint32_t tx = stage_tx;
      const uint32_t tx_later = stage_tx + (withhold_kb >= 0 ? 16u : 0u);
      for (int tile = worker; tile < total_tiles && ok; tile += n_workers) {
        int m_tile, n_tile, seg, kb0, nkb, e;
        bool own;
        decode(tile, m_tile, n_tile, seg, kb0, nkb, own, e);
        const int b_row = MODE == EPI_SWIGLU ? e * 2 * N + n_tile * 128 : e * N + n_tile * block_n;
        for (int kq = 0; kq < nkb; ++kq) {
          const int kb = kb0 + kq;
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, wait_limit)) { ok = false; break; }
          const uint32_t sa = base + stage * SB;
          if constexpr (CG == 2) {
            // both CTAs' copies count on the leader's barrier, which alone expects them
            if (rank == 0) mbar_expect_tx(full_bar(stage), tx);
            tx = tx_later;
            const uint32_t fb = map_rank(full_bar(stage), 0);
            if (a_mn) {
              tma_load_2d_pair(sa, &tmap_a, fb, m_tile * BLOCK_M, kb * BLOCK_K);
              tma_load_2d_pair(sa + MN_BOX_BYTES, &tmap_a, fb, m_tile * BLOCK_M + 64, kb * BLOCK_K);
            } else {
              tma_load_2d_pair(sa, &tmap_a, fb, kb * BLOCK_K, m_tile * BLOCK_M);
            }
            if (b_mn) {
              const int n0 = n_tile * block_n + 128 * (int)rank;
              tma_load_2d_pair(sa + A_STAGE_BYTES, &tmap_b, fb, n0, e * Kd + kb * BLOCK_K);
              tma_load_2d_pair(sa + A_STAGE_BYTES + MN_BOX_BYTES, &tmap_b, fb, n0 + 64, e * Kd + kb * BLOCK_K);
            } else {      // rows 128 .. 255 of the B tile: the next columns, or (SWIGLU) the up rows of the same hidden units
              tma_load_2d_pair(sa + A_STAGE_BYTES, &tmap_b, fb, kb * BLOCK_K, b_row + (int)rank * (MODE == EPI_SWIGLU ? N : 128));
            }
            ++issued;
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
            continue;
          }
          mbar_expect_tx(full_bar(stage), stage_tx);
          // fault injection (tests only): the copies of K block `withhold_kb` of this CTA's first tile are never issued,
          // so the stage never fills and the waits downstream run out
          if (!(withhold_kb >= 0 && tile == worker && kq == withhold_kb)) {
            if (a_mn) {
              tma_load_2d(sa, &tmap_a, full_bar(stage), m_tile * BLOCK_M, kb * BLOCK_K);
              tma_load_2d(sa + MN_BOX_BYTES, &tmap_a, full_bar(stage), m_tile * BLOCK_M + 64, kb * BLOCK_K);
            } else {
              tma_load_2d(sa, &tmap_a, full_bar(stage), kb * BLOCK_K, m_tile * BLOCK_M);
            }
            if (b_mn) {      // B is [n_experts * Kd, N]: the expert's rows are its K range
              for (int i = 0; i < b_boxes; ++i)
                tma_load_2d(sa + A_STAGE_BYTES + i * MN_BOX_BYTES, &tmap_b, full_bar(stage), n_tile * block_n + 64 * i, e * Kd + kb * BLOCK_K);
            } else {
              tma_load_2d(sa + A_STAGE_BYTES, &tmap_b, full_bar(stage), kb * BLOCK_K, b_row);
            }
            if (MODE == EPI_SWIGLU)     // second half of the B tile: the up rows of the same 128 hidden units (box = 128 rows)
              tma_load_2d(sa + A_STAGE_BYTES + 128 * BLOCK_K * 2, &tmap_b, full_bar(stage), kb * BLOCK_K, b_row + N);
          }
          ++issued;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok) {
        if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 1); }
        *abort_flag = 1;
      }
      if (*abort_flag) {
        // drain: give this CTA's copies still in flight a bounded time to land before the CTA exits
        int s = stage; uint32_t ph = phase;
        for (int i = 0; i < min(issued, STAGES); ++i) {
          if (--s < 0) { s = STAGES - 1; ph ^= 1u; }
          for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
            if (mbar_try_wait(full_bar(s), ph)) break;
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      int stage = 0; uint32_t phase = 0;
      int acc = 0; uint32_t acc_phase = 0;
      bool ok = true, issued_any = false;
      auto commit = [&](uint32_t bar) { if constexpr (CG == 2) umma_commit_pair(bar); else umma_commit(bar); };
      auto wait = [&](uint32_t bar, uint32_t ph) {
        return CG == 2 ? mbar_wait_cluster(bar, ph, abort_flag, wait_limit) : mbar_wait(bar, ph, abort_flag, wait_limit);
      };
      for (int tile = worker; tile < total_tiles && ok; tile += n_workers) {
        if (!wait(tempty_bar(acc), acc_phase ^ 1u)) { ok = false; break; }
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)acc * MAX_BLOCK_N;
        int m_tile_, n_tile_, seg_, kb0_, nkb, e_;
        bool own_;
        decode(tile, m_tile_, n_tile_, seg_, kb0_, nkb, own_, e_);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!wait(full_bar(stage), phase)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = base + stage * SB;
          const uint64_t adesc = a_mn ? make_smem_desc_mn(sa) : make_smem_desc(sa);
          const uint64_t bdesc = b_mn ? make_smem_desc_mn(sa + A_STAGE_BYTES) : make_smem_desc(sa + A_STAGE_BYTES);
          // K-major: 16 elements = 32 bytes along K inside the swizzled row, +2 in the address field
          constexpr uint32_t astep = a_mn ? MN_KSTEP : 2u, bstep = b_mn ? MN_KSTEP : 2u;
#pragma unroll
          for (int k = 0; k < BLOCK_K / UMMA_K; ++k) {
            if constexpr (CG == 2) umma_bf16_pair(tmem_d, adesc + (uint64_t)(astep * k), bdesc + (uint64_t)(bstep * k), idesc, (kb | k) != 0 ? 1u : 0u);
            else umma_bf16(tmem_d, adesc + (uint64_t)(astep * k), bdesc + (uint64_t)(bstep * k), idesc, (kb | k) != 0 ? 1u : 0u);
          }
          commit(empty_bar(stage));
          issued_any = true;
          if (++stage == STAGES) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        commit(tfull_bar(acc));
        if (++acc == ACC_STAGES) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) {
        if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 2); }
        *abort_flag = 1;
      }
      if (*abort_flag && issued_any) {
        // the MMAs already issued may still read shared memory and write tensor memory: one more commit tracks them
        // all; wait for it (bounded) before the CTA frees its tensor memory
        commit(drain_bar);
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(drain_bar, 0)) break;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    const int quarter = warp & 3;                 // TMEM lanes [32*quarter, 32*quarter+32) belong to this warp
    constexpr int EWQ = epi_warps_of(MODE) / 4;   // warps per lane quarter
    const int half = (warp - 2) >> 2;             // which of the EWQ warps of the quarter: takes chunks half, half+EWQ, ...
    const int n_chunks = block_n >> 5;
    int acc = 0; uint32_t acc_phase = 0;
    bool ok = true;
    for (int tile = worker; tile < total_tiles && ok; tile += n_workers) {
      int m_tile, n_tile, seg, kb0_, nkb, e_;
      bool own;
      decode(tile, m_tile, n_tile, seg, kb0_, nkb, own, e_);
      // warp-uniform outcome: the tensor-memory loads below need the whole warp
      if (!__all_sync(0xffffffffu, mbar_wait(tfull_bar(acc), acc_phase, abort_flag, wait_limit))) { ok = false; break; }
      tc_fence_after();
      const int row = m_tile * BLOCK_M + quarter * 32 + lane;
      bool row_ok = row < M_valid && own;
      size_t out_row = (size_t)row;
      float scale = 1.0f;
      size_t tok_row = (size_t)row;
      if ((MODE == EPI_OUTPROJ || (MODE == EPI_INPROJ && ep.row_token != nullptr)) && row_ok) {
        const int tok = __ldg(ep.row_token + row);      // rows are written at their token's position
        row_ok = tok >= 0;
        if (row_ok) {
          out_row = (size_t)tok;
          if (MODE == EPI_OUTPROJ) scale = __ldg(ep.row_scale + tok);
        }
      }
      if (MODE == EPI_XPROJ && ep.row_token != nullptr && row_ok) {
        // per-expert x Proj at top-1: delta_r stays in expert order (it feeds the grouped dt Proj), B and C go to the token's row
        const int tok = __ldg(ep.row_token + row);
        row_ok = tok >= 0;
        tok_row = row_ok ? (size_t)tok : 0;
      }
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * MAX_BLOCK_N;
      const int n_base = n_tile * block_n;
      uint32_t ra[32], rb[32];
      float4 bq[8];
      if constexpr (row_out(MODE)) {
        uint4* stage = reinterpret_cast<uint4*>(out_stage + (warp - 2) * 1024);
        const int orow = row_ok ? (int)out_row : -1;
        if constexpr (MODE == EPI_SWIGLU) {
          // accumulator columns [0,128) = gate, [128,256) = up; this warp takes the 32-column groups 2 half and 2 half + 1
          for (int cc = 0; cc < 2; ++cc) {
            tmem_ld32_issue(taddr + (2 * half + cc) * 32, ra);
            tmem_ld32_issue(taddr + 128 + (2 * half + cc) * 32, rb);
            tmem_ld_wait(ra);
            tmem_ld_wait(rb);
            stage_rows32<MODE>(stage, cc, ra, rb, true, 1.0f, lane);
          }
          __syncwarp();
          flush_rows64(ep, stage, orow, n_tile * 128 + half * 64, N, lane);
          __syncwarp();
        } else {
          // pairs of adjacent chunks 2 half, 2 half + 4; the next chunk's load is in flight while one is staged
          int ch = 2 * half;
          if (ch < n_chunks) tmem_ld32_issue(taddr + ch * 32, ra);
          while (ch < n_chunks) {
            const bool act = MODE == EPI_INPROJ && n_base + ch * 32 >= ep.R;      // (the boundary is a multiple of 64)
            tmem_ld_wait(ra);
            if (ch + 1 < n_chunks) tmem_ld32_issue(taddr + (ch + 1) * 32, rb);
            stage_rows32<MODE>(stage, 0, ra, ra, act, scale, lane);
            if (ch + 1 < n_chunks) {
              tmem_ld_wait(rb);
              if (ch + 4 < n_chunks) tmem_ld32_issue(taddr + (ch + 4) * 32, ra);
              stage_rows32<MODE>(stage, 1, rb, rb, act, scale, lane);
            }
            __syncwarp();
            flush_rows64(ep, stage, orow, n_base + ch * 32, min(N, n_base + min(ch + 2, n_chunks) * 32), lane);
            __syncwarp();
            ch += 4;
          }
        }
      }
      if constexpr (EWQ == 4) {
        // sixteen warps: at most two chunks each, one register buffer (the register file has no room for two)
        uint4* stage = reinterpret_cast<uint4*>(out_stage + (warp - 2) * 1024);
        const int c0 = 2 * half;                       // this warp's chunks: c0 and c0 + 1
        int n_pieces = 0;
        for (int cc = 0; cc < 2 && c0 + cc < n_chunks; ++cc) {
          tmem_ld32_issue(taddr + (c0 + cc) * 32, ra);
          load_bias<MODE>(ep, n_base + (c0 + cc) * 32, N, bq);
          tmem_ld_wait(ra);
          softplus_stage_bf16(stage, 4 * cc, ra, bq, lane);
          n_pieces += 4;
        }
        if (n_pieces > 0) {
          __syncwarp();
          softplus_flush_bf16<MODE>(ep, stage, m_tile * BLOCK_M + quarter * 32, M_valid, n_base + c0 * 32, N, n_pieces, lane);
          __syncwarp();
        }
      }
      // weight-gradient mode: problem `seg` owns its own rows of C; an empty K range leaves zeros
      Epilogue epl = ep;
      if (MODE == EPI_F32 && k_seg) epl.C = reinterpret_cast<float*>(ep.C) + (size_t)seg * M_max * ep.ldc;
      const bool zero_acc = MODE == EPI_F32 && nkb <= 0;
      int ch = (row_out(MODE) || EWQ == 4) ? n_chunks : half;
      if (ch < n_chunks) tmem_ld32_issue(taddr + ch * 32, ra);
      // two register buffers: while one chunk is processed the next chunk's tensor-memory load is in flight
      while (ch < n_chunks) {
        load_bias<MODE>(ep, n_base + ch * 32, N, bq);     // in flight together with the tensor-memory load
        tmem_ld_wait(ra);
        if (ch + EWQ < n_chunks) tmem_ld32_issue(taddr + (ch + EWQ) * 32, rb);
        if (zero_acc) {
#pragma unroll
          for (int i = 0; i < 32; ++i) ra[i] = 0u;
        }
        if (f32_out(MODE)) epi_softplus32<MODE>(epl, out_stage + (warp - 2) * 1024, m_tile * BLOCK_M + quarter * 32, own ? M_valid : 0, n_base + ch * 32, N, ra, bq, lane);
        else if (row_ok) epi_xproj32(ep, out_row, tok_row, n_base + ch * 32, N, ra);
        ch += EWQ;
        if (ch >= n_chunks) break;
        load_bias<MODE>(ep, n_base + ch * 32, N, bq);
        tmem_ld_wait(rb);
        if (ch + EWQ < n_chunks) tmem_ld32_issue(taddr + (ch + EWQ) * 32, ra);
        if (zero_acc) {
#pragma unroll
          for (int i = 0; i < 32; ++i) rb[i] = 0u;
        }
        if (f32_out(MODE)) epi_softplus32<MODE>(epl, out_stage + (warp - 2) * 1024, m_tile * BLOCK_M + quarter * 32, own ? M_valid : 0, n_base + ch * 32, N, rb, bq, lane);
        else if (row_ok) epi_xproj32(ep, out_row, tok_row, n_base + ch * 32, N, rb);
        ch += EWQ;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { if (CG == 2) mbar_arrive_cluster(map_rank(tempty_bar(acc), 0)); else mbar_arrive(tempty_bar(acc)); }
      if (++acc == ACC_STAGES) { acc = 0; acc_phase ^= 1u; }
    }
    if (!ok && lane == 0) {
      if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 3); }
      *abort_flag = 1;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();                      // neither CTA leaves while the other may still signal it or read its operands
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if constexpr (CG == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

}  // namespace

namespace {
// instruction descriptor: D = f32, A = B = bf16, operand majorness (1 = MN-major) at bits 15 / 16, N >> 3 at bit 17, M >> 4 at bit 24
uint32_t make_idesc(int block_n, bool a_mn, bool b_mn, int block_m = BLOCK_M) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) | ((uint32_t)(block_n >> 3) << 17) |
         ((uint32_t)(block_m >> 4) << 24);
}

// One persistent CTA pair per two SMs (a cluster of two), or one CTA per SM.
template <typename... P, typename... Args>
cudaError_t launch_workers(void (*kern)(P...), int cg, long long tiles, int num_sms, int threads, int smem, cudaStream_t st, Args... args) {
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const long long slots = num_sms / cg;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(cg * (tiles < slots ? tiles : slots)));
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2]{};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cg; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cg > 1 ? 2 : 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
}  // namespace

cudaError_t launch_gemm_tc(const void* A, int lda, const void* Bw, int ldb, int n_experts, int M_max, int N, int Kd,
                           const int32_t* tile_expert, const int32_t* num_m_tiles_dev, const Epilogue& epi,
                           int32_t* status, cudaStream_t st, bool test_stall, bool b_mn, const int32_t* pad_offsets) {
  // N tile: a multiple of 32 (epilogue column groups) and of 16 (UMMA N for M = 128), at most 256
  const bool swiglu = epi.mode == EPI_SWIGLU;      // N output columns from 2N rows of B per expert, loaded as two boxes of 128 rows
  if (swiglu && (N % 128 != 0 || MAX_BLOCK_N != 256 || b_mn)) return cudaErrorInvalidValue;
  if (epi.mode == EPI_XPROJ && !tile_expert && !epi.row_token && lda == Kd && ldb == Kd && x_proj_applicable(M_max, N, Kd))
    return launch_x_proj(A, Bw, M_max, N, Kd, epi, status, st, test_stall);
  if (epi.mode == EPI_SOFTPLUS && lda == Kd && ldb == Kd && epi.ldc == N && dt_proj_applicable(N, Kd))
    return launch_dt_proj(A, Bw, M_max, N, Kd, epi, status, st, test_stall);
  if (b_mn && n_experts > 1 && Kd % BLOCK_K != 0) return cudaErrorInvalidValue;      // a K block must not run into the next expert
  int block_n = (swiglu || N >= MAX_BLOCK_N) ? MAX_BLOCK_N : (N + 31) / 32 * 32;
  if (epi.mode == EPI_XPROJ && block_n > XPROJ_BLOCK_N) block_n = XPROJ_BLOCK_N;
  int num_sms = 0;
  cudaError_t e = current_device_sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  // CTA pairs: a pair fetches each B tile once for 256 rows (per CTA 32 KB a stage instead of 48).  An expert with an odd number of row
  // tiles ends in a pair that is half empty; measured from 1 to 16 row tiles an expert, pairs are faster all the same (4300 tokens
  // over 8 experts: 2-3 % of the layer) as long as the experts average a full tile; below that single CTAs spread over more SMs.
  // (The softplus output ops, few K blocks a tile, are slower on pairs: 69 us against 58 at 16384 x 4096 x 128.)
  const bool pair_mode = epi.mode == EPI_STORE || epi.mode == EPI_INPROJ || epi.mode == EPI_OUTPROJ || swiglu;
  const int cg = pair_mode && pad_offsets && M_max >= n_experts * 2 * BLOCK_M && block_n == MAX_BLOCK_N ? 2 : 1;
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, A, (uint64_t)M_max, (uint64_t)Kd, (uint64_t)lda, BLOCK_M)) return cudaErrorInvalidValue;
  const bool ok = b_mn ? make_tmap(&tb, Bw, (uint64_t)n_experts * Kd, (uint64_t)N, (uint64_t)ldb, BLOCK_K)
                       : make_tmap(&tb, Bw, (uint64_t)n_experts * (swiglu ? 2 * N : N), (uint64_t)Kd, (uint64_t)ldb,
                                   swiglu || cg == 2 ? 128u : (uint32_t)block_n);
  if (!ok) return cudaErrorInvalidValue;
  const int n_tiles = swiglu ? N / 128 : (N + block_n - 1) / block_n;
  const int m_tiles = (M_max + BLOCK_M - 1) / BLOCK_M;
  auto go = [&](auto kern) {
    return launch_workers(kern, cg, (long long)(cg == 2 ? (m_tiles + n_experts) / 2 : m_tiles) * n_tiles, num_sms, threads_of(epi.mode),
                          smem_bytes_of(epi.mode, cg), st, ta, tb, M_max, N, Kd, block_n, make_idesc(block_n, false, b_mn, cg * BLOCK_M), tile_expert,
                          num_m_tiles_dev, epi, status, test_stall ? WAIT_LIMIT_TEST : WAIT_LIMIT, test_stall ? 1 : -1, nullptr, 1,
                          pad_offsets, n_experts);
  };
  if (b_mn) {
    if (epi.mode != EPI_STORE) return cudaErrorInvalidValue;      // data gradients leave as they are
    return cg == 2 ? go(gemm_tc_kernel<EPI_STORE, 2, MN_B>) : go(gemm_tc_kernel<EPI_STORE, 1, MN_B>);
  }
  constexpr int NO = MN_NONE;
  if (cg == 2) return go(epi.mode == EPI_STORE ? gemm_tc_kernel<EPI_STORE, 2, NO> : epi.mode == EPI_INPROJ ? gemm_tc_kernel<EPI_INPROJ, 2, NO>
                         : epi.mode == EPI_OUTPROJ ? gemm_tc_kernel<EPI_OUTPROJ, 2, NO> : gemm_tc_kernel<EPI_SWIGLU, 2, NO>);
  return go(epi.mode == EPI_STORE ? gemm_tc_kernel<EPI_STORE, 1, NO> : epi.mode == EPI_XPROJ ? gemm_tc_kernel<EPI_XPROJ, 1, NO>
            : epi.mode == EPI_INPROJ ? gemm_tc_kernel<EPI_INPROJ, 1, NO> : epi.mode == EPI_OUTPROJ ? gemm_tc_kernel<EPI_OUTPROJ, 1, NO>
            : epi.mode == EPI_F32 ? gemm_tc_kernel<EPI_F32, 1, NO> : epi.mode == EPI_SWIGLU ? gemm_tc_kernel<EPI_SWIGLU, 1, NO>
            : epi.mode == EPI_SOFTPLUS_ROWS ? gemm_tc_kernel<EPI_SOFTPLUS_ROWS, 1, NO> : gemm_tc_kernel<EPI_SOFTPLUS, 1, NO>);
}

namespace {
// pieces of at least eight K blocks, as many as keep one tile per SM, none of them empty
int wgrad_pieces(int rows, long long tiles, int num_sms) {
  const int num_kb = (rows + BLOCK_K - 1) / BLOCK_K;
  int n = 1;
  while ((n + 1) * tiles <= num_sms && num_kb / (n + 1) >= 8) ++n;
  const int per = (num_kb + n - 1) / n;
  return (num_kb + per - 1) / per;
}
long long wgrad_tiles(int P, int Q) {
  const int block_n = Q >= MAX_BLOCK_N ? MAX_BLOCK_N : (Q + 31) / 32 * 32;
  return (long long)((P + BLOCK_M - 1) / BLOCK_M) * ((Q + block_n - 1) / block_n);
}
}  // namespace

bool gemm_tc_wgrad_adds(int rows, int P, int Q) {
  int num_sms = 0;
  return current_device_sm_count(&num_sms) == cudaSuccess && wgrad_pieces(rows, wgrad_tiles(P, Q), num_sms) > 1;
}

// Weight gradient on the tensor cores: C[s][P, Q] (fp32) = sum over the rows r of segment s of X[r, p] Y[r, q], X [rows, P] and
// Y [rows, Q] bf16 as the layer holds them (token rows outermost): both operands are MN-major tiles, nothing is transposed in
// memory.  seg: n_seg + 1 device offsets, multiples of 64 (the padded expert segments; rows outside are never read).
// seg == nullptr: one sum over all rows; with too few output tiles to fill the GPU (the shared x Proj / dt Proj: 32 tiles
// against 16384 rows) the rows are cut into pieces that add into C.
cudaError_t launch_gemm_tc_wgrad(const void* X, const void* Y, int rows, const int32_t* seg, int n_seg, int P, int Q, float* C,
                                 int32_t* status, cudaStream_t st) {
  const int block_n = Q >= MAX_BLOCK_N ? MAX_BLOCK_N : (Q + 31) / 32 * 32;
  CUtensorMap ta, tb;
  if (!make_tmap(&ta, X, (uint64_t)rows, (uint64_t)P, (uint64_t)P, BLOCK_K)) return cudaErrorInvalidValue;
  if (!make_tmap(&tb, Y, (uint64_t)rows, (uint64_t)Q, (uint64_t)Q, BLOCK_K)) return cudaErrorInvalidValue;
  int num_sms = 0;
  cudaError_t e = current_device_sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  const long long tiles = wgrad_tiles(P, Q);
  Epilogue epi{EPI_F32, C, Q, nullptr, nullptr, nullptr, 0, 0, nullptr, nullptr};
  if (!seg) {
    n_seg = wgrad_pieces(rows, tiles, num_sms);
    epi.accumulate = n_seg > 1;                      // (C was zeroed by the caller)
  }
  const int cg = seg && block_n == MAX_BLOCK_N && P >= 2 * BLOCK_M ? 2 : 1;
  const long long units = (long long)n_seg * ((P + cg * BLOCK_M - 1) / (cg * BLOCK_M)) * ((Q + block_n - 1) / block_n);
  return launch_workers(cg == 2 ? gemm_tc_kernel<EPI_F32, 2, MN_BOTH> : gemm_tc_kernel<EPI_F32, 1, MN_BOTH>, cg, units, num_sms, threads_of(EPI_F32), smem_bytes_of(EPI_F32, cg), st,
                        ta, tb, P, Q, rows, block_n, make_idesc(block_n, true, true, cg * BLOCK_M), nullptr, nullptr, epi, status, WAIT_LIMIT, -1, seg, n_seg,
                        nullptr, 0);
}

}  // namespace rom
