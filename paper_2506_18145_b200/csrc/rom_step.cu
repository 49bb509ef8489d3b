// Single-token step of the layer (recurrent inference) for a few tokens per expert, bf16: five launches, chained by programmatic
// dependent launch, against the eight of the general sequence.
//
//   step_route    : one block per token: logits in fp64 (exact products, the same order for every expert), softmax, top-K
//                   (one or two tokens: inside the In Proj, four launches)
//   step_gemm<IN> : grouped [Conv Proj | Gate Proj] of the selected experts; at top-1 its output op also runs the short conv
//                   on the caller's window of H (step_conv does both for K > 1, where H is a sum over experts)
//   step_xproj    : x Proj -> delta_r | B | C, clusters of eight CTAs that share the contracted index
//   step_dt_scan  : dt Proj + softplus, one step of the recurrence on the caller's state, skip, gate
//   step_gemm<OUT>: grouped Out Proj, times the gate (K > 1: rows summed by step_combine)
//
// What bounds it: the weights of the selected experts, read once (HBM), and below that latency -- every stage waits for the one
// before.  With a handful of tokens per expert a 128-row tensor tile is nearly all padding and one CTA per 256 columns leaves
// most SMs idle (out_proj of one token: 8 CTAs, 26 us for 16 MB).  Here the weights are the M operand of mma.m16n8k16 and the
// tokens its N = 8 columns: a block owns 16 or 32 weight rows and splits the contracted index over its warps, so that one token
// already spreads over 128 to 256 blocks; lanes read 16 consecutive bytes of a weight row straight into fragments (the
// contracted index is permuted inside a 32-wide block, alike for both operands).  Every kernel requests what does not depend on
// its predecessor (states, small weights, and for the Out Proj its first weight tiles) before it waits.
// The predecessor's predecessors are complete by then: every kernel triggers its successor only after its own wait.
#include "rom_tc_ptx.cuh"

namespace rom {
namespace {

constexpr int NST = 16;
constexpr int kStepMaxTokens = 512, kStepMaxAssign = 2048;
// Assignments from which the weights are streamed (step_tc).  us a step, register-fed / streamed, 2048 channels, 8 experts, top-1:
// 1: 23.1 / 43.7, 2: 33.3 / 49.4, 3: 44.1 / 54.3, 4: 55.4 / 61.5, 5: 59.7 / 65.8, 8: 77.8 / 77.5, 16: 121.6 / 91.0; 16 experts 3: 49.4 / 59.8,
// 4: 60.0 / 64.6; 1024 channels, 8 experts 4: 30.7 / 37.0, 5: 33.3 / 38.5, 8: 39.1 / 42.1.  By these times the line would lie at eight; it
// stays at four because the two kernels add in different orders and a sequence's result is the same in every batch from four on.
constexpr int kStreamMin = 4;
constexpr float kLog2e = 1.4426950408889634f;
typedef __nv_bfloat16 bf16;

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// One 32-wide block of the contracted index: q0 / q1 = rows g / g + 8 of the weights, xq = token g, each 8 consecutive elements
// at 8 t.  The pairs (0,1), (2,3) feed the first MMA, (4,5), (6,7) the second.
__device__ __forceinline__ void mma_block(float (&d)[4], const uint4& q0, const uint4& q1, const uint4& xq) {
  mma_bf16(d, q0.x, q1.x, q0.y, q1.y, xq.x, xq.y);
  mma_bf16(d, q0.z, q1.z, q0.w, q1.w, xq.z, xq.w);
}
// weights are read once per step: keep them out of the way of the activations in L1
__device__ __forceinline__ uint4 ld_stream(const bf16* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
// activations of an earlier kernel of the chain
__device__ __forceinline__ uint4 ld_act(const bf16* p) {
  uint4 v;
  asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}

// ---------------------------------------------------------------------------------------------- router
constexpr int kRouteWarps = 8;
struct RouteArgs { const bf16* x; const bf16* W_r; const float* b_r; int Dm, E, K, gate_mode; int32_t* idx_ws; float* gates_ws; int32_t* idx_out; int32_t* status; };
struct RouteSmem { double part[kRouteWarps][kMaxE], lg[kMaxE], pr[kMaxE]; };

// logits of one token in lg, by a block of eight warps: products widened before they are multiplied (exact whatever the operands'
// exponents, as in the forward's router), every expert summed in the same order
__device__ __forceinline__ void route_logits(const RouteArgs& p, int t, RouteSmem& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, E = p.E;
  // warp w takes the 8-element groups w * 32 + lane, ...
  for (int e0 = 0; e0 < E; e0 += 8) {
    double acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0;
    for (int d = (warp * 32 + lane) * 8; d < p.Dm; d += 2048) {
      V16<bf16> q;
      float xv[8];
      double xd[8];
      q.load(p.x + (size_t)t * p.Dm + d);
      V16<bf16> wq[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) wq[e].load(p.W_r + (size_t)min(e0 + e, E - 1) * p.Dm + d);
      q.get(xv);
#pragma unroll
      for (int i = 0; i < 8; ++i) xd[i] = (double)xv[i];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float wv[8];
        wq[e].get(wv);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[e] = fma(xd[i], (double)wv[i], acc[e]);
      }
    }
    // transposed sums over the lanes: 8 values -> lane keeps value (lane & 7) after three exchanges, then two plain ones
    {
      double a4[4], a2[2], a1;
      const bool s0 = lane & 1, s1 = lane & 2, s2 = lane & 4;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const double send = s2 ? acc[i] : acc[4 + i], keep = s2 ? acc[4 + i] : acc[i];
        a4[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const double send = s1 ? a4[i] : a4[2 + i], keep = s1 ? a4[2 + i] : a4[i];
        a2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
      }
      const double send = s0 ? a2[0] : a2[1], keep = s0 ? a2[1] : a2[0];
      a1 = keep + __shfl_xor_sync(0xffffffffu, send, 1);
      a1 += __shfl_xor_sync(0xffffffffu, a1, 8);
      a1 += __shfl_xor_sync(0xffffffffu, a1, 16);
      if (lane < 8 && e0 + lane < kMaxE) s.part[warp][e0 + lane] = a1;
    }
  }
  __syncthreads();
  if (threadIdx.x < E) {
    const int e = threadIdx.x;
    double v = p.b_r ? (double)p.b_r[e] : 0.0;
#pragma unroll
    for (int w = 0; w < kRouteWarps; ++w) v += s.part[w][e];
    s.lg[e] = v;
  }
  __syncthreads();
}
// the k-th expert: largest logit not taken yet, ties to the lowest id, NaN below everything
__device__ __forceinline__ int route_pick(const double* lg, int E, unsigned long long& taken) {
  int best = -1; double bestv = -INFINITY;
  for (int e = 0; e < E; ++e) {
    if ((taken >> e) & 1ull) continue;
    double v = lg[e];
    if (v != v) v = -INFINITY;
    if (best < 0 || v > bestv) { best = e; bestv = v; }
  }
  taken |= 1ull << best;
  return best;
}
// logits, softmax, top-K and gates of one token, written out
__device__ __forceinline__ void route_token(const RouteArgs& p, int t, RouteSmem& s) {
  const int E = p.E, K = p.K;
  route_logits(p, t, s);
  if (threadIdx.x < E) {
    double m = -INFINITY;
    for (int j = 0; j < E; ++j) { const double v = s.lg[j]; if (v > m) m = v; }      // NaN never raises m
    s.pr[threadIdx.x] = exp(s.lg[threadIdx.x] - m);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double denom = 0.0, gsum = 0.0, gsel[kMaxK];
    for (int e = 0; e < E; ++e) denom += s.pr[e];
    unsigned long long taken = 0ull;
    int isel[kMaxK];
    for (int k = 0; k < K; ++k) {
      isel[k] = route_pick(s.lg, E, taken);
      gsel[k] = s.pr[isel[k]] / denom;
      gsum += gsel[k];
    }
    for (int k = 0; k < K; ++k) {
      p.idx_ws[t * K + k] = isel[k];
      if (p.idx_out) p.idx_out[t * K + k] = isel[k];
      p.gates_ws[t * K + k] = (float)(p.gate_mode == 1 ? gsel[k] / gsum : gsel[k]);
    }
  }
}
__global__ void __launch_bounds__(kRouteWarps * 32)
step_route(const RouteArgs p) {
  __shared__ RouteSmem s;
  pdl_trigger();                        // the first kernel of the chain: nothing before it is pending
  if (blockIdx.x == 0 && threadIdx.x < kStatusInts) p.status[threadIdx.x] = 0;
  route_token(p, blockIdx.x, s);
}

// ---------------------------------------------------------------------------------------------- projections
enum StepGemm { STEP_IN = 0, STEP_OUT = 1 };
struct StepGemmArgs {
  const bf16* x; int ldx;               // activation rows: IN: x [B, Dm]; OUT: Yg [B, De]
  const bf16* W; int Kd, n_rows;        // weights [E, n_rows, Kd]
  const int32_t* idx; const float* gates; int B, K, E;
  bf16* C; int ldc;                     // IN: XZ [B K, 2 De]; OUT: out [B, Dm] (K == 1) or Op [B K, Dm]
  // IN at top-1: the short conv
  int De; const bf16* w_conv; const float* b_conv; float* conv_state; int dconv; bf16* U;
  int tile_rows;                        // step_tc: rows per weight tile
};

// ROUTE (the In Proj of one or two tokens, while all its blocks are resident at once and there are few logits): every block finds the
// experts itself, 32 KB of router weights from the L2 with 8 experts, which takes less than a launch and the tables in between; one more
// block writes the routing out for the kernels to come.  With the window, taps and gate of a thread's output requested beside the weights and the tokens' operands of
// step_dt_scan beside delta_r: one token of 2048 channels 28.1 -> 23.1 us, of 1280 23.6 -> 20.0, top-2 of 16 experts 45.4 -> 41.6, two
// tokens 37.0 -> 33.3 (routing inside without the limit on the blocks: 37.7 and 45.5 for the last two, second waves route again).
// Every block reads all E rows of the router for every token: us a step, launch of its own / inside: one token, 8 experts of 2048 channels
// 21.0 / 19.4, 16 20.3 / 20.0, 24 21.8 / 22.0, 64 33.4 / 35.0; 64 of 1024 (one block an SM) 24.2 / 21.1, 64 of 1280 29.2 / 27.1, 64 of 1536 26.9 / 29.5; two
// tokens, 4 of 1024 16.2 / 15.6, 8 of 512 13.2 / 13.1, 8 of 1024 15.4 / 15.6, 16 of 1024 18.2 / 19.2, 64 of 1024 25.2 / 34.4.
bool route_inside_pays(int B, int K, int E, int Dm, int De, int num_sms) {
  const int slots = B * K < E ? B * K : E;
  if (B > 2 || (2 * De / 32 + 1) * slots > 2 * num_sms) return false;
  return B == 1 ? Dm <= 1280 || E * Dm <= 24 * 1536 : E * Dm <= 4096;
}
template <int MODE, int RT, int WARPS, bool ROUTE = false>
__global__ void __launch_bounds__(WARPS * 32, MODE == STEP_IN ? 2 : 1)
step_gemm(const StepGemmArgs p, const RouteArgs rt) {
  constexpr int ROWS = RT * 16, COLS = 8, PITCH = ROWS + 4, PAIRS = ROWS / 2;
  constexpr int U = RT == 2 ? 4 : 8;                 // 32-wide blocks in flight per warp
  static_assert(kStreamMin <= COLS + 1 && COLS * PAIRS <= WARPS * 32, "an expert's tokens are one group, an output pair a thread");
  static_assert(!ROUTE || (MODE == STEP_IN && WARPS == kRouteWarps), "");
  __shared__ __align__(16) float red[WARPS][COLS][PITCH];
  __shared__ int list[kStreamMin];                   // assignments of this block's expert
  __shared__ unsigned long long mask;
  __shared__ int count;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
  const int row0 = blockIdx.x * ROWS;
  const int nkb = p.Kd / 32;

  if (ROUTE) pdl_trigger();                          // the first kernel of the chain
  else if (MODE == STEP_IN) { pdl_wait(); pdl_trigger(); }      // (OUT: the routing tables are two kernels back, complete already)
  // the blockIdx.y-th selected expert and its assignments (in whatever order: a token's column does not matter)
  const int A = p.B * p.K;
  int mine = -1;                                     // thread a < A: the expert of assignment a
  if constexpr (ROUTE) {
    __shared__ RouteSmem rs;
    if (blockIdx.x == gridDim.x - 1) {
      if (blockIdx.y) return;
      if (threadIdx.x < kStatusInts) rt.status[threadIdx.x] = 0;
      for (int t = 0; t < p.B; ++t) { route_token(rt, t, rs); __syncthreads(); }
      return;
    }
    for (int t = 0; t < p.B; ++t) {
      route_logits(rt, t, rs);
      const int k = (int)threadIdx.x - t * p.K;      // thread t K + k walks the picks up to its own
      unsigned long long taken = 0ull;
      if (k >= 0 && k < p.K)
        for (int q = 0; q <= k; ++q) mine = route_pick(rs.lg, p.E, taken);
    }
  } else if (threadIdx.x < A) {
    mine = p.idx[threadIdx.x];
  }
  if (threadIdx.x == 0) { mask = 0ull; count = 0; }
  __syncthreads();
  if (mine >= 0) atomicOr(&mask, 1ull << mine);
  __syncthreads();
  unsigned long long mk = mask;
  for (int i = 0; i < (int)blockIdx.y && mk; ++i) mk &= mk - 1;
  if (!mk) {
    if (MODE == STEP_OUT) { pdl_wait(); pdl_trigger(); }
    return;
  }
  const int e = __ffsll(mk) - 1;
  if (mine == e) list[atomicAdd(&count, 1)] = threadIdx.x;
  __syncthreads();
  const int m = count;                               // tokens of this block
  const bf16* wrow[RT][2];
#pragma unroll
  for (int r = 0; r < RT; ++r)
#pragma unroll
    for (int h = 0; h < 2; ++h) wrow[r][h] = p.W + ((size_t)e * p.n_rows + row0 + r * 16 + h * 8 + g) * p.Kd + 8 * t4;

  // output of this thread: two adjacent rows of one token, and what it takes besides the products, requested with the weights
  const int j_out = threadIdx.x / PAIRS, row_out = row0 + (threadIdx.x % PAIRS) * 2;
  const bool has_out = j_out < m;
  const int a_out = has_out ? list[j_out] : 0;
  const bool conv = MODE == STEP_IN && p.U != nullptr && has_out && row_out < p.De;
  float2 win[3], taps[4], ub = make_float2(0.0f, 0.0f);
  float gate = 1.0f;
  float* const st = p.conv_state + (size_t)a_out * (p.dconv - 1) * p.De + row_out;
  auto fetch_out = [&]() {
    if (conv) {
      if (p.b_conv) ub = make_float2(p.b_conv[row_out], p.b_conv[row_out + 1]);
#pragma unroll
      for (int q = 0; q < 3; ++q)
        if (q < p.dconv - 1) win[q] = *reinterpret_cast<const float2*>(st + (size_t)q * p.De);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < p.dconv) taps[q] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p.w_conv + (size_t)q * p.De + row_out));
    }
    if (MODE == STEP_OUT && has_out && p.K == 1) gate = p.gates[a_out];
  };

  bool waited = MODE == STEP_IN;
  const int tok_g = g < m ? list[g] / p.K : -1;
  const bf16* xrow = tok_g >= 0 ? p.x + (size_t)tok_g * p.ldx + 8 * t4 : nullptr;
  float acc[RT][4] = {};
  for (int kb0 = warp; kb0 < nkb; kb0 += WARPS * U) {
    uint4 wq[U][RT][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int kb = min(kb0 + u * WARPS, nkb - 1);      // past the end: the last block again, against zero activations
#pragma unroll
      for (int r = 0; r < RT; ++r) { wq[u][r][0] = ld_stream(wrow[r][0] + kb * 32); wq[u][r][1] = ld_stream(wrow[r][1] + kb * 32); }
    }
    if (kb0 == warp) fetch_out();
    if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int kb = kb0 + u * WARPS;
      const uint4 xq = (xrow && kb < nkb) ? ld_act(xrow + kb * 32) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int r = 0; r < RT; ++r) mma_block(acc[r], wq[u][r][0], wq[u][r][1], xq);
    }
  }
  if (warp >= nkb) fetch_out();                      // (a warp without a block of the contracted index)
  if (!waited) { pdl_wait(); pdl_trigger(); }
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    red[warp][2 * t4][r * 16 + g] = acc[r][0];
    red[warp][2 * t4 + 1][r * 16 + g] = acc[r][1];
    red[warp][2 * t4][r * 16 + g + 8] = acc[r][2];
    red[warp][2 * t4 + 1][r * 16 + g + 8] = acc[r][3];
  }
  __syncthreads();
  if (!has_out) return;
  // sums over the warps, output op
  float2 v = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int w = 0; w < WARPS; ++w) {
    const float2 q = *reinterpret_cast<const float2*>(&red[w][j_out][row_out - row0]);
    v.x += q.x; v.y += q.y;
  }
  const size_t a = a_out;
  const int row = row_out;
  if (MODE == STEP_OUT) {
    *reinterpret_cast<__nv_bfloat162*>(p.C + a * p.ldc + row) = __floats2bfloat162_rn(v.x * gate, v.y * gate);
  } else if (p.U == nullptr) {                       // K > 1: rows of the assignment, summed over the slots by step_conv
    *reinterpret_cast<__nv_bfloat162*>(p.C + a * p.ldc + row) = __floats2bfloat162_rn(v.x, v.y);
  } else if (row >= p.De) {                          // Gate Proj row, activated
    *reinterpret_cast<__nv_bfloat162*>(p.C + a * p.ldc + row) = __floats2bfloat162_rn(silu_fast(v.x), silu_fast(v.y));
  } else {
    // Conv Proj row: H (rounded to the storage type), the conv over the caller's window, and the window moved on
    const __nv_bfloat162 hb = __floats2bfloat162_rn(v.x, v.y);
    const float2 h = __bfloat1622float2(hb);
    float2 u = ub;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < p.dconv) {
        const float2 hv = q < p.dconv - 1 ? win[q < 3 ? q : 2] : h;
        u.x = fmaf(taps[q].x, hv.x, u.x); u.y = fmaf(taps[q].y, hv.y, u.y);
      }
    *reinterpret_cast<__nv_bfloat162*>(p.U + a * p.De + row) = __floats2bfloat162_rn(silu_fast(u.x), silu_fast(u.y));
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (q + 1 < p.dconv - 1) *reinterpret_cast<float2*>(st + (size_t)q * p.De) = win[q + 1];
    *reinterpret_cast<float2*>(st + (size_t)(p.dconv - 2) * p.De) = h;
  }
}

// The same for more assignments, where the weights of most experts are walked and streaming them is all that counts: tcgen05 with
// the weights as the M = 128 operand and an expert's tokens (16, 32 or 64 columns, at most TC_N per pass) as N.  One persistent CTA
// per SM takes (expert, 128 weight rows) tiles; warp 0 keeps a ring of operand stages full of weights (128 x 128 by two TMA loads),
// warps 6..9 put the tokens' rows beside them (16-byte loads on their indices into the swizzled layout: nothing is permuted in
// memory, and the TMA unit is left to the weights -- gather4 loads cost it about 28 ns a row, more than the weights of the stage),
// warp 1 issues the MMAs, warps 2..5 drain the accumulator (lane = weight row, column = token; double-buffered) while the next tile
// streams.  The register-fed kernel above reached 3.6 TB/s at 64 tokens (268 MB in 74 us), waiting on its own sums and output ops.
constexpr int TC_N = 64;                             // token columns per pass
constexpr int TC_W_HALF = 128 * BLOCK_K * 2, TC_X_HALF = TC_N * BLOCK_K * 2;      // a stage: two 64-wide K blocks of both operands
constexpr int TC_A_BYTES = 2 * TC_W_HALF, TC_STAGE = TC_A_BYTES + 2 * TC_X_HALF;
constexpr int TC_STAGES = 4;
constexpr int TC_X_FLIGHT = 2;                       // stages of token rows in flight (at most TC_STAGES - 2)
constexpr int TC_SMEM = TC_STAGES * TC_STAGE + 1024;
constexpr int TC_THREADS = 320;

template <int MODE>
__global__ void __launch_bounds__(TC_THREADS, 1)
step_tc(const __grid_constant__ CUtensorMap tmap_w, const StepGemmArgs p, int32_t* __restrict__ status, uint32_t wait_limit, bool stall) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ int cnt[kMaxE], off[kMaxE + 1], fill[kMaxE], act[kMaxE], n_act_s;
  __shared__ short list[kStepMaxAssign], tok[kStepMaxAssign];      // assignments by expert, and their tokens
  __shared__ __align__(8) unsigned long long bars[2 * TC_STAGES + 5];
  __shared__ uint32_t tmem_s;
  __shared__ int abort_s;
  volatile int* abort_flag = &abort_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
  auto empty_bar = [&](int s) { return smem_u32(&bars[TC_STAGES + s]); };
  auto tfull_bar = [&](int a) { return smem_u32(&bars[2 * TC_STAGES + a]); };
  auto tempty_bar = [&](int a) { return smem_u32(&bars[2 * TC_STAGES + 2 + a]); };
  const uint32_t drain_bar = smem_u32(&bars[2 * TC_STAGES + 4]);

  if (MODE == STEP_IN) { pdl_wait(); pdl_trigger(); }      // OUT: the routing is two kernels back; the wait comes before the activations
  if (tid == 0) {
    for (int s = 0; s < TC_STAGES; ++s) { mbar_init(full_bar(s), 1 + 4); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 4); }
    mbar_init(drain_bar, 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid < kMaxE) { cnt[tid] = 0; fill[tid] = 0; }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)), "r"(2 * TC_N) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_s;
  // assignments of every expert (in whatever order: a token's column does not matter)
  const int A = p.B * p.K;
  for (int a = tid; a < A; a += TC_THREADS) atomicAdd(&cnt[p.idx[a]], 1);
  __syncthreads();
  auto cols = [](int m) { return m > 32 ? 64 : m > 16 ? 32 : 16; };      // N of a pass over m tokens
  if (tid == 0) {
    int o = 0, n = 0;
    for (int e = 0; e < p.E; ++e) { off[e] = o; o += cnt[e]; if (cnt[e]) act[n++] = e; }
    n_act_s = n;
  }
  __syncthreads();
  for (int a = tid; a < A; a += TC_THREADS) {
    const int e = p.idx[a], at = off[e] + atomicAdd(&fill[e], 1);
    list[at] = (short)a; tok[at] = (short)(a / p.K);
  }
  __syncthreads();
  const int tpe = (p.n_rows + p.tile_rows - 1) / p.tile_rows;      // weight tiles per expert
  const int total = n_act_s * tpe;
  const int num_kb = (p.Kd + 2 * BLOCK_K - 1) / (2 * BLOCK_K);      // stages of 128; d_model may leave half of the last one
  // every weight tile starts at its own K block: in step the CTAs would all read the same 128-byte column of rows that are a power of two
  // apart.  The start depends on the tile's rows alone, so a token's sums do not depend on the CTA, i.e. on the batch around it.
  auto rot_of = [&](int w) { return (w % tpe * 5) % num_kb; };
  auto k_of = [&](int kb, int rot) { return (kb + rot < num_kb ? kb + rot : kb + rot - num_kb) * 2 * BLOCK_K; };

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the weights (nothing here depends on the launch before)
    if (lane == 0) {
    int stage = 0, issued = 0; uint32_t phase = 0;
    bool ok = true;
    // fault injection (tests only): from the second stage on 16 bytes are expected that never come
    uint32_t tx = 2 * p.tile_rows * BLOCK_K * 2;
    const uint32_t tx_later = tx + (stall ? 16u : 0u);
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const int e = act[w / tpe], row = e * p.n_rows + (w % tpe) * p.tile_rows, rot = rot_of(w);
      for (int n0 = 0; n0 < cnt[e] && ok; n0 += TC_N)
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, wait_limit)) { ok = false; break; }
          const int k0 = k_of(kb, rot);
          mbar_expect_tx(full_bar(stage), tx);
          tx = tx_later;
          tma_load_2d(base + stage * TC_STAGE, &tmap_w, full_bar(stage), k0, row);
          tma_load_2d(base + stage * TC_STAGE + TC_W_HALF, &tmap_w, full_bar(stage), k0 + BLOCK_K, row);
          ++issued;
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
        }
    }
    if (!ok) {
      if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 4); }
      *abort_flag = 1;
    }
    if (*abort_flag) {                               // give the copies still in flight a bounded time to land before the CTA exits
      for (int i = 0; i < min(issued, TC_STAGES); ++i) {
        if (--stage < 0) { stage = TC_STAGES - 1; phase ^= 1u; }
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(full_bar(stage), phase)) break;
      }
    }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      int acc = 0; uint32_t acc_phase = 0;
      bool ok = true, issued_any = false;
      for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
        const int e = act[w / tpe], rot = rot_of(w);
        for (int n0 = 0; n0 < cnt[e] && ok; n0 += TC_N) {
          const int n16 = cols(min(cnt[e] - n0, TC_N));
          const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n16 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
          if (!mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag, wait_limit)) { ok = false; break; }
          tc_fence_after();
          for (int kb = 0; kb < num_kb; ++kb) {
            if (!mbar_wait(full_bar(stage), phase, abort_flag, wait_limit)) { ok = false; break; }
            tc_fence_after();
            const int halves = k_of(kb, rot) + BLOCK_K < p.Kd ? 2 : 1;
            for (int hf = 0; hf < halves; ++hf) {
              const uint64_t adesc = make_smem_desc(base + stage * TC_STAGE + hf * TC_W_HALF);
              const uint64_t bdesc = make_smem_desc(base + stage * TC_STAGE + TC_A_BYTES + hf * TC_X_HALF);
#pragma unroll
              for (int k = 0; k < BLOCK_K / UMMA_K; ++k)
                umma_bf16(tmem_base + acc * TC_N, adesc + (uint64_t)(2 * k), bdesc + (uint64_t)(2 * k), idesc, (kb | hf | k) != 0 ? 1u : 0u);
            }
            umma_commit(empty_bar(stage));
            issued_any = true;
            if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          umma_commit(tfull_bar(acc));
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
      }
      if (!ok) {
        if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 5); }
        *abort_flag = 1;
      }
      if (*abort_flag && issued_any) {
        umma_commit(drain_bar);
        for (uint32_t it = 0; it < (wait_limit >> 2); ++it)
          if (mbar_try_wait(drain_bar, 0)) break;
      }
    }
  } else if (warp >= 6) {
    // ---------------------------------------------------------------- token rows of every stage: 128 threads, 16-byte pieces
    const int l = tid - 6 * 32, lrow = l >> 3, chunk = l & 7;
    if (MODE == STEP_OUT) { pdl_wait(); pdl_trigger(); }
    int stage = 0, pub = 0, pending = 0; uint32_t phase = 0;
    bool ok = true;
    auto publish = [&]() {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full_bar(pub));
      if (++pub == TC_STAGES) pub = 0;
      --pending;
    };
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const int e = act[w / tpe], rot = rot_of(w);
      for (int n0 = 0; n0 < cnt[e] && ok; n0 += TC_N) {
        const int m = min(cnt[e] - n0, TC_N), nq = cols(m) >> 4;      // 16-row groups: 1, 2 or 4 pieces per thread and stage
        const bf16* src[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) src[q] = p.x + (size_t)tok[off[e] + n0 + min(lrow + 16 * q, m - 1)] * p.ldx + chunk * 8;      // (rows past the last token repeat it)
        for (int kb = 0; kb < num_kb; ++kb) {
          ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, wait_limit));
          if (!ok) break;
          const uint32_t dst = base + stage * TC_STAGE + TC_A_BYTES + lrow * 128 + ((chunk ^ (lrow & 7)) << 4);
          const int k0 = k_of(kb, rot);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < nq) {
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q * 16 * 128), "l"(src[q] + k0) : "memory");
              if (k0 + BLOCK_K < p.Kd)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + TC_X_HALF + q * 16 * 128), "l"(src[q] + k0 + BLOCK_K) : "memory");
            }
          asm volatile("cp.async.commit_group;" ::: "memory");
          if (++stage == TC_STAGES) { stage = 0; phase ^= 1u; }
          // the stage of TC_X_FLIGHT copies ago has landed: publish it to the tensor cores
          if (++pending > TC_X_FLIGHT) {
            asm volatile("cp.async.wait_group %0;" ::"n"(TC_X_FLIGHT) : "memory");
            publish();
          }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    while (pending > 0) publish();
    if (!ok && lane == 0) {
      if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 7); }
      *abort_flag = 1;
    }
  } else {
    // ---------------------------------------------------------------- output: lane = weight row, column = token
    const int quarter = warp & 3;
    int acc = 0; uint32_t acc_phase = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < total && ok; w += gridDim.x) {
      const int e = act[w / tpe], r = quarter * 32 + lane, row = (w % tpe) * p.tile_rows + r;
      const bool row_ok = r < p.tile_rows && row < p.n_rows;      // (rows of the stage beyond the tile keep what they hold)
      const bool conv = MODE == STEP_IN && p.U != nullptr && row < p.De && row_ok;
      float wv[4], bias = 0.0f;
      if (conv) {
        if (p.b_conv) bias = p.b_conv[row];
#pragma unroll
        for (int q = 0; q < 4; ++q) wv[q] = q < p.dconv ? to_f32(p.w_conv[(size_t)q * p.De + row]) : 0.0f;
      }
      for (int n0 = 0; n0 < cnt[e] && ok; n0 += TC_N) {
        const int m = min(cnt[e] - n0, TC_N);
        const short* mine = list + off[e] + n0;
        if (!__all_sync(0xffffffffu, mbar_wait(tfull_bar(acc), acc_phase, abort_flag, wait_limit))) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)acc * TC_N;
        for (int c0 = 0; c0 < m; c0 += 32) {
          uint32_t r[32];
          tmem_ld32_issue(taddr + c0, r);
          tmem_ld_wait(r);
          const int mm = m - c0;
#pragma unroll
          for (int jb = 0; jb < 32; jb += 8) {
            if (jb >= mm) break;
            if (conv) {
              float win[8][3];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float* st = p.conv_state + (size_t)mine[c0 + min(jb + j, mm - 1)] * (p.dconv - 1) * p.De + row;
#pragma unroll
                for (int q = 0; q < 3; ++q) win[j][q] = q < p.dconv - 1 ? st[(size_t)q * p.De] : 0.0f;
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (jb + j >= mm) break;
                const size_t a = mine[c0 + jb + j];
                // Conv Proj row: H (rounded to the storage type), the conv over the caller's window, and the window moved on
                const float h = to_f32(__float2bfloat16_rn(__uint_as_float(r[jb + j])));
                float u = bias;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  if (q >= p.dconv) break;
                  u = fmaf(wv[q], q < p.dconv - 1 ? win[j][q < 3 ? q : 2] : h, u);
                }
                p.U[a * p.De + row] = __float2bfloat16_rn(silu_fast(u));
                float* st = p.conv_state + a * (p.dconv - 1) * p.De + row;
#pragma unroll
                for (int q = 0; q < 2; ++q)
                  if (q + 1 < p.dconv - 1) st[(size_t)q * p.De] = win[j][q + 1];
                st[(size_t)(p.dconv - 2) * p.De] = h;
              }
            } else if (row_ok) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (jb + j >= mm) break;
                const size_t a = mine[c0 + jb + j];
                float v = __uint_as_float(r[jb + j]);
                if (MODE == STEP_IN && p.U != nullptr) v = silu_fast(v);      // Gate Proj row
                if (MODE == STEP_OUT && p.K == 1) v *= p.gates[a];
                p.C[a * p.ldc + row] = __float2bfloat16_rn(v);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty_bar(acc));
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) {
      if (!*abort_flag) { atomicExch(status + kStatCode, ROM_ERR_DEVICE_TIMEOUT); atomicExch(status + kStatWhere, 6); }
      *abort_flag = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * TC_N) : "memory");
  }
}

// K > 1: H and Z of a token are sums over its slots (ascending), then the conv as above and G = SiLU(Z).  Two channels per thread.
__global__ void __launch_bounds__(128)
step_conv(const bf16* __restrict__ XZ, int K, int De, const bf16* __restrict__ w_conv, const float* __restrict__ b_conv,
          float* __restrict__ conv_state, int dconv, bf16* __restrict__ U, bf16* __restrict__ Zs) {
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) * 2;
  const size_t b = blockIdx.y;
  const bool in = c < De;
  float* st = conv_state + b * (size_t)(dconv - 1) * De + c;
  float2 win[3], w[4], u = make_float2(0.0f, 0.0f);
  if (in) {                                          // the window and the taps do not depend on the launch before
    if (b_conv) u = make_float2(b_conv[c], b_conv[c + 1]);
    for (int q = 0; q < dconv - 1; ++q) win[q] = *reinterpret_cast<const float2*>(st + (size_t)q * De);
    for (int q = 0; q < dconv; ++q) w[q] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(w_conv + (size_t)q * De + c));
  }
  pdl_wait();
  pdl_trigger();
  if (!in) return;
  float2 h = make_float2(0.0f, 0.0f), z = h;
  for (int k = 0; k < K; ++k) {
    const bf16* r = XZ + (b * K + k) * (size_t)(2 * De) + c;
    const float2 hv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(r)), zv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(r + De));
    h.x += hv.x; h.y += hv.y; z.x += zv.x; z.y += zv.y;
  }
  for (int q = 0; q < dconv; ++q) {
    const float2 hv = q < dconv - 1 ? win[q] : h;
    u.x = fmaf(w[q].x, hv.x, u.x); u.y = fmaf(w[q].y, hv.y, u.y);
  }
  *reinterpret_cast<__nv_bfloat162*>(U + b * De + c) = __floats2bfloat162_rn(silu_fast(u.x), silu_fast(u.y));
  *reinterpret_cast<__nv_bfloat162*>(Zs + b * De + c) = __floats2bfloat162_rn(silu_fast(z.x), silu_fast(z.y));
  for (int q = 0; q + 1 < dconv - 1; ++q) *reinterpret_cast<float2*>(st + (size_t)q * De) = win[q + 1];
  *reinterpret_cast<float2*>(st + (size_t)(dconv - 2) * De) = h;
}

// ---------------------------------------------------------------------------------------------- x Proj
// 16 weight rows and up to 16 tokens a cluster of eight CTAs, which share the contracted index: its 32-wide blocks are dealt out to the
// CTAs and their warps, the partial sums meet in shared memory (warps, in order) and across the cluster (CTAs, in order; the order is
// the same for every batch).  What bounds it: latency; a row is 2 De bytes, and one block per 16 rows and 8 tokens, as before, took
// 131 KB of weights through one SM (7.8 us from the end of the In Proj at 64 tokens).  us a step, before / 64, 32, 16, 8 tokens a
// cluster: 64 tokens of 2048 channels 101.9 / 101.7, 103.6, 100.1, 103.3; 8 tokens 74.3 / 71.5, 71.9, 71.1, 71.5; 1 token 23.6 / -, -,
// 23.2, -; 4 of 1024 35.1 / -, -, 33.2, -.
constexpr int XC = 8, X_TOK = 16, X_WARPS = 8;
__global__ void __launch_bounds__(X_WARPS * 32)
step_xproj(const bf16* __restrict__ U, const bf16* __restrict__ W, int De, int R, bf16* __restrict__ delta_r, float* __restrict__ Bm,
           float* __restrict__ Cm, int B) {
  constexpr int ROWS = 16, NG = X_TOK / 8, KB = 2;      // KB: blocks of a warp in flight
  __shared__ __align__(16) float red[X_WARPS][X_TOK][ROWS + 1];
  __shared__ float part[X_TOK][ROWS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
  const int rank = (int)cluster_rank(), row0 = blockIdx.y * ROWS, tb = blockIdx.z * X_TOK, nt = min(X_TOK, B - tb);
  const int nkb = De / 32, lo = nkb * rank / XC, hi = nkb * (rank + 1) / XC;
  const bf16* w0 = W + (size_t)(row0 + g) * De + 8 * t4;
  const bf16* w1 = w0 + (size_t)8 * De;
  const uint4 zero4 = make_uint4(0, 0, 0, 0);
  float acc[NG][4] = {};
  bool waited = false;
  for (int kb0 = lo + warp; kb0 < hi; kb0 += X_WARPS * KB) {
    uint4 q0[KB], q1[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int kb = kb0 + k * X_WARPS;
      q0[k] = kb < hi ? ld_stream(w0 + kb * 32) : zero4;
      q1[k] = kb < hi ? ld_stream(w1 + kb * 32) : zero4;
    }
    if (!waited) { pdl_wait(); pdl_trigger(); waited = true; }
    uint4 xq[NG][KB];                  // (all of them requested before the first is used)
#pragma unroll
    for (int n = 0; n < NG; ++n)
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        const int kb = kb0 + k * X_WARPS;
        xq[n][k] = n * 8 + g < nt && kb < hi ? ld_act(U + (size_t)(tb + n * 8 + g) * De + 8 * t4 + kb * 32) : zero4;
      }
#pragma unroll
    for (int n = 0; n < NG; ++n)
#pragma unroll
      for (int k = 0; k < KB; ++k) mma_block(acc[n], q0[k], q1[k], xq[n][k]);
  }
  if (!waited) { pdl_wait(); pdl_trigger(); }
#pragma unroll
  for (int n = 0; n < NG; ++n) {
    if (n * 8 >= nt) break;
    float (*r)[ROWS + 1] = red[warp] + n * 8 + 2 * t4;
    r[0][g] = acc[n][0]; r[1][g] = acc[n][1]; r[0][g + 8] = acc[n][2]; r[1][g + 8] = acc[n][3];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nt * ROWS; i += X_WARPS * 32) {
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < X_WARPS; ++w) v += red[w][i / ROWS][i % ROWS];
    part[i / ROWS][i % ROWS] = v;
  }
  cluster_sync();
  // CTA q finishes tokens q, q + 8, ...
  for (int i = threadIdx.x; i < X_TOK / XC * ROWS; i += X_WARPS * 32) {
    const int t = (i / ROWS) * XC + rank, r = i % ROWS, row = row0 + r;
    if (t >= nt) continue;
    float q[XC], v = 0.0f;
#pragma unroll
    for (int c = 0; c < XC; ++c) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(q[c]) : "r"(map_rank(smem_u32(&part[t][r]), c)) : "memory");
#pragma unroll
    for (int c = 0; c < XC; ++c) v += q[c];
    const size_t tok = tb + t;
    if (row < R) delta_r[tok * R + row] = __float2bfloat16_rn(v);
    else if (row < R + NST) Bm[tok * NST + row - R] = v;
    else Cm[tok * NST + row - R - NST] = v;
  }
  cluster_sync();                      // nobody leaves while its sums may still be read
}

// ---------------------------------------------------------------------------------------------- dt Proj + recurrence
// A warp takes 16 channels x 8 tokens: Delta by MMA, then one (channel half, token) at a time with four lanes per channel (four
// states each), so that states move as whole 512-byte rows.  The states (the traffic that counts: 8 KB in and out per warp), A and
// the dt weights are requested before the wait; B, C, u and the gate of the block's tokens right after it, into shared memory (read
// token by token each was waited for: 64 sequences 104.1 -> 101.6 us a step, 200: 158.1 -> 147.6).
template <bool ZOH>
__global__ void __launch_bounds__(128, 4)
step_dt_scan(const bf16* __restrict__ delta_r, const bf16* __restrict__ W_dt, const float* __restrict__ b_dt, int R,
             const float* __restrict__ A, const float* __restrict__ Bm, const float* __restrict__ Cm, const float* __restrict__ D,
             const bf16* __restrict__ U, const bf16* __restrict__ Z, int ldz, float* __restrict__ ssm_state, bf16* __restrict__ Yg, int B, int De) {
  __shared__ float dls[4][8][17], ys[4][8][17];
  __shared__ __align__(16) float bcs[8][2 * NST];
  __shared__ __align__(16) bf16 us[8][64], zs[8][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t4 = lane & 3;
  const int c0 = (blockIdx.x * 4 + warp) * 16;
  const int tb = blockIdx.y * 8, nt = min(8, B - tb);
  const uint4 zero4 = make_uint4(0, 0, 0, 0);
  float4* hp = reinterpret_cast<float4*>(ssm_state) + ((size_t)tb * De + c0 + g) * 4 + t4;      // token tl, half hf: + (tl De + 8 hf) 4
  float4 h[8][2];
#pragma unroll
  for (int tl = 0; tl < 8; ++tl)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) h[tl][hf] = tl < nt ? hp[((size_t)tl * De + 8 * hf) * 4] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  uint4 wq[4][2];                                    // the first 128 columns of the dt weights
#pragma unroll
  for (int kb = 0; kb < 4; ++kb) {
    const bool in = kb * 32 + 8 * t4 < R;
    wq[kb][0] = in ? ld_stream(W_dt + (size_t)(c0 + g) * R + kb * 32 + 8 * t4) : zero4;
    wq[kb][1] = in ? ld_stream(W_dt + (size_t)(c0 + g + 8) * R + kb * 32 + 8 * t4) : zero4;
  }
  const float4 a0 = __ldg(reinterpret_cast<const float4*>(A + (size_t)(c0 + g) * NST) + t4), a1 = __ldg(reinterpret_cast<const float4*>(A + (size_t)(c0 + 8 + g) * NST) + t4);
  const float av[2][4] = {{a0.x, a0.y, a0.z, a0.w}, {a1.x, a1.y, a1.z, a1.w}};
  const float bias[2] = {b_dt ? b_dt[c0 + g] : 0.0f, b_dt ? b_dt[c0 + 8 + g] : 0.0f}, Dc[2] = {D ? D[c0 + g] : 0.0f, D ? D[c0 + 8 + g] : 0.0f};
  pdl_wait();
  pdl_trigger();
  // what the tokens need besides, in flight with delta_r: token by token these loads would be waited for one after another
  const int tid = threadIdx.x, pt = tid >> 3, pc = tid & 7;      // threads 0..63: eight 16-byte pieces a token
  uint4 q_bc = zero4, q_uz = zero4;
  if ((pt & 7) < nt) {
    const size_t t = tb + (pt & 7);
    if (pt < 8) q_bc = reinterpret_cast<const uint4*>((pc < 4 ? Bm : Cm) + t * NST)[pc & 3];
    const int cb = blockIdx.x * 64 + 8 * pc;
    q_uz = *reinterpret_cast<const uint4*>(pt < 8 ? U + t * De + cb : Z + t * ldz + cb);
  }
  float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  const bool tok_ok = g < nt;
  const bf16* dr = delta_r + (size_t)(tb + g) * R + 8 * t4;
#pragma unroll
  for (int kb = 0; kb < 4; ++kb) {
    if (kb * 32 >= R) break;
    mma_block(acc, wq[kb][0], wq[kb][1], (tok_ok && kb * 32 + 8 * t4 < R) ? ld_act(dr + kb * 32) : zero4);
  }
  for (int kb = 4; kb * 32 < R; ++kb) {
    const bool in = kb * 32 + 8 * t4 < R;
    const uint4 q0 = in ? ld_stream(W_dt + (size_t)(c0 + g) * R + kb * 32 + 8 * t4) : zero4;
    const uint4 q1 = in ? ld_stream(W_dt + (size_t)(c0 + g + 8) * R + kb * 32 + 8 * t4) : zero4;
    mma_block(acc, q0, q1, (tok_ok && in) ? ld_act(dr + kb * 32) : zero4);
  }
  if (pt < 8) { *reinterpret_cast<uint4*>(&bcs[pt][4 * pc]) = q_bc; *reinterpret_cast<uint4*>(&us[pt][8 * pc]) = q_uz; }
  else *reinterpret_cast<uint4*>(&zs[pt - 8][8 * pc]) = q_uz;
#pragma unroll
  for (int j = 0; j < 4; ++j) dls[warp][2 * t4 + (j & 1)][g + 8 * (j >> 1)] = softplus_fast(acc[j] + bias[j >> 1]);
  __syncthreads();
  float a2[2][4], nk[2][4];
#pragma unroll
  for (int hf = 0; hf < 2; ++hf)
#pragma unroll
    for (int i = 0; i < 4; ++i) { a2[hf][i] = av[hf][i] * kLog2e; nk[hf][i] = -1.0f / av[hf][i]; }
#pragma unroll
  for (int tl = 0; tl < 8; ++tl) {
    if (tl >= nt) break;
    const float4 b4 = *reinterpret_cast<const float4*>(&bcs[tl][4 * t4]), c4 = *reinterpret_cast<const float4*>(&bcs[tl][NST + 4 * t4]);
    const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int cl = warp * 16 + 8 * hf + g;
      const float uu = to_f32(us[tl][cl]), dl = dls[warp][tl][8 * hf + g];
      float hv[4] = {h[tl][hf].x, h[tl][hf].y, h[tl][hf].z, h[tl][hf].w};
      float y = 0.0f;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float a = ex2_ftz(dl * a2[hf][i]);
        if (ZOH) {
          const float w = (uu * nk[hf][i]) * bb[i];
          hv[i] = fmaf(a, hv[i] - w, w);
        } else {
          hv[i] = fmaf(a, hv[i], (dl * uu) * bb[i]);
        }
        y = fmaf(cc[i], hv[i], y);
      }
      hp[((size_t)tl * De + 8 * hf) * 4] = make_float4(hv[0], hv[1], hv[2], hv[3]);
      y += __shfl_xor_sync(0xffffffffu, y, 1);
      y += __shfl_xor_sync(0xffffffffu, y, 2);
      if (t4 == 0) ys[warp][tl][8 * hf + g] = fmaf(Dc[hf], uu, y) * to_f32(zs[tl][cl]);
    }
  }
  __syncwarp();
  if (g < nt) {                                      // lane (token g, channels 4 t4 ..)
    const float* y4 = &ys[warp][g][4 * t4];
    __nv_bfloat162 lo = __floats2bfloat162_rn(y4[0], y4[1]), hi = __floats2bfloat162_rn(y4[2], y4[3]);
    *reinterpret_cast<uint2*>(Yg + (size_t)(tb + g) * De + c0 + 4 * t4) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
  }
}

// out[t, :] = sum_k gate_k Op[t K + k, :]
__global__ void __launch_bounds__(128)
step_combine(const bf16* __restrict__ Op, const float* __restrict__ gates, bf16* __restrict__ out, int Dm, int K) {
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) * 2;
  const size_t t = blockIdx.y;
  pdl_wait();
  if (c >= Dm) return;
  float2 acc = make_float2(0.0f, 0.0f);
  for (int k = 0; k < K; ++k) {
    const float gk = gates[t * K + k];
    const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(Op + (t * K + k) * (size_t)Dm + c));
    acc.x = fmaf(gk, v.x, acc.x); acc.y = fmaf(gk, v.y, acc.y);
  }
  *reinterpret_cast<__nv_bfloat162*>(out + t * Dm + c) = __floats2bfloat162_rn(acc.x, acc.y);
}

// Launch that may begin while the kernel before it on the stream drains (it waits in griddepcontrol.wait).
template <typename... P, typename... Args>
cudaError_t launch_chained_smem(void (*kern)(P...), dim3 grid, int threads, int smem, cudaStream_t st, bool chained, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.dynamicSmemBytes = smem;
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

template <typename... P, typename... Args>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, int threads, cudaStream_t st, bool chained, Args... args) {
  return launch_chained_smem(kern, grid, threads, 0, st, chained, args...);
}

template <int MODE>
cudaError_t launch_step_tc(const StepGemmArgs& a, int num_sms, int32_t* status, bool test_stall, cudaStream_t st) {
  CUtensorMap tw;
  if (!make_tmap(&tw, a.W, (uint64_t)a.E * a.n_rows, (uint64_t)a.Kd, (uint64_t)a.Kd, a.tile_rows)) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(step_tc<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
  if (e != cudaSuccess) return e;
  return launch_chained_smem(step_tc<MODE>, dim3(num_sms), TC_THREADS, TC_SMEM, st, true, tw, a, status,
                             test_stall ? WAIT_LIMIT_TEST : WAIT_LIMIT, test_stall);
}

// Rows per weight tile: the multiple of 16 in 96 .. 128 for which the CTAs' rounds x rows is smallest when every expert is selected
// (d_model 2048, 8 experts: 112 rows make the in_proj 4.0 rounds of tiles, where 128 need 4 rounds for 3.46).  Not a function of the
// batch, which would show in the last bits of every token's result.
int pick_tile_rows(int E, int n_rows, int num_sms) {
  int best = 128;
  long long cost = -1;
  for (int h = 128; h >= 96; h -= 16) {
    const long long tiles = (long long)E * ((n_rows + h - 1) / h), c = (tiles + num_sms - 1) / num_sms * h;
    if (cost < 0 || c < cost) { cost = c; best = h; }
  }
  return best;
}

template <int MODE, int RT, int WARPS>
cudaError_t launch_step_gemm(const StepGemmArgs& a, dim3 grid, cudaStream_t st) {
  return launch_chained(step_gemm<MODE, RT, WARPS>, grid, WARPS * 32, st, true, a, RouteArgs{});
}

}  // namespace

bool step_small_applicable(const rom_config& c) {
  // (the fault injection stalls the second operand stage of a kernel with bounded waits: the general sequence serves it below
  // kStreamMin, where there is no such kernel here, and up to 128 columns, which are one stage)
  const bool flags_ok = c.flags == 0 || (c.flags == ROM_FLAG_TEST_STALL && c.B * c.K >= kStreamMin && c.d_model > 2 * BLOCK_K);
  return c.dtype == ROM_BF16 && flags_ok && c.small_proj_experts <= 1 && c.L == 1 && c.B <= kStepMaxTokens && c.B * c.K <= kStepMaxAssign &&
         c.dt_rank % 16 == 0;
}

cudaError_t launch_step_small(const rom_config& c, const rom_weights& w, const void* x, float* conv_state, float* ssm_state, void* out,
                              int32_t* topk_idx_out, float* gates, char* W, const WsLayout& lay, cudaStream_t st) {
  const int B = c.B, De = c.d_inner, Dm = c.d_model, R = c.dt_rank, K = c.K;
  int32_t* idx = reinterpret_cast<int32_t*>(W + lay.topk_idx);
  bf16* XZ = reinterpret_cast<bf16*>(W + lay.XZp);
  bf16* U = reinterpret_cast<bf16*>(W + lay.U);
  bf16* Zs = reinterpret_cast<bf16*>(W + lay.Zs);
  bf16* dr = reinterpret_cast<bf16*>(W + lay.delta_r);
  bf16* Yg = reinterpret_cast<bf16*>(W + lay.Ygp);
  bf16* Op = reinterpret_cast<bf16*>(W + lay.Op);
  float* Bm = reinterpret_cast<float*>(W + lay.Bm);
  float* Cm = reinterpret_cast<float*>(W + lay.Cm);
  const RouteArgs rt{(const bf16*)x, (const bf16*)w.W_r, w.b_r, Dm, c.E, K, c.gate_mode, idx, gates, topk_idx_out, reinterpret_cast<int32_t*>(W + lay.status)};
  int num_sms = 0;
  cudaError_t e = current_device_sm_count(&num_sms);
  if (e != cudaSuccess) return e;
  const int slots = B * K < c.E ? B * K : c.E;      // selected experts at most
  // few assignments: latency counts, the register-fed kernel spreads them over more blocks; more: stream the weights
  const bool stream = B * K >= kStreamMin, route_inside = !stream && route_inside_pays(B, K, c.E, Dm, De, num_sms);
  if (!route_inside && (e = launch_chained(step_route, dim3(B), kRouteWarps * 32, st, false, rt)) != cudaSuccess) return e;
  StepGemmArgs a{};
  a.x = (const bf16*)x; a.ldx = Dm; a.W = (const bf16*)w.W_inz; a.Kd = Dm; a.n_rows = 2 * De;
  a.idx = idx; a.gates = gates; a.B = B; a.K = K; a.E = c.E; a.C = XZ; a.ldc = 2 * De; a.De = De;
  if (K == 1) { a.w_conv = (const bf16*)w.w_conv; a.b_conv = w.b_conv; a.conv_state = conv_state; a.dconv = c.d_conv; a.U = U; }
  int32_t* status = reinterpret_cast<int32_t*>(W + lay.status);
  a.tile_rows = pick_tile_rows(c.E, 2 * De, num_sms);
  if (stream) e = launch_step_tc<STEP_IN>(a, num_sms, status, c.flags & ROM_FLAG_TEST_STALL, st);
  else if (route_inside) e = launch_chained(step_gemm<STEP_IN, 2, 8, true>, dim3(2 * De / 32 + 1, slots), 256, st, false, a, rt);
  else e = launch_step_gemm<STEP_IN, 2, 8>(a, dim3(2 * De / 32, slots), st);
  if (e != cudaSuccess) return e;
  if (K > 1 && (e = launch_chained(step_conv, dim3((De / 2 + 127) / 128, B), 128, st, true, (const bf16*)XZ, K, De, (const bf16*)w.w_conv, w.b_conv, conv_state,
                                   c.d_conv, U, Zs)) != cudaSuccess) return e;
  {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(XC, (R + 2 * NST) / 16, (B + X_TOK - 1) / X_TOK);
    cfg.blockDim = dim3(X_WARPS * 32);
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = XC; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    count_launch();
    if ((e = cudaLaunchKernelEx(&cfg, step_xproj, (const bf16*)U, (const bf16*)w.W_x, De, R, dr, Bm, Cm, B)) != cudaSuccess) return e;
  }
  auto scan = c.disc_mode == 0 ? step_dt_scan<true> : step_dt_scan<false>;
  if ((e = launch_chained(scan, dim3(De / 64, (B + 7) / 8), 128, st, true, (const bf16*)dr, (const bf16*)w.W_dt, w.b_dt, R, w.A, (const float*)Bm, (const float*)Cm, w.D,
                          (const bf16*)U, (const bf16*)(K == 1 ? XZ + De : Zs), K == 1 ? 2 * De : De, ssm_state, Yg, B, De)) != cudaSuccess) return e;
  StepGemmArgs ao{};
  ao.x = Yg; ao.ldx = De; ao.W = (const bf16*)w.W_out; ao.Kd = De; ao.n_rows = Dm; ao.idx = idx; ao.gates = gates; ao.B = B; ao.K = K; ao.E = c.E;
  ao.C = K == 1 ? (bf16*)out : Op; ao.ldc = Dm;
  ao.tile_rows = pick_tile_rows(c.E, Dm, num_sms);
  if (stream) e = launch_step_tc<STEP_OUT>(ao, num_sms, status, false, st);
  else e = launch_step_gemm<STEP_OUT, 1, 16>(ao, dim3(Dm / 16, slots), st);
  if (e != cudaSuccess) return e;
  if (K > 1) return launch_chained(step_combine, dim3((Dm / 2 + 127) / 128, B), 128, st, true, (const bf16*)Op, (const float*)gates, (bf16*)out, Dm, K);
  return cudaSuccess;
}

}  // namespace rom
