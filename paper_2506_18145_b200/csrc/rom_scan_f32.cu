// Selective scan for fp32 storage, A per channel and state (same arithmetic and arguments as rom_scan.cu), below 32768 channels: one launch,
// every exponential evaluated once.
//
// What bounds it: the accurate expf and expm1f of an update (about 45 instructions with the rest of it), and for short sequences the
// latency of the launches and of the steps, which depend on one another.  The general kernel cuts a sequence into chunks, whose
// exponentials it evaluates twice, in three launches.  Here the steps of four channels are spread over the warps of a block: a thread
// keeps the decays and inputs of 16 steps of one state in registers and what they do to a state, h -> P h + E, meets in shared memory;
// every thread composes the segments before its own, sweeps its 16 steps and the 16 lanes of a channel exchange their products with C
// until each holds one output.  256 steps of 512 channels: 26.7 -> 10 us (one launch of 128 blocks); 2 x 2048 of 1024: 293 -> 175;
// 24 x 1024 of 1024: 1112 -> 828.  It is not the faster one everywhere: long sequences of few channels (the general kernel's chunks fill
// the SMs), many channels with B-bar = Delta B, and counts that fill the general kernel's blocks evenly (f32_one_launch, rom_scan.cu).
#include "rom_scan_args.cuh"

namespace rom {
namespace {

constexpr int NST = 16;
constexpr int CB = 4;              // channels per block
constexpr int TS = 16;             // steps per segment
constexpr int PAIRS = CB * NST;    // threads per segment

template <int SEG>              // most segments at a time
struct F32Smem {
  float B[SEG * TS][NST], C[SEG * TS][NST];
  float d[SEG * TS][CB], u[SEG * TS][CB];
  float2 map[SEG][PAIRS];          // what a segment does to the state before it: h -> x h + y
  float carry[PAIRS];              // state before the block's next SEG segments
};

template <int SEG, bool ZOH, bool CKPT>
__global__ void __launch_bounds__(SEG * PAIRS, 16 / SEG)
scan_f32_kernel(const ScanArgs p) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  F32Smem<SEG>& s = *reinterpret_cast<F32Smem<SEG>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, n = lane & 15, seg = tid / PAIRS, n_seg = blockDim.x / PAIRS;
  const int pr = tid % PAIRS, cl = pr >> 4, c0 = blockIdx.x * CB, c = c0 + cl;      // this thread: state n of channel c
  const int De = p.De, L = p.L, round = n_seg * TS;
  const size_t tok0 = (size_t)blockIdx.y * L;
  const float av = __ldg(p.A + (size_t)c * NST + n), nik = -1.0f / av;
  const float d_skip = p.D ? __ldg(p.D + c) : 0.0f;
  const float* __restrict__ zp = static_cast<const float*>(p.z);
  if (seg == 0) s.carry[pr] = p.h0 ? p.h0[((size_t)blockIdx.y * De + c) * NST + n] : 0.0f;

  const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float4 rb, rc, rd;               // next round: B, C rows (four threads each); Delta and u rows by the first 2 * round threads
  auto fetch = [&](int t0) {
    const int t = t0 + (tid >> 2);
    const bool in = t < L;
    rb = in ? __ldg(reinterpret_cast<const float4*>(p.Bm + (tok0 + t) * NST) + (tid & 3)) : zero4;
    rc = in ? __ldg(reinterpret_cast<const float4*>(p.Cm + (tok0 + t) * NST) + (tid & 3)) : zero4;
    const int td = t0 + (tid >> 1);
    rd = zero4;
    if (tid < 2 * round && td < L) rd = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>((tid & 1) ? p.u : p.delta) + (tok0 + td) * De + c0));
  };
  fetch(0);
  for (int t0 = 0; t0 < L; t0 += round) {
    reinterpret_cast<float4*>(s.B)[tid] = rb;
    reinterpret_cast<float4*>(s.C)[tid] = rc;
    if (tid < 2 * round) *reinterpret_cast<float4*>((tid & 1) ? s.u[tid >> 1] : s.d[tid >> 1]) = rd;
    __syncthreads();
    if (t0 + round < L) fetch(t0 + round);
    // the output this thread will write: step n of its segment
    const int t_out = t0 + seg * TS + n;
    float z = 1.0f;
    if (zp && t_out < L) z = __ldg(zp + (p.z_row ? (size_t)__ldg(p.z_row + tok0 + t_out) : tok0 + t_out) * p.ldz + c);

    // ---- decays and inputs of the segment; what it does to a state
    float a[TS], b[TS], P = 1.0f, E = 0.0f;
#pragma unroll
    for (int i = 0; i < TS; ++i) {
      const int r = seg * TS + i;
      const float dl = s.d[r][cl], uu = s.u[r][cl], x = dl * av;
      a[i] = expf(x);
      b[i] = ZOH ? -expm1f(x) * nik * (s.B[r][n] * uu) : s.B[r][n] * (dl * uu);
      E = fmaf(a[i], E, b[i]);
      P *= a[i];
    }
    if (__any_sync(0xffffffffu, P == 0.0f)) {      // none of the decays zero, but their product: an infinite state stays infinite, as step by step
      bool zero = false;
#pragma unroll
      for (int i = 0; i < TS; ++i) zero |= a[i] == 0.0f;
      if (P == 0.0f && !zero) P = __int_as_float(1);
    }
    s.map[seg][pr] = make_float2(P, E);
    __syncthreads();
    float h = s.carry[pr];
    for (int k = 0; k < seg; ++k) { const float2 m = s.map[k][pr]; h = fmaf(m.x, h, m.y); }

    // ---- states and outputs
#pragma unroll
    for (int i = 0; i < TS; ++i) {
      if (CKPT && i % kScanCkpt == 0) {
        const int t = t0 + seg * TS + i;
        if (t < L) p.ckpt[(((size_t)blockIdx.y * p.nck + t / kScanCkpt) * De + c) * NST + n] = h;
      }
      h = fmaf(a[i], h, b[i]);
      a[i] = s.C[seg * TS + i][n] * h;
    }
    // sums over the 16 states: a lane gives half of its steps and keeps the others, four times, and is left with step n
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1)
#pragma unroll
      for (int i = 0; i < o; ++i) {
        const float give = (n & o) ? a[i] : a[i + o], keep = (n & o) ? a[i + o] : a[i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
    if (t_out < L) {
      float y = fmaf(d_skip, s.u[seg * TS + n][cl], a[0]);
      if (zp) y *= p.gate_activated ? z : z / (1.0f + expf(-z));
      float* yp = static_cast<float*>(p.y) + c;
      if (p.y_rows == nullptr) yp[(tok0 + t_out) * De] = y;
      else
        for (int k = 0; k < p.K; ++k) yp[(size_t)__ldg(p.y_rows + (tok0 + t_out) * p.K + k) * De] = y;
    }
    __syncthreads();               // everything of this round has been read
    if (seg == n_seg - 1) {
      s.carry[pr] = h;
      if (p.h_last && t0 + round >= L) p.h_last[((size_t)blockIdx.y * De + c) * NST + n] = h;
    }
  }
}

template <int SEG, bool ZOH, bool CKPT>
cudaError_t launch_one(const ScanArgs& a, int B, cudaStream_t st) {
  constexpr int smem = (int)sizeof(F32Smem<SEG>);
  const cudaError_t e = cudaFuncSetAttribute(scan_f32_kernel<SEG, ZOH, CKPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const int segs = (a.L + TS - 1) / TS;
  const dim3 grid(a.De / CB, B);
  launch_k((long long)grid.x * grid.y <= 148, scan_f32_kernel<SEG, ZOH, CKPT>, grid, PAIRS * (segs < SEG ? segs : SEG), smem, st, a);
  count_launch();
  return cudaGetLastError();
}

// Segments per round: all 16 while every SM has one block at most (the fewest rounds), less where blocks share an SM, so that one
// computes while another waits at its barriers (4 x 1024 steps of 1024 channels: 160 us with 16, 152 with 8, 149 with 4; 2048 steps of
// 512: 46, 50, 63).
template <bool ZOH, bool CKPT>
cudaError_t launch_segs(const ScanArgs& a, int B, cudaStream_t st) {
  const long long blocks = (long long)B * (a.De / CB);
  return blocks <= 148 ? launch_one<16, ZOH, CKPT>(a, B, st) : blocks <= 2 * 148 ? launch_one<8, ZOH, CKPT>(a, B, st) : launch_one<4, ZOH, CKPT>(a, B, st);
}

}  // namespace

cudaError_t launch_scan_f32(const ScanArgs& a, int B, bool zoh, bool ckpt, cudaStream_t st) {
  if (ckpt) return zoh ? launch_segs<true, true>(a, B, st) : launch_segs<false, true>(a, B, st);
  return zoh ? launch_segs<true, false>(a, B, st) : launch_segs<false, false>(a, B, st);
}

}  // namespace rom
