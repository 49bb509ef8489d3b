// Selective scan for bf16 storage with few channels (same arithmetic and arguments as rom_scan.cu): one launch, every exponential
// evaluated once.
//
// Few channels fill the SMs only when a sequence is cut along time, and the chunked form (rom_scan_warp.cu) then evaluates nearly every
// exponential twice: 16 of the special-function unit's cycles a warp-wide update against ten of the fp32 pipe.  Here a block owns 32
// channels of one sequence, and its twelve warps take tiles of eight steps in turn.  A warp runs its tile from a zero state (a lane holds
// 4 states of 4 adjacent channels, as in rom_scan_warp.cuh) and keeps what a state before the tile would add to the outputs, C times the
// running product of the decays: 16 values a lane and step, which registers cannot hold for eight steps.  They go to tensor memory (128
// columns a warp; no matrix instruction runs).  The state then comes from the warp before, P h + E goes on to the next warp at once, and
// one multiply-add an update brings the outputs up to date; nothing of that depends on the step before.
// Values that are not finite: where the decays of a tile multiply to zero, none of them zero, an infinite state would become NaN, and an
// infinite C meets the two parts of a state one by one.  A state that is not finite is there to the end: the last tile looks at it, every
// tile at its C, and a block that has seen one goes over its sequence again step by step.  (Looked at tile by tile the states cost 4 %.  With a NaN
// in every sequence 16384 steps of 4096 channels take 2.1 ms; all by one warp a block 3.1.)
// Measured against the chunked form, in the layer: 4 x 2048 steps of 2048 channels 164 -> 146 us, 16384 of 4096 593 -> 524; as rom_scan 3 x 1017 of
// 3072 95 -> 82.  What bounds it: issue (9.5 instructions an update at up to 72 %), the fp32 pipe (nine operations of an update) and latency: twelve
// warps an SM.
// Tried (us of a layer of 4 x 2048 steps of 2048 channels; this form 300, in chunks 317): decays and inputs both in tensor memory with eight
// warps of 255 registers (seven operations, but two warps a scheduler) 309, that with the second sweep beside the next tile's first 352;
// decays alone and the inputs formed twice, sixteen warps 317; B and C twice in shared memory for the packed pairs 319; Delta and u staged
// as bf16 307; the outputs from the zero state in tensor memory as well 315; the carry in the layout of the registers 309 (spills).
#include "rom_scan_warp.cuh"
#include "rom_tc_ptx.cuh"

namespace rom {
namespace {

constexpr int W = 12;             // warps per block (of WCH channels)
constexpr int TM_COLS = 512;      // tensor memory columns (a power of two): 128 for each of a lane quarter's three warps

struct RingTile {
  float4 dl[CK][8], u[CK][8];     // Delta, u of 4 channels; group g of step r sits at g ^ r
  float4 b[CK][4], c[CK][4];
  float4 y[CK][32];               // partial sums of 4 channels over one lane's states; lane l of step r at ysw(l, r)
};
struct RingSmem {
  RingTile tile[W];
  float4 carry[W][4][32];         // state before the tile of warp w
  float D[WCH];
  uint32_t tmem;
  int odd;                        // a state or a C that is not finite has turned up
};

__device__ __forceinline__ void tm_store16(uint32_t at, const float2 (&a)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(at), "f"(a[0].x), "f"(a[0].y), "f"(a[1].x), "f"(a[1].y), "f"(a[2].x), "f"(a[2].y), "f"(a[3].x), "f"(a[3].y),
        "f"(a[4].x), "f"(a[4].y), "f"(a[5].x), "f"(a[5].y), "f"(a[6].x), "f"(a[6].y), "f"(a[7].x), "f"(a[7].y)
      : "memory");
}
__device__ __forceinline__ void tm_store_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void bar_sync(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void block_sync() { asm volatile("bar.sync %0, %1;" ::"n"(W), "n"(W * 32) : "memory"); }      // (0 .. W - 1: the warps')
__device__ __forceinline__ void bar_arrive(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// The block's channels again, step by step, the warps still in turns.  (A function of its own, so that the kernel's registers do not feel it.)
struct StepSmem {
  WarpTile tile[W];
  float4 carry[W][4][32];
};
struct TilesInTurns {
  StepSmem& sm;
  const int warp, lane;
  static constexpr int STRIDE = W * CK;
  __device__ int first() const { return warp * CK; }
  __device__ void take(float2 (&h)[4][2], int t0) const {
    if (t0 == 0) return;
    __syncwarp();
    bar_sync(warp);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 x = sm.carry[warp][2 * j][lane], y = sm.carry[warp][2 * j + 1][lane];
      h[0][j] = make_float2(x.x, y.x); h[1][j] = make_float2(x.y, y.y); h[2][j] = make_float2(x.z, y.z); h[3][j] = make_float2(x.w, y.w);
    }
  }
  __device__ void give(const float2 (&h)[4][2], int t0, int L) const {
    if (t0 + CK >= L) return;
    const int nx = warp + 1 == W ? 0 : warp + 1;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      sm.carry[nx][2 * j][lane] = make_float4(h[0][j].x, h[1][j].x, h[2][j].x, h[3][j].x);
      sm.carry[nx][2 * j + 1][lane] = make_float4(h[0][j].y, h[1][j].y, h[2][j].y, h[3][j].y);
    }
    bar_arrive(nx);
  }
  __device__ bool has_last(int L) const { return (L - 1) / CK % W == warp; }
};
template <typename TD, bool ZOH, bool CKPT, bool SLOTS>
__device__ __noinline__ void scan_stepwise(const ScanArgs& p, StepSmem& sm) {
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  scan_warp_channels<TD, ZOH, CKPT ? SCAN_FULL_CKPT : SCAN_FULL, SLOTS>(p, sm.tile[warp], blockIdx.x * WCH, blockIdx.y, 0, TilesInTurns{sm, warp, lane});
}

template <typename TD, bool ZOH, bool CKPT, bool SLOTS>
__global__ void __launch_bounds__(W * 32, 1)
scan_ring_kernel(const __grid_constant__ ScanArgs p) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RingSmem& sm = *reinterpret_cast<RingSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  RingTile& s = sm.tile[warp];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm.tmem)), "r"(TM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  const int De = p.De, L = p.L;
  const int c_warp = blockIdx.x * WCH;
  const size_t b = blockIdx.y, tok0 = b * L;
  const int NT = (L + CK - 1) / CK;

  // ---- compute role: channels c0 .. c0+3 (pairs), states 4q .. 4q+3
  const int q = lane & 3, cg = lane >> 2;
  const int c0 = c_warp + 4 * cg;
  float2 a2[8], kin[8];           // [4 states x 2 pairs]
  {
    float av[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 a4 = __ldg(reinterpret_cast<const float4*>(p.A + (size_t)(c0 + i) * NST) + q);
      av[i][0] = a4.x; av[i][1] = a4.y; av[i][2] = a4.z; av[i][3] = a4.w;
      if (warp == 0) sm.carry[0][i][lane] = p.h0 ? load4_any(p.h0 + (b * De + c0 + i) * NST + 4 * q) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        a2[2 * n + j] = make_float2(av[2 * j][n] * kLog2e, av[2 * j + 1][n] * kLog2e);
        kin[2 * n + j] = make_float2(-1.0f / av[2 * j][n], -1.0f / av[2 * j + 1][n]);
      }
  }
  if (warp == 0) {
    if (lane == 0) sm.odd = 0;
    sm.D[lane] = p.D ? __ldg(p.D + c_warp + lane) : 0.0f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_trigger();      // (only now: the product that follows takes its tensor memory before it waits for this kernel)
  const uint32_t tm = sm.tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * 128;

  // ---- loader / output role: step lt of every tile, channels lc .. lc+7
  const int lt = lane >> 2, l8 = lane & 3, lc = c_warp + 8 * l8;
  const bf16* __restrict__ zp = static_cast<const bf16*>(p.z);
  Raw8<TD> r_d;
  Raw8<bf16> r_u, cur_u, cur_z, cur_z2;
  float4 r_b, r_c;
  int cur_row = 0, cur_row2 = 0;
  auto fetch = [&](int t0) {
    const int t = t0 + lt;
    const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (t < L) {
      r_d.load(static_cast<const TD*>(p.delta) + (tok0 + t) * De + lc);
      r_u.load(static_cast<const bf16*>(p.u) + (tok0 + t) * De + lc);
    } else {
      r_d.zero(); r_u.zero();
    }
    r_b = t < L ? __ldg(reinterpret_cast<const float4*>(p.Bm + (tok0 + t0) * NST) + lane) : zero4;
    r_c = t < L ? __ldg(reinterpret_cast<const float4*>(p.Cm + (tok0 + t0) * NST) + lane) : zero4;
  };
  auto fetch_rows = [&](int t0) {      // rows of the gate and of the output (their indices a sweep ahead of what they lead to)
    const int t = t0 + lt;
    if (t < L) {
      if constexpr (SLOTS) {
        const int32_t* zr = p.z_row + (tok0 + t) * p.K;
        cur_row = __ldg(zr); cur_row2 = __ldg(zr + 1);
      } else {
        cur_row = p.y_rows ? __ldg(p.y_rows + (tok0 + t) * p.K) : (int)(tok0 + t);
      }
    }
  };
  if (warp < NT) fetch(warp * CK);
  for (int tile = warp; tile < NT; tile += W) {
    const int t0 = tile * CK;
    {
      float d[8], uu[8];
      r_d.get(d); r_u.get(uu);
      if (!ZOH) {
#pragma unroll
        for (int i = 0; i < 8; ++i) uu[i] *= d[i];
      }
      s.dl[lt][(2 * l8) ^ lt] = make_float4(d[0], d[1], d[2], d[3]);
      s.dl[lt][(2 * l8 + 1) ^ lt] = make_float4(d[4], d[5], d[6], d[7]);
      s.u[lt][(2 * l8) ^ lt] = make_float4(uu[0], uu[1], uu[2], uu[3]);
      s.u[lt][(2 * l8 + 1) ^ lt] = make_float4(uu[4], uu[5], uu[6], uu[7]);
      reinterpret_cast<float4*>(s.b)[lane] = r_b;
      reinterpret_cast<float4*>(s.c)[lane] = r_c;
      cur_u = r_u;
    }
    fetch_rows(t0);
    {      // (by vote or by lane, as the instance's registers like it: fp32 Delta with the hold 153 us by lane, 141 by vote, 4096 steps of 4096 channels)
      constexpr bool VOTE = ZOH && sizeof(TD) == 4;
      const bool odd = !(fabsf((r_c.x + r_c.y) + (r_c.z + r_c.w)) < __int_as_float(0x7f800000));
      if (VOTE ? __any_sync(0xffffffffu, odd) : odd) sm.odd = 1;
    }
    __syncwarp();
    // ---- from a zero state: outputs, what a state before the tile adds to them (C times the running product of the decays, to tensor
    // memory) and what the tile does to it
    float2 E[8], P[8];
    {
      float4 nd = s.dl[0][cg], nu = s.u[0][cg], nb = s.b[0][q], nc = s.c[0][q];
#pragma unroll
      for (int r = 0; r < CK; ++r) {
        const float4 d4 = nd, u4 = nu, b4 = nb, c4 = nc;
        if (r + 1 < CK) { nd = s.dl[r + 1][cg ^ (r + 1)]; nu = s.u[r + 1][cg ^ (r + 1)]; nb = s.b[r + 1][q]; nc = s.c[r + 1][q]; }
        const float2 dl[2] = {make_float2(d4.x, d4.y), make_float2(d4.z, d4.w)}, uu[2] = {make_float2(u4.x, u4.y), make_float2(u4.z, u4.w)};
        const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, cc[4] = {c4.x, c4.y, c4.z, c4.w};
        float2 cp[8], acc[2];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int k = 2 * n + j;
            const float2 x = __fmul2_rn(dl[j], a2[k]);
            const float2 a = make_float2(ex2_ftz(x.x), ex2_ftz(x.y));
            const float2 uB = __fmul2_rn(uu[j], dup(bb[n]));
            if (ZOH) {             // w = -B u / A, h <- a (h - w) + w
              const float2 w = __fmul2_rn(uB, kin[k]);
              E[k] = __ffma2_rn(a, r == 0 ? __fmul2_rn(w, dup(-1.0f)) : __ffma2_rn(w, dup(-1.0f), E[k]), w);
            } else {
              E[k] = r == 0 ? uB : __ffma2_rn(a, E[k], uB);
            }
            P[k] = r == 0 ? a : __fmul2_rn(P[k], a);
            cp[k] = __fmul2_rn(dup(cc[n]), P[k]);
            acc[j] = n == 0 ? __fmul2_rn(dup(cc[n]), E[k]) : __ffma2_rn(dup(cc[n]), E[k], acc[j]);
          }
        s.y[r][ysw(lane, r)] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
        tm_store16(tm + 16 * r, cp);
      }
    }
    if (t0 + lt < L && zp) {
      if constexpr (SLOTS) {
        cur_z.load(zp + (size_t)cur_row * p.ldz + lc);
        cur_z2.load(zp + (size_t)cur_row2 * p.ldz + lc);
      } else {
        cur_z.load(zp + (p.z_row ? (size_t)__ldg(p.z_row + tok0 + t0 + lt) : tok0 + t0 + lt) * p.ldz + lc);
      }
    }
    if (tile + W < NT) fetch(t0 + W * CK);
    __syncwarp();                 // (the lanes part in a last tile cut short; the barrier and the waits below take the whole warp)
    float2 h[8];
    // ---- the state before the tile arrives, the one behind it leaves
    if (tile > 0) bar_sync(warp);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 x = sm.carry[warp][2 * j][lane], y = sm.carry[warp][2 * j + 1][lane];
      h[j] = make_float2(x.x, y.x); h[2 + j] = make_float2(x.y, y.y); h[4 + j] = make_float2(x.z, y.z); h[6 + j] = make_float2(x.w, y.w);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) E[k] = __ffma2_rn(P[k], h[k], E[k]);
    {
      const float4 e[4] = {make_float4(E[0].x, E[2].x, E[4].x, E[6].x), make_float4(E[0].y, E[2].y, E[4].y, E[6].y),
                           make_float4(E[1].x, E[3].x, E[5].x, E[7].x), make_float4(E[1].y, E[3].y, E[5].y, E[7].y)};
      if (tile + 1 < NT) {
        const int nx = warp + 1 == W ? 0 : warp + 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) sm.carry[nx][i][lane] = e[i];
        bar_arrive(nx);
      } else {
        float nf = 0.0f;
#pragma unroll
        for (int i = 0; i < 4; ++i) nf = fmaf(e[i].x, 0.0f, fmaf(e[i].y, 0.0f, fmaf(e[i].z, 0.0f, fmaf(e[i].w, 0.0f, nf))));
        if (__any_sync(0xffffffffu, !(nf == 0.0f))) sm.odd = 1;
        else if (p.h_last && !sm.odd)
#pragma unroll
          for (int i = 0; i < 4; ++i) store4_any(p.h_last + (b * De + c0 + i) * NST + 4 * q, e[i]);
      }
    }
    if (CKPT) {
      float* at = p.ckpt + ((b * p.nck + tile) * De + c0) * NST + 4 * q;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        *reinterpret_cast<float4*>(at + (2 * j) * NST) = make_float4(h[j].x, h[2 + j].x, h[4 + j].x, h[6 + j].x);
        *reinterpret_cast<float4*>(at + (2 * j + 1) * NST) = make_float4(h[j].y, h[2 + j].y, h[4 + j].y, h[6 + j].y);
      }
    }
    // ---- what the state before the tile adds to the outputs
    {
      tm_store_wait();
      uint32_t v[2][32];
      tmem_ld32_issue(tm, v[0]);
#pragma unroll
      for (int r2 = 0; r2 < CK / 2; ++r2) {
        tmem_ld_wait(v[r2 & 1]);
        if (r2 + 1 < CK / 2) tmem_ld32_issue(tm + 32 * (r2 + 1), v[(r2 + 1) & 1]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int r = 2 * r2 + i;
          float4 y4 = s.y[r][ysw(lane, r)];
          const uint32_t* vr = v[r2 & 1] + 16 * i;
#pragma unroll
          for (int n = 0; n < 4; ++n) {      // (single: the values of the load take two moves into the pair of a packed sum)
            y4.x = fmaf(__uint_as_float(vr[4 * n]), h[2 * n].x, y4.x); y4.y = fmaf(__uint_as_float(vr[4 * n + 1]), h[2 * n].y, y4.y);
            y4.z = fmaf(__uint_as_float(vr[4 * n + 2]), h[2 * n + 1].x, y4.z); y4.w = fmaf(__uint_as_float(vr[4 * n + 3]), h[2 * n + 1].y, y4.w);
          }
          s.y[r][ysw(lane, r)] = y4;
        }
      }
    }
    __syncwarp();
    // ---- y = (sum over the four lanes + D u) * gate, rounded, written to the K rows of the token
    const int t = t0 + lt;
    if (t < L) {
      float o[8], uu[8], zz[8];
      cur_u.get(uu);
      if (zp) {
        cur_z.get(zz);
        if (SLOTS) {
          float z2[8];
          cur_z2.get(z2);
#pragma unroll
          for (int i = 0; i < 8; ++i) zz[i] += z2[i];
          for (int k = 2; k < p.K; ++k) {
            V16<bf16> zk;
            zk.load(zp + (size_t)__ldg(p.z_row + (tok0 + t) * p.K + k) * p.ldz + lc);
            zk.get(z2);
#pragma unroll
            for (int i = 0; i < 8; ++i) zz[i] += z2[i];
          }
        }
        if (SLOTS || !p.gate_activated) {
#pragma unroll
          for (int i = 0; i < 8; ++i) zz[i] = silu_fast(zz[i]);
        }
      }
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int g4 = 8 * l8 + 4 * hf;
        const float4 x0 = s.y[lt][ysw(g4, lt)], x1 = s.y[lt][ysw(g4 + 1, lt)], x2 = s.y[lt][ysw(g4 + 2, lt)], x3 = s.y[lt][ysw(g4 + 3, lt)];
        const float4 D4 = reinterpret_cast<const float4*>(sm.D)[2 * l8 + hf];
        float2 v0 = __fadd2_rn(__fadd2_rn(make_float2(x0.x, x0.y), make_float2(x1.x, x1.y)), __fadd2_rn(make_float2(x2.x, x2.y), make_float2(x3.x, x3.y)));
        float2 v1 = __fadd2_rn(__fadd2_rn(make_float2(x0.z, x0.w), make_float2(x1.z, x1.w)), __fadd2_rn(make_float2(x2.z, x2.w), make_float2(x3.z, x3.w)));
        v0 = __ffma2_rn(make_float2(D4.x, D4.y), make_float2(uu[4 * hf], uu[4 * hf + 1]), v0);
        v1 = __ffma2_rn(make_float2(D4.z, D4.w), make_float2(uu[4 * hf + 2], uu[4 * hf + 3]), v1);
        if (zp) {
          v0 = __fmul2_rn(v0, make_float2(zz[4 * hf], zz[4 * hf + 1]));
          v1 = __fmul2_rn(v1, make_float2(zz[4 * hf + 2], zz[4 * hf + 3]));
        }
        o[4 * hf] = v0.x; o[4 * hf + 1] = v0.y; o[4 * hf + 2] = v1.x; o[4 * hf + 3] = v1.y;
      }
      bf16* y = static_cast<bf16*>(p.y) + lc;
      V16<bf16>::store(y + (size_t)cur_row * De, o);
      if (SLOTS) V16<bf16>::store(y + (size_t)cur_row2 * De, o);
      if (p.y_rows)
        for (int k = SLOTS ? 2 : 1; k < p.K; ++k) V16<bf16>::store(y + (size_t)__ldg(p.y_rows + (tok0 + t) * p.K + k) * De, o);
    }
    __syncwarp();
  }
  tc_fence_before();
  block_sync();
  const bool odd = sm.odd;
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(TM_COLS));
  }
  if (odd) {
    block_sync();      // (everybody has read what lay there)
    scan_stepwise<TD, ZOH, CKPT, SLOTS>(p, *reinterpret_cast<StepSmem*>(smem_raw));
  }
}

template <typename TD, bool ZOH, bool CKPT, bool SLOTS>
cudaError_t launch_one(const ScanArgs& a, int B, cudaStream_t st) {
  constexpr int smem = (int)(sizeof(RingSmem) > sizeof(StepSmem) ? sizeof(RingSmem) : sizeof(StepSmem));
  const cudaError_t e = cudaFuncSetAttribute(scan_ring_kernel<TD, ZOH, CKPT, SLOTS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  launch_k(a.early != 0, scan_ring_kernel<TD, ZOH, CKPT, SLOTS>, dim3(a.De / WCH, B), W * 32, smem, st, a);
  count_launch();
  return cudaGetLastError();
}
template <typename TD, bool ZOH, bool CKPT>
cudaError_t launch_slots(const ScanArgs& a, int B, cudaStream_t st) {
  if (a.z_row && a.K > 1) {
    if constexpr (sizeof(TD) == 2 && !CKPT) return launch_one<TD, ZOH, CKPT, true>(a, B, st);
    else return cudaErrorInvalidValue;
  }
  return launch_one<TD, ZOH, CKPT, false>(a, B, st);
}
}  // namespace

cudaError_t launch_scan_ring(const ScanArgs& a, int B, bool zoh, bool delta_fp32, bool ckpt, cudaStream_t st) {
  if (delta_fp32) {
    if (ckpt) return cudaErrorInvalidValue;
    return zoh ? launch_slots<float, true, false>(a, B, st) : launch_slots<float, false, false>(a, B, st);
  }
  if (ckpt) return zoh ? launch_slots<bf16, true, true>(a, B, st) : launch_slots<bf16, false, true>(a, B, st);
  return zoh ? launch_slots<bf16, true, false>(a, B, st) : launch_slots<bf16, false, false>(a, B, st);
}

}  // namespace rom
