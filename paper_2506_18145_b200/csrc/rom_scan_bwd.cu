// Backward of the selective scan (Section 3.1 recurrence; Section 5.1 trains the layer end to end).
//
// Forward:  h_t = a_t h_{t-1} + b_t u_t,  y_t = sum_n C_t,n h_t,n + D u_t,  out_t = y_t * SiLU(z_t)   (gate optional)
//           a = exp(Delta A);  b = expm1(Delta A)/A * B (zero-order hold)  or  Delta B.
// Reverse, with g = dLoss/dh_t carried from later steps and e_t = dout_t * SiLU(z_t):
//           g += C_t e_t;  dC_t = sum_c e_t h_t;  dA-bar = g h_{t-1};  db = g u_t;  du_t = sum_n g b + D e_t;  g <- a_t g.
// With w = -u B / A the zero-order-hold step is h_t = a (h_{t-1} - w) + w, and everything that passes through the exponent is
// g p with p = a (h_{t-1} - w):  dDelta = sum_n A g p,  dA = Delta g p + r w  with  r = g (a - 1) / A,  dB = r u,  du = sum_n r B.
//
// The reverse sweep needs h_{t-1} and h_t at every step.  The state at the start of every CK = 8 steps is kept in the workspace
// (checkpoints, written by a forward scan: the layer's recomputed forward, or the state-only passes of rom_scan_backward); the
// reverse kernel walks the checkpoints backwards, recomputes eight states into shared memory and sweeps them in reverse.
//
// A long sequence with few channels is cut into coarse chunks that run in parallel, as in the forward scan: the gradient
// recurrence is linear in g.  A pre-pass runs it per chunk from a zero gradient (the gradient that leaves the chunk's start, and
// the sum of Delta), a chain kernel composes the true gradient at the end of every chunk.
//
// What bounds the reverse kernel: the fp32 pipe.  Per state and step it needs about 23 fp32 lane operations (6 recomputed
// forward, 17 reverse) and two exponentials, so the layout is chosen to add as little as possible: a thread owns 4 states of 4
// adjacent channels (packed pairs along the states), so that the sums over channels (dB, dC) start as accumulation in
// registers and the sums over states (dDelta, du, y) need four lanes only; the former finish with a transposed 7-shuffle
// reduction per step, the latter are left in the shared-memory slot of the state just consumed and added by the lane that owns
// the output.  A warp owns 32 channels and everything it touches: no block barrier.  Shared memory (81 KB per block of four
// warps) allows two blocks per SM, and the 16 independent updates per thread and step hide the latencies.
// All arithmetic is fp32; the fp32 configuration uses the accurate exp / expm1, the bf16 one a single ex2.approx per state
// and step (exp(x) - 1 by subtraction: with Delta A down to -5e-4 that is still good to a few 1e-4 relative).
#include "rom_scan_args.cuh"

namespace rom {
namespace {

constexpr int NST = 16;
constexpr int CK = kScanCkpt;     // steps per checkpoint
constexpr int WCH = 32;           // channels per warp
constexpr int WPB = 4;            // warps per block
constexpr int BT = WPB * 32;
constexpr int BCH = WPB * WCH;    // channels per block
constexpr float kLog2e = 1.4426950408889634f, kLn2 = 0.6931471805599453f;

struct WarpSmem {
  float4 h[CK][4][32];            // [step][channel of the thread][lane]: state before the step; later the step's partial sums
  float4 dl[CK][8], u[CK][8], e[CK][8];     // Delta, u, e of 4 channels; group g of step r sits at g ^ r
  float4 bc[2][CK][4];            // B, C
};
constexpr int BWD_SMEM = WPB * (int)sizeof(WarpSmem);
constexpr int BLOCKS_PER_SM = 2;

struct BwdArgs {
  const void* dy; const void* u; const void* delta; const float* A; const float* Bm; const float* Cm; const float* D;
  const void* z; const float* dh_last;
  void* du; float* ddelta; float* dA; float* dBm; float* dCm; float* dD; void* dz; float* dh0;
  void* dpre; float* db_dt;       // dpre != nullptr: the gradient goes through Delta = softplus(pre) and leaves as dpre (ddelta unused)
  const float* ckpt;              // [B, nck, De, 16]
  int L, De, nck;
  int ldz;                        // row pitch (elements) of z and dz
  const int32_t* dz_rows; int K;  // rows of dz that take token t: dz_rows[t K + k]; nullptr: row t
  int Lc, ncc;                    // coarse chunks (blockIdx.z): chunk j covers steps [j Lc, (j+1) Lc); Lc is a multiple of 16
  float* g_in;                    // [B, ncc, De, 16] state gradient at the end of every coarse chunk (ncc > 1)
  int Lp, mp;                     // pre-pass: every coarse chunk in mp pieces of Lp steps (the last ones shorter or empty)
  float* q_start; float* sum_delta;         // pre-pass outputs: [B, ncc, mp, De, 16] and [B, ncc, mp, De]
};

template <bool PRECISE> __device__ __forceinline__ float sigmoid_f(float v) {
  return PRECISE ? 1.0f / (1.0f + expf(-v)) : rcp_ftz(1.0f + ex2_ftz(-kLog2e * v));
}
// 1 - exp(-x), x >= 0 (the derivative of softplus expressed in its result)
template <bool PRECISE> __device__ __forceinline__ float one_minus_exp(float x) {
  if (PRECISE) return -expm1f(-x);
  // series below 1/4 (next term x^5/720, 1.4e-6 relative), subtraction above
  const float s = x * fmaf(x, -fmaf(x, -fmaf(x, -fmaf(x, -1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f), 0.5f), 1.0f);
  return x < 0.25f ? s : 1.0f - ex2_ftz(-kLog2e * x);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }      // a - b
// exp(Delta A) of a pair of states, and exp - 1; a2 holds A log2(e) (A itself when PRECISE)
template <bool PRECISE> __device__ __forceinline__ float2 exp_pair(float2 x) {
  return PRECISE ? make_float2(expf(x.x), expf(x.y)) : make_float2(ex2_ftz(x.x), ex2_ftz(x.y));
}

template <typename T, typename TD, bool ZOH>
__global__ void __launch_bounds__(BT, BLOCKS_PER_SM)
scan_bwd_kernel(const BwdArgs p) {
  pdl_sync();
  constexpr bool PRECISE = sizeof(T) == 4;
  extern __shared__ __align__(16) unsigned char bwd_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WarpSmem& s = reinterpret_cast<WarpSmem*>(bwd_smem)[warp];
  const int De = p.De, L = p.L;
  const int c_warp = blockIdx.x * BCH + warp * WCH;
  if (c_warp >= De) return;                      // d_inner is a multiple of 64: a warp's 32 channels are all in or all out
  const size_t b = blockIdx.y;
  const int cj = blockIdx.z;
  const int k_lo = cj * (p.Lc / CK), k_hi = min(k_lo + p.Lc / CK, p.nck);

  // ---- compute role: channels c0 .. c0+3, states 4q .. 4q+3
  const int q = lane & 3, cg = lane >> 2;
  const int c0 = c_warp + 4 * cg;
  float2 a2[4][2], nik[4][2], g[4][2], dA[4][2];      // A (log2 e), -1/A, gradient carried, dA
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 av = *reinterpret_cast<const float4*>(p.A + (size_t)(c0 + i) * NST + 4 * q);
    const float sc = PRECISE ? 1.0f : kLog2e;
    a2[i][0] = make_float2(av.x * sc, av.y * sc); a2[i][1] = make_float2(av.z * sc, av.w * sc);
    nik[i][0] = make_float2(-1.0f / av.x, -1.0f / av.y); nik[i][1] = make_float2(-1.0f / av.z, -1.0f / av.w);
    float4 gv = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (p.ncc > 1) gv = *reinterpret_cast<const float4*>(p.g_in + ((b * p.ncc + cj) * De + c0 + i) * NST + 4 * q);
    else if (p.dh_last) gv = *reinterpret_cast<const float4*>(p.dh_last + (b * De + c0 + i) * NST + 4 * q);
    g[i][0] = make_float2(gv.x, gv.y); g[i][1] = make_float2(gv.z, gv.w);
    dA[i][0] = make_float2(0.0f, 0.0f); dA[i][1] = dA[i][0];
  }
  // ---- loader / output role: step lt of every checkpoint interval, channels lc .. lc+7 (four lanes per row: a load's quarter-warp
  // touches two rows of global memory, not eight)
  const int lt = lane >> 2, l8 = lane & 3, lc = c_warp + 8 * l8;
  float Dv[8], dDacc[8], dbacc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { Dv[i] = p.D ? p.D[lc + i] : 0.0f; dDacc[i] = 0.0f; dbacc[i] = 0.0f; }
  const T* __restrict__ up = static_cast<const T*>(p.u);
  const T* __restrict__ dyp = static_cast<const T*>(p.dy);
  const T* __restrict__ zp = static_cast<const T*>(p.z);
  const TD* __restrict__ dlp = static_cast<const TD*>(p.delta);

  Raw8<TD> r_dl; Raw8<T> r_u, r_dy, r_z, cur_dy, cur_z;
  float4 r_b, r_c, r_h[4];
  int r_row = 0, cur_row = 0;      // first output row of dz of this lane's step
  auto fetch = [&](int k) {
    const int t = k * CK + lt;
    if (t < L) {
      r_row = p.dz_rows ? __ldg(p.dz_rows + (b * L + t) * p.K) : (int)(b * L + t);
      const size_t row = b * L + t;
      r_dl.load(dlp + row * De + lc); r_u.load(up + row * De + lc); r_dy.load(dyp + row * De + lc);
      if (zp) r_z.load(zp + row * p.ldz + lc);
    } else {
      r_dl.zero(); r_u.zero(); r_dy.zero(); r_z.zero();
    }
    // eight steps of B and C: 128 consecutive floats each, four per lane
    const int tb = k * CK + (lane >> 2);
    const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    r_b = tb < L ? __ldg(reinterpret_cast<const float4*>(p.Bm + (b * L + k * CK) * NST) + lane) : zero4;
    r_c = tb < L ? __ldg(reinterpret_cast<const float4*>(p.Cm + (b * L + k * CK) * NST) + lane) : zero4;
#pragma unroll
    for (int i = 0; i < 4; ++i) r_h[i] = __ldg(reinterpret_cast<const float4*>(p.ckpt + ((b * p.nck + k) * De + c0 + i) * NST) + q);
  };
  fetch(k_hi - 1);

  for (int k = k_hi - 1; k >= k_lo; --k) {
    // ---- stage the interval: e = dout * SiLU(z) is the gradient arriving at y; steps past the end are all zero (they change nothing)
    float2 h[4][2];
    {
      float dl[8], uu[8], dy[8];
      r_dl.get(dl); r_u.get(uu); r_dy.get(dy);
      s.dl[lt][(2 * l8) ^ lt] = make_float4(dl[0], dl[1], dl[2], dl[3]);
      s.dl[lt][(2 * l8 + 1) ^ lt] = make_float4(dl[4], dl[5], dl[6], dl[7]);
      s.u[lt][(2 * l8) ^ lt] = make_float4(uu[0], uu[1], uu[2], uu[3]);
      s.u[lt][(2 * l8 + 1) ^ lt] = make_float4(uu[4], uu[5], uu[6], uu[7]);
      if (zp) {
        float zz[8];
        r_z.get(zz);
#pragma unroll
        for (int i = 0; i < 8; ++i) dy[i] *= zz[i] * sigmoid_f<PRECISE>(zz[i]);
      }
      s.e[lt][(2 * l8) ^ lt] = make_float4(dy[0], dy[1], dy[2], dy[3]);
      s.e[lt][(2 * l8 + 1) ^ lt] = make_float4(dy[4], dy[5], dy[6], dy[7]);
      reinterpret_cast<float4*>(s.bc[0])[lane] = r_b;
      reinterpret_cast<float4*>(s.bc[1])[lane] = r_c;
      cur_dy = r_dy; cur_z = r_z; cur_row = r_row;
#pragma unroll
      for (int i = 0; i < 4; ++i) { h[i][0] = make_float2(r_h[i].x, r_h[i].y); h[i][1] = make_float2(r_h[i].z, r_h[i].w); }
    }
    __syncwarp();
    if (k > k_lo) fetch(k - 1);

    // ---- the interval's states, from its checkpoint
#pragma unroll 4
    for (int r = 0; r < CK; ++r) {
      const float4 dl4 = s.dl[r][cg ^ r], u4 = s.u[r][cg ^ r], B4 = s.bc[0][r][q];
      const float dlv[4] = {dl4.x, dl4.y, dl4.z, dl4.w}, uv[4] = {u4.x, u4.y, u4.z, u4.w};
      const float2 Bv[2] = {make_float2(B4.x, B4.y), make_float2(B4.z, B4.w)};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        s.h[r][i][lane] = make_float4(h[i][0].x, h[i][0].y, h[i][1].x, h[i][1].y);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float2 x = __fmul2_rn(dup(dlv[i]), a2[i][j]);
          const float2 a = exp_pair<PRECISE>(x);
          const float2 uB = __fmul2_rn(dup(ZOH ? uv[i] : uv[i] * dlv[i]), Bv[j]);
          if (!ZOH) {
            h[i][j] = __ffma2_rn(a, h[i][j], uB);
          } else if (PRECISE) {
            const float2 nem1 = make_float2(-expm1f(x.x), -expm1f(x.y));
            h[i][j] = __ffma2_rn(a, h[i][j], __fmul2_rn(__fmul2_rn(nem1, nik[i][j]), uB));
          } else {
            const float2 w = __fmul2_rn(nik[i][j], uB);
            h[i][j] = __ffma2_rn(a, sub2(h[i][j], w), w);
          }
        }
      }
    }

    // ---- reverse sweep
#pragma unroll 2
    for (int r = CK - 1; r >= 0; --r) {
      const float4 dl4 = s.dl[r][cg ^ r], u4 = s.u[r][cg ^ r], e4 = s.e[r][cg ^ r], B4 = s.bc[0][r][q], C4 = s.bc[1][r][q];
      const float dlv[4] = {dl4.x, dl4.y, dl4.z, dl4.w}, uv[4] = {u4.x, u4.y, u4.z, u4.w}, ev[4] = {e4.x, e4.y, e4.z, e4.w};
      const float2 Bv[2] = {make_float2(B4.x, B4.y), make_float2(B4.z, B4.w)}, Cv[2] = {make_float2(C4.x, C4.y), make_float2(C4.z, C4.w)};
      float2 dB[2], dC[2];
      float ddv[4], duv[4], yv[4];
      float4 hp4[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) hp4[i] = s.h[r][i][lane];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 hp[2] = {make_float2(hp4[i].x, hp4[i].y), make_float2(hp4[i].z, hp4[i].w)};
        const float2 dl = dup(dlv[i]), uu = dup(uv[i]), ee = dup(ev[i]);
        float2 dd, du, yy;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float2 x = __fmul2_rn(dl, a2[i][j]);
          const float2 a = exp_pair<PRECISE>(x);
          yy = j == 0 ? __fmul2_rn(Cv[j], h[i][j]) : __ffma2_rn(Cv[j], h[i][j], yy);
          dC[j] = i == 0 ? __fmul2_rn(ee, h[i][j]) : __ffma2_rn(ee, h[i][j], dC[j]);
          const float2 gg = __ffma2_rn(Cv[j], ee, g[i][j]);
          if (ZOH) {
            const float2 w = __fmul2_rn(nik[i][j], __fmul2_rn(uu, Bv[j]));
            const float2 gp = __fmul2_rn(gg, __fmul2_rn(a, sub2(hp[j], w)));
            const float2 oma = PRECISE ? make_float2(-expm1f(x.x), -expm1f(x.y)) : sub2(dup(1.0f), a);      // 1 - a
            const float2 rr = __fmul2_rn(__fmul2_rn(gg, oma), nik[i][j]);
            dd = j == 0 ? __fmul2_rn(a2[i][j], gp) : __ffma2_rn(a2[i][j], gp, dd);
            du = j == 0 ? __fmul2_rn(rr, Bv[j]) : __ffma2_rn(rr, Bv[j], du);
            dB[j] = i == 0 ? __fmul2_rn(rr, uu) : __ffma2_rn(rr, uu, dB[j]);
            dA[i][j] = __ffma2_rn(dl, gp, dA[i][j]);
            dA[i][j] = __ffma2_rn(rr, w, dA[i][j]);
          } else {
            const float2 gp = __fmul2_rn(gg, __fmul2_rn(a, hp[j]));
            const float2 gB = __fmul2_rn(gg, Bv[j]);
            dd = j == 0 ? __fmul2_rn(a2[i][j], gp) : __ffma2_rn(a2[i][j], gp, dd);
            du = j == 0 ? gB : __fadd2_rn(du, gB);
            const float2 ud = dup(uv[i] * dlv[i]);
            dB[j] = i == 0 ? __fmul2_rn(gg, ud) : __ffma2_rn(gg, ud, dB[j]);
            dA[i][j] = __ffma2_rn(dl, gp, dA[i][j]);
          }
          g[i][j] = __fmul2_rn(gg, a);
          h[i][j] = hp[j];
        }
        yv[i] = yy.x + yy.y;
        const float dsum = (dd.x + dd.y) * (PRECISE ? 1.0f : kLn2), usum = du.x + du.y;
        if (ZOH) { ddv[i] = dsum; duv[i] = usum; }
        else { ddv[i] = fmaf(usum, uv[i], dsum); duv[i] = usum * dlv[i]; }        // b = Delta B: du = Delta sum g B, dDelta += u sum g B
      }
      // partial sums over this lane's states, into the slot of the state that every lane has now consumed
      __syncwarp();
      s.h[r][0][ysw(lane, r)] = make_float4(ddv[0], ddv[1], ddv[2], ddv[3]);
      s.h[r][1][ysw(lane, r)] = make_float4(duv[0], duv[1], duv[2], duv[3]);
      s.h[r][2][ysw(lane, r)] = make_float4(yv[0], yv[1], yv[2], yv[3]);
      // sums over the warp's channels: 8 values (4 dB, 4 dC of the lane's states) over the 8 channel groups; three exchange
      // steps halve the values a lane keeps while adding its partner's, so every lane ends with ONE fully reduced value
      {
        const float v[8] = {dB[0].x, dB[0].y, dB[1].x, dB[1].y, dC[0].x, dC[0].y, dC[1].x, dC[1].y};
        const bool b2 = lane & 4, b3 = lane & 8, b4 = lane & 16;
        float w4[4], w2[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float send = b2 ? v[i] : v[4 + i], keep = b2 ? v[4 + i] : v[i];
          w4[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float send = b3 ? w4[i] : w4[2 + i], keep = b3 ? w4[2 + i] : w4[i];
          w2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
        const float send = b4 ? w2[0] : w2[1], keep = b4 ? w2[1] : w2[0];
        const float tot = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        const int t = k * CK + r;
        float* dst = (b2 ? p.dCm : p.dBm) + (b * L + t) * NST + 4 * q + (b3 ? 2 : 0) + (b4 ? 1 : 0);
        if (t < L) atomicAdd(dst, tot);
      }
    }
    __syncwarp();

    // ---- outputs of step lt, channels lc .. lc+7: the four lanes' partial sums of each value
    {
      float dd[8], du[8], yy[8], dl[8], uu[8], ee[8];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int grp = 2 * l8 + hf;
        float4 acc[3];
#pragma unroll
        for (int v = 0; v < 3; ++v) {
          const float4 x0 = s.h[lt][v][ysw(grp * 4, lt)], x1 = s.h[lt][v][ysw(grp * 4 + 1, lt)], x2 = s.h[lt][v][ysw(grp * 4 + 2, lt)], x3 = s.h[lt][v][ysw(grp * 4 + 3, lt)];
          acc[v] = make_float4((x0.x + x1.x) + (x2.x + x3.x), (x0.y + x1.y) + (x2.y + x3.y), (x0.z + x1.z) + (x2.z + x3.z), (x0.w + x1.w) + (x2.w + x3.w));
        }
        dd[4 * hf] = acc[0].x; dd[4 * hf + 1] = acc[0].y; dd[4 * hf + 2] = acc[0].z; dd[4 * hf + 3] = acc[0].w;
        du[4 * hf] = acc[1].x; du[4 * hf + 1] = acc[1].y; du[4 * hf + 2] = acc[1].z; du[4 * hf + 3] = acc[1].w;
        yy[4 * hf] = acc[2].x; yy[4 * hf + 1] = acc[2].y; yy[4 * hf + 2] = acc[2].z; yy[4 * hf + 3] = acc[2].w;
        const float4 d4 = s.dl[lt][grp ^ lt], u4 = s.u[lt][grp ^ lt], e4 = s.e[lt][grp ^ lt];
        dl[4 * hf] = d4.x; dl[4 * hf + 1] = d4.y; dl[4 * hf + 2] = d4.z; dl[4 * hf + 3] = d4.w;
        uu[4 * hf] = u4.x; uu[4 * hf + 1] = u4.y; uu[4 * hf + 2] = u4.z; uu[4 * hf + 3] = u4.w;
        ee[4 * hf] = e4.x; ee[4 * hf + 1] = e4.y; ee[4 * hf + 2] = e4.z; ee[4 * hf + 3] = e4.w;
      }
      const int t = k * CK + lt;
      if (t < L) {
        const size_t row = b * L + t;
#pragma unroll
        for (int i = 0; i < 8; ++i) { du[i] = fmaf(Dv[i], ee[i], du[i]); dDacc[i] = fmaf(ee[i], uu[i], dDacc[i]); }
        Raw8<T>::store(static_cast<T*>(p.du) + row * De + lc, du);
        if (zp) {
          float zz[8], dy[8], o[8];
          cur_z.get(zz); cur_dy.get(dy);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float sg = sigmoid_f<PRECISE>(zz[i]);
            o[i] = dy[i] * fmaf(Dv[i], uu[i], yy[i]) * sg * (1.0f + zz[i] * (1.0f - sg));
          }
          Raw8<T>::store(static_cast<T*>(p.dz) + (size_t)cur_row * p.ldz + lc, o);
          if (p.dz_rows)
            for (int kk = 1; kk < p.K; ++kk) Raw8<T>::store(static_cast<T*>(p.dz) + (size_t)__ldg(p.dz_rows + row * p.K + kk) * p.ldz + lc, o);
        }
        if (p.dpre) {
#pragma unroll
          for (int i = 0; i < 8; ++i) { dd[i] *= one_minus_exp<PRECISE>(dl[i]); dbacc[i] += dd[i]; }
          Raw8<T>::store(static_cast<T*>(p.dpre) + row * De + lc, dd);
        } else {
          Raw8<float>::store(p.ddelta + row * De + lc, dd);
        }
      }
    }
    __syncwarp();
  }

#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      atomicAdd(p.dA + (size_t)(c0 + i) * NST + 4 * q + 2 * j, dA[i][j].x);
      atomicAdd(p.dA + (size_t)(c0 + i) * NST + 4 * q + 2 * j + 1, dA[i][j].y);
    }
    if (p.dh0 && cj == 0)
      *reinterpret_cast<float4*>(p.dh0 + (b * De + c0 + i) * NST + 4 * q) = make_float4(g[i][0].x, g[i][0].y, g[i][1].x, g[i][1].y);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) { dDacc[i] += __shfl_xor_sync(0xffffffffu, dDacc[i], o); dbacc[i] += __shfl_xor_sync(0xffffffffu, dbacc[i], o); }
    if (lt == 0 && p.dD) atomicAdd(p.dD + lc + i, dDacc[i]);
    if (lt == 0 && p.dpre) atomicAdd(p.db_dt + lc + i, dbacc[i]);
  }
}

// Pre-pass of the chunk-parallel form, one piece of a coarse chunk per blockIdx.z: from a zero gradient, the gradient that leaves the
// piece's start (g <- a_t (g + C_t e_t), t descending) and the sum of Delta over it.  A lane owns all 16 states of one
// channel, a warp 32 channels; eight steps are staged at a time, the next eight in flight.  Bound by the special-function unit
// (one exponential per state and step against three fp32 operations).
struct PreSmem { float2 de[CK][32]; float4 c[CK][4]; };
template <typename T, typename TD>
__global__ void __launch_bounds__(BT)
scan_bwd_prepass_kernel(const BwdArgs p) {
  pdl_sync();
  constexpr bool PRECISE = sizeof(T) == 4;
  __shared__ PreSmem sm[WPB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PreSmem& s = sm[warp];
  const int De = p.De;
  const int c_warp = blockIdx.x * BCH + warp * WCH;
  if (c_warp >= De) return;
  const size_t b = blockIdx.y;
  const int cj = blockIdx.z / p.mp + 1, piece = blockIdx.z % p.mp;      // chunk 0's start gradient is nobody's input
  const int c_hi = min((cj + 1) * p.Lc, p.L), t_lo = min(cj * p.Lc + piece * p.Lp, c_hi), t_hi = min(t_lo + p.Lp, c_hi);
  const int c = c_warp + lane;
  const int lt = lane & 7, l8 = lane >> 3, lc = c_warp + 8 * l8;
  float2 a2[8], g[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 av = *reinterpret_cast<const float4*>(p.A + (size_t)c * NST + 4 * i);
    const float sc = PRECISE ? 1.0f : kLog2e;
    a2[2 * i] = make_float2(av.x * sc, av.y * sc); a2[2 * i + 1] = make_float2(av.z * sc, av.w * sc);
    g[2 * i] = make_float2(0.0f, 0.0f); g[2 * i + 1] = g[2 * i];
  }
  float sd = 0.0f;
  const T* __restrict__ dyp = static_cast<const T*>(p.dy);
  const T* __restrict__ zp = static_cast<const T*>(p.z);
  const TD* __restrict__ dlp = static_cast<const TD*>(p.delta);
  Raw8<TD> r_dl; Raw8<T> r_dy, r_z; float4 r_c;
  auto fetch = [&](int t0) {
    const int t = t0 + lt;
    if (t < t_hi) {
      const size_t row = b * p.L + t;
      r_dl.load(dlp + row * De + lc); r_dy.load(dyp + row * De + lc);
      if (zp) r_z.load(zp + row * p.ldz + lc);
    } else {
      r_dl.zero(); r_dy.zero(); r_z.zero();
    }
    r_c = t0 + (lane >> 2) < t_hi ? __ldg(reinterpret_cast<const float4*>(p.Cm + (b * p.L + t0) * NST) + lane) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  };
  int t0 = t_lo + (t_hi - t_lo - 1) / CK * CK;      // (an empty piece: t_lo, every step past the end)
  fetch(t0);
  for (; t0 >= t_lo; t0 -= CK) {
    {
      float dl[8], dy[8];
      r_dl.get(dl); r_dy.get(dy);
      if (zp) {
        float zz[8];
        r_z.get(zz);
#pragma unroll
        for (int i = 0; i < 8; ++i) dy[i] *= zz[i] * sigmoid_f<PRECISE>(zz[i]);
      }
      // channel pairs of an 8-channel group rotated by the step: the eight lanes of a store fall into different banks
      float4* row = reinterpret_cast<float4*>(&s.de[lt][0]);
#pragma unroll
      for (int i = 0; i < 4; ++i) row[(4 * l8 + i) ^ lt] = make_float4(dl[2 * i], dy[2 * i], dl[2 * i + 1], dy[2 * i + 1]);
      reinterpret_cast<float4*>(s.c)[lane] = r_c;
    }
    __syncwarp();
    if (t0 > t_lo) fetch(t0 - CK);
#pragma unroll
    for (int r = CK - 1; r >= 0; --r) {
      const float2 de = s.de[r][((((lane >> 1) ^ r)) << 1) | (lane & 1)];
      sd += de.x;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 C4 = s.c[r][i];
        const float2 x0 = __fmul2_rn(dup(de.x), a2[2 * i]), x1 = __fmul2_rn(dup(de.x), a2[2 * i + 1]);
        g[2 * i] = __fmul2_rn(__ffma2_rn(make_float2(C4.x, C4.y), dup(de.y), g[2 * i]), exp_pair<PRECISE>(x0));
        g[2 * i + 1] = __fmul2_rn(__ffma2_rn(make_float2(C4.z, C4.w), dup(de.y), g[2 * i + 1]), exp_pair<PRECISE>(x1));
      }
    }
    __syncwarp();
  }
  const size_t o = ((b * p.ncc + cj) * p.mp + piece) * De + c;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4*>(p.q_start + o * NST + 4 * i) = make_float4(g[2 * i].x, g[2 * i].y, g[2 * i + 1].x, g[2 * i + 1].y);
  p.sum_delta[o] = sd;
}

// Composes the gradient over the pieces of the coarse chunks (the recurrence is linear): with P_s = exp(A sum_delta_s), from dh_last,
//   g <- P_s g + q_start[s]  for s = ncc mp - 1 down to mp;  what stands before a coarse chunk's last piece is its g_in.
__global__ void __launch_bounds__(256)
scan_bwd_chain_kernel(const float* __restrict__ A, const float* __restrict__ dh_last, const float* __restrict__ q_start,
                      const float* __restrict__ sum_delta, float* __restrict__ g_in, int B, int De, int ncc, int mp) {
  pdl_sync();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * De * NST) return;
  const int n = (int)(i % NST);
  const int c = (int)((i / NST) % De);
  const size_t b = (size_t)(i / ((long long)NST * De));
  const float a = A[(size_t)c * NST + n];
  float g = dh_last ? dh_last[i] : 0.0f;
  constexpr int G = 8;             // pieces whose loads are in flight together
  for (int s0 = ncc * mp - 1; s0 >= mp; s0 -= G) {
    float qv[G], sv[G];
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const size_t sq = b * ncc * mp + max(s0 - k, mp);
      sv[k] = __ldg(sum_delta + sq * De + c);
      qv[k] = __ldg(q_start + (sq * De + c) * NST + n);
    }
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const int s = s0 - k;
      if (s < mp) break;
      if ((s + 1) % mp == 0) g_in[((b * ncc + s / mp) * De + c) * NST + n] = g;
      g = fmaf(expf(a * sv[k]), g, qv[k]);
    }
  }
  g_in[(b * ncc * De + c) * NST + n] = g;
}
// The same for the states (rom_scan_backward, where no forward scan has left checkpoints): h_in[0] = h0, h_in[j+1] = P_j h_in[j] + h_end[j].
__global__ void __launch_bounds__(256)
scan_bwd_chain_states_kernel(const float* __restrict__ A, const float* __restrict__ h0, const float* __restrict__ h_end,
                             const float* __restrict__ sum_delta, float* __restrict__ h_in, int B, int De, int ncc) {
  pdl_sync();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)B * De * NST) return;
  const int n = (int)(i % NST);
  const int c = (int)((i / NST) % De);
  const size_t b = (size_t)(i / ((long long)NST * De));
  const float a = A[(size_t)c * NST + n];
  float h = h0 ? h0[i] : 0.0f;
  for (int j = 0; j < ncc; ++j) {
    const size_t sq = b * ncc + j;
    h_in[(sq * De + c) * NST + n] = h;
    h = fmaf(expf(a * sum_delta[sq * De + c]), h, h_end[(sq * De + c) * NST + n]);
  }
}

// Coarse chunks per sequence: the count (at most 32, chunks of at least 64 steps) for which the reverse kernel's blocks best
// fill whole waves of two blocks per SM (148 SMs assumed); the pre-pass costs about a fifth of the reverse kernel, so one chunk
// (no pre-pass) is kept when it already fills 80 % of its waves.  A function of the sizes only (workspace sizing = launch).
int coarse_chunks(int B, int De, int L, int* Lc_out) {
  const long long blocks1 = (long long)B * ((De + BCH - 1) / BCH), slots = 148 * BLOCKS_PER_SM;
  int ncc = 1;
  double best = 0.0;
  for (int n = 1; n <= 32 && (n == 1 || (L + n - 1) / n >= 64); ++n) {
    const long long blocks = blocks1 * n;
    double fill = (double)blocks / (double)((blocks + slots - 1) / slots * slots);
    if (n == 1) fill *= 1.2;
    if (fill > best + 0.02) { best = fill; ncc = n; }
    if (blocks > 2 * slots) break;
  }
  int Lc = (L + ncc - 1) / ncc;
  Lc = (Lc + 15) / 16 * 16;
  *Lc_out = Lc;
  return (L + Lc - 1) / Lc;
}

// Pieces of a coarse chunk in the pre-pass (at most 8): the coarse chunks fill the reverse kernel's two blocks per SM and leave the
// pre-pass, which has four, with an uneven few.  The count minimises a model measured on this kernel: ns a step with so many blocks to
// an SM, and 160 ns of the chain kernel for every piece of a sequence.  Both kernels, us, one piece / by the rule: 16384 steps of 4096
// channels 363 / 294 (4 pieces), 3 x 1371 of 2048 55.6 / 48.2 (3), 2 x 6000 of 2048 142 / 120 (4), 5 x 800 of 3584 60 / 48 (5).
int prepass_pieces(int B, int De, int Lc, int ncc, int* Lp_out) {
  const long long blocks1 = (long long)B * ((De + BCH - 1) / BCH) * (ncc - 1);
  int best = 1;
  long long best_t = 0;
  for (int m = 1; m <= 8; ++m) {
    const long long k = (blocks1 * m + 147) / 148, Lp = ((Lc + m - 1) / m + CK - 1) / CK * CK;
    const long long t = Lp * (k <= 1 ? 133 : k == 2 ? 197 : k == 3 ? 275 : 90 * k) + 160LL * ncc * m;
    if (m == 1 || t < best_t) { best = m; best_t = t; *Lp_out = (int)Lp; }
  }
  return best;
}

}  // namespace

size_t scan_bwd_ckpt_floats(int B, int De, int L) { return (size_t)B * ((L + CK - 1) / CK) * De * NST; }

size_t scan_bwd_ws_bytes(int B, int De, int L) {
  int Lc = 0;
  const int ncc = coarse_chunks(B, De, L, &Lc);
  size_t floats = scan_bwd_ckpt_floats(B, De, L);
  if (ncc > 1) {
    int Lp = 0;
    floats += (size_t)B * ncc * De * (3 * NST + 1 + (NST + 1) * (size_t)prepass_pieces(B, De, Lc, ncc, &Lp));
  }
  return align_up(sizeof(float) * floats, 256);
}

void scan_bwd_zero(const rom_config& c, const ScanBwd& s, ZeroList& z) {
  auto add = [&](float* p, long long n) { if (p) { z.p[z.count] = p; z.n[z.count++] = n; } };
  add(s.dA, (long long)c.d_inner * NST);
  add(s.dBm, (long long)c.B * c.L * NST);
  add(s.dCm, (long long)c.B * c.L * NST);
  add(s.dD, c.d_inner);
  add(s.dpre ? s.db_dt : nullptr, c.d_inner);
}

cudaError_t launch_scan_backward(const rom_config& c, const ScanBwd& s, cudaStream_t st) {
  const int nck = (c.L + CK - 1) / CK;
  int Lc = 0;
  const int ncc = coarse_chunks(c.B, c.d_inner, c.L, &Lc);
  int Lp = 0;
  const int mp = prepass_pieces(c.B, c.d_inner, Lc, ncc, &Lp);
  const size_t n_fine = scan_bwd_ckpt_floats(c.B, c.d_inner, c.L), n_coarse = (size_t)c.B * ncc * c.d_inner * NST;
  float* g_in = s.ckpt + n_fine;
  float* h_end = g_in + n_coarse;
  float* h_in = h_end + n_coarse;
  float* q_start = h_in + n_coarse;
  float* sum_delta_h = q_start + n_coarse * mp;
  float* sum_delta = sum_delta_h + (size_t)c.B * ncc * c.d_inner;
  const BwdArgs a{s.dy, s.u, s.delta, s.A, s.Bm, s.Cm, s.D, s.z, s.dh_last, s.du, s.ddelta, s.dA, s.dBm, s.dCm, s.dD, s.dz, s.dh0, s.dpre, s.db_dt,
                  s.ckpt, c.L, c.d_inner, nck, s.ldz, s.dz_rows, s.K, Lc, ncc, g_in, Lp, mp, q_start, sum_delta};
  cudaError_t e = cudaSuccess;
  const bool zoh = c.disc_mode == 0, bf = c.dtype == ROM_BF16;
  const long long n_thr = (long long)c.B * c.d_inner * NST;
  const unsigned chain_blocks = (unsigned)((n_thr + 255) / 256);
  if (!s.ckpt_ready) {
    // no forward scan has left checkpoints: state-only passes of the forward kernel (chunk end states, chain, checkpoints)
    if (!s.delta_fp32) return cudaErrorInvalidValue;
    const float* delta = static_cast<const float*>(s.delta);
    const float* h_start = s.h0;
    if (ncc > 1) {
      if ((e = launch_scan_states(c, s.u, delta, s.A, s.Bm, Lc, ncc, nullptr, h_end, sum_delta_h, nullptr, 0, st)) != cudaSuccess) return e;
      launch_k(scan_bwd_chain_states_kernel, chain_blocks, 256, 0, st, s.A, s.h0, h_end, sum_delta_h, h_in, c.B, c.d_inner, ncc);
      count_launch();
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      h_start = h_in;
    }
    if ((e = launch_scan_states(c, s.u, delta, s.A, s.Bm, Lc, ncc, h_start, nullptr, nullptr, s.ckpt, nck, st)) != cudaSuccess) return e;
  }
  const dim3 grid((c.d_inner + BCH - 1) / BCH, c.B, ncc);
  if (ncc > 1) {
    const dim3 pgrid(grid.x, grid.y, (ncc - 1) * mp);
    if (!bf) launch_k(scan_bwd_prepass_kernel<float, float>, pgrid, BT, 0, st, a);
    else if (s.delta_fp32) launch_k(scan_bwd_prepass_kernel<__nv_bfloat16, float>, pgrid, BT, 0, st, a);
    else launch_k(scan_bwd_prepass_kernel<__nv_bfloat16, __nv_bfloat16>, pgrid, BT, 0, st, a);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    launch_k(scan_bwd_chain_kernel, chain_blocks, 256, 0, st, s.A, s.dh_last, q_start, sum_delta, g_in, c.B, c.d_inner, ncc, mp);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  auto kern = !bf ? (zoh ? scan_bwd_kernel<float, float, true> : scan_bwd_kernel<float, float, false>)
              : s.delta_fp32 ? (zoh ? scan_bwd_kernel<__nv_bfloat16, float, true> : scan_bwd_kernel<__nv_bfloat16, float, false>)
                             : (zoh ? scan_bwd_kernel<__nv_bfloat16, __nv_bfloat16, true> : scan_bwd_kernel<__nv_bfloat16, __nv_bfloat16, false>);
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BWD_SMEM)) != cudaSuccess) return e;
  launch_k(kern, grid, BT, BWD_SMEM, st, a);
  count_launch();
  return cudaGetLastError();
}

}  // namespace rom
