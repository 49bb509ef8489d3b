// Scalar-decay recurrence of the Mamba2-style block (rom_mamba2.cu) in its chunked matrix form, bf16 storage, 64 channels per head:
//   per head:  h_t = exp(dt_t A) h_{t-1} + dt_t x_t (x) B_t,   y_t = C_t h_t + D x_t,   out = y * SiLU(z)
// With S_t the running sum of dt A inside a chunk of 64 steps and h the state before the chunk,
//   y_t = sum_{s <= t} (C_t . B_s) exp(S_t - S_s) dt_s x_s  +  exp(S_t) C_t h  (+ D x_t on the diagonal),
//   h  <- exp(S_64) h + sum_s exp(S_64 - S_s) dt_s x_s (x) B_s.
// The decay is one number per head and step, so all of this is small matrix products over x, which is bf16 as stored: the
// element-wise selective-scan kernel spent two fp32 operations per state, step and channel plus the shared-memory traffic of B and
// C on what is 64 x 64 x 64 here (0.47 ms for 16384 steps of 4096 channels, with 0.10 ms to write Delta out per channel).
//
// Precision: x enters exactly; every other operand is computed in fp32 and fed as the sum of three bf16 terms (24 bits), products
// accumulate in fp32 -- the tensor cores replace fp32 arithmetic, not its precision.  (Terms of the state product below 2^-24 of
// the leading one are dropped: six of nine.)  S_t - S_s is a difference of running sums, and an fp32 sum would leave the decay
// between two late steps with the rounding of all that came before (units of S, where the recurrence has those of S_t - S_s): S_t is
// summed in fp64 and kept as two floats, the low one of s folded into dt_s.  Steps of a decay below 2^-256 count as 2^-256: a product
// with one of them is 0 in fp32 either way, and |S| stays below 2^14.  (One more fp32 addition per table entry: recurrence 251 -> 254 us
// at 16384 steps of 4096 channels.)
//
// A warp owns one head of one segment of the sequence and carries h (64 x 16, fp32) in accumulator registers; everything is kept
// transposed (Y^T = X^T G^T, h^T) so that h^T is the A operand of the next chunk as it stands and G^T, C and B fragments are
// computed element-wise in registers.  A block is eight heads of the same steps: they share C . B (one 64 x 64 table per chunk)
// and the B, C rows.  x and z come by cp.async (x a chunk ahead), the gated rows leave through the z tile.  A long sequence is
// cut into segments: a first launch runs them state-only from zero, a small kernel chains the segment states, the second launch
// is the full pass.
#include <type_traits>

#include "rom_internal.cuh"

namespace rom {
namespace {

typedef __nv_bfloat16 bf16;
constexpr int Q = 64, P = 64, NST = 16, HPB = 8, BT = HPB * 32;
constexpr int CBP = 72, NP = 68;                     // row pitches (floats) of the C . B table and of the transposed B, C rows
constexpr float kLog2e = 1.4426950408889634f;

struct SsdSmem {
  bf16 x[HPB][2][Q * P];                             // rows of 128 bytes, 16-byte pieces at piece ^ (row & 7)
  bf16 z[HPB][Q * P];
  float cb[Q * CBP];                                 // [t][s]
  float Bt[NST * NP], Ct[NST * NP];                  // [n][step]
  float S[HPB][Q], Sl[HPB][Q], dt[HPB][Q];           // running sum of dt A log2(e), its low part; dt 2^-Sl
};
struct SsdStateSmem {
  bf16 x[HPB][2][Q * P];
  float Bt[NST * NP];
  float S[HPB][Q], Sl[HPB][Q], dt[HPB][Q];
};

struct SsdArgs {
  const bf16* xc; const float* Bm; const float* Cm;  // [T, De], [T, 16]
  const bf16* zx; int W; int dt_col;                 // projection rows: z at column 0, dt at dt_col
  const float* dt_bias; const float* A; const float* D;
  bf16* y; int L, De, H;
  int seg_chunks, nseg;                              // chunks per segment
  const int32_t* nonfinite;                          // set when some x is not finite
  float* h_seg; float* s_seg;                        // [B, nseg, H, 1024] states in fragment order; [B, nseg, H] log2 decay of the segment
};

__device__ __forceinline__ uint32_t sptr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void ldsm_t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stsm_t(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// (v0, v1) as three packed bf16 pairs whose sum is v to 24 bits
__device__ __forceinline__ void split3(float v0, float v1, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(v1), "f"(v0));
  v0 -= __uint_as_float(hi << 16); v1 -= __uint_as_float(hi & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(mid) : "f"(v1), "f"(v0));
  v0 -= __uint_as_float(mid << 16); v1 -= __uint_as_float(mid & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(v1), "f"(v0));
}

// STATE: only the segment's end state from zero and its total decay (the chunks after the last segment boundary are not needed).
// CHECK: the outputs again, for a call whose conv has seen an x that is not finite (otherwise the launch ends at once): in a block on the
// diagonal the zero weights of the steps before such an x must not meet it.  A launch of its own, since the test inside the loops costs
// every call: 8 us of 202 where it looks x over, 5 to 15 where a flag skips that.  With this launch the layer takes 1149 us as without.
template <bool STATE, bool CHECK>
__global__ void __launch_bounds__(BT, 1)
ssd_kernel(const SsdArgs p) {
  pdl_sync();
  if (CHECK && *p.nonfinite == 0) return;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using Smem = typename std::conditional<STATE, SsdStateSmem, SsdSmem>::type;
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t4 = lane & 3;
  const int head = blockIdx.x * HPB + warp, seg = blockIdx.y;
  const size_t b = blockIdx.z;
  const int n_chunks = (p.L + Q - 1) / Q;
  const int c_lo = seg * p.seg_chunks, c_hi = min(c_lo + p.seg_chunks, n_chunks);
  const size_t tok_b = b * p.L;

  float h[4][2][4];                                  // h^T: rows p = 16 m + g (+ 8), columns n = 8 nt + 2 t4 (+ 1)
  const size_t seg_at = (b * p.nseg + seg) * p.H + head;
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) h[m][nt][i] = (!STATE && seg > 0) ? p.h_seg[seg_at * 1024 + (m * 8 + nt * 4 + i) * 32 + lane] : 0.0f;
  const float a2 = p.A[head] * kLog2e, bias = p.dt_bias ? p.dt_bias[head] : 0.0f, Dh = p.D ? p.D[head] : 0.0f;
  float s_total = 0.0f;

  // ---- loads: x and z tiles by cp.async, B / C rows and dt through registers, all a chunk ahead
  auto fetch_tile = [&](bf16* dst, const bf16* src, size_t ld, int c) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = i * 4 + (lane >> 3), pc = lane & 7, t = c * Q + r;
      cp16(sptr(dst + r * P) + ((pc ^ (r & 7)) << 4), src + (tok_b + min(t, p.L - 1)) * ld + (size_t)head * P + pc * 8, t < p.L);
    }
  };
  float4 rb, rc;
  bf16 rd[2];
  auto fetch_small = [&](int c) {
    const int t = c * Q + (tid >> 2);
    const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    rb = t < p.L ? __ldg(reinterpret_cast<const float4*>(p.Bm + (tok_b + t) * NST) + (tid & 3)) : z4;
    rc = (!STATE && t < p.L) ? __ldg(reinterpret_cast<const float4*>(p.Cm + (tok_b + t) * NST) + (tid & 3)) : z4;
#pragma unroll
    for (int j = 0; j < 2; ++j) rd[j] = p.zx[(tok_b + min(c * Q + lane + 32 * j, p.L - 1)) * p.W + p.dt_col + head];
  };
  fetch_tile(sm.x[warp][c_lo & 1], p.xc, p.De, c_lo);
  asm volatile("cp.async.commit_group;" ::: "memory");
  fetch_small(c_lo);

  for (int c = c_lo; c < c_hi; ++c) {
    if constexpr (!STATE) fetch_tile(sm.z[warp], p.zx, p.W, c);
    if (c + 1 < c_hi) fetch_tile(sm.x[warp][(c + 1) & 1], p.xc, p.De, c + 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    {
      const int r = tid >> 2, q4 = (tid & 3) * 4;
      const float bv[4] = {rb.x, rb.y, rb.z, rb.w}, cv[4] = {rc.x, rc.y, rc.z, rc.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        sm.Bt[(q4 + i) * NP + r] = bv[i];
        if constexpr (!STATE) sm.Ct[(q4 + i) * NP + r] = cv[i];
      }
      // dt and the running sum of dt A (base-2 logarithm of the decay); steps past the end of the sequence do nothing
      float d[2];
      double s[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        d[j] = c * Q + lane + 32 * j < p.L ? softplus_f(to_f32(rd[j]) + bias) : 0.0f;
        const float x = d[j] * a2;
        s[j] = x < -256.0f ? -256.0 : (double)x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double v = __shfl_up_sync(0xffffffffu, s[j], o);
          if (lane >= o) s[j] += v;
        }
      }
      s[1] += __shfl_sync(0xffffffffu, s[0], 31);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float hi = (float)s[j], lo = (float)(s[j] - (double)hi);
        sm.S[warp][lane + 32 * j] = hi;
        sm.Sl[warp][lane + 32 * j] = lo;
        sm.dt[warp][lane + 32 * j] = d[j] * exp2f(-lo);
      }
    }
    if (c + 1 < c_hi) fetch_small(c + 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");      // x of this chunk (committed an iteration ago)
    __syncthreads();
    if constexpr (!STATE) {
      // C . B of the chunk, 4 x 4 per thread, lower triangle
      const int t0 = (tid >> 4) * 4, s0 = (tid & 15) * 4;
      if (s0 <= t0) {
        float acc[4][4] = {};
#pragma unroll
        for (int n = 0; n < NST; ++n) {
          const float4 cq = *reinterpret_cast<const float4*>(sm.Ct + n * NP + t0), bq = *reinterpret_cast<const float4*>(sm.Bt + n * NP + s0);
          const float cv[4] = {cq.x, cq.y, cq.z, cq.w}, bv[4] = {bq.x, bq.y, bq.z, bq.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(cv[i], bv[j], acc[i][j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(sm.cb + (t0 + i) * CBP + s0) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
      }
      __syncthreads();
    }
    const bf16* xs = sm.x[warp][c & 1];
    const float* Sw = sm.S[warp];
    const float* dw = sm.dt[warp];
    // A fragments of X^T: rows p = 16 m .., columns s = 16 ks ..
    auto load_x = [&](int ks, uint32_t (&xa)[4][4]) {
      const int s = ks * 16 + (lane & 7) + ((lane >> 4) << 3);
#pragma unroll
      for (int m = 0; m < 4; ++m) ldsm_t(sptr(xs + s * P) + (((2 * m + ((lane >> 3) & 1)) ^ (s & 7)) << 4), xa[m]);
    };

    if constexpr (!STATE) {
#pragma unroll 1
      for (int th = 0; th < 2; ++th) {               // 32 output steps at a time: t = 32 th + 8 tj + g
        float acc[4][4][4] = {};                     // [m][tj]: rows p, columns t = .. + 2 t4 (+ 1)
        // the state before the chunk: Y^T += h^T (exp(S_t) C_t)^T
        if (c > 0) {
          uint32_t ce[4][3][2];
#pragma unroll
          for (int tj = 0; tj < 4; ++tj) {
            const int t = 32 * th + 8 * tj + g;
            const float e = ex2_ftz(Sw[t]);
#pragma unroll
            for (int k = 0; k < 2; ++k)
              split3(sm.Ct[(8 * k + 2 * t4) * NP + t] * e, sm.Ct[(8 * k + 2 * t4 + 1) * NP + t] * e, ce[tj][0][k], ce[tj][1][k], ce[tj][2][k]);
          }
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            uint32_t ha[3][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
              split3(h[m][nt][0], h[m][nt][1], ha[0][2 * nt], ha[1][2 * nt], ha[2][2 * nt]);
              split3(h[m][nt][2], h[m][nt][3], ha[0][2 * nt + 1], ha[1][2 * nt + 1], ha[2][2 * nt + 1]);
            }
#pragma unroll
            for (int u = 2; u >= 0; --u)             // smallest products first
#pragma unroll
              for (int v = 2 - u; v >= 0; --v)
#pragma unroll
                for (int tj = 0; tj < 4; ++tj) mma(acc[m][tj], ha[u], ce[tj][v][0], ce[tj][v][1]);
          }
        }
        // steps of the chunk itself: Y^T += X^T G^T
#pragma unroll 1
        for (int ks = 0; ks < 2 * th + 2; ++ks) {
          uint32_t xa[4][4];
          load_x(ks, xa);
          bool bad = false;
          if (CHECK && ks >= 2 * th) {
            uint32_t mx = 0u;
#pragma unroll
            for (int m = 0; m < 4; ++m)
#pragma unroll
              for (int i = 0; i < 4; ++i) mx = __vmaxu2(mx, xa[m][i] & 0x7f807f80u);
            bad = __any_sync(0xffffffffu, (mx >> 16) == 0x7f80u || (mx & 0xffffu) == 0x7f80u);
          }
          const int s0 = 16 * ks + 2 * t4;
          const float2 S0 = *reinterpret_cast<const float2*>(Sw + s0), S1 = *reinterpret_cast<const float2*>(Sw + s0 + 8);
          const float2 d0 = *reinterpret_cast<const float2*>(dw + s0), d1 = *reinterpret_cast<const float2*>(dw + s0 + 8);
#pragma unroll
          for (int tj = 0; tj < 4; ++tj) {
            const int jt = 4 * th + tj;
            if (jt < 2 * ks) continue;               // (warp-uniform) all of it is above the diagonal
            const int t = 8 * jt + g;
            const float St = Sw[t], Sl = sm.Sl[warp][t];
            const float2 q0 = *reinterpret_cast<const float2*>(sm.cb + t * CBP + s0), q1 = *reinterpret_cast<const float2*>(sm.cb + t * CBP + s0 + 8);
            float v[4] = {q0.x * ex2_ftz((St - S0.x) + Sl) * d0.x, q0.y * ex2_ftz((St - S0.y) + Sl) * d0.y,
                          q1.x * ex2_ftz((St - S1.x) + Sl) * d1.x, q1.y * ex2_ftz((St - S1.y) + Sl) * d1.y};
            if (jt < 2 * ks + 2) {                   // on the diagonal: later steps out, the skip term in
              const int sv[4] = {s0, s0 + 1, s0 + 8, s0 + 9};
#pragma unroll
              for (int i = 0; i < 4; ++i) v[i] = sv[i] > t ? 0.0f : sv[i] == t ? v[i] + Dh : v[i];
            }
            uint32_t gb[3][2];
            split3(v[0], v[1], gb[0][0], gb[1][0], gb[2][0]);
            split3(v[2], v[3], gb[0][1], gb[1][1], gb[2][1]);
            if (CHECK && bad && jt < 2 * ks + 2) {            // one step s of the block at a time, kept by the steps t >= s
#pragma unroll 1
              for (int i = 0; i < 16; ++i) {
                const uint32_t keep = t4 == ((i & 7) >> 1) ? ((i & 1) ? 0xffff0000u : 0x0000ffffu) : 0u;
                const uint32_t k0 = i < 8 ? keep : 0u, k1 = i < 8 ? 0u : keep;
                const bool in0 = 8 * jt + 2 * t4 >= 16 * ks + i, in1 = 8 * jt + 2 * t4 + 1 >= 16 * ks + i;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                  const uint32_t xi[4] = {xa[m][0] & k0, xa[m][1] & k0, xa[m][2] & k1, xa[m][3] & k1};
                  float d[4] = {acc[m][tj][0], acc[m][tj][1], acc[m][tj][2], acc[m][tj][3]};
#pragma unroll
                  for (int u = 2; u >= 0; --u) mma(d, xi, gb[u][0] & k0, gb[u][1] & k1);
                  if (in0) { acc[m][tj][0] = d[0]; acc[m][tj][2] = d[2]; }
                  if (in1) { acc[m][tj][1] = d[1]; acc[m][tj][3] = d[3]; }
                }
              }
              continue;
            }
#pragma unroll
            for (int u = 2; u >= 0; --u)
#pragma unroll
              for (int m = 0; m < 4; ++m) mma(acc[m][tj], xa[m], gb[u][0], gb[u][1]);
          }
        }
        // gate and round, in place of the z tile
        if (th == 0) {
          asm volatile("cp.async.wait_group 0;" ::: "memory");
          __syncwarp();
        }
#pragma unroll
        for (int tp = 0; tp < 2; ++tp)
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int t = 32 * th + 16 * tp + (lane & 7) + ((lane >> 4) << 3);
            const uint32_t addr = sptr(sm.z[warp] + t * P) + (((2 * m + ((lane >> 3) & 1)) ^ (t & 7)) << 4);
            uint32_t zr[4], o[4];
            ldsm_t(addr, zr);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float y0 = acc[m][2 * tp + (i >> 1)][2 * (i & 1)], y1 = acc[m][2 * tp + (i >> 1)][2 * (i & 1) + 1];
              const float z0 = __uint_as_float(zr[i] << 16), z1 = __uint_as_float(zr[i] & 0xffff0000u);
              const __nv_bfloat162 r = __floats2bfloat162_rn(y0 * silu_fast(z0), y1 * silu_fast(z1));
              o[i] = *reinterpret_cast<const uint32_t*>(&r);
            }
            stsm_t(addr, o[0], o[1], o[2], o[3]);
          }
      }
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int r = i * 4 + (lane >> 3), pc = lane & 7, t = c * Q + r;
        if (t < p.L)
          *reinterpret_cast<uint4*>(p.y + (tok_b + t) * p.De + (size_t)head * P + pc * 8) =
              *reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(sm.z[warp] + r * P) + ((pc ^ (r & 7)) << 4));
      }
      __syncwarp();
    }

    // ---- the state after the chunk
    const float S63 = Sw[Q - 1], Sl63 = sm.Sl[warp][Q - 1], dec = ex2_ftz(S63);
    s_total += S63;
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) h[m][nt][i] *= dec;
#pragma unroll 1
    for (int ks = 0; ks < 4; ++ks) {
      uint32_t xa[4][4];
      load_x(ks, xa);
      const int s0 = 16 * ks + 2 * t4;
      const float2 S0 = *reinterpret_cast<const float2*>(Sw + s0), S1 = *reinterpret_cast<const float2*>(Sw + s0 + 8);
      const float2 d0 = *reinterpret_cast<const float2*>(dw + s0), d1 = *reinterpret_cast<const float2*>(dw + s0 + 8);
      const float f[4] = {ex2_ftz((S63 - S0.x) + Sl63) * d0.x, ex2_ftz((S63 - S0.y) + Sl63) * d0.y,
                          ex2_ftz((S63 - S1.x) + Sl63) * d1.x, ex2_ftz((S63 - S1.y) + Sl63) * d1.y};
#pragma unroll
      for (int nt = 0; nt < 2; ++nt) {
        const float2 b0 = *reinterpret_cast<const float2*>(sm.Bt + (8 * nt + g) * NP + s0), b1 = *reinterpret_cast<const float2*>(sm.Bt + (8 * nt + g) * NP + s0 + 8);
        uint32_t wb[3][2];
        split3(f[0] * b0.x, f[1] * b0.y, wb[0][0], wb[1][0], wb[2][0]);
        split3(f[2] * b1.x, f[3] * b1.y, wb[0][1], wb[1][1], wb[2][1]);
#pragma unroll
        for (int u = 2; u >= 0; --u)
#pragma unroll
          for (int m = 0; m < 4; ++m) mma(h[m][nt], xa[m], wb[u][0], wb[u][1]);
      }
    }
    __syncthreads();                                 // the shared tables are free for the next chunk
  }
  if constexpr (STATE) {
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) p.h_seg[seg_at * 1024 + (m * 8 + nt * 4 + i) * 32 + lane] = h[m][nt][i];
    if (lane == 0) p.s_seg[seg_at] = s_total;
  }
}

// Start state of every segment, in place over the end states: h_in[0] = 0, h_in[j + 1] = 2^s_seg[j] h_in[j] + h_end[j].
__global__ void __launch_bounds__(256)
ssd_chain(float* __restrict__ h_seg, const float* __restrict__ s_seg, int H, int nseg, long long total) {
  pdl_sync();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;      // (sequence, head, element)
  if (i >= total) return;
  const int el = (int)(i & 1023);
  const long long bh = i >> 10;
  const int head = (int)(bh % H);
  const size_t b = (size_t)(bh / H);
  float* hp = h_seg + (b * nseg * H + head) * 1024 + el;
  const float* sp = s_seg + b * nseg * H + head;
  const size_t hs = (size_t)H * 1024;
  constexpr int G = 8;                               // segments whose loads are in flight together
  float cur = 0.0f;
  for (int j0 = 0; j0 < nseg; j0 += G) {
    float end[G], dec[G];
#pragma unroll
    for (int j = 0; j < G; ++j) {
      const bool in = j0 + j + 1 < nseg;             // nobody needs the last segment's end
      end[j] = in ? hp[(j0 + j) * hs] : 0.0f;
      dec[j] = in ? exp2f(sp[(size_t)(j0 + j) * H]) : 0.0f;
    }
#pragma unroll
    for (int j = 0; j < G; ++j) {
      if (j0 + j >= nseg) break;
      hp[(j0 + j) * hs] = cur;
      cur = fmaf(dec[j], cur, end[j]);
    }
  }
}

// Chunks per segment: whole sequences when (sequences x head groups) fill the SMs to 80 %, else the split (segments of at least
// two chunks) whose blocks best fill whole waves of one block per SM (148 assumed: workspace sizing and launch agree).
int segment_chunks(int B, int H, int L) {
  const int n_chunks = (L + Q - 1) / Q;
  const long long blocks1 = (long long)B * (H / HPB);
  int best = n_chunks;
  double best_fill = 0.0;
  for (int n = 1; n <= 64 && (n == 1 || n_chunks / n >= 2); ++n) {
    const int per = (n_chunks + n - 1) / n, ns = (n_chunks + per - 1) / per;
    const long long blocks = blocks1 * ns;
    double fill = (double)blocks / (double)((blocks + 147) / 148 * 148) * ((double)n_chunks / ((double)per * ns));
    if (n == 1) fill *= 1.25;                        // no state-only launch
    if (fill > best_fill + 0.01) { best_fill = fill; best = per; }
    if (blocks >= 2 * 148) break;
  }
  return best;
}

}  // namespace

bool ssd_applicable(const rom_config& c, int headdim) {
  return c.dtype == ROM_BF16 && headdim == P && c.d_state == NST && (c.d_inner / P) % HPB == 0 && !(c.flags & ROM_FLAG_SIMT_GEMM);
}

size_t ssd_ws_floats(const rom_config& c) {
  const int H = c.d_inner / P, per = segment_chunks(c.B, H, c.L), nseg = ((c.L + Q - 1) / Q + per - 1) / per;
  return nseg > 1 ? (size_t)c.B * nseg * H * 1025 : 0;
}

cudaError_t launch_ssd(const rom_config& c, const void* xc, const float* Bm, const float* Cm, const void* zx, int W, int dt_col, const float* dt_bias,
                       const float* A, const float* D, void* y, float* ws, const int32_t* nonfinite, cudaStream_t st) {
  const int H = c.d_inner / P, per = segment_chunks(c.B, H, c.L), nseg = ((c.L + Q - 1) / Q + per - 1) / per;
  const SsdArgs a{(const bf16*)xc, Bm, Cm, (const bf16*)zx, W, dt_col, dt_bias, A, D, (bf16*)y, c.L, c.d_inner, H, per, nseg,
                  nonfinite, ws, ws + (size_t)c.B * nseg * H * 1024};
  cudaError_t e;
  if (nseg > 1) {
    if ((e = cudaFuncSetAttribute(ssd_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SsdStateSmem))) != cudaSuccess) return e;
    launch_k(ssd_kernel<true, false>, dim3(H / HPB, nseg - 1, c.B), BT, sizeof(SsdStateSmem), st, a);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const long long total = (long long)c.B * H * 1024;
    launch_k(ssd_chain, (unsigned)((total + 255) / 256), 256, 0, st, a.h_seg, a.s_seg, H, nseg, total);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  for (auto kern : {ssd_kernel<false, false>, ssd_kernel<false, true>}) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SsdSmem))) != cudaSuccess) return e;
    launch_k(kern, dim3(H / HPB, nseg, c.B), BT, sizeof(SsdSmem), st, a);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace rom
