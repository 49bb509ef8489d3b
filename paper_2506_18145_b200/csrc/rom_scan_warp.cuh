// What one warp of the bf16 scan does: 32 channels of one chunk of one sequence, step by step (rom_scan_warp.cu, which says why; rom_scan_ring.cu
// for sequences with values that are not finite).
#pragma once

#include <type_traits>

#include "rom_scan_args.cuh"

namespace rom {
namespace {

typedef __nv_bfloat16 bf16;
constexpr int NST = 16;
constexpr int CK = kScanCkpt;     // steps per tile
constexpr int WCH = 32;           // channels per warp
constexpr float kLog2e = 1.4426950408889634f;

struct WarpTile {
  float4 dl[CK][8], u[CK][8];     // Delta, u of 4 channels; group g of step r sits at g ^ r
  float4 b[CK][4], c[CK][4];
  float D[WCH];                   // skip factors (zeros without)
  float4 y[CK][32];               // partial sums of 4 channels over one lane's states; lane l of step r at ysw(l, r)
};

// Which tiles of its chunk a warp takes: all of them, the state staying with it.  (rom_scan_ring.cu: warps in turns, which hand it on.)
struct AllTiles {
  static constexpr int STRIDE = CK;
  __device__ int first() const { return 0; }
  __device__ void take(float2 (&)[4][2], int) const {}
  __device__ void give(const float2 (&)[4][2], int, int) const {}
  __device__ bool has_last(int) const { return true; }
};

// SLOTS: the gate of a token is SiLU of the sum of its K >= 2 rows z_row[t K + k], which are also its output rows (y_rows).
template <typename TD, bool ZOH, int MODE, bool SLOTS, typename Tiles = AllTiles>
__device__ __forceinline__ void scan_warp_channels(const ScanArgs& p, WarpTile& s, const int c_warp, const int seq, const int chunk, const Tiles& tiles = {}) {
  constexpr int STRIDE = Tiles::STRIDE;
  constexpr bool FIRST = MODE == SCAN_FIRST || MODE == SCAN_FIRST_CKPT;
  const int lane = threadIdx.x & 31, De = p.De;
  const bool so = MODE == SCAN_STATE || MODE == SCAN_CKPT || (FIRST && chunk != 0);      // this block only produces states
  const int t_first = chunk == 0 ? 0 : p.L0 + (chunk - 1) * p.Lc;
  const int L = min(chunk == 0 ? p.L0 : p.Lc, p.L - t_first);      // steps of this chunk (<= 0: an empty chunk)
  const size_t sc = (size_t)seq * p.nch + chunk;            // index of the (sequence, chunk) state
  const size_t tok0 = (size_t)seq * p.L + (size_t)t_first;

  // ---- compute role: channels c0 .. c0+3 (pairs), states 4q .. 4q+3
  const int q = lane & 3, cg = lane >> 2;
  const int c0 = c_warp + 4 * cg;
  constexpr bool SECOND = MODE == SCAN_FULL || MODE == SCAN_FULL_CKPT;      // may be the second launch of the chunked scan
  float2 a2[4][2], kin[4][2], h[4][2], sdel[2];
  const float d_skip = !so && p.D ? __ldg(p.D + c_warp + lane) : 0.0f;      // (in flight with A: put down below)
  {
    float av[4][4], hv[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 a4 = __ldg(reinterpret_cast<const float4*>(p.A + (size_t)(c0 + i) * NST) + q);
      float4 h4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (p.h0 && !(FIRST && so)) h4 = load4_any(p.h0 + ((FIRST ? (size_t)seq : sc) * De + c0 + i) * NST + 4 * q);
      av[i][0] = a4.x; av[i][1] = a4.y; av[i][2] = a4.z; av[i][3] = a4.w;
      hv[i][0] = h4.x; hv[i][1] = h4.y; hv[i][2] = h4.z; hv[i][3] = h4.w;
    }
    if (SECOND && p.chain_end) {      // the state this chunk starts from: h <- exp(A sum Delta_j) h + h_end[j] over the chunks before
      const size_t s0 = sc - chunk;
      const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      for (int k0 = 0; k0 < chunk; k0 += 4) {      // four chunks' loads in flight; past the last one: the identity
        float4 d4[4], e4[4][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const size_t sk = s0 + k0 + k;
          const bool in = k0 + k < chunk;
          // (chunk 0's end state is the true one and nothing precedes it: its sum is not kept)
          d4[k] = in && k0 + k > 0 ? __ldg(reinterpret_cast<const float4*>(p.chain_sum + sk * De + c0)) : zero4;
#pragma unroll
          for (int i = 0; i < 4; ++i) e4[k][i] = in ? __ldg(reinterpret_cast<const float4*>(p.chain_end + (sk * De + c0 + i) * NST) + q) : zero4;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float dk[4] = {d4[k].x, d4[k].y, d4[k].z, d4[k].w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float ev[4] = {e4[k][i].x, e4[k][i].y, e4[k][i].z, e4[k][i].w};
#pragma unroll
            for (int n = 0; n < 4; ++n) hv[i][n] = fmaf(expf(av[i][n] * dk[i]), hv[i][n], ev[n]);
          }
        }
      }
    }
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        a2[n][j] = make_float2(av[2 * j][n] * kLog2e, av[2 * j + 1][n] * kLog2e);
        kin[n][j] = make_float2(-1.0f / av[2 * j][n], -1.0f / av[2 * j + 1][n]);
        h[n][j] = make_float2(hv[2 * j][n], hv[2 * j + 1][n]);
      }
    sdel[0] = make_float2(0.0f, 0.0f); sdel[1] = sdel[0];
  }
  auto put_state = [&](float* dst, auto any_tag) {      // [De, 16] state array of one (sequence, chunk or checkpoint); any: the caller's
    auto put = [&](float* at, float4 v) { if constexpr (decltype(any_tag)::value) store4_any(at, v); else *reinterpret_cast<float4*>(at) = v; };
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      put(dst + (size_t)(c0 + 2 * j) * NST + 4 * q, make_float4(h[0][j].x, h[1][j].x, h[2][j].x, h[3][j].x));
      put(dst + (size_t)(c0 + 2 * j + 1) * NST + 4 * q, make_float4(h[0][j].y, h[1][j].y, h[2][j].y, h[3][j].y));
    }
  };
  if (!so) s.D[lane] = d_skip;
  // ---- loader / output role: step lt of every tile, channels lc .. lc+7
  // (four lanes per row: a load's quarter-warp touches two rows of global memory, not eight)
  const int lt = lane >> 2, l8 = lane & 3, lc = c_warp + 8 * l8, t_own = tiles.first();
  const bf16* __restrict__ zp = so ? nullptr : static_cast<const bf16*>(p.z);
  const TD* dptr = static_cast<const TD*>(p.delta) + (tok0 + t_own + lt) * De + lc;
  const bf16* uptr = static_cast<const bf16*>(p.u) + (tok0 + t_own + lt) * De + lc;
  const float4* bptr = reinterpret_cast<const float4*>(p.Bm + (tok0 + t_own) * NST) + lane;
  const float4* cptr = reinterpret_cast<const float4*>(p.Cm + (tok0 + t_own) * NST) + lane;

  Raw8<TD> r_d;
  Raw8<bf16> r_u, r_z, r_z2, cur_u, cur_z, cur_z2;
  float4 r_b, r_c;
  int r_row = 0, cur_row = 0, r_row2 = 0, cur_row2 = 0;      // first output rows of this lane's step
  int z_i0 = 0, z_i1 = 0;          // SLOTS: rows of the next tile to fetch: their indices are a tile ahead, so that nothing waits for them
  auto fetch_rows = [&](int t0) {
    if (SLOTS && t0 + lt < L) {
      const int32_t* zr = p.z_row + (tok0 + t0 + lt) * p.K;
      z_i0 = __ldg(zr);
      z_i1 = __ldg(zr + 1);
    }
  };
  auto fetch = [&](int t0) {
    const int t = t0 + lt;
    const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (t < L) {
      r_d.load(dptr); r_u.load(uptr);
      if (!so) {
        if constexpr (SLOTS) {     // gate rows by slot; the third and later ones are fetched where they are added
          r_row = z_i0; r_row2 = z_i1;
          r_z.load(zp + (size_t)z_i0 * p.ldz + lc);
          r_z2.load(zp + (size_t)z_i1 * p.ldz + lc);
        } else {
          r_row = p.y_rows ? __ldg(p.y_rows + (tok0 + t) * p.K) : (int)(tok0 + t);
          if (zp) r_z.load(zp + (p.z_row ? (size_t)__ldg(p.z_row + tok0 + t) : tok0 + t) * p.ldz + lc);
        }
      }
    } else {                       // steps past the end change nothing
      r_d.zero(); r_u.zero();
    }
    dptr += (size_t)STRIDE * De; uptr += (size_t)STRIDE * De;
    const bool in = t0 + (lane >> 2) < L;
    r_b = in ? __ldg(bptr) : zero4;
    if (!so) r_c = in ? __ldg(cptr) : zero4;
    bptr += STRIDE * 4; cptr += STRIDE * 4;
    if (SLOTS && !so) fetch_rows(t0 + STRIDE);
  };

  auto run = [&](auto so_tag) {
    constexpr bool SO = decltype(so_tag)::value;
    constexpr bool CKPT = MODE == SCAN_CKPT || MODE == SCAN_FULL_CKPT || (MODE == SCAN_FIRST_CKPT && !SO);
    // from a zero state and with nothing read before the end, the state is carried times -A: one product less an update (16384 steps of
    // 4096 channels 280 -> 272 us for the first launch, 4 x 2048 of 2048 75.4 -> 73.8)
    constexpr bool SCALED = ZOH && SO && !CKPT;
    if (SLOTS && !SO) fetch_rows(t_own);
    fetch(t_own);
    for (int t0 = t_own; t0 < L; t0 += STRIDE) {
      {
        float d[8], uu[8];
        r_d.get(d); r_u.get(uu);
        if (!ZOH) {                // B-bar = Delta B: the input enters as Delta u
#pragma unroll
          for (int i = 0; i < 8; ++i) uu[i] *= d[i];
        }
        s.dl[lt][(2 * l8) ^ lt] = make_float4(d[0], d[1], d[2], d[3]);
        s.dl[lt][(2 * l8 + 1) ^ lt] = make_float4(d[4], d[5], d[6], d[7]);
        s.u[lt][(2 * l8) ^ lt] = make_float4(uu[0], uu[1], uu[2], uu[3]);
        s.u[lt][(2 * l8 + 1) ^ lt] = make_float4(uu[4], uu[5], uu[6], uu[7]);
        reinterpret_cast<float4*>(s.b)[lane] = r_b;
        if (!SO) { reinterpret_cast<float4*>(s.c)[lane] = r_c; cur_u = r_u; cur_z = r_z; cur_row = r_row; if (SLOTS) { cur_z2 = r_z2; cur_row2 = r_row2; } }
      }
      __syncwarp();
      if (t0 + STRIDE < L) fetch(t0 + STRIDE);
      tiles.take(h, t0);
      if constexpr (CKPT) put_state(p.ckpt + ((size_t)seq * p.nck + (size_t)((t_first + t0) / CK)) * De * NST, std::false_type{});
      // the next step's operands are requested before this step's arithmetic: a load issued behind a step's exponentials waits
      // for all of them in the queue that both share
      float4 nd = s.dl[0][cg], nu = s.u[0][cg], nb = s.b[0][q], nc = SO ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : s.c[0][q];
      constexpr int UF = SO ? 4 : CK;      // (state-only: nothing orders the steps, and eight at once are slower)
#pragma unroll UF
      for (int r = 0; r < CK; ++r) {
        const float4 d4 = nd, u4 = nu, b4 = nb, c4 = nc;
        if (r + 1 < CK) {
          nd = s.dl[r + 1][cg ^ (r + 1)]; nu = s.u[r + 1][cg ^ (r + 1)]; nb = s.b[r + 1][q];
          if (!SO) nc = s.c[r + 1][q];
        }
        const float2 dl[2] = {make_float2(d4.x, d4.y), make_float2(d4.z, d4.w)}, uu[2] = {make_float2(u4.x, u4.y), make_float2(u4.z, u4.w)};
        const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, cc[4] = {c4.x, c4.y, c4.z, c4.w};
        float2 acc[2];
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const float2 x = __fmul2_rn(dl[j], a2[n][j]);
            const float2 a = make_float2(ex2_ftz(x.x), ex2_ftz(x.y));
            const float2 uB = __fmul2_rn(uu[j], dup(bb[n]));
            if (SCALED) {
              h[n][j] = __ffma2_rn(a, __ffma2_rn(uB, dup(-1.0f), h[n][j]), uB);
            } else if (ZOH) {      // w = -B u / A, h <- a (h - w) + w
              const float2 w = __fmul2_rn(uB, kin[n][j]);
              h[n][j] = __ffma2_rn(a, __ffma2_rn(w, dup(-1.0f), h[n][j]), w);
            } else {
              h[n][j] = __ffma2_rn(a, h[n][j], uB);
            }
            if (!SO) acc[j] = n == 0 ? __fmul2_rn(dup(cc[n]), h[n][j]) : __ffma2_rn(dup(cc[n]), h[n][j], acc[j]);
          }
        if (SO) { sdel[0] = __fadd2_rn(sdel[0], dl[0]); sdel[1] = __fadd2_rn(sdel[1], dl[1]); }
        else s.y[r][ysw(lane, r)] = make_float4(acc[0].x, acc[0].y, acc[1].x, acc[1].y);
      }
      tiles.give(h, t0, L);
      __syncwarp();
      if (!SO) {
        // y = (sum over the four lanes + D u) * gate, rounded, written to the K rows of the token
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
            const float4 D4 = reinterpret_cast<const float4*>(s.D)[2 * l8 + hf];
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
    }
    if constexpr (SCALED)
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j) h[n][j] = __fmul2_rn(h[n][j], kin[n][j]);
  };
  if constexpr (MODE == SCAN_STATE || MODE == SCAN_CKPT) run(std::true_type{});
  else if constexpr (FIRST) { if (so) run(std::true_type{}); else run(std::false_type{}); }
  else run(std::false_type{});

  const bool chained = SECOND && p.chain_end;
  if (p.h_last && (!chained || chunk == p.nch - 1) && tiles.has_last(L)) {
    put_state(p.h_last + (chained ? (size_t)seq : sc) * De * NST, std::true_type{});
    if (so && q == 0 && p.sum_delta) *reinterpret_cast<float4*>(p.sum_delta + sc * De + c0) = make_float4(sdel[0].x, sdel[0].y, sdel[1].x, sdel[1].y);
  }
}

}  // namespace
}  // namespace rom
