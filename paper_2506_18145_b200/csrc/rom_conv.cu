// Un-permute + sum over the selected experts (indicator only, Section 4.2 equation for H_t), then the
// causal depthwise short convolution with SiLU (Section 3.1, U = SiLU(DWConv(H, W_conv))).
// Also the gate-weighted combine of the Out Proj rows (Section 4.2 equation for O_t).
//
// Both are HBM-bound streaming kernels: one 16-byte vector of channels per thread, consecutive
// threads on consecutive vectors, a sliding window of the previous k-1 rows kept in registers.
#include "rom_internal.cuh"

namespace rom {
namespace {

template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> { static constexpr int N = 8; };
template <> struct Vec<float> { static constexpr int N = 4; };

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
__device__ __forceinline__ void store_vec(__nv_bfloat16* p, const float (&v)[8]) {
  uint4 q;
  uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(p) = q;
}
__device__ __forceinline__ void store_vec(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// One 16-byte vector kept as loaded; converted to fp32 only when used.
template <typename T> struct RawVec;
template <> struct RawVec<__nv_bfloat16> {
  uint4 q;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { q = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void zero() { q = make_uint4(0, 0, 0, 0); }
  __device__ __forceinline__ void get(float (&v)[8]) const {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};
template <> struct RawVec<float> {
  float4 q;
  __device__ __forceinline__ void load(const float* p) { q = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void zero() { q = make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
  __device__ __forceinline__ void get(float (&v)[4]) const { v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w; }
};

// Sum over the K slots of a token of one 16-byte vector of a [rows, ld] matrix (fp32 accumulation).
template <typename T, int V, int KT>
__device__ __forceinline__ void load_sum(const T* M, int ld, const int32_t* row_of_assign, int K, size_t t, int c0, float (&h)[V]) {
  if constexpr (KT == 1) {
    load_vec(M + (size_t)__ldg(row_of_assign + t) * ld + c0, h);
  } else {
    const int kk = KT > 0 ? KT : K;
#pragma unroll
    for (int i = 0; i < V; ++i) h[i] = 0.0f;
#pragma unroll
    for (int k = 0; k < kk; ++k) {
      float v[V];
      load_vec(M + (size_t)__ldg(row_of_assign + t * kk + k) * ld + c0, v);
#pragma unroll
      for (int i = 0; i < V; ++i) h[i] += v[i];
    }
  }
}

// One thread: one 16-byte vector of channels, TCH consecutive time steps of one sequence.  All rows it
// needs (TCH + 3 of H, TCH of Z when Zs != nullptr) are loaded before anything is consumed, so the
// memory system sees TCH + 3 independent requests per thread.  KT > 0 fixes K at compile time.
constexpr int TCH = 8;

template <typename T, int KT>
__global__ void __launch_bounds__(128)
conv_silu_kernel(const T* __restrict__ XZp, const int32_t* __restrict__ row_of_assign, const T* __restrict__ w_conv,
                 const float* __restrict__ b_conv, T* __restrict__ U, T* __restrict__ Zs, int L, int De, int K, int dconv) {
  pdl_sync();
  constexpr int V = Vec<T>::N;
  const int c0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (c0 >= De) return;
  const int b = blockIdx.z;
  const int tb = blockIdx.y * TCH;
  const int ld = 2 * De;
  const size_t tok0 = (size_t)b * L;

  // rows tb-3 .. tb+TCH-1 of H.  K = 1, 2: kept as raw 16-byte words (row indices first, then all rows in
  // flight at once), converted and summed over the slots on use; other K: summed over the slots as they arrive.
  constexpr int NR = TCH + 3;
  constexpr bool RAWP = KT == 1 || KT == 2;
  constexpr int KS = RAWP ? KT : 1;
  RawVec<T> raw[RAWP ? NR : 1][KS];
  int32_t rix[RAWP ? NR : 1][KS];
  float hsum[RAWP ? 1 : NR][V];
  if constexpr (RAWP) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int t = tb - 3 + r;
#pragma unroll
      for (int k = 0; k < KS; ++k)
        rix[r][k] = (t >= 0 && t < L) ? (row_of_assign ? __ldg(row_of_assign + (tok0 + t) * KS + k) : (int32_t)(tok0 + t)) : -1;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        if (rix[r][k] >= 0) raw[r][k].load(XZp + (size_t)rix[r][k] * ld + c0);
        else raw[r][k].zero();
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int t = tb - 3 + r;
      if (t >= 0 && t < L) load_sum<T, V, KT>(XZp, ld, row_of_assign, K, tok0 + t, c0, hsum[r]);
      else {
#pragma unroll
        for (int i = 0; i < V; ++i) hsum[r][i] = 0.0f;
      }
    }
  }
  auto hrow = [&](int r, float (&out)[V]) {
    if constexpr (RAWP) {
      raw[r][0].get(out);
      if constexpr (KS == 2) {
        float v2[V];
        raw[r][1].get(v2);
#pragma unroll
        for (int i = 0; i < V; ++i) out[i] += v2[i];
      }
    } else {
#pragma unroll
      for (int i = 0; i < V; ++i) out[i] = hsum[r][i];
    }
  };
  // taps right-aligned into 4 slots: slot 3 multiplies the current token
  float w[4][V];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int src = j - (4 - dconv);
    if (src >= 0) load_vec(w_conv + (size_t)src * De + c0, w[j]);
    else {
#pragma unroll
      for (int i = 0; i < V; ++i) w[j][i] = 0.0f;
    }
  }
  float bias[V];
#pragma unroll
  for (int i = 0; i < V; ++i) bias[i] = b_conv ? b_conv[c0 + i] : 0.0f;

#pragma unroll
  for (int r = 0; r < TCH; ++r) {
    const int t = tb + r;
    if (t >= L) break;
    float u[V], h0[V], h1[V], h2[V], h3[V];
    hrow(r, h0); hrow(r + 1, h1); hrow(r + 2, h2); hrow(r + 3, h3);
#pragma unroll
    for (int i = 0; i < V; ++i) {
      float pre = bias[i];
      pre = fmaf(w[0][i], h0[i], pre);
      pre = fmaf(w[1][i], h1[i], pre);
      pre = fmaf(w[2][i], h2[i], pre);
      pre = fmaf(w[3][i], h3[i], pre);
      u[i] = sizeof(T) == 2 ? silu_fast(pre) : silu_f(pre);
    }
    store_vec(U + (tok0 + t) * De + c0, u);
  }
  if (Zs != nullptr) {
    // G = SiLU(sum over the selected experts of the Gate Proj rows) (indicator only), one row per token
    if constexpr (KS == 2) {
      // the Gate rows of the TCH tokens: same row indices as H, all requested before any is used
#pragma unroll
      for (int r = 0; r < TCH; ++r) {
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          if (rix[r + 3][k] >= 0) raw[r][k].load(XZp + De + (size_t)rix[r + 3][k] * ld + c0);
          else raw[r][k].zero();
        }
      }
#pragma unroll
      for (int r = 0; r < TCH; ++r) {
        const int t = tb + r;
        if (t >= L) break;
        float zsum[V];
        hrow(r, zsum);
#pragma unroll
        for (int i = 0; i < V; ++i) zsum[i] = sizeof(T) == 2 ? silu_fast(zsum[i]) : silu_f(zsum[i]);
        store_vec(Zs + (tok0 + t) * De + c0, zsum);
      }
    } else {
#pragma unroll
      for (int r = 0; r < TCH; ++r) {
        const int t = tb + r;
        if (t >= L) break;
        float zsum[V];
        load_sum<T, V, KT>(XZp + De, ld, row_of_assign, K, tok0 + t, c0, zsum);
#pragma unroll
        for (int i = 0; i < V; ++i) zsum[i] = sizeof(T) == 2 ? silu_fast(zsum[i]) : silu_f(zsum[i]);
        store_vec(Zs + (tok0 + t) * De + c0, zsum);
      }
    }
  }
}

// The same for many tokens and K = 1 or 2 in bf16, without the gate: a thread walks seg steps with the last four rows of H in registers
// as packed fp32 pairs, and the next four rows are in flight while four are used (their indices four rows earlier still).  HBM-bound
// (two or three 16-byte vectors per output vector); in the kernel above a thread loads 11 rows for 8 steps, computes, and ends, so that
// loads and arithmetic overlap only between blocks and every row is widened for each of its four taps.  K = 2, 64 x 1024 steps of 3072
// channels: 317 -> 239 us (5.1 TB/s), 8 x 4096 of 4096: 211 -> 163; K = 1, 16384 of 4096: 70 -> 61.  More blocks per SM (96 and 128
// registers) spill and are slower than the kernel above.
template <int KT>
__global__ void __launch_bounds__(128, KT == 1 ? 4 : 3)
conv_silu_roll_kernel(const __nv_bfloat16* __restrict__ XZp, const int32_t* __restrict__ row_of_assign, const __nv_bfloat16* __restrict__ w_conv,
                      const float* __restrict__ b_conv, __nv_bfloat16* __restrict__ U, int L, int De, int dconv, int seg) {
  typedef __nv_bfloat16 T;
  pdl_sync();
  const int c0 = (blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (c0 >= De) return;
  const int tb = blockIdx.y * seg, te = min(tb + seg, L);
  const int ld = 2 * De;
  const size_t tok0 = (size_t)blockIdx.z * L;
  const T* __restrict__ H = XZp + c0;

  auto index = [&](int t, int k) -> int32_t {      // rows outside the sequence: -1 (zeros)
    if (t < 0 || t >= te) return -1;
    return row_of_assign ? __ldg(row_of_assign + (tok0 + t) * KT + k) : (int32_t)(tok0 + t);
  };
  auto fetch = [&](RawVec<T>& r, int32_t ix) {
    if (ix >= 0) r.load(H + (size_t)ix * ld);
    else r.zero();
  };
  auto widen = [&](const RawVec<T> (&r)[KT], float2 (&h)[4]) {
    float v[8];
    r[0].get(v);
#pragma unroll
    for (int i = 0; i < 4; ++i) h[i] = make_float2(v[2 * i], v[2 * i + 1]);
    if constexpr (KT == 2) {
      r[1].get(v);
#pragma unroll
      for (int i = 0; i < 4; ++i) h[i] = __fadd2_rn(h[i], make_float2(v[2 * i], v[2 * i + 1]));
    }
  };

  RawVec<T> nxt[4][KT], halo[3][KT];
  int32_t ix[4][KT];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < KT; ++k) fetch(halo[r][k], index(tb - 3 + r, k));
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int k = 0; k < KT; ++k) { fetch(nxt[r][k], index(tb + r, k)); ix[r][k] = index(tb + 4 + r, k); }

  // taps right-aligned into 4 slots: slot 3 multiplies the current token
  float2 w[4][4], bias[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int src = j - (4 - dconv);
    float v[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (src >= 0) load_vec(w_conv + (size_t)src * De + c0, v);
#pragma unroll
    for (int i = 0; i < 4; ++i) w[j][i] = make_float2(v[2 * i], v[2 * i + 1]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) bias[i] = b_conv ? make_float2(__ldg(b_conv + c0 + 2 * i), __ldg(b_conv + c0 + 2 * i + 1)) : make_float2(0.0f, 0.0f);

  float2 h[4][4];      // row t of H in slot t & 3 (tb is a multiple of four)
#pragma unroll
  for (int r = 0; r < 3; ++r) widen(halo[r], h[r + 1]);
  T* out = U + (tok0 + tb) * De + c0;
  for (int t0 = tb; t0 < te; t0 += 4) {
    RawVec<T> cur[4][KT];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        cur[r][k] = nxt[r][k];
        fetch(nxt[r][k], ix[r][k]);
        ix[r][k] = index(t0 + 8 + r, k);
      }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      widen(cur[r], h[r]);
      float u[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float2 pre = bias[i];
#pragma unroll
        for (int j = 0; j < 4; ++j) pre = __ffma2_rn(w[j][i], h[(r + 1 + j) & 3][i], pre);
        u[2 * i] = silu_fast(pre.x);
        u[2 * i + 1] = silu_fast(pre.y);
      }
      if (t0 + r < te) store_vec(out, u);
      out += De;
    }
  }
}

// Single-token step of the short convolution: one thread = one 16-byte vector of channels of one sequence.
// conv_state [B, dconv-1, De] fp32 holds H of the previous dconv-1 tokens, oldest first; it is shifted by one and
// the new H appended.  Taps are applied in the same order as in conv_silu_kernel (right-aligned into 4 slots).
template <typename T>
__global__ void __launch_bounds__(128)
conv_step_kernel(const T* __restrict__ XZp, const int32_t* __restrict__ row_of_assign, const T* __restrict__ w_conv,
                 const float* __restrict__ b_conv, float* __restrict__ conv_state, T* __restrict__ U, T* __restrict__ Zs,
                 int De, int K, int dconv) {
  pdl_sync();
  constexpr int V = Vec<T>::N;
  const int c0 = (blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (c0 >= De) return;
  const size_t b = blockIdx.y;
  const int ld = 2 * De;
  float win[4][V];                       // slot 3 = the current token, slots 4-dconv .. 2 = the state rows
  if (row_of_assign) load_sum<T, V, 0>(XZp, ld, row_of_assign, K, b, c0, win[3]);
  else load_vec(XZp + b * ld + c0, win[3]);
  float* st = conv_state + b * (size_t)(dconv - 1) * De + c0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int src = j - (4 - dconv);     // state row feeding slot j
#pragma unroll
    for (int i = 0; i < V; ++i) win[j][i] = src >= 0 ? st[(size_t)src * De + i] : 0.0f;
  }
  float u[V];
#pragma unroll
  for (int i = 0; i < V; ++i) u[i] = b_conv ? b_conv[c0 + i] : 0.0f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int src = j - (4 - dconv);
    if (src < 0) continue;
    float w[V];
    load_vec(w_conv + (size_t)src * De + c0, w);
#pragma unroll
    for (int i = 0; i < V; ++i) u[i] = fmaf(w[i], win[j][i], u[i]);
  }
#pragma unroll
  for (int i = 0; i < V; ++i) u[i] = sizeof(T) == 2 ? silu_fast(u[i]) : silu_f(u[i]);
  store_vec(U + b * De + c0, u);
  // new state: drop the oldest row, append the current H
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const int dst = j - (4 - dconv);
    if (dst < 0) continue;
#pragma unroll
    for (int i = 0; i < V; ++i) st[(size_t)dst * De + i] = win[j + 1][i];
  }
  if (Zs != nullptr) {
    float zsum[V];
    load_sum<T, V, 0>(XZp + De, ld, row_of_assign, K, b, c0, zsum);
#pragma unroll
    for (int i = 0; i < V; ++i) zsum[i] = sizeof(T) == 2 ? silu_fast(zsum[i]) : silu_f(zsum[i]);
    store_vec(Zs + b * De + c0, zsum);
  }
}

// out[t, :] = sum_k gates[t,k] * Op[row_of_assign[t*K+k], :], slots added in ascending k.
template <typename T>
__global__ void __launch_bounds__(256)
combine_kernel(const T* __restrict__ Op, const int32_t* __restrict__ row_of_assign, const float* __restrict__ gates,
               T* __restrict__ out, int Dm, int K, long long total_vec) {
  pdl_sync();
  constexpr int V = Vec<T>::N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total_vec) return;
  const int vpr = Dm / V;
  const long long t = i / vpr;
  const int c0 = (int)(i % vpr) * V;
  float acc[V];
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0.0f;
  for (int k = 0; k < K; ++k) {
    const int row = __ldg(row_of_assign + t * K + k);
    const float g = __ldg(gates + t * K + k);
    float v[V];
    load_vec(Op + (size_t)row * Dm + c0, v);
#pragma unroll
    for (int j = 0; j < V; ++j) acc[j] = fmaf(g, v[j], acc[j]);
  }
  store_vec(out + t * Dm + c0, acc);
}

// The same in bf16 for top-2: a warp per token, four 16-byte pieces of both rows in flight per lane.  HBM-bound (three rows a token); with
// one piece to a thread, behind its row indices, 32768 tokens of 2048 channels took 76 us, here 53.5; 65536 of 1536 113 -> 83; 3051 8.2 -> 6.6.
__global__ void __launch_bounds__(128)
combine_pair_kernel(const __nv_bfloat16* __restrict__ Op, const int32_t* __restrict__ row_of_assign, const float* __restrict__ gates,
                    __nv_bfloat16* __restrict__ out, int Dm, long long Tn) {
  pdl_sync();
  typedef V16<__nv_bfloat16> Vec8;
  constexpr int G = 4;
  const int lane = threadIdx.x & 31, nv = Dm / 8;
  const long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (t >= Tn) return;
  const int2 rows = __ldg(reinterpret_cast<const int2*>(row_of_assign) + t);
  const float g0 = __ldg(gates + 2 * t), g1 = __ldg(gates + 2 * t + 1);
  const __nv_bfloat16 *p0 = Op + (size_t)rows.x * Dm, *p1 = Op + (size_t)rows.y * Dm;
  for (int v0 = lane; v0 < nv; v0 += 32 * G) {
    Vec8 a[G], b[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const int v = min(v0 + 32 * i, nv - 1);      // (past the end: loaded and not used)
      a[i].load(p0 + (size_t)v * 8);
      b[i].load(p1 + (size_t)v * 8);
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      float x[8], y[8];
      a[i].get(x); b[i].get(y);
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = fmaf(g1, y[j], fmaf(g0, x[j], 0.0f));
      if (v0 + 32 * i < nv) Vec8::store(out + t * Dm + (size_t)(v0 + 32 * i) * 8, x);
    }
  }
}

// Per-expert x Proj / dt Proj: one thread per float4 of a token's [Delta | B | C] row; the K slots are added in
// ascending order, then (Delta only) the shared bias and the softplus.
template <typename T>
__global__ void __launch_bounds__(256)
small_combine_kernel(const float* __restrict__ Bp, const float* __restrict__ Cp, const float* __restrict__ Dpre,
                     const int32_t* __restrict__ row_of_assign, const float* __restrict__ b_dt, float* __restrict__ Bm,
                     float* __restrict__ Cm, T* __restrict__ Delta, int De, int N, int K, long long total_vec) {
  pdl_sync();
  constexpr bool PRECISE = sizeof(T) == 4;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total_vec) return;
  const int vpr = (De + 2 * N) / 4;
  const long long t = i / vpr;
  const int c0 = (int)(i % vpr) * 4;
  const float* src; float* dst = nullptr; int ld, col;
  if (c0 < De) { src = Dpre; ld = De; col = c0; }
  else if (c0 < De + N) { src = Bp; dst = Bm; ld = N; col = c0 - De; }
  else { src = Cp; dst = Cm; ld = N; col = c0 - De - N; }
  float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int k = 0; k < K; ++k) {
    const int row = __ldg(row_of_assign + t * K + k);
    const float4 v = __ldg(reinterpret_cast<const float4*>(src + (size_t)row * ld + col));
    acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
  }
  if (c0 < De) {
    const float4 b = b_dt ? __ldg(reinterpret_cast<const float4*>(b_dt + col)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (PRECISE) acc = make_float4(softplus_f(acc.x + b.x), softplus_f(acc.y + b.y), softplus_f(acc.z + b.z), softplus_f(acc.w + b.w));
    else acc = make_float4(softplus_fast(acc.x + b.x), softplus_fast(acc.y + b.y), softplus_fast(acc.z + b.z), softplus_fast(acc.w + b.w));
    T* d = Delta + (size_t)t * ld + col;
    d[0] = from_f32<T>(acc.x); d[1] = from_f32<T>(acc.y); d[2] = from_f32<T>(acc.z); d[3] = from_f32<T>(acc.w);
    return;
  }
  *reinterpret_cast<float4*>(dst + (size_t)t * ld + col) = acc;
}

}  // namespace

template <typename T>
cudaError_t launch_conv_t(const rom_config& c, const void* XZp, const int32_t* row_of_assign, const void* w_conv,
                          const float* b_conv, void* U, void* Zs, cudaStream_t st) {
  constexpr int V = Vec<T>::N;
  const int threads = 128;
  dim3 grid((c.d_inner / V + threads - 1) / threads, (c.L + TCH - 1) / TCH, c.B);
  auto args = [&](auto kern) {
    launch_k(kern, grid, threads, 0, st, (const T*)XZp, row_of_assign, (const T*)w_conv, b_conv, (T*)U, (T*)Zs, c.L, c.d_inner, c.K, c.d_conv);
  };
  if constexpr (sizeof(T) == 2) {
    // 64 steps to a thread once that leaves three waves of four blocks per SM, else 32 (4 x 2048 steps of 2048 channels: 20 us, 22.6
    // with 64); the short walk of the kernel above where even those do not give every SM a block
    const long long cols = (long long)grid.x * c.B;
    const int seg = cols * ((c.L + 63) / 64) >= 148 * 12 ? 64 : 32;
    const dim3 g2(grid.x, (c.L + seg - 1) / seg, c.B);
    if (c.K <= 2 && Zs == nullptr && cols * g2.y >= 148) {
      launch_k(c.K == 1 ? conv_silu_roll_kernel<1> : conv_silu_roll_kernel<2>, g2, threads, 0, st, (const T*)XZp, row_of_assign,
               (const T*)w_conv, b_conv, (T*)U, c.L, c.d_inner, c.d_conv, seg);
      count_launch();
      return cudaGetLastError();
    }
  }
  if (c.K == 1) args(conv_silu_kernel<T, 1>);
  else if (c.K == 2) args(conv_silu_kernel<T, 2>);
  else args(conv_silu_kernel<T, 0>);
  count_launch();
  return cudaGetLastError();
}

// Zs: [T, d_inner] sum over the K slots of the Gate Proj rows, or nullptr (not produced).
cudaError_t launch_conv(const rom_config& c, const void* XZp, const int32_t* row_of_assign, const void* w_conv,
                        const float* b_conv, void* U, void* Zs, cudaStream_t st) {
  if (c.B > 65535 || (c.L + TCH - 1) / TCH > 65535) return cudaErrorInvalidConfiguration;
  return c.dtype == ROM_BF16 ? launch_conv_t<__nv_bfloat16>(c, XZp, row_of_assign, w_conv, b_conv, U, Zs, st)
                             : launch_conv_t<float>(c, XZp, row_of_assign, w_conv, b_conv, U, Zs, st);
}

cudaError_t launch_combine(const rom_config& c, const void* Op, const int32_t* row_of_assign, const float* gates,
                           void* out, cudaStream_t st) {
  const bool bf = c.dtype == ROM_BF16;
  const int V = bf ? 8 : 4;
  const long long total = (long long)c.B * c.L * (c.d_model / V);
  const int threads = 256;
  const unsigned blocks = (unsigned)((total + threads - 1) / threads);
  if (bf && c.K == 2)
    launch_k(combine_pair_kernel, (unsigned)(((long long)c.B * c.L + 3) / 4), 128, 0, st, (const __nv_bfloat16*)Op, row_of_assign, gates, (__nv_bfloat16*)out,
             c.d_model, (long long)c.B * c.L);
  else if (bf)
    launch_k(combine_kernel<__nv_bfloat16>, blocks, threads, 0, st, (const __nv_bfloat16*)Op, row_of_assign, gates, (__nv_bfloat16*)out,
                                                             c.d_model, c.K, total);
  else
    launch_k(combine_kernel<float>, blocks, threads, 0, st, (const float*)Op, row_of_assign, gates, (float*)out, c.d_model, c.K, total);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_small_combine(const rom_config& c, const float* Bp, const float* Cp, const float* Dpre,
                                 const int32_t* row_of_assign, const float* b_dt, float* Bm, float* Cm, void* Delta,
                                 cudaStream_t st) {
  const long long total = (long long)c.B * c.L * ((c.d_inner + 2 * c.d_state) / 4);
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if (c.dtype == ROM_F32)
    launch_k(small_combine_kernel<float>, blocks, 256, 0, st, Bp, Cp, Dpre, row_of_assign, b_dt, Bm, Cm, (float*)Delta, c.d_inner, c.d_state, c.K, total);
  else
    launch_k(small_combine_kernel<__nv_bfloat16>, blocks, 256, 0, st, Bp, Cp, Dpre, row_of_assign, b_dt, Bm, Cm, (__nv_bfloat16*)Delta, c.d_inner, c.d_state, c.K, total);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_conv_step(const rom_config& c, const void* XZp, const int32_t* row_of_assign, const void* w_conv,
                             const float* b_conv, float* conv_state, void* U, void* Zs, cudaStream_t st) {
  const bool bf = c.dtype == ROM_BF16;
  const int V = bf ? 8 : 4;
  const int threads = 128;
  dim3 grid((c.d_inner / V + threads - 1) / threads, c.B);
  if (bf)
    launch_k(conv_step_kernel<__nv_bfloat16>, grid, threads, 0, st, (const __nv_bfloat16*)XZp, row_of_assign, (const __nv_bfloat16*)w_conv, b_conv,
                                                            conv_state, (__nv_bfloat16*)U, (__nv_bfloat16*)Zs, c.d_inner, c.K, c.d_conv);
  else
    launch_k(conv_step_kernel<float>, grid, threads, 0, st, (const float*)XZp, row_of_assign, (const float*)w_conv, b_conv, conv_state,
                                                     (float*)U, (float*)Zs, c.d_inner, c.K, c.d_conv);
  count_launch();
  return cudaGetLastError();
}

}  // namespace rom
