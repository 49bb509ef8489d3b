// Kernels of the layer's backward pass other than the scan's (rom_scan_bwd.cu) and, on the tensor path, the projections' data and
// weight gradients (rom_gemm_tc.cu, on weights and activations as stored): the sum over a token's slots, the reverse of the gate-weighted
// combine, conv / router reverses; for the plain-FMA path transposed weights (its data gradients are the forward's grouped GEMMs on
// them) and the weight gradients (sums over tokens).
//
// Section 5.1 trains the layer end to end and Appendix A.3 trains the router through the gate values; the equations
// differentiated are those of Sections 3.1 and 4.2 (forward: rom_api.cu).  All
// sums are fp32, weight gradients leave in fp32, and sums that cross thread blocks use floating-point atomics (their last bits
// vary from run to run).
#include <type_traits>

#include "rom_internal.cuh"

namespace rom {
namespace {

template <typename T> struct VecN { static constexpr int N = 16 / sizeof(T); };

__device__ __forceinline__ void ldv(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 q = *reinterpret_cast<const uint4*>(p);
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
}
__device__ __forceinline__ void ldv(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void stv(__nv_bfloat16* p, const float (&v)[8]) {
  uint4 q;
  uint32_t* w = reinterpret_cast<uint32_t*>(&q);
#pragma unroll
  for (int i = 0; i < 4; ++i) { const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]); w[i] = *reinterpret_cast<const uint32_t*>(&h); }
  *reinterpret_cast<uint4*>(p) = q;
}
__device__ __forceinline__ void stv(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }

// out[b][c][r] = in[b][r][c]
template <typename T>
__global__ void __launch_bounds__(256)
transpose_kernel(const T* __restrict__ in, T* __restrict__ out, int R, int C) {
  pdl_sync();
  __shared__ T tile[32][33];
  const size_t base = (size_t)blockIdx.z * R * C;
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[i][threadIdx.x] = in[base + (size_t)r * C + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < C) out[base + (size_t)c * R + r] = tile[threadIdx.x][i];
  }
}

__global__ void __launch_bounds__(256)
zero_kernel(const ZeroList z) {
  pdl_sync();
  float* p = z.p[blockIdx.y];
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < z.n[blockIdx.y]; i += (long long)gridDim.x * 256) p[i] = 0.0f;
}

// dst[t, :] = sum_k src[row_of_assign[t*K + k], :]  (ascending k, fp32 accumulation), rows `width` wide
template <typename T>
__global__ void __launch_bounds__(256)
slot_sum_kernel(const T* __restrict__ src, const int32_t* __restrict__ row_of_assign, T* __restrict__ dst, int width, int K, long long total_vec) {
  pdl_sync();
  constexpr int V = VecN<T>::N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total_vec) return;
  const int vpr = width / V;
  const long long t = i / vpr;
  const int c0 = (int)(i % vpr) * V;
  float acc[V];
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0.0f;
  for (int k = 0; k < K; ++k) {
    float v[V];
    ldv(src + (size_t)row_of_assign[t * K + k] * width + c0, v);
#pragma unroll
    for (int j = 0; j < V; ++j) acc[j] += v[j];
  }
  stv(dst + t * width + c0, acc);
}

// Reverse of O_t = sum_k gate_k * (Yg_t W_out,k): with back_k = dO_t W_out,k (rows of dYgu, expert order),
//   dYg_t = sum_k gate_k back_k,  dgate_k = <back_k, Yg_t>;  and the operand of the Out Proj weight gradient, gate_k Yg_t: written
// over the token's rows of Ygp, or (rowscale != nullptr) left as it is with the gate of every padded row in rowscale.
template <typename T>
__global__ void __launch_bounds__(128)
combine_bwd_kernel(const T* __restrict__ dYgu, T* Ygp, const int32_t* __restrict__ row_of_assign,
                   const float* __restrict__ gates, T* __restrict__ dYg, float* __restrict__ dgate, float* __restrict__ rowscale,
                   int De, int K) {
  pdl_sync();
  __shared__ float red[kMaxK][4];
  const size_t t = blockIdx.x;
  int rows[kMaxK]; float g[kMaxK], part[kMaxK];
  for (int k = 0; k < K; ++k) { rows[k] = row_of_assign[t * K + k]; g[k] = gates[t * K + k]; part[k] = 0.0f; }
  const T* yg = Ygp + (size_t)rows[0] * De;          // the K rows of a token hold the same gated scan output
  constexpr int V = V16<T>::N;
  {
    for (int i = threadIdx.x; i < De / V; i += blockDim.x) {
      V16<T> q;
      float y[V], acc[V];
      ldv(yg + (size_t)i * V, y);
#pragma unroll
      for (int j = 0; j < V; ++j) acc[j] = 0.0f;
      for (int k = 0; k < K; ++k) {
        float bv[V];
        q.load(dYgu + (size_t)rows[k] * De + (size_t)i * V); q.get(bv);
#pragma unroll
        for (int j = 0; j < V; ++j) { acc[j] = fmaf(g[k], bv[j], acc[j]); part[k] = fmaf(bv[j], y[j], part[k]); }
      }
      V16<T>::store(dYg + t * De + (size_t)i * V, acc);
      if (!rowscale) {
        for (int k = 0; k < K; ++k) {
          float sv[V];
#pragma unroll
          for (int j = 0; j < V; ++j) sv[j] = g[k] * y[j];
          V16<T>::store(Ygp + (size_t)rows[k] * De + (size_t)i * V, sv);
        }
      }
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < K; ++k) {
    float v = part[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[k][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < K) {
    const int k = threadIdx.x;
    dgate[t * K + k] = (red[k][0] + red[k][1]) + (red[k][2] + red[k][3]);
    if (rowscale) rowscale[rows[k]] = g[k];
  }
}

// The same in bf16 for top-1 and top-2, the scaled rows written: a warp per token, four 16-byte pieces of every row in flight and no
// block barrier.  HBM-bound (2 K + 2 rows a token); with the experts of a token in a loop of unknown length and one block per token,
// 16384 tokens of 4096 channels took 123 us, here 90 (82 at the copy bandwidth); 4113 of 2048 at top-2 22 -> 16.
template <int KT>
__global__ void __launch_bounds__(128)
combine_bwd_warp_kernel(const __nv_bfloat16* __restrict__ dYgu, __nv_bfloat16* Ygp, const int32_t* __restrict__ row_of_assign,
                        const float* __restrict__ gates, __nv_bfloat16* __restrict__ dYg, float* __restrict__ dgate, int De, long long Tn) {
  pdl_sync();
  typedef V16<__nv_bfloat16> Vec;
  const int lane = threadIdx.x & 31;
  const long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5);
  if (t >= Tn) return;
  size_t rows[KT];
  float g[KT], part[KT];
#pragma unroll
  for (int k = 0; k < KT; ++k) { rows[k] = (size_t)__ldg(row_of_assign + t * KT + k); g[k] = __ldg(gates + t * KT + k); part[k] = 0.0f; }
  const int nv = De / 8;
  constexpr int G = 4;
  for (int v0 = lane; v0 < nv; v0 += 32 * G) {
    Vec y[G], b[G][KT];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const int v = min(v0 + 32 * i, nv - 1);      // (past the end: loaded and not used)
      y[i].q = *reinterpret_cast<const uint4*>(Ygp + rows[0] * De + (size_t)v * 8);      // the K rows of a token hold the same gated scan output
#pragma unroll
      for (int k = 0; k < KT; ++k) b[i][k].load(dYgu + rows[k] * De + (size_t)v * 8);
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      if (v0 + 32 * i >= nv) break;
      float yv[8], acc[8];
      y[i].get(yv);
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        float bv[8];
        b[i][k].get(bv);
#pragma unroll
        for (int j = 0; j < 8; ++j) { acc[j] = fmaf(g[k], bv[j], k == 0 ? 0.0f : acc[j]); part[k] = fmaf(bv[j], yv[j], part[k]); }
      }
      Vec::store(dYg + t * De + (size_t)(v0 + 32 * i) * 8, acc);
#pragma unroll
      for (int k = 0; k < KT; ++k) {
        float sv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) sv[j] = g[k] * yv[j];
        Vec::store(Ygp + rows[k] * De + (size_t)(v0 + 32 * i) * 8, sv);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < KT; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part[k] += __shfl_xor_sync(0xffffffffu, part[k], o);
    if (lane == 0) dgate[t * KT + k] = part[k];
  }
}

// dxdbl[t, R + j] = dB[t, j] (j < N) or dC[t, j - N]: the B | C part of the gradient of (delta, B, C) = U W_x
template <typename T>
__global__ void __launch_bounds__(256)
pack_bc_kernel(const float* __restrict__ dBm, const float* __restrict__ dCm, T* __restrict__ dxdbl, long long Tn, int R, int N) {
  pdl_sync();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Tn * 2 * N) return;
  const long long t = i / (2 * N);
  const int j = (int)(i % (2 * N));
  dxdbl[t * (R + 2 * N) + R + j] = from_f32<T>(j < N ? dBm[t * N + j] : dCm[t * N + (j - N)]);
}

// Reverse of U = SiLU(b + sum_j w[j] H[t - (k-1-j)]):
//   g_t = dU_t SiLU'(pre_t);  dH_tau = sum_j w[j] g_{tau + (k-1-j)};  dw[j] = sum_t g_t H[t - (k-1-j)];  db = sum_t g_t.
// H is the left half of HZ ([T, 2 De]); dU = dU1 + dU2 (scan part + x Proj part); dH of token t goes to the left half of the K
// rows of dHZ that row_of_assign names (the operand of the grouped Conv/Gate gradients).
// A thread walks `seg` steps of four channels (two packed pairs) with a window of the last k-1 rows of H and of the k-1 rows of
// dH still being collected; three rows of four steps are in flight while four are used.  Bound by HBM (24 bytes per token and
// four channels at bf16) at one walk per element: one channel per thread with two-byte loads took 0.96 ms at 16384 x 4096
// channels (0.56 TB/s), bound by its load and exponential instructions.  bf16: four blocks to an SM by register limit (158 otherwise), so
// that 516 blocks are one wave: 4113 tokens of 2048 channels 30.9 -> 24.7 us, 16384 of 4096 135.6 -> 133.8.  There issue slots were 70 %
// busy: groups that are all the thread's own carry no tests, 133.8 -> 121.7 us, 24.7 -> 23.5.
template <typename T> struct Raw4;
template <> struct Raw4<__nv_bfloat16> {
  uint2 q;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { q = __ldg(reinterpret_cast<const uint2*>(p)); }
  __device__ __forceinline__ void zero() { q = make_uint2(0, 0); }
  __device__ __forceinline__ void get(float2 (&v)[2]) const {
    v[0] = make_float2(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u));
    v[1] = make_float2(__uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, const float2 (&v)[2]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0].x, v[0].y), b = __floats2bfloat162_rn(v[1].x, v[1].y);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  }
};
template <> struct Raw4<float> {
  float4 q;
  __device__ __forceinline__ void load(const float* p) { q = __ldg(reinterpret_cast<const float4*>(p)); }
  __device__ __forceinline__ void zero() { q = make_float4(0.0f, 0.0f, 0.0f, 0.0f); }
  __device__ __forceinline__ void get(float2 (&v)[2]) const { v[0] = make_float2(q.x, q.y); v[1] = make_float2(q.z, q.w); }
  static __device__ __forceinline__ void store(float* p, const float2 (&v)[2]) { *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y); }
};
// SiLU'(v) = s (1 + v (1 - s)), s = sigmoid(v)
template <bool PRECISE> __device__ __forceinline__ float dsilu(float v) {
  const float s = PRECISE ? 1.0f / (1.0f + expf(-v)) : rcp_ftz(1.0f + ex2_ftz(-1.4426950408889634f * v));
  return s * fmaf(v, 1.0f - s, 1.0f);
}

template <typename T, int KC>
__global__ void __launch_bounds__(128, sizeof(T) == 2 ? 4 : 2)
conv_bwd_kernel(const T* __restrict__ HZ, const T* __restrict__ w_conv, const float* __restrict__ b_conv, const T* __restrict__ dU1,
                const T* __restrict__ dU2, T* __restrict__ dHZ, const int32_t* __restrict__ row_of_assign, float* __restrict__ dw,
                float* __restrict__ db, int L, int De, int K, int seg) {
  pdl_sync();
  constexpr bool PRECISE = sizeof(T) == 4;
  constexpr int G = 4;
  const int c = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (c >= De) return;
  const size_t tok0 = (size_t)blockIdx.z * L;
  const int t0 = blockIdx.y * seg, t1 = min(t0 + seg, L), t_end = min(t1 + KC - 1, L);
  const int ld = 2 * De;
  float2 w[KC][2], dwl[KC][2], hw[KC - 1][2], dacc[KC - 1][2], bias[2], dbl[2];
  const float2 zero2 = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int j = 0; j < KC; ++j) {
    Raw4<T> r;
    r.load(w_conv + (size_t)j * De + c); r.get(w[j]);
    dwl[j][0] = zero2; dwl[j][1] = zero2;
  }
  bias[0] = b_conv ? make_float2(b_conv[c], b_conv[c + 1]) : zero2;
  bias[1] = b_conv ? make_float2(b_conv[c + 2], b_conv[c + 3]) : zero2;
  dbl[0] = zero2; dbl[1] = zero2;
#pragma unroll
  for (int j = 0; j < KC - 1; ++j) {      // hw[j] = H[t - (KC-1) + j] before step t
    Raw4<T> r;
    const int t = t0 - (KC - 1) + j;
    if (t >= 0) r.load(HZ + (tok0 + t) * ld + c); else r.zero();
    r.get(hw[j]);
    dacc[j][0] = zero2; dacc[j][1] = zero2;
  }
  auto put = [&](int tau, const float2 (&v)[2]) {
    for (int k = 0; k < K; ++k) Raw4<T>::store(dHZ + (size_t)__ldg(row_of_assign + (tok0 + tau) * K + k) * ld + c, v);
  };
  Raw4<T> rh[G], r1[G], r2[G];
  auto fetch = [&](int tg) {
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const size_t t = tok0 + min(tg + i, t_end - 1);
      rh[i].load(HZ + t * ld + c); r1[i].load(dU1 + t * De + c); r2[i].load(dU2 + t * De + c);
    }
  };
  auto group = [&](int tg, auto inner) {      // inner: every step is this thread's own
    constexpr bool INNER = decltype(inner)::value;
    Raw4<T> ch[G], c1[G], c2[G];
#pragma unroll
    for (int i = 0; i < G; ++i) { ch[i] = rh[i]; c1[i] = r1[i]; c2[i] = r2[i]; }
    if (tg + G < t_end) fetch(tg + G);
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const int t = tg + i;
      if (!INNER && t >= t_end) break;
      float2 hz[2], d1[2], d2[2], g[2], o[2];
      ch[i].get(hz); c1[i].get(d1); c2[i].get(d2);
      const bool own = INNER || t < t1;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float2 pre = __ffma2_rn(w[KC - 1][v], hz[v], bias[v]);
#pragma unroll
        for (int j = 0; j < KC - 1; ++j) pre = __ffma2_rn(w[j][v], hw[j][v], pre);
        g[v] = __fmul2_rn(__fadd2_rn(d1[v], d2[v]), make_float2(dsilu<PRECISE>(pre.x), dsilu<PRECISE>(pre.y)));
        if (own) {
          dbl[v] = __fadd2_rn(dbl[v], g[v]);
#pragma unroll
          for (int j = 0; j < KC - 1; ++j) dwl[j][v] = __ffma2_rn(g[v], hw[j][v], dwl[j][v]);
          dwl[KC - 1][v] = __ffma2_rn(g[v], hz[v], dwl[KC - 1][v]);
        }
        // dacc[i] collects dH of step t - (KC-1) + i; with this step's term, index 0 is complete
        o[v] = __ffma2_rn(w[0][v], g[v], dacc[0][v]);
#pragma unroll
        for (int j = 0; j + 1 < KC - 1; ++j) dacc[j][v] = __ffma2_rn(w[j + 1][v], g[v], dacc[j + 1][v]);
        dacc[KC - 2][v] = __fmul2_rn(w[KC - 1][v], g[v]);
#pragma unroll
        for (int j = 0; j + 1 < KC - 1; ++j) hw[j][v] = hw[j + 1][v];
        hw[KC - 2][v] = hz[v];
      }
      if (t - (KC - 1) >= t0) put(t - (KC - 1), o);
    }
  };
  fetch(t0);
  int tg = t0;
  for (; tg + G <= t1; tg += G) group(tg, std::true_type{});
  for (; tg < t_end; tg += G) group(tg, std::false_type{});
  // steps whose later neighbours do not exist (end of the sequence): what has been collected is final
#pragma unroll
  for (int i = 0; i < KC - 1; ++i) {
    const int tau = t_end - (KC - 1) + i;
    if (tau >= t0 && tau < t1) put(tau, dacc[i]);
  }
#pragma unroll
  for (int j = 0; j < KC; ++j) atomicAdd(reinterpret_cast<float4*>(dw + (size_t)j * De + c), make_float4(dwl[j][0].x, dwl[j][0].y, dwl[j][1].x, dwl[j][1].y));
  atomicAdd(reinterpret_cast<float4*>(db + c), make_float4(dbl[0].x, dbl[0].y, dbl[1].x, dbl[1].y));
}

// Reverse of the gate values with the selected set held fixed, one thread per token: with P = Softmax(X W_r) as the router left
// it, dP[idx_k] = dgate_k (gate_mode 0) or (dgate_k - sum_j dgate_j gate_j) / sum_j P[idx_j] (gate_mode 1),
// dlogit = P (dP - sum_e dP_e P_e).  Writes dlogit [T, E] (fp32) and adds db_r.
__global__ void __launch_bounds__(128)
router_bwd_kernel(const float* __restrict__ P, const int32_t* __restrict__ idx, const float* __restrict__ gates, const float* __restrict__ dgate,
                  float* __restrict__ dlogit, float* __restrict__ db_r, long long Tn, int E, int K, int gate_mode) {
  pdl_sync();
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = t < Tn;
  const float* p = P + (in ? t : 0) * E;
  int sel[kMaxK]; float ds[kMaxK];
  float S = 1.0f, dot = 0.0f, mean = 0.0f;
  for (int k = 0; k < K; ++k) { sel[k] = in ? idx[t * K + k] : 0; ds[k] = in ? dgate[t * K + k] : 0.0f; }
  if (gate_mode == 1) {
    S = 0.0f;
    for (int k = 0; k < K; ++k) { S += p[sel[k]]; dot = fmaf(ds[k], in ? gates[t * K + k] : 0.0f, dot); }
    for (int k = 0; k < K; ++k) ds[k] = (ds[k] - dot) / S;
  }
  for (int k = 0; k < K; ++k) mean = fmaf(ds[k], p[sel[k]], mean);
  for (int e = 0; e < E; ++e) {
    float dP = 0.0f;
    for (int k = 0; k < K; ++k) dP += sel[k] == e ? ds[k] : 0.0f;
    float dl = in ? p[e] * (dP - mean) : 0.0f;
    if (in) dlogit[t * E + e] = dl;
    if (db_r) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
      if ((threadIdx.x & 31) == 0) atomicAdd(db_r + e, dl);
    }
  }
}

// dx[t, :] = sum_k dxp[row(t,k), :] + sum_e dlogit[t, e] W_r[e, :]
template <typename T>
__global__ void __launch_bounds__(256)
dx_kernel(const T* __restrict__ dxp, const int32_t* __restrict__ row_of_assign, const float* __restrict__ dlogit, const T* __restrict__ W_r,
          T* __restrict__ dx, int Dm, int E, int K, long long total_vec) {
  pdl_sync();
  constexpr int V = VecN<T>::N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total_vec) return;
  const int vpr = Dm / V;
  const long long t = i / vpr;
  const int c0 = (int)(i % vpr) * V;
  float acc[V];
#pragma unroll
  for (int j = 0; j < V; ++j) acc[j] = 0.0f;
  for (int k = 0; k < K; ++k) {
    float v[V];
    ldv(dxp + (size_t)row_of_assign[t * K + k] * Dm + c0, v);
#pragma unroll
    for (int j = 0; j < V; ++j) acc[j] += v[j];
  }
  for (int e = 0; e < E; ++e) {
    const float dl = dlogit[t * E + e];
    float v[V];
    ldv(W_r + (size_t)e * Dm + c0, v);
#pragma unroll
    for (int j = 0; j < V; ++j) acc[j] = fmaf(dl, v[j], acc[j]);
  }
  stv(dx + t * Dm + c0, acc);
}

// The same in bf16 for 4, 8 or 16 experts at top-1 and top-2: a thread keeps its 8 columns of W_r and walks seg tokens, four in flight
// (their row indices four tokens earlier still).  Above, every vector of dx reads and widens all E of W_r, about 170 instructions: 16384
// tokens of 2048 channels with 8 experts 58 us, here 38 (20 at the copy bandwidth), 4113 of 1024 at top-2 11.6 -> 8.9.  Eight tokens to a
// thread: with 16 and 32 the former takes 36 and 35, the latter 11.6 and 19.9 (too few threads).  Other counts in the next larger form, with
// zero rows of W_r, gain nothing (whole backward of 8192 tokens of 768 channels, 6 experts: 831.5 us above, 831.2 padded; top-2 979 / 987; 12
// experts 863 / 862): their dlogit rows are no longer 16-byte pieces.
template <int NE, int KT>
__global__ void __launch_bounds__(128, NE <= 8 ? 4 : 2)
dx_walk_kernel(const __nv_bfloat16* __restrict__ dxp, const int32_t* __restrict__ row_of_assign, const float* __restrict__ dlogit,
               const __nv_bfloat16* __restrict__ W_r, __nv_bfloat16* __restrict__ dx, int Dm, int seg, long long Tn) {
  pdl_sync();
  typedef V16<__nv_bfloat16> Vec;
  constexpr int G = 4;
  constexpr bool WIDE = NE <= 8;       // W_r widened once; 16 experts stay as stored
  const int nv = Dm / 8;
  const long long id = (long long)blockIdx.x * 128 + threadIdx.x;
  const int c0 = (int)(id % nv) * 8;
  const long long tb = id / nv * seg, te = min(tb + seg, Tn);
  if (tb >= Tn) return;
  Vec wr[NE];
  float2 w[WIDE ? NE : 1][4];
#pragma unroll
  for (int e = 0; e < NE; ++e) wr[e].load(W_r + (size_t)e * Dm + c0);
  auto pairs = [](const Vec& q, float2 (&o)[4]) {
    float v[8];
    q.get(v);
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = make_float2(v[2 * i], v[2 * i + 1]);
  };
  if constexpr (WIDE) {
#pragma unroll
    for (int e = 0; e < NE; ++e) pairs(wr[e], w[e]);
  }
  int32_t ix[G][KT];
  Vec nxt[G][KT];
  auto index = [&](long long t0) {
#pragma unroll
    for (int i = 0; i < G; ++i)
#pragma unroll
      for (int k = 0; k < KT; ++k) ix[i][k] = __ldg(row_of_assign + min(t0 + i, te - 1) * KT + k);      // (past the end: the last token again)
  };
  auto fetch = [&]() {
#pragma unroll
    for (int i = 0; i < G; ++i)
#pragma unroll
      for (int k = 0; k < KT; ++k) nxt[i][k].load(dxp + (size_t)ix[i][k] * Dm + c0);
  };
  index(tb);
  fetch();
  index(tb + G);
  for (long long t0 = tb; t0 < te; t0 += G) {
    Vec cur[G][KT];
#pragma unroll
    for (int i = 0; i < G; ++i)
#pragma unroll
      for (int k = 0; k < KT; ++k) cur[i][k] = nxt[i][k];
    fetch();
    index(t0 + 2 * G);
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const long long t = min(t0 + i, te - 1);
      float4 dl[NE / 4];
#pragma unroll
      for (int q = 0; q < NE / 4; ++q) dl[q] = __ldg(reinterpret_cast<const float4*>(dlogit + t * NE) + q);
      float2 acc[4], v[4];
      pairs(cur[i][0], acc);
      if constexpr (KT == 2) {
        pairs(cur[i][1], v);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = __fadd2_rn(acc[j], v[j]);
      }
#pragma unroll
      for (int e = 0; e < NE; ++e) {
        const float f = (e & 3) == 0 ? dl[e / 4].x : (e & 3) == 1 ? dl[e / 4].y : (e & 3) == 2 ? dl[e / 4].z : dl[e / 4].w;
        if constexpr (!WIDE) pairs(wr[e], v);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] = __ffma2_rn(make_float2(f, f), WIDE ? w[WIDE ? e : 0][j] : v[j], acc[j]);
      }
      if (t0 + i < te) {
        const float o[8] = {acc[0].x, acc[0].y, acc[1].x, acc[1].y, acc[2].x, acc[2].y, acc[3].x, acc[3].y};
        Vec::store(dx + t * Dm + c0, o);
      }
    }
  }
}

// dW_r[e, d] = sum_t dlogit[t, e] x[t, d]: a thread owns four columns of x and eight experts over a slab of tokens (x is read
// once per eight experts; the slab's dlogit values sit in shared memory), one 16-byte atomic per slab, expert and four columns.
constexpr int RSLAB = 64;
template <typename T>
__global__ void __launch_bounds__(128)
router_wgrad_kernel(const float* __restrict__ dlogit, const T* __restrict__ x, float* __restrict__ dW_r, long long Tn, int Dm, int E) {
  pdl_sync();
  __shared__ float dl[RSLAB][8];
  const int e0 = blockIdx.y * 8;
  const long long t0 = (long long)blockIdx.z * RSLAB;
  const int nt = (int)min((long long)RSLAB, Tn - t0);
  for (int i = threadIdx.x; i < RSLAB * 8; i += blockDim.x) {
    const int r = i >> 3, e = e0 + (i & 7);
    dl[r][i & 7] = (r < nt && e < E) ? dlogit[(t0 + r) * E + e] : 0.0f;
  }
  __syncthreads();
  const int d = (blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (d >= Dm) return;
  float2 acc[8][2];
#pragma unroll
  for (int e = 0; e < 8; ++e) { acc[e][0] = make_float2(0.0f, 0.0f); acc[e][1] = acc[e][0]; }
  constexpr int G = 8;
  for (int r0 = 0; r0 < nt; r0 += G) {
    Raw4<T> raw[G];
#pragma unroll
    for (int i = 0; i < G; ++i) raw[i].load(x + (t0 + min(r0 + i, nt - 1)) * Dm + d);
#pragma unroll
    for (int i = 0; i < G; ++i) {      // rows past the slab's end repeat its last token with a zero factor
      float2 v[2];
      raw[i].get(v);
      const float4 f0 = *reinterpret_cast<const float4*>(&dl[r0 + i][0]), f1 = *reinterpret_cast<const float4*>(&dl[r0 + i][4]);
      const float f[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        acc[e][0] = __ffma2_rn(make_float2(f[e], f[e]), v[0], acc[e][0]);
        acc[e][1] = __ffma2_rn(make_float2(f[e], f[e]), v[1], acc[e][1]);
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if (e0 + e < E) atomicAdd(reinterpret_cast<float4*>(dW_r + (size_t)(e0 + e) * Dm + d), make_float4(acc[e][0].x, acc[e][0].y, acc[e][1].x, acc[e][1].y));
}

// Weight gradient of a (grouped) projection: C[s][p, q] = sum over the rows r of segment s of scale[r] X[r, p] Y[r, q]
// (X, Y row-major with the contracted index, the token row, outermost).  64 x 64 outputs per block, 4 x 4 per thread,
// 16 rows per step through shared memory; fp32 accumulation and output.  seg == nullptr: one segment [0, rows_total).
template <typename T>
__global__ void __launch_bounds__(256)
wgrad_kernel(const T* __restrict__ X, int ldx, const T* __restrict__ Y, int ldy, const float* __restrict__ scale,
             const int32_t* __restrict__ seg, int rows_total, int P, int Q, float* __restrict__ C) {
  pdl_sync();
  __shared__ float Xs[16][64 + 4];
  __shared__ float Ys[16][64 + 4];
  const int s = blockIdx.z;
  const int r0 = seg ? seg[s] : 0, r1 = seg ? seg[s + 1] : rows_total;
  const int p0 = blockIdx.y * 64, q0 = blockIdx.x * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int lr = threadIdx.x >> 4, lc = (threadIdx.x & 15) * 4;       // loader: row lr of the step, 4 consecutive columns from lc
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  for (int r = r0; r < r1; r += 16) {
    const int row = r + lr;
    const bool in = row < r1;
    const float sc = (in && scale) ? scale[row] : 1.0f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + lc + j, q = q0 + lc + j;
      Xs[lr][lc + j] = (in && p < P) ? sc * to_f32(X[(size_t)row * ldx + p]) : 0.0f;
      Ys[lr][lc + j] = (in && q < Q) ? to_f32(Y[(size_t)row * ldy + q]) : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      float xa[4], yb[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { xa[i] = Xs[kk][ty * 4 + i]; yb[i] = Ys[kk][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xa[i], yb[j], acc[i][j]);
    }
    __syncthreads();
  }
  float* Cs = C + (size_t)s * P * Q;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + ty * 4 + i, q = q0 + tx * 4 + j;
      if (p < P && q < Q) Cs[(size_t)p * Q + q] = acc[i][j];
    }
}

}  // namespace

cudaError_t launch_transpose(int dtype, const void* in, void* out, int batch, int R, int C, cudaStream_t st) {
  const dim3 grid((C + 31) / 32, (R + 31) / 32, batch), block(32, 8);
  if (dtype == ROM_BF16) launch_k(transpose_kernel<__nv_bfloat16>, grid, block, 0, st, (const __nv_bfloat16*)in, (__nv_bfloat16*)out, R, C);
  else launch_k(transpose_kernel<float>, grid, block, 0, st, (const float*)in, (float*)out, R, C);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_zero(const ZeroList& z, cudaStream_t st) {
  launch_k(zero_kernel, dim3(64, z.count), 256, 0, st, z);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_slot_sum(int dtype, const void* src, const int32_t* row_of_assign, void* dst, long long Tn, int width, int K, cudaStream_t st) {
  const long long total = Tn * (width / (dtype == ROM_BF16 ? 8 : 4));
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if (dtype == ROM_BF16) launch_k(slot_sum_kernel<__nv_bfloat16>, blocks, 256, 0, st, (const __nv_bfloat16*)src, row_of_assign, (__nv_bfloat16*)dst, width, K, total);
  else launch_k(slot_sum_kernel<float>, blocks, 256, 0, st, (const float*)src, row_of_assign, (float*)dst, width, K, total);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_combine_bwd(int dtype, const void* dYgu, void* Ygp, const int32_t* row_of_assign, const float* gates, void* dYg,
                               float* dgate, float* rowscale, long long Tn, int De, int K, cudaStream_t st) {
  if (dtype == ROM_BF16 && !rowscale && K <= 2)
    launch_k(K == 1 ? combine_bwd_warp_kernel<1> : combine_bwd_warp_kernel<2>, (unsigned)((Tn + 3) / 4), 128, 0, st, (const __nv_bfloat16*)dYgu,
             (__nv_bfloat16*)Ygp, row_of_assign, gates, (__nv_bfloat16*)dYg, dgate, De, Tn);
  else if (dtype == ROM_BF16)
    launch_k(combine_bwd_kernel<__nv_bfloat16>, (unsigned)Tn, 128, 0, st, (const __nv_bfloat16*)dYgu, (__nv_bfloat16*)Ygp, row_of_assign, gates,
                                                                  (__nv_bfloat16*)dYg, dgate, rowscale, De, K);
  else
    launch_k(combine_bwd_kernel<float>, (unsigned)Tn, 128, 0, st, (const float*)dYgu, (float*)Ygp, row_of_assign, gates, (float*)dYg, dgate,
                                                          rowscale, De, K);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_pack_bc(int dtype, const float* dBm, const float* dCm, void* dxdbl, long long Tn, int R, int N, cudaStream_t st) {
  const unsigned blocks = (unsigned)((Tn * 2 * N + 255) / 256);
  if (dtype == ROM_BF16) launch_k(pack_bc_kernel<__nv_bfloat16>, blocks, 256, 0, st, dBm, dCm, (__nv_bfloat16*)dxdbl, Tn, R, N);
  else launch_k(pack_bc_kernel<float>, blocks, 256, 0, st, dBm, dCm, (float*)dxdbl, Tn, R, N);
  count_launch();
  return cudaGetLastError();
}

template <typename T>
static void launch_conv_bwd_t(const rom_config& c, const void* HZ, const void* w_conv, const float* b_conv, const void* dU1, const void* dU2, void* dHZ,
                              const int32_t* row_of_assign, float* dw, float* db, cudaStream_t st) {
  // 64 steps per thread (three of them walked twice), 32 when that leaves SMs idle
  const unsigned gx = (c.d_inner / 4 + 127) / 128;
  const int seg = (long long)gx * c.B * ((c.L + 63) / 64) >= 4 * 148 ? 64 : 32;
  const dim3 grid(gx, (c.L + seg - 1) / seg, c.B);
  auto go = [&](auto kern) {
    launch_k(kern, grid, 128, 0, st, (const T*)HZ, (const T*)w_conv, b_conv, (const T*)dU1, (const T*)dU2, (T*)dHZ, row_of_assign, dw, db, c.L, c.d_inner, c.K, seg);
  };
  if (c.d_conv == 4) go(conv_bwd_kernel<T, 4>);
  else if (c.d_conv == 3) go(conv_bwd_kernel<T, 3>);
  else go(conv_bwd_kernel<T, 2>);
}
cudaError_t launch_conv_bwd(const rom_config& c, const void* HZ, const void* w_conv, const float* b_conv, const void* dU1, const void* dU2,
                            void* dHZ, const int32_t* row_of_assign, float* dw, float* db, cudaStream_t st) {
  if (c.dtype == ROM_BF16) launch_conv_bwd_t<__nv_bfloat16>(c, HZ, w_conv, b_conv, dU1, dU2, dHZ, row_of_assign, dw, db, st);
  else launch_conv_bwd_t<float>(c, HZ, w_conv, b_conv, dU1, dU2, dHZ, row_of_assign, dw, db, st);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_router_bwd(const rom_config& c, const void* x, const float* probs, const int32_t* idx, const float* gates, const float* dgate,
                              float* dlogit, float* db_r, float* dW_r, cudaStream_t st) {
  const long long Tn = (long long)c.B * c.L;
  launch_k(router_bwd_kernel, (unsigned)((Tn + 127) / 128), 128, 0, st, probs, idx, gates, dgate, dlogit, db_r, Tn, c.E, c.K, c.gate_mode);
  count_launch();
  const dim3 wgrid((c.d_model / 4 + 127) / 128, (c.E + 7) / 8, (unsigned)((Tn + RSLAB - 1) / RSLAB));
  if (c.dtype == ROM_BF16) launch_k(router_wgrad_kernel<__nv_bfloat16>, wgrid, 128, 0, st, dlogit, (const __nv_bfloat16*)x, dW_r, Tn, c.d_model, c.E);
  else launch_k(router_wgrad_kernel<float>, wgrid, 128, 0, st, dlogit, (const float*)x, dW_r, Tn, c.d_model, c.E);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_dx(const rom_config& c, const void* dxp, const int32_t* row_of_assign, const float* dlogit, const void* W_r, void* dx,
                      cudaStream_t st) {
  const long long total = (long long)c.B * c.L * (c.d_model / (c.dtype == ROM_BF16 ? 8 : 4));
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if (c.dtype == ROM_BF16 && c.K <= 2 && (c.E == 4 || c.E == 8 || c.E == 16)) {
    const long long Tn = (long long)c.B * c.L, nv = c.d_model / 8;
    const int seg = 8;
    const unsigned wb = (unsigned)((nv * ((Tn + seg - 1) / seg) + 127) / 128);
    auto go = [&](auto kern) { launch_k(kern, wb, 128, 0, st, (const __nv_bfloat16*)dxp, row_of_assign, dlogit, (const __nv_bfloat16*)W_r, (__nv_bfloat16*)dx, c.d_model, seg, Tn); };
    if (c.K == 1) go(c.E == 4 ? dx_walk_kernel<4, 1> : c.E == 8 ? dx_walk_kernel<8, 1> : dx_walk_kernel<16, 1>);
    else go(c.E == 4 ? dx_walk_kernel<4, 2> : c.E == 8 ? dx_walk_kernel<8, 2> : dx_walk_kernel<16, 2>);
  } else if (c.dtype == ROM_BF16)
    launch_k(dx_kernel<__nv_bfloat16>, blocks, 256, 0, st, (const __nv_bfloat16*)dxp, row_of_assign, dlogit, (const __nv_bfloat16*)W_r, (__nv_bfloat16*)dx,
                                                   c.d_model, c.E, c.K, total);
  else
    launch_k(dx_kernel<float>, blocks, 256, 0, st, (const float*)dxp, row_of_assign, dlogit, (const float*)W_r, (float*)dx, c.d_model, c.E, c.K, total);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_wgrad(int dtype, const void* X, int ldx, const void* Y, int ldy, const float* scale, const int32_t* seg, int n_seg,
                         int rows_total, int P, int Q, float* C, cudaStream_t st) {
  const dim3 grid((Q + 63) / 64, (P + 63) / 64, n_seg);
  if (dtype == ROM_BF16)
    launch_k(wgrad_kernel<__nv_bfloat16>, grid, 256, 0, st, (const __nv_bfloat16*)X, ldx, (const __nv_bfloat16*)Y, ldy, scale, seg, rows_total, P, Q, C);
  else
    launch_k(wgrad_kernel<float>, grid, 256, 0, st, (const float*)X, ldx, (const float*)Y, ldy, scale, seg, rows_total, P, Q, C);
  count_launch();
  return cudaGetLastError();
}

}  // namespace rom
