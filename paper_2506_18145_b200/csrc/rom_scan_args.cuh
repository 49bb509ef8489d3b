// Arguments and helpers shared by the selective-scan kernels (rom_scan.cu, rom_scan_warp.cu, rom_scan_bwd.cu).
#pragma once

#include "rom_internal.cuh"

namespace rom {

struct ScanArgs {
  const void* u; const void* delta; const float* A; const float* Bm; const float* Cm; const float* D;
  const void* z; int ldz; const int32_t* z_row /* [T] or, warp kernel with K > 1, [T, K]: rows summed */; const float* h0; void* y; float* h_last; const int32_t* y_rows;
  int K, L, De;
  int Lc, nch;          // chunk length and chunks per sequence (nch == 1: Lc == L); blockIdx.z = chunk
  int L0;               // length of chunk 0; chunk j >= 1 covers steps [L0 + (j-1) Lc, L0 + j Lc)
  float* sum_delta;     // state-only blocks: [B*nch, De] sum of Delta over the chunk
  int gate_activated;   // z already holds SiLU(gate pre-activation): multiply only
  int chunk_off;        // chunk of blockIdx.z == 0
  float* ckpt;          // MODE 3..5: [B, nck, De, 16] state at the start of every kScanCkpt steps (nck per sequence)
  int nck;
  int scalar_a;         // A[c, :] is one value per channel (scalar-per-head decay of a Mamba2-style block): one exponential
                        // per channel and step instead of one per state (only with B-bar = Delta B)
  // second launch of the chunked scan (SCAN_FULL, SCAN_FULL_CKPT): [B, nch, De, 16] end states of the chunks before (chunk 0: true;
  // others: from a zero state) and their [B, nch, De] sums of Delta, from which a block chains its own initial state; h_last is then
  // [B, De, 16], written by the last chunk
  const float* chain_end;
  const float* chain_sum;
  int early;            // warp kernel: the kernel before lets nobody in before its blocks end
};

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
// Slot of lane l's partial sums of step r: conflict-free both for a quarter-warp of writers (eight lanes, one step) and of readers
// (lanes l = 8 g + const, two steps).
__device__ __forceinline__ int ysw(int l, int r) { return l ^ (2 * (l >> 3) + (r & 1)); }

// What a scan launch does.  SCAN_FULL: outputs.  SCAN_STATE: state only (h_last and sum_delta of every chunk).  SCAN_FIRST: first
// launch of the chunked scan: chunk 0 in full from the caller's initial state (h0 indexed by sequence), the others state-only
// from a zero state.  SCAN_CKPT: state only from the given chunk-start states, storing the state at the start of every kScanCkpt
// steps (backward pass).  SCAN_FULL_CKPT, SCAN_FIRST_CKPT: SCAN_FULL and SCAN_FIRST with those stores beside the outputs.
enum ScanMode : int { SCAN_FULL = 0, SCAN_STATE = 1, SCAN_FIRST = 2, SCAN_CKPT = 3, SCAN_FULL_CKPT = 4, SCAN_FIRST_CKPT = 5 };

// rom_scan_warp.cu: bf16 storage, A per channel and state.  grid_z chunks per sequence from a.chunk_off on.
cudaError_t launch_scan_warp(const ScanArgs& a, int B, int grid_z, bool zoh, bool delta_fp32, ScanMode mode, cudaStream_t st);

// rom_scan_ring.cu: the whole scan in one launch; bf16 storage, A per channel and state.  ckpt: with checkpoints (delta in bf16).
cudaError_t launch_scan_ring(const ScanArgs& a, int B, bool zoh, bool delta_fp32, bool ckpt, cudaStream_t st);

// rom_scan_f32.cu: the whole scan in one launch; fp32 storage, A per channel and state.
cudaError_t launch_scan_f32(const ScanArgs& a, int B, bool zoh, bool ckpt, cudaStream_t st);

}  // namespace rom
