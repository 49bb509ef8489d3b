// Selective scan for bf16 storage (same arithmetic and arguments as rom_scan.cu): one warp owns 32 channels of one chunk of one
// sequence, a lane 4 states of 4 adjacent channels (rom_scan_warp.cuh).
//
// What bounds it: per state update one exponential on the special-function unit (16 per clock and SM), six fp32 lane operations
// (128 per clock and SM) and the bytes that shared memory returns to registers (128 per clock and SM, one copy per lane).  With
// 8 states of one channel per lane the B and C of every step cost 8 bytes per update -- as much time as the exponential -- and the
// sums over states a shuffle and its selects.  Here the 16 updates of a lane and step share 16 bytes of B, 16 of C and 32 of
// (Delta, u): 4 bytes per update; packed pairs run along the channels, so Delta and u need no duplication and the sums over a
// lane's states no horizontal add; the four lanes of a channel leave their partial sums in shared memory, where the lane that
// writes the output adds them (1 byte per update each way, no shuffles).  A warp is self-contained (no block barrier), eight steps
// are staged at a time while the next eight are in flight in registers, and twelve warps fit an SM (sixteen at 128 registers, without
// the operands of the next step ahead: 1.30 ms against 1.04 at 64 x 1024 steps of 3072 channels; eight at 255: 1.16).
// Measured there: 1.39 ms for 8 states per lane, 1.27 with this layout and a loader that touched eight rows per quarter-warp (75 % of
// the shared-memory pipe's wavefronts), 1.04 with four loader lanes per row: 69 % of the special-function peak.
#include "rom_scan_warp.cuh"

namespace rom {
namespace {

constexpr int WPB = 4;            // warps per block
constexpr int BT = WPB * 32;

template <typename TD, bool ZOH, int MODE, bool SLOTS>
__global__ void __launch_bounds__(BT, 3)
scan_warp_kernel(const ScanArgs p) {
  constexpr bool FIRST = MODE == SCAN_FIRST || MODE == SCAN_FIRST_CKPT;
  pdl_wait();
  if (!FIRST) pdl_trigger();      // (the second launch comes in as the blocks of the first end: see launch_mode)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int c_warp = blockIdx.x * BT + warp * WCH;
  if (c_warp >= p.De) return;     // d_inner is a multiple of 64: a warp's 32 channels are all in or all out
  scan_warp_channels<TD, ZOH, MODE, SLOTS>(p, reinterpret_cast<WarpTile*>(smem_raw)[warp], c_warp, blockIdx.y, blockIdx.z + p.chunk_off);
}

// A scan is launched early only behind a kernel that lets nobody in before its blocks end: let in while they run, few blocks per SM
// pile up on the first SMs to drain (+40 % at 256 blocks).  Behind such a kernel (the dt Proj; the first launch of a chunked scan) the
// launch itself is hidden: 4 x 2048 steps of 2048 channels 5 us less for the two.
template <typename TD, bool ZOH, int MODE>
cudaError_t launch_mode(const ScanArgs& a, int B, int grid_z, cudaStream_t st) {
  constexpr int smem = WPB * (int)sizeof(WarpTile);
  const dim3 grid((a.De + BT - 1) / BT, B, grid_z);
  if (a.z_row && a.K > 1) {
    if constexpr (sizeof(TD) == 2 && (MODE == SCAN_FULL || MODE == SCAN_FIRST)) launch_k(a.early != 0, scan_warp_kernel<TD, ZOH, MODE, true>, grid, BT, smem, st, a);
    else return cudaErrorInvalidValue;
  } else {
    launch_k(a.early != 0, scan_warp_kernel<TD, ZOH, MODE, false>, grid, BT, smem, st, a);
  }
  count_launch();
  return cudaGetLastError();
}
// fp32 Delta: rom_scan and the state passes of rom_scan_backward; bf16 Delta: the layer, whose backward takes checkpoints from the full scan.
template <typename TD, bool ZOH>
cudaError_t launch_any(const ScanArgs& a, int B, int grid_z, ScanMode mode, cudaStream_t st) {
  if (mode == SCAN_FULL) return launch_mode<TD, ZOH, SCAN_FULL>(a, B, grid_z, st);
  if (mode == SCAN_FIRST) return launch_mode<TD, ZOH, SCAN_FIRST>(a, B, grid_z, st);
  if constexpr (sizeof(TD) == 4) {
    if (mode == SCAN_STATE) return launch_mode<TD, ZOH, SCAN_STATE>(a, B, grid_z, st);
    if (mode == SCAN_CKPT) return launch_mode<TD, ZOH, SCAN_CKPT>(a, B, grid_z, st);
  } else {
    if (mode == SCAN_FULL_CKPT) return launch_mode<TD, ZOH, SCAN_FULL_CKPT>(a, B, grid_z, st);
    if (mode == SCAN_FIRST_CKPT) return launch_mode<TD, ZOH, SCAN_FIRST_CKPT>(a, B, grid_z, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_scan_warp(const ScanArgs& a, int B, int grid_z, bool zoh, bool delta_fp32, ScanMode mode, cudaStream_t st) {
  if (delta_fp32) return zoh ? launch_any<float, true>(a, B, grid_z, mode, st) : launch_any<float, false>(a, B, grid_z, mode, st);
  return zoh ? launch_any<bf16, true>(a, B, grid_z, mode, st) : launch_any<bf16, false>(a, B, grid_z, mode, st);
}

}  // namespace rom
