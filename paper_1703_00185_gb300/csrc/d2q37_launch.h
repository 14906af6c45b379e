// Host-side launchers of the sm_103a kernels (d2q37_kernels.cu), used by the
// C ABI (d2q37_api.cu).  Each launcher enqueues on `stream` and returns the
// number of kernels it launched, or -1 if a launch failed.
#pragma once

#include <type_traits>

#include <cuda_runtime.h>

#include "d2q37_lattice.cuh"

namespace d2q37 {

// Copy the quadrature constants to the current device's constant memory.
cudaError_t upload_shell_consts(const ShellConsts& c);

int sm_count();  // of the current device

// Launch; dependent: as a programmatic dependent of the kernel before it in the
// stream.  Such a grid may be resident while earlier kernels still write what it
// reads: after its griddepcontrol.wait those writes are visible to its ordinary
// loads, but not to loads through the read-only path, whose data must not change
// while the grid lives.  So no pointer of a kernel launched here is const
// __restrict__ (which lets the compiler take that path, and move a load above
// the wait).  The FP64 ones load populations from L2: store_images reads row 3 of
// the edge columns back, and with it the wall rows of the same sector, which
// wall_band_kernel may be writing, into the L1 of an SM where the next grid waits.
template <class... A>
inline bool launch_pdl(void (*kernel)(A...), dim3 grid, int block, int smem, cudaStream_t stream, bool dependent,
                       std::common_type_t<A>... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess;
}

int launch_wrap(double* buf, const StepParams& p, cudaStream_t stream);
int launch_propagate(const double* src, double* dst, const StepParams& p, cudaStream_t stream);
int launch_bc(const double* src, double* dst, const StepParams& p, cudaStream_t stream);
int launch_collide(double* buf, const StepParams& p, cudaStream_t stream);
// overlap: the wall-band kernel (walls only) is launched as a programmatic
// dependent of the sites kernel and starts in its tail; false: after it.
// chain: the first kernel may be launched as a programmatic dependent of whatever
// kernel precedes it in the stream (it waits for it before its first access).
// alone: no other stream's grids are expected beside it.
int launch_fused(const double* src, double* dst, const StepParams& p, cudaStream_t stream, bool overlap = true,
                 bool chain = false, bool alone = false);
int launch_fields(const double* buf, double* rho, double* u, double* T, const StepParams& p, cudaStream_t stream,
                  bool chain = false);
// Rayleigh-Taylor initial state, FP64 or FP32 deviations; yi: device, the
// interface of every column.
int launch_init_rayleigh_taylor(void* buf, bool fp32, const double* yi, double T_top, double T_bot,
                                unsigned long long seed, const StepParams& p, cudaStream_t stream);

// FP32 deviation storage (d2q37_kernels_fp32.cu).
// wide_fp64 selects FP64 (true) or double-float (false) for the wide terms.
cudaError_t upload_shell_consts32(const ShellConsts32& c);
int launch_wrap32(float* buf, const StepParams& p, cudaStream_t stream);
int launch_propagate32(const float* src, float* dst, const StepParams& p, cudaStream_t stream);
int launch_bc32(const float* src, float* dst, const StepParams& p, cudaStream_t stream);
int launch_collide32(float* buf, const StepParams& p, bool wide_fp64, cudaStream_t stream);
int launch_fused32(const float* src, float* dst, const StepParams& p, bool wide_fp64, cudaStream_t stream,
                   bool chain = false);
int launch_fields32(const float* buf, double* rho, double* u, double* T, const StepParams& p, cudaStream_t stream,
                    bool chain = false);
// Batched fused step over a table of n lattices (BatchEntry, device memory),
// tiles of block_y rows; block_y in {64, 128, 256}; grid = number of blocks
// of the grid-stride loop.  *_blocks_per_sm: resident blocks per SM.
// tile_entry: owning entry of every tile (device, tiles values), or null
// for a binary search over the table's tile0.  common (FP64): when every
// lattice shares tau and g, their collision constants (passed as a kernel
// argument), else null.
int launch_batch_fused(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity,
                       int block_y, int grid, const Collision* common, cudaStream_t stream);
int batch_blocks_per_sm(int block_y);
// The batched FP64 step with one block per tile (see BatchLaunch); uniform:
// every lattice has the collision constants L.common.  tab: the BatchEntry
// table for tiles of block_y rows (device).
// tile_entry: owning lattice of every site tile (device), or null for a search.
// Small batches run the table kernel instead.
int launch_batch_tiles(const BatchLaunch& L, bool uniform, const BatchEntry* tab, const int* tile_entry, int parity,
                       int block_y, cudaStream_t stream);
// The (column, wall) groups one wall tile holds.
int batch_wall_groups_per_tile(int block_y);
int launch_batch_fused32(const BatchEntry* tab, const int* tile_entry, int n, long long tiles, int parity,
                         int block_y, int grid, bool wide_fp64, cudaStream_t stream);
int batch32_blocks_per_sm(int block_y, bool wide_fp64);
// The same in FP32 storage (BatchLaunch32); tiles: grid size.
int launch_batch_tiles32(const BatchLaunch32& L, const BatchEntry* tab, const int* tile_entry, int tiles, int parity,
                         int block_y, bool wide_fp64, cudaStream_t stream);

// Populations l0 .. l0 + count - 1 between contiguous FP64 [count][Lx][Ly]
// planes and the FP32 deviation frame (d = f - w_l).
int launch_planes_to_frame32(float* frame, const double* planes, int l0, int count, const StepParams& p,
                             cudaStream_t stream);
int launch_frame32_to_planes(double* planes, const float* frame, int l0, int count, const StepParams& p,
                             cudaStream_t stream);

}  // namespace d2q37
