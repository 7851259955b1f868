// voxtet_slices.cuh -- host interface of the slice-unit kernel (voxtet_slices.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

#include "voxtet_batch.cuh"
#include "voxtet_device.cuh"

namespace voxtet {

constexpr int kSuBlock = 128;   // threads per block, and tets per tile (one per thread)
constexpr int kSuSlices = 32;   // slices a thread takes per window (5 blocks per SM)
constexpr int kSuSlicesSmall = 16;  // the smaller capacity: less shared memory, 7 blocks per SM
constexpr int kSuRows = 1024;   // x-rows per slice of a tet's box in one window
constexpr int kSuMaxGroup = 7;  // log2 of the most threads that share a tet (a whole block)

// log2 of the threads that share a tet in the slice-unit kernel, from the mesh's size and the grid
// it goes to (side: the lattice's voxels per axis; ry: rows per slice; slab: the slices produced): a tet of a mesh that
// fills its grid spans about w = side / cbrt(n_tets / 6) slices.
//   - As many threads as make one window hold w slices (`slices` a thread).  Measured on GB300, 64
//     meshes of 1k-1M tets on 64^3-512^3 grids: 1.54 ms with this many threads, 1.94 with a
//     quarter, 1.60 with three times as many (every thread of a group repeats the tet's setup).
//   - More if the tiles of kSuBlock >> lg tets would occupy fewer than half of `blocks` (the
//     resident blocks; 0: this does not matter): 56,679 tets at 256^3 (443 tiles for 1064 blocks)
//     25.7 us with two threads a tet, 29.3 with one or four; 1,244 tets at 512^3 (10 tiles) 40 us
//     with 64 threads, 77 us with the first rule alone.
//   - More if a tile or two per resident block would be uneven (su_share_more).
//   - Never more than w: they would have no slice to take (4,200 tets at 64^3: 62 us up to 16
//     threads a tet, 78 with 64).
int su_group_log2(long long n_tets, int side, int ry, int slab, int slices, long long blocks);

// Enqueue the slice-unit kernel for p on `stream`: variant = (list << 2) | (strict << 1) | cull;
// slices = the slices a thread takes per window (kSuSlicesSmall or kSuSlices); list = the tets are
// those k_slab_list listed; spread = over all resident blocks, if need be in tiles of fewer tets (lists
// always are).  Returns VOXTET_OK or VOXTET_ERR_CUDA.
int launch_slices(const Params &p, int variant, int slices, bool spread, int sms, cudaStream_t stream);

// Enqueue the slice-unit kernel over a batch's jobs (tile_base: the jobs' tile offsets, tiles of
// kSuBlock >> lg tets); its resident blocks per SM (0 on a CUDA error).
int launch_slices_batched(BatchHeader *bh, const JobDesc *jobs, const unsigned long long *tile_base, int *status,
                          bool strict, bool cull, int sms, cudaStream_t stream);
int slices_batched_blocks(bool strict, bool cull);

// Shared memory of one block of the slice-unit kernel with that slice capacity.
size_t slices_smem_bytes(int slices);

}  // namespace voxtet
