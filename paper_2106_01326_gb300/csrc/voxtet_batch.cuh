// voxtet_batch.cuh -- the device table of a batch of meshes.
//
// A batch is a device table of jobs, each a complete single-mesh problem (its own Params, snap
// arguments and workspace slice with the single-mesh layout).  One launch per kernel type covers
// all jobs; units of work (prologue chunks, tiles) are numbered across the batch and a unit's job
// is found in host-built prefix sums.
#pragma once
#include "voxtet_device.cuh"

namespace voxtet {

struct SnapArgsK {  // the snap's scalars (see snap_one)
  double ox, oy, oz, h, scale, mul;
  int use_mul, fast;
};

struct JobDesc {
  Params p;
  SnapArgsK s;
  const void *verts;     // float32 or (fixed) int32 lattice coordinates
  int fixed;
  int clear;             // 1: the grid is zeroed first
  long long grid_words;  // 0 for a rejected job
};

struct BatchHeader {
  int n_jobs;
  int pad0;
  unsigned long long total_tiles;
  unsigned long long total_prep;  // chunks of zeroing and snapping
  unsigned long long tile_counter;
  unsigned long long chunk;  // tiles a block claims at a time
  unsigned long long reserved[27];
};
static_assert(sizeof(BatchHeader) == 256, "batch header is 256 bytes");

// Largest j in [0, n) with base[j] <= x (base ascending, base[0] = 0), found by the 32 lanes of a
// warp together: each step narrows the range 32 times with one load per lane, so up to 1024 jobs
// take two dependent loads where a bisection takes ten.
__device__ __forceinline__ int find_job_warp(const unsigned long long *base, int n, unsigned long long x) {
  const int lane = threadIdx.x & 31;
  int lo = 0, size = n;  // the answer is in [lo, lo + size)
  while (size > 1) {
    const int step = (size + 31) >> 5;
    const int i = lo + lane * step;
    const bool le = lane * step < size && base[i] <= x;  // true for lane 0, and for a prefix of the lanes
    const int last = 31 - __clz(__ballot_sync(0xFFFFFFFFu, le));
    lo += last * step;
    size = min(step, size - last * step);
  }
  return lo;
}

}  // namespace voxtet
