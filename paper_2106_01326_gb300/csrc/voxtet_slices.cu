// voxtet_slices.cu -- the slice-unit kernel of the voxelizer (scanline step and OR writes).
//
// The operation is the same as the span kernel's (voxtet.cu): every voxel-centre sample
// of a tet's bounding box that passes the closed (or strict) point-in-tetrahedron test of
// Section 4, Theorem 1 is set, the samples of one x-row solved at once as an interval
// (Section 3, "Voxelization", per row instead of per sample).  Only the distribution of
// the work differs.  A block takes a tile of kSuBlock tets, one per thread, and
//   (1) sets each tet up once: checked load, sample box, exact orientation from the
//       64-bit face normals, the four faces' single-precision filter data (a record in
//       shared memory), and for every z-slice of the box the exact range of candidate
//       rows (the cross-section's y-extent, narrowed exactly by faces parallel to x);
//   (2) counting-sorts the tile's (tet, slice) units by their row count, so the 32 lanes
//       of a warp walk units of the same length and stay in step (a block-wide exclusive
//       scan over per-warp bucket counters is the work distributor);
//   (3) walks each unit's rows: per row the four face bounds, the tightest upper and
//       lower bound certified once each (the filter of Section 4's orientation values,
//       voxtet_rows.cuh), and the interval ORed into the grid's words.
// What bounds it: instruction issue, the L1 data path (record loads of random slots, the
// ORs) and, on finer grids, the rate at which an SM can send ORs to L2.  Measured on GB300
// with timing-only copies, 1.3 M-tet sliver mesh at 512^3 (258 us): load, classification and
// face data 58 us, the slices' row ranges 29, the sort 14, the units' record loads 28, the
// rows' bounds 61, the ORs 68.  Biased bounds (no separate bracket), one add-and-round per
// side, 16-word records and the rows' range from four lines took the kernel from 274 to 257 us
// there and from 1027 to 1002 us at 1024^3 (212 M warp instructions against 221 M).
// Tets this kernel does not take -- zero volume (skipped), wider than 2^20 lattice
// units or use_filter = 0 (exact kernel), or more than kSuSlices slices or kSuRows rows
// per slice (listed at the back of the tet queue for the span kernel) -- are counted or
// queued exactly as the span kernel would.  Rows the filter cannot certify go to the
// same row queue, solved afterwards by the exact kernel.
#include <cuda_runtime.h>

#include <atomic>

#include "voxtet.h"
#include "tet_math.cuh"
#include "voxtet_device.cuh"
#include "voxtet_rows.cuh"
#include "voxtet_slices.cuh"

namespace voxtet {

constexpr int kSuWarps = kSuBlock / 32;
constexpr int kSuBuckets = 64;                           // row counts 1..63 one bucket each, >= 64 together
constexpr int kSuCounters = kSuBuckets * kSuWarps;       // bucket-major, one counter per warp of each bucket
constexpr int kSuRec = 20;  // floats per tet record: 16 used; 5 groups of 16 bytes, an odd number,
                            // so that lanes loading records of random slots spread over all banks
constexpr int kSuStage = 64;                             // staged uncertain rows per block (about 5 per tile)
constexpr uint32_t kSuEmpty = 0xFFFFFFFFu;               // a slice without candidate rows
static_assert(kSuBlock == 128 && kSuSlices <= 32 && kSuRows == 1024, "unit fields: 7 + 5 bits; rows in 10 bits");

// Tet record (kSuRec words per slot): alpha' of the four faces | beta | gamma | E of the upper
// and of the lower side, i0 | (na - 1) << 16 | upper slots << 30, j0 | (l0 - z0) << 16.  Upper faces fill the slots from the
// front and lower faces from the back; a face parallel to x leaves a neutral upper slot (alpha' =
// +infinity) between them.  Slot 0 is always an upper face and slot 3 a lower one.
constexpr int kRecB = 4, kRecG = 8, kRecEU = 12, kRecEL = 13, kRecX = 14, kRecYZ = 15;
constexpr int kSuColumns = 1 << 14;  // most samples along x of a tet's box (14 bits hold na - 1)

// Shared memory of one block (dynamic), for tets of at most SL slices.
template <int SL>
struct SuSmem {
  float rec[kSuBlock * kSuRec];
  // per tet slot, slice k of its tet: b_lo | (n - 1) << 10, or kSuEmpty
  uint32_t slice[SL][kSuBlock];
  // the tile's units sorted by row count, longest first: slot | k << 7 | b_lo << 12 | (n - 1) << 22
  uint32_t unit[kSuBlock * SL];
  uint32_t hist[kSuCounters];  // unit counts, then (after the scan) cursors
  uint32_t total;
  uint32_t warp_tot[kSuWarps];
  RowStageN<kSuStage> stage;
  long long tile;
};

// 16-slice tiles fit 7 blocks per SM (228 KB, 1 KB reserved per block), 32-slice tiles 5
static_assert(sizeof(SuSmem<kSuSlicesSmall>) <= 31 * 1024, "slice-unit kernel shared memory: seven blocks per SM");
static_assert(sizeof(SuSmem<kSuSlices>) <= 44 * 1024 + 512, "slice-unit kernel shared memory: five blocks per SM");

// Counter of a unit with n rows emitted by warp w: longer units first.
__device__ __forceinline__ int su_counter(int n, int w) {
  return (kSuBuckets - min(n, kSuBuckets)) * kSuWarps + w;
}

// Phase (1) for tet t of this thread (t < 0: none).  Returns the slices whose entries it
// wrote to sm.slice (0 if the tet has no unit here); counts each unit in its counter (no
// rank is needed here, so the count does not wait on the shared-memory atomic).
template <bool STRICT, bool CULL, int SL>
__device__ __forceinline__ int su_setup(const Params &p, long long t, SuSmem<SL> &sm, TileCounters &ctr) {
  const int tid = threadIdx.x, warp = tid >> 5;
  if (t < 0) return 0;
  int3 V[4];
  if (!load_tet(p, t, V, ctr.err)) return 0;
  Box bx;
  const int E = tet_box(V, p.sh, p.rx, p.ry, p.z0, p.z1, bx);
  const bool empty = bx.na <= 0 || bx.nb <= 0 || bx.nc <= 0;
  if (E > kNarrowExtent) {  // wider than 2^20 lattice units: 128-bit sign, exact kernel
    if (v6_sign(V, E) == 0) {
      ++ctr.degenerate;
      return 0;
    }
    if (empty) return 0;
    ++ctr.wide;
    const unsigned k = atomicAdd(&p.hdr->tetq_count, 1u);
    p.tetq[k] = (uint32_t)t;
    return 0;
  }
  // E <= 2^20: edges below 2^21, normals below 2^43, V6 and every face value below 1.5 * 2^62
  const int e1x = V[1].x - V[0].x, e1y = V[1].y - V[0].y, e1z = V[1].z - V[0].z;
  const int e2x = V[2].x - V[0].x, e2y = V[2].y - V[0].y, e2z = V[2].z - V[0].z;
  const int e3x = V[3].x - V[0].x, e3y = V[3].y - V[0].y, e3z = V[3].z - V[0].z;
  i64 n1x = (i64)e2y * e3z - (i64)e2z * e3y, n1y = (i64)e2z * e3x - (i64)e2x * e3z, n1z = (i64)e2x * e3y - (i64)e2y * e3x;
  i64 n2x = (i64)e3y * e1z - (i64)e3z * e1y, n2y = (i64)e3z * e1x - (i64)e3x * e1z, n2z = (i64)e3x * e1y - (i64)e3y * e1x;
  i64 n3x = (i64)e1y * e2z - (i64)e1z * e2y, n3y = (i64)e1z * e2x - (i64)e1x * e2z, n3z = (i64)e1x * e2y - (i64)e1y * e2x;
  i64 v6 = (i64)e1x * n1x + (i64)e1y * n1y + (i64)e1z * n1z;
  if (v6 == 0) {
    ++ctr.degenerate;
    return 0;
  }
  if (empty) return 0;
  if (p.exact_all || bx.nb > kMaxFilterRows) {
    const unsigned k = atomicAdd(&p.hdr->tetq_count, 1u);
    p.tetq[k] = (uint32_t)t;
    return 0;
  }
  if (bx.nc > SL || bx.nb > kSuRows || bx.na > kSuColumns) {  // the span kernel takes it (list mode)
    const unsigned k = atomicAdd(&p.hdr->listq_count, 1u);
    p.tetq[p.n_tets - 1 - k] = (uint32_t)t;
    return 0;
  }
  // Orientation (Lemma 1.1): for V6 < 0 every orientation value of an inside point is <= 0,
  // so negating the normals (and V6) gives the positively oriented form of the same faces.
  if (v6 < 0) {
    n1x = -n1x; n1y = -n1y; n1z = -n1z;
    n2x = -n2x; n2y = -n2y; n2z = -n2z;
    n3x = -n3x; n3y = -n3y; n3z = -n3z;
    v6 = -v6;
  }
  // lam_m at the box's lowest sample P0 (tet_math.cuh): lam_m = (P0 - V0) . n_m for m = 1..3,
  // lam_0 = V6 - lam_1 - lam_2 - lam_3 with n_0 = -(n_1 + n_2 + n_3); sums that may wrap
  // transiently are formed in unsigned arithmetic (exact modulo 2^64, and the result fits)
  const int s = 1 << (p.sh - 1);
  const i64 qx = (i64)(s + (bx.i0 << p.sh)) - V[0].x;
  const i64 qy = (i64)(s + (bx.j0 << p.sh)) - V[0].y;
  const i64 qz = (i64)(s + (bx.l0 << p.sh)) - V[0].z;
  i64 L[4], Nx[4], Ny[4], Nz[4];
  L[1] = qx * n1x + qy * n1y + qz * n1z;
  L[2] = qx * n2x + qy * n2y + qz * n2z;
  L[3] = qx * n3x + qy * n3y + qz * n3z;
  L[0] = wrap_sub<i64>(wrap_sub<i64>(wrap_sub<i64>(v6, L[1]), L[2]), L[3]);
  Nx[1] = n1x; Ny[1] = n1y; Nz[1] = n1z;
  Nx[2] = n2x; Ny[2] = n2y; Nz[2] = n2z;
  Nx[3] = n3x; Ny[3] = n3y; Nz[3] = n3z;
  Nx[0] = wrap_sub<i64>(wrap_sub<i64>(wrap_sub<i64>(0, n1x), n2x), n3x);
  Ny[0] = wrap_sub<i64>(wrap_sub<i64>(wrap_sub<i64>(0, n1y), n2y), n3y);
  Nz[0] = wrap_sub<i64>(wrap_sub<i64>(wrap_sub<i64>(0, n1z), n2z), n3z);
  // Filter data per face (lam = L + D . (a, b, c) with D = 2s n) into the record's upper or
  // lower slots; a face parallel to x (Dx = 0) is an exact condition on the rows of each
  // slice below instead (at most two such faces).  Every live tet has a face with Dx < 0
  // and one with Dx > 0 (the four gradients sum to zero, at most two vanish).
  float *rec = sm.rec + tid * kSuRec;
  const float fb = (float)(bx.nb - 1), fc = (float)(bx.nc - 1);
  float eU = 0.f, eL = 0.f;
  int cu = 0, cl = 3;
  i64 zL0 = 0, zDy0 = 0, zDz0 = 0, zL1 = 0, zDy1 = 0, zDz1 = 0;
  int nz = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (Nx[m] != 0) {
      float a, b, g;
      const float e = face_bound<STRICT>(L[m], Nx[m], Ny[m], Nz[m], p.sh, fb, fc, a, b, g);
      const bool up = Nx[m] < 0;
      const int o = up ? cu++ : cl--;
      if (up) eU = fmaxf(eU, e);
      else eL = fmaxf(eL, e);
      rec[o] = a;
      rec[kRecB + o] = b;
      rec[kRecG + o] = g;
    } else {
      const i64 Dy = Ny[m] << p.sh, Dz = Nz[m] << p.sh;
      if (nz == 0) {
        zL0 = L[m]; zDy0 = Dy; zDz0 = Dz;
      } else {
        zL1 = L[m]; zDy1 = Dy; zDz1 = Dz;
      }
      ++nz;
    }
  }
  for (; cu <= cl; ++cu) {
    rec[cu] = __int_as_float(0x7f800000);
    rec[kRecB + cu] = 0.f;
    rec[kRecG + cu] = 0.f;
  }
  rec[kRecEU] = eU;
  rec[kRecEL] = eL;
  rec[kRecX] = __uint_as_float((uint32_t)bx.i0 | ((uint32_t)(bx.na - 1) << 16) | ((uint32_t)cu << 30));
  rec[kRecYZ] = __uint_as_float((uint32_t)bx.j0 | ((uint32_t)(bx.l0 - p.z0) << 16));
  // Candidate rows of each slice: the cross-section's y-extent (a superset of the rows with
  // samples), narrowed exactly by the faces parallel to x.  Each unit is counted (no rank is
  // needed here, so the count does not wait on the shared-memory atomic).
  RowRange R;
  if (CULL) {
    row_range(V, bx, p.sh, R);
  } else {
    R.kL0 = R.kL1 = R.kU0 = R.kU1 = 0.f;
    R.aL0 = R.aL1 = 0.f;
    R.aU0 = R.aU1 = fb;
  }
  int units = 0;
  float cf = 0.f;
  for (int k = 0; k < bx.nc; ++k, cf += 1.f) {
    float flo, fhi;
    slice_range(R, cf, fb, flo, fhi);
    bool any = flo <= fhi;
    uint32_t b_lo = __float_as_uint(flo) - kMagicBits, n1 = __float_as_uint(fhi) - __float_as_uint(flo);
    if (nz > 0 && any) {
      int lo = (int)b_lo, hi = (int)(b_lo + n1);
      narrow_by_row_constraint<STRICT>(zL0 + zDz0 * (i64)k, zDy0, lo, hi);
      if (nz > 1) narrow_by_row_constraint<STRICT>(zL1 + zDz1 * (i64)k, zDy1, lo, hi);
      any = lo <= hi;
      b_lo = (uint32_t)lo;
      n1 = (uint32_t)(hi - lo);
    }
    if (any) {
      atomicAdd(&sm.hist[su_counter((int)n1 + 1, warp)], 1u);
      ++units;
    }
    sm.slice[k][tid] = any ? b_lo | (n1 << 10) : kSuEmpty;
  }
  return units ? bx.nc : 0;
}

// Block-wide exclusive prefix sum of one value per thread (all threads call it); `total`
// gets the sum.  Uses sm.warp_tot; ends with the block in step.
template <int SL>
__device__ __forceinline__ uint32_t su_block_scan(SuSmem<SL> &sm, uint32_t v, uint32_t &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) sm.warp_tot[warp] = x;
  __syncthreads();
  uint32_t before = x - v;
  total = 0;
#pragma unroll
  for (int w = 0; w < kSuWarps; ++w) {
    const uint32_t t = sm.warp_tot[w];
    if (w < warp) before += t;
    total += t;
  }
  __syncthreads();
  return before;
}

// Phase (3): rows b0 .. b0 + n - 1 of slice k of the tet in `slot` (tet index t).
template <bool STRICT, bool CLAMP, int SL>
__device__ __forceinline__ void su_walk(const Params &p, SuSmem<SL> &sm, int slot, long long t, int k, int b0, int n) {
  const float4 *R = reinterpret_cast<const float4 *>(sm.rec + slot * kSuRec);
  const float4 qa = R[0], qb = R[1], qg = R[2], qi = R[3];
  const float cf = (float)k, INF = __int_as_float(0x7f800000);
  const uint32_t xx = __float_as_uint(qi.z), yz = __float_as_uint(qi.w);
  const uint32_t nup = xx >> 30;
  const bool up1 = nup >= 2, up2 = nup >= 3;
  const float a1 = __fmaf_rn(qg.y, cf, qa.y), a2 = __fmaf_rn(qg.z, cf, qa.z);
  RowFaces f;
  f.aU0 = __fmaf_rn(qg.x, cf, qa.x);
  f.bU0 = qb.x;
  f.aU1 = up1 ? a1 : INF;
  f.bU1 = up1 ? qb.y : 0.f;
  f.aU2 = up2 ? a2 : INF;
  f.bU2 = up2 ? qb.z : 0.f;
  f.aL0 = __fmaf_rn(qg.w, cf, qa.w);
  f.bL0 = qb.w;
  f.aL1 = up1 ? -INF : a1;
  f.bL1 = up1 ? 0.f : qb.y;
  f.aL2 = up2 ? -INF : a2;
  f.bL2 = up2 ? 0.f : qb.z;
  f.eU = qi.x;
  f.eL = qi.y;
  row_magic<STRICT>(f, (int)(xx & 0xFFFFu), (int)((xx >> 16) & 0x3FFFu));
  // rows of the slab from its first: below 2^32 for every accepted grid
  const uint32_t r0 = ((yz >> 16) + (uint32_t)k) * (uint32_t)p.ry + (yz & 0xFFFFu) + (uint32_t)b0;
  uint32_t *const row = p.out + (size_t)r0 * (uint32_t)p.W - kMagicWord;
  uint32_t off = 0;
  float bf = (float)b0;
  // uncertain rows are collected as bits, 32 rows at a time, and queued after the rows, so
  // that the row loop has no call in it
  for (int s0 = 0; s0 < n; s0 += 32) {
    const int s1 = min(n, s0 + 32);
    uint32_t amb = 0;
    for (int r = s0; r < s1; ++r) {
      uint32_t lo, hi;
      bool live;
      amb |= (uint32_t)row_bounds<STRICT, CLAMP>(f, bf, lo, hi, live) << (r - s0);
      row_or(row, off, lo, hi, live);
      bf += 1.f;
      off += (uint32_t)p.W;
    }
    while (amb) {
      const int j = __ffs(amb) - 1;
      amb &= amb - 1u;
      queue_row_staged(p, sm.stage, t, b0 + s0 + j, k);
    }
  }
}

template <bool STRICT, bool CULL, bool CLAMP, bool STRIDED, int SL>
__global__ void __launch_bounds__(kSuBlock, SL == kSuSlicesSmall ? 7 : 5) k_slices(Params p) {
  chain_wait();  // vertices snapped, header zeroed
  chain_release();
  extern __shared__ __align__(16) unsigned char su_dyn_smem[];
  SuSmem<SL> &sm = *reinterpret_cast<SuSmem<SL> *>(su_dyn_smem);
  const int tid = threadIdx.x;
  TileCounters ctr;
  for (int i = tid; i < kSuCounters; i += kSuBlock) sm.hist[i] = 0u;
  if (tid == 0) sm.stage.n = 0;
  for (;;) {
    if (tid == 0) sm.tile = (long long)atomicAdd(&p.hdr->tile_counter, 1ull);
    __syncthreads();
    const long long tile = sm.tile;
    long long base, t;
    if (STRIDED) {  // slab launches: tile k holds tets k + j * tile_stride
      if (tile >= p.tile_stride) break;
      base = tile;
      t = base + (long long)tid * p.tile_stride;
    } else {
      base = tile * kSuBlock;
      if (base >= p.n_tets) break;
      t = base + tid;
    }
    if (t >= p.n_tets) t = -1;
    // (1) set up this thread's tet and its slices' row ranges; count units per counter
    const int nc = su_setup<STRICT, CULL, SL>(p, t, sm, ctr);
    __syncthreads();
    // (2) exclusive scan of the counters (two per thread) into cursors, then every unit to
    // its place (a cursor per counter: units of one counter come from one warp)
    {
      const uint32_t c0 = sm.hist[2 * tid], c1 = sm.hist[2 * tid + 1];
      uint32_t all = 0;
      const uint32_t before = su_block_scan(sm, c0 + c1, all);
      sm.hist[2 * tid] = before;
      sm.hist[2 * tid + 1] = before + c0;
      if (tid == 0) sm.total = all;
      __syncthreads();
    }
    const uint32_t total = sm.total;
#pragma unroll 4
    for (int k = 0; k < nc; ++k) {
      const uint32_t e = sm.slice[k][tid];
      if (e == kSuEmpty) continue;
      const int n = (int)(e >> 10) + 1;
      const uint32_t pos = atomicAdd(&sm.hist[su_counter(n, tid >> 5)], 1u);
      sm.unit[pos] = (uint32_t)tid | ((uint32_t)k << 7) | (e << 12);
    }
    __syncthreads();
    if (tid == 0) ctr.spans += total;
    sm.hist[2 * tid] = 0u;  // ready for the next tile's counts (a barrier comes before them)
    sm.hist[2 * tid + 1] = 0u;
    // (3) walk the units, longest first; a warp takes 32 neighbouring units of the order
    for (uint32_t i = tid; i < total; i += kSuBlock) {
      const uint32_t u = sm.unit[i];
      const int slot = (int)(u & 127u), k = (int)((u >> 7) & 31u);
      const int b0 = (int)((u >> 12) & 1023u), n = (int)(u >> 22) + 1;
      const long long tt = STRIDED ? base + (long long)slot * p.tile_stride : base + slot;
      ctr.rows += (unsigned)n;
      su_walk<STRICT, CLAMP, SL>(p, sm, slot, tt, k, b0, n);
    }
    flush_stage(p, sm.stage);
  }
  flush_counters(p.hdr, ctr);
}

// ------------------------------------------------------------------ host side

typedef void (*SuKernel)(Params);

template <int SL>
static SuKernel su_kernel(int v) {
  switch (v) {
    case 0: return k_slices<false, false, false, false, SL>;
    case 1: return k_slices<false, false, true, false, SL>;
    case 2: return k_slices<false, true, false, false, SL>;
    case 3: return k_slices<false, true, true, false, SL>;
    case 4: return k_slices<true, false, false, false, SL>;
    case 5: return k_slices<true, false, true, false, SL>;
    case 6: return k_slices<true, true, false, false, SL>;
    case 7: return k_slices<true, true, true, false, SL>;
    case 8: return k_slices<false, false, false, true, SL>;
    case 9: return k_slices<false, false, true, true, SL>;
    case 10: return k_slices<false, true, false, true, SL>;
    case 11: return k_slices<false, true, true, true, SL>;
    case 12: return k_slices<true, false, false, true, SL>;
    case 13: return k_slices<true, false, true, true, SL>;
    case 14: return k_slices<true, true, false, true, SL>;
    default: return k_slices<true, true, true, true, SL>;
  }
}

constexpr int kSuMaxDevices = 64;
static int g_su_occ[kSuMaxDevices][2][16];  // resident blocks per SM per capacity and variant, 0 = not yet queried
static std::atomic<int> g_su_lock{0};

size_t slices_smem_bytes(int slices) {
  return slices <= kSuSlicesSmall ? sizeof(SuSmem<kSuSlicesSmall>) : sizeof(SuSmem<kSuSlices>);
}

int launch_slices(const Params &p_in, int variant, int slices, int sms, cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kSuMaxDevices) return VOXTET_ERR_CUDA;
  const int c = slices <= kSuSlicesSmall ? 0 : 1;
  SuKernel kern = c == 0 ? su_kernel<kSuSlicesSmall>(variant & 15) : su_kernel<kSuSlices>(variant & 15);
  const size_t smem = slices_smem_bytes(slices);
  int occ = g_su_occ[dev][c][variant & 15];
  if (occ == 0) {
    while (g_su_lock.exchange(1)) {
    }
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(kern),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kSuBlock, smem);
    if (e == cudaSuccess && occ < 1) occ = 1;
    if (e == cudaSuccess) g_su_occ[dev][c][variant & 15] = occ;
    g_su_lock.store(0);
    if (e != cudaSuccess) return VOXTET_ERR_CUDA;
  }
  Params p = p_in;
  const bool strided = (variant & 8) != 0;
  long long grid = (long long)sms * occ;
  long long tiles = (p.n_tets + kSuBlock - 1) / kSuBlock;
  p.tile_stride = 0;
  if (strided) {  // at least one tile per resident block (see the span kernel's slab launches)
    long long stride = tiles;
    if (stride < grid) stride = p.n_tets < grid ? p.n_tets : grid;
    p.tile_stride = stride;
    tiles = stride;
  }
  if (grid > tiles) grid = tiles;
  if (grid < 1) grid = 1;
  return launch_chained(kern, (unsigned)grid, kSuBlock, smem, stream, p) == cudaSuccess ? VOXTET_OK : VOXTET_ERR_CUDA;
}

}  // namespace voxtet
