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
// Where a mesh has too few tets for a thread each to fill the chip, or tets of more slices than a
// thread takes, a group of 2^lg threads shares a tet and its slices (su_group_log2); slices or rows
// past that are taken in further windows of the same tile, by the tets that have them.  A batch's jobs run in one launch
// (k_slices_batched), a thin slab's tets from a list (LIST).
// What bounds it: instruction issue and, on finer grids, the rate at which ORs reach L2, half of
// them across the dies.  Measured on GB300, 1.3 M-tet sliver mesh: 257 us a call at 512^3, 990 at
// 1024^3 (rows ORed in pairs of words).  Timing-only copies of a form that ORed single words at both
// sizes: at 512^3 261 us a call, of these 65 for the ORs, 100 for the rest of the rows, 45 for the
// slices' row ranges and the sort, 40 for load, classification and face data; at 1024^3 1020 us, 505
// for the ORs (213 M of them) and 360 for the rest of the rows.  ORing a tile's rows in shared memory
// first and the words once into the grid took 9 times fewer ORs but a sixth more instructions (302 and
// 1100 us).
// Tets wider than 2^20 lattice units (or all, use_filter = 0) go to the exact kernel, zero-volume
// ones are counted; rows the filter cannot certify go to the row queue, as in the span kernel.
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>

#include "voxtet.h"
#include "tet_math.cuh"
#include "voxtet_device.cuh"
#include "voxtet_rows.cuh"
#include "voxtet_slices.cuh"

namespace voxtet {

constexpr int kSuWarps = kSuBlock / 32;
constexpr int kSuBuckets = 64;                           // row counts 1..63 one bucket each, >= 64 together
constexpr int kSuCounters = kSuBuckets * kSuWarps;       // bucket-major, one counter per warp of each bucket
constexpr int kSuRec = 20;  // floats per tet record: 5 groups of 16 bytes, an odd number, so that
                            // lanes loading records of random slots spread over all banks
constexpr int kSuStage = 64;                             // staged uncertain rows per block (about 5 per tile)
constexpr uint32_t kSuEmpty = 0xFFFFFFFFu;               // a slice without candidate rows
static_assert(kSuBlock == 128 && kSuSlices <= 32 && kSuRows == 1024, "unit fields: 7 + 5 bits; rows in 10 bits");

// Tet record (kSuRec words per slot): alpha' of the four faces | beta | gamma | E of the upper
// side (sign bit: slot 1 is an upper face) and of the lower side (sign bit: slot 2 is an upper
// face), i0 | (na - 1) << 16, j0 | (l0 - z0) << 16 | the four faces' E.  Upper faces fill the slots from the
// front and lower faces from the back; a face parallel to x leaves a neutral upper slot (alpha' =
// +infinity) between them.  Slot 0 is always an upper face and slot 3 a lower one.
constexpr int kRecB = 4, kRecG = 8, kRecEU = 12, kRecEL = 13, kRecX = 14, kRecYZ = 15, kRecE = 16;

// Shared memory of one block (dynamic), for tets of at most SL slices.
template <int SL>
struct SuSmem {
  float rec[kSuBlock * kSuRec];
  // per tet slot, slice k of its tet: b_lo | (n - 1) << 10, or kSuEmpty
  uint32_t slice[SL][kSuBlock];
  // the tile's units sorted by row count, longest first: slot | k << 7 | b_lo << 12 | (n - 1) << 22
  uint32_t unit[kSuBlock * SL];
  uint32_t hist[kSuCounters];  // unit counts, then (after the scan) cursors
  uint32_t warp_tot[kSuWarps];
  RowStageN<kSuStage> stage;
  long long tile;
  int c0, r0;            // the current window: slices from c0, rows from r0 of each tet's box
  int next_c0, next_r0;  // the window after it (0, 0: the tile is done)
  // the current window's tets, 2^lg threads each: all tile_tets of the tile (n_sel = 0, lg = tile_lg) or the
  // n_sel at places place[buf] of it; those of the next window are collected in the other list.
  // (Read from here where they are used: held across the phases they cost the row loop registers.)
  int lg, tile_lg, tile_tets, n_sel, n_next, buf;
  uint8_t place[2][kSuBlock];
  // the block's counters but for the rows, since the last flush
  unsigned long long spans;
  unsigned degenerate, wide;
  int err;
};

// 16-slice tiles fit 7 blocks per SM (228 KB, 1 KB reserved per block), 32-slice tiles 5
static_assert(sizeof(SuSmem<kSuSlicesSmall>) <= 31 * 1024, "slice-unit kernel shared memory: seven blocks per SM");
static_assert(sizeof(SuSmem<kSuSlices>) <= 44 * 1024 + 512, "slice-unit kernel shared memory: five blocks per SM");

// Counter of a unit with n rows emitted by warp w: longer units first.
__device__ __forceinline__ int su_counter(int n, int w) {
  return (kSuBuckets - min(n, kSuBuckets)) * kSuWarps + w;
}

// Phase (1) for tet t of this thread's group (t < 0: none).  The group's 2^lg threads each set
// the tet up and take its slices c0 + sub, c0 + sub + 2^lg, ... (sub = the thread within its
// group), at most SL of them: a window of SL 2^lg slices from c0.  Returns the entries it wrote
// to sm.slice (0 if none); counts each unit in its counter (no rank is needed here, so the
// count does not wait on the shared-memory atomic).  `more` is set if the tet has slices past
// the window; a window also covers at most kSuRows rows per slice, from row r0 of the box, and
// `tall` is set if the tet's box has rows past it (both alike for all threads of a group).  A tet is
// counted (or queued) once, by its group's first thread in its first window; zero-volume and wide
// tets and errors, all rare, in shared memory, so that the counters take no registers.
template <bool STRICT, bool CULL, bool TALL, int SL>
__device__ __forceinline__ int su_setup(const Params &p, long long t, SuSmem<SL> &sm, bool &more, bool &tall) {
  const int tid = threadIdx.x, warp = tid >> 5;
  if (t < 0) return 0;
  const int lg = sm.lg;
  const bool first = ((tid & ((1 << lg) - 1)) | sm.c0 | (TALL ? sm.r0 : 0)) == 0;
  int3 V[4];
  {
    int err = 0;
    const bool valid = load_tet(p, t, V, err);
    if (err) atomicOr(&sm.err, err);
    if (!valid) return 0;
  }
  Box bx;
  const int E = tet_box(V, p.sh, p.rx, p.ry, p.z0, p.z1, bx);
  const bool empty = bx.na <= 0 || bx.nb <= 0 || bx.nc <= 0;
  if (E > kNarrowExtent) {  // wider than 2^20 lattice units: 128-bit sign, exact kernel
    if (!first) return 0;
    if (v6_sign(V, E) == 0) {
      atomicAdd(&sm.degenerate, 1u);
      return 0;
    }
    if (empty) return 0;
    atomicAdd(&sm.wide, 1u);
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
    if (first) atomicAdd(&sm.degenerate, 1u);
    return 0;
  }
  if (empty) return 0;
  if (p.exact_all || bx.nb > kMaxFilterRows) {
    if (!first) return 0;
    const unsigned k = atomicAdd(&p.hdr->tetq_count, 1u);
    p.tetq[k] = (uint32_t)t;
    return 0;
  }
  tall = TALL && bx.nb > sm.r0 + kSuRows;
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
      rec[kRecE + o] = e;
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
    rec[kRecE + cu] = 0.f;
  }
  rec[kRecEU] = __int_as_float(__float_as_int(eU) | (cu >= 2 ? (int)0x80000000 : 0));
  rec[kRecEL] = __int_as_float(__float_as_int(eL) | (cu >= 3 ? (int)0x80000000 : 0));
  rec[kRecX] = __uint_as_float((uint32_t)bx.i0 | ((uint32_t)(bx.na - 1) << 16));
  rec[kRecYZ] = __uint_as_float((uint32_t)bx.j0 | ((uint32_t)(bx.l0 - p.z0) << 16));
  // Candidate rows of each slice: the cross-section's y-extent (a superset of the rows with
  // samples), narrowed exactly by the faces parallel to x.  Each unit is counted (no rank is
  // needed here, so the count does not wait on the shared-memory atomic).
  RowRange R;
  if (CULL) {
    row_range(V, bx, p.sh, R);
  } else {
    R.kL0 = R.kL1 = R.kU0 = R.kU1 = R.z0 = R.z1 = 0.f;
    R.aL0 = R.aL1 = 0.f;
    R.aU0 = R.aU1 = fb;
  }
  const int c0 = sm.c0, r0 = TALL ? sm.r0 : 0;
  const int sub = tid & ((1 << lg) - 1);
  const float row0 = (float)r0, row1 = TALL ? fminf(fb, (float)(r0 + kSuRows - 1)) : fb;
  const uint32_t row0_bits = kMagicBits + (uint32_t)r0;
  const int step = 1 << lg, k_end = min(bx.nc, c0 + (SL << lg));
  more = bx.nc > k_end;
  int units = 0, kk = 0;
  float cf = (float)(c0 + sub);
  const float cstep = (float)step;
  for (int k = c0 + sub; k < k_end; k += step, cf += cstep, ++kk) {
    float flo, fhi;
    slice_range(R, cf, row0, row1, flo, fhi);
    bool any = flo <= fhi;
    uint32_t b_lo = __float_as_uint(flo) - row0_bits, n1 = __float_as_uint(fhi) - __float_as_uint(flo);
    if (nz > 0 && any) {
      int lo = (int)b_lo + r0, hi = lo + (int)n1;
      narrow_by_row_constraint<STRICT>(zL0 + zDz0 * (i64)k, zDy0, lo, hi);
      if (nz > 1) narrow_by_row_constraint<STRICT>(zL1 + zDz1 * (i64)k, zDy1, lo, hi);
      any = lo <= hi;
      b_lo = (uint32_t)(lo - r0);
      n1 = (uint32_t)(hi - lo);
    }
    if (any) {
      atomicAdd(&sm.hist[su_counter((int)n1 + 1, warp)], 1u);
      ++units;
    }
    sm.slice[kk][tid] = any ? b_lo | (n1 << 10) : kSuEmpty;
  }
  return units ? kk : 0;
}

// Block-wide exclusive prefix sum of one value per thread (all threads call it); `total`
// gets the sum.  Uses sm.warp_tot, which no thread may write again before the next barrier.
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
  return before;
}

// The tet at place i of a launch (below `end`, else -1): tet i, or the i-th listed one.
template <bool LIST>
__device__ __forceinline__ long long su_tet(const Params &p, long long i, long long end) {
  if (i >= end) return -1;
  return LIST ? (long long)p.tetq[p.n_tets - 1 - i] : i;
}

// Place in the tile of the tet whose threads in the current window include `slot`.
template <int SL>
__device__ __forceinline__ int su_place(const SuSmem<SL> &sm, int slot) {
  const int g = slot >> sm.lg;
  return sm.n_sel ? (int)sm.place[sm.buf][g] : g;
}

// ... and in the launch.
template <int SL>
__device__ __forceinline__ long long su_launch_place(const SuSmem<SL> &sm, int slot) {
  return sm.tile * sm.tile_tets + su_place(sm, slot);
}

// Phase (3): rows b0 .. b0 + n - 1 of slice k of the tet in `slot`.
template <bool STRICT, bool PAIRS, bool LIST, bool BATCH, int SL>
__device__ __forceinline__ void su_walk(const Params &p, SuSmem<SL> &sm, int slot, int k, int b0, int n) {
  const float4 *R = reinterpret_cast<const float4 *>(sm.rec + slot * kSuRec);
  const float4 qa = R[0], qb = R[1], qg = R[2], qi = R[3];
  const float cf = (float)k, INF = __int_as_float(0x7f800000);
  const uint32_t xx = __float_as_uint(qi.z), yz = __float_as_uint(qi.w);
  const bool up1 = __float_as_int(qi.x) < 0, up2 = __float_as_int(qi.y) < 0;
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
  f.eU = fabsf(qi.x);
  f.eL = fabsf(qi.y);
  row_magic<STRICT>(f, (int)(xx & 0xFFFFu), (int)(xx >> 16));
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
    const float b_end = bf + (float)(s1 - s0);
#pragma unroll 1
    do {
      uint32_t lo, hi;
      bool live;
      bool a = row_bounds<STRICT>(f, bf, lo, hi, live);
      if (a) {
        a = row_refine<STRICT>(f, R[kRecE / 4], up1, up2, bf);
        live = !a && __uint_as_float(lo) <= __uint_as_float(hi);
      }
      amb = amb + amb + (a ? 1u : 0u);  // the last row in the lowest bit
      if (PAIRS) row_or_pairs(row, off, lo, hi, live);
      else row_or<BATCH>(row, off, lo, hi, live);
      bf += 1.f;
      off += (uint32_t)p.W;
    } while (bf != b_end);
    while (amb) {
      const int j = __ffs(amb) - 1;
      amb &= amb - 1u;
      queue_row_staged(p, sm.stage, su_tet<LIST>(p, su_launch_place(sm, slot), p.n_tets), b0 + s1 - 1 - j, k);
    }
  }
}

// Phases (1)-(3) of one window of tile sm.tile.  The first window holds its kSuBlock >> tile_lg tets
// (those at places below `end`), 2^tile_lg threads each; a further one the tets with slices or rows
// past the window before, by as many threads each as there are for them.  (A few wide tets among many
// small ones would else leave most of the block idle in window after window, with all tets set up
// again in each: 20 tets of 300-500 slices next to each other in a 663,000-tet mesh at 512^3 1726 ->
// 1145 us, 20 such tets spread over it 725 -> 332.)
// All threads of the block call it, in step; if it returns true, su_next_window is to be asked before
// another tile is claimed.  The caller's loop claims a tile or moves to the tile's next window: a loop
// of its own around these phases cost the row loop its reconvergence (measured on GB300, sliver mesh
// at 512^3: 26.7 -> 15.9 active lanes, 262 -> 440 us).
template <bool STRICT, bool CULL, bool PAIRS, bool TALL, bool LIST, bool BATCH, int SL>
__device__ __forceinline__ bool su_pass(const Params &p, long long end, SuSmem<SL> &sm, unsigned &rows) {
  const int tid = threadIdx.x;
  // (1) set up this thread's tet and its slices' row ranges; count units per counter
  bool more = false, tall = false;
  const int n_sel = sm.n_sel, lg = sm.lg;
  int g = tid >> lg;
  const bool any = g < (n_sel ? n_sel : sm.tile_tets);
  if (n_sel && any) g = sm.place[sm.buf][g];
  const long long t = any ? su_tet<LIST>(p, sm.tile * sm.tile_tets + g, end) : -1;
  const int nc = su_setup<STRICT, CULL, TALL, SL>(p, t, sm, more, tall);
  bool again;
  {
    const bool any_more = __syncthreads_or(more);
    const bool any_tall = TALL && p.ry > kSuRows && __syncthreads_or(tall);
    again = any_more || any_tall || n_sel;
    if ((more || tall) && (tid & ((1 << sm.lg) - 1)) == 0)
      sm.place[sm.buf ^ 1][atomicAdd(&sm.n_next, 1)] = (uint8_t)su_place(sm, tid);
    if (tid == 0) {
      sm.stage.n = 0;  // flushed by the previous window; every thread has passed a barrier since
      // every slice of these rows first, then the next rows
      sm.next_c0 = any_more ? sm.c0 + (SL << sm.lg) : 0;
      if (TALL) sm.next_r0 = any_more ? sm.r0 : any_tall ? sm.r0 + kSuRows : 0;
    }
  }
  // (2) exclusive scan of the counters (two per thread) into cursors, then every unit to
  // its place (a cursor per counter: units of one counter come from one warp)
  const uint32_t h0 = sm.hist[2 * tid], h1 = sm.hist[2 * tid + 1];
  uint32_t total = 0;
  const uint32_t before = su_block_scan(sm, h0 + h1, total);
  sm.hist[2 * tid] = before;
  sm.hist[2 * tid + 1] = before + h0;
  __syncthreads();
#pragma unroll 4
  for (int k = 0; k < nc; ++k) {
    const uint32_t e = sm.slice[k][tid];
    if (e == kSuEmpty) continue;
    const int n = (int)(e >> 10) + 1;
    const uint32_t pos = atomicAdd(&sm.hist[su_counter(n, tid >> 5)], 1u);
    sm.unit[pos] = (uint32_t)tid | ((uint32_t)k << 7) | (e << 12);
  }
  __syncthreads();
  if (tid == 0) sm.spans += total;
  sm.hist[2 * tid] = 0u;  // ready for the next tile's counts (a barrier comes before them)
  sm.hist[2 * tid + 1] = 0u;
  // (3) walk the units, longest first; a warp takes 32 neighbouring units of the order
  const int c0 = sm.c0, r0 = TALL ? sm.r0 : 0;
  for (uint32_t i = tid; i < total; i += kSuBlock) {
    const uint32_t u = sm.unit[i];
    const int slot = (int)(u & 127u);
    const int k = c0 + ((int)((u >> 7) & 31u) << lg) + (slot & ((1 << lg) - 1));
    const int b0 = (int)((u >> 12) & 1023u) + r0, n = (int)(u >> 22) + 1;
    rows += (unsigned)n;
    su_walk<STRICT, PAIRS, LIST, BATCH, SL>(p, sm, slot, k, b0, n);
  }
  flush_stage(p, sm.stage);
  return again;
}

// The block's first thread moves to the tile's next window, after su_pass returned true; true if the
// tile is done.
template <int SL>
__device__ __forceinline__ bool su_next_window(SuSmem<SL> &sm) {
  const int n = sm.n_next;  // 0: the tile is done
  sm.c0 = sm.next_c0;
  sm.r0 = sm.next_r0;
  sm.n_sel = n;
  sm.n_next = 0;
  sm.buf ^= 1;
  sm.lg = n ? __clz(n - 1) - (32 - kSuMaxGroup) : sm.tile_lg;  // the most with n << lg <= kSuBlock
  return n == 0;
}

template <int SL>
__device__ __forceinline__ void su_begin(SuSmem<SL> &sm, int tile_lg, int tile_tets) {
  for (int i = threadIdx.x; i < kSuCounters; i += kSuBlock) sm.hist[i] = 0u;
  if (threadIdx.x == 0) {
    sm.stage.n = 0;
    sm.c0 = sm.r0 = sm.next_c0 = sm.next_r0 = 0;
    sm.n_sel = sm.n_next = sm.buf = 0;
    sm.lg = sm.tile_lg = tile_lg;
    sm.tile_tets = tile_tets;
    sm.spans = 0;
    sm.degenerate = sm.wide = 0u;
    sm.err = 0;
  }
}

// Adds the block's counters to a mesh's header (and its error bits to `status`) and resets them.  All
// threads call it, a barrier after the counted work and one before the next.
template <int SL>
__device__ __forceinline__ void su_flush(Header *hdr, SuSmem<SL> &sm, unsigned &rows, int *status = nullptr) {
  unsigned long long sum = rows;
  rows = 0;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, d);
  if ((threadIdx.x & 31) == 0 && sum) atomicAdd(&hdr->rows, sum);
  if (threadIdx.x == 0) {
    if (sm.spans) atomicAdd(&hdr->spans, sm.spans);
    if (sm.degenerate) atomicAdd(&hdr->degenerate, (unsigned long long)sm.degenerate);
    if (sm.wide) atomicAdd(&hdr->wide, (unsigned long long)sm.wide);
    if (sm.err) {
      atomicOr(&hdr->status_bits, sm.err);
      if (status) atomicOr(status, sm.err);
    }
    sm.spans = 0;
    sm.degenerate = sm.wide = 0u;
    sm.err = 0;
  }
}

// Should twice as many threads share a tet as 2^lg, for tiles of about even work over `blocks`
// resident blocks: `tiles` now, `rows` a tet.  Every thread repeats the tet's setup, about 10 rows'
// worth: up to four tiles a block while that adds less than a fifth.  Measured on GB300: a 4096^3
// torus of 198,529 tets in slabs of 64 slices 5.41, 4.59, 4.27 and 4.28 ms with 4, 8, 16 and 32 threads
// a tet (875 to 7000 tiles for 760 blocks); 196,608 tets at 512^3 144 -> 133 us with two; but a
// 30-slice slab of about 50 rows a tet 56 -> 61 us with two.
static __host__ __device__ __forceinline__ bool su_share_more(long long tiles, long long blocks, float rows, int lg) {
  return tiles < 4 * blocks && 50.0f * (float)((2 << lg) - 1) < rows;
}

// Tets per tile where a slab of few slices leaves its tets to few threads each: as many as give each of
// `blocks` blocks a tile, if that is fewer than a tile's threads have room for.  (Full tiles put a few
// coarse tets, each with hundreds of rows of many words, on a few of the SMs: 384 tets in one slice of a
// 2048^3 grid 191 -> 136 us, 3,072 in one of 512^3 28.7 -> 25.0; spans 159 and 26.9.)
static __host__ __device__ __forceinline__ int su_tile_tets(long long tets, int lg, long long blocks) {
  const long long room = kSuBlock >> lg, even = (tets + blocks - 1) / blocks;
  return (int)(even < 1 ? 1 : even < room ? even : room);
}

// LIST: the tets are the hdr->listq_count ones listed at the back of p.tetq.  PAIRS: rows are ORed in
// pairs of words.
template <bool STRICT, bool CULL, bool PAIRS, bool LIST, int SL>
__global__ void __launch_bounds__(kSuBlock, SL == kSuSlicesSmall ? 7 : 5) k_slices(Params p) {
  chain_wait();  // vertices snapped, header zeroed, tets listed
  chain_release();
  extern __shared__ __align__(16) unsigned char su_dyn_smem[];
  SuSmem<SL> &sm = *reinterpret_cast<SuSmem<SL> *>(su_dyn_smem);
  unsigned rows = 0;
  const long long end = LIST ? (long long)p.hdr->listq_count : p.n_tets;
  int lg = p.lg;
  if (LIST && end > 0) {  // as su_group_log2, with the slab's tets counted and their slices and rows added up
    const float slab = (float)(p.z1 - p.z0), per_tet = 0.5f * (float)p.hdr->list_rows / (float)end;
    const float slices = (float)p.hdr->list_slices / (float)end;
    while (lg < kSuMaxGroup && (float)(SL << lg) < slices) ++lg;
    while (lg < kSuMaxGroup && (float)(1 << lg) < slab &&
           (((end << lg) / kSuBlock) * 2 < (long long)gridDim.x ||
            su_share_more((end << lg) / kSuBlock, (long long)gridDim.x, per_tet, lg)))
      ++lg;
  }
  su_begin(sm, lg, LIST ? su_tile_tets(end, lg, (long long)gridDim.x) : p.tile_tets);
  bool again = false;
  for (;;) {
    if (threadIdx.x == 0 && (!again || su_next_window(sm))) sm.tile = (long long)atomicAdd(&p.hdr->tile_counter, 1ull);
    __syncthreads();
    if (sm.tile * sm.tile_tets >= end) break;
    again = su_pass<STRICT, CULL, PAIRS, SL == kSuSlices, LIST, false, SL>(p, end, sm, rows);
  }
  su_flush(p.hdr, sm, rows);
}

// The tiles of every job of a batch, claimed from one counter bh->chunk at a time; a claim's job is
// found in the per-job tile offsets by one warp.  A job's device-detected errors also go to its
// status word.
template <bool STRICT, bool CULL>
__global__ void __launch_bounds__(kSuBlock, 7) k_slices_batched(BatchHeader *bh, const JobDesc *jobs,
                                                               const unsigned long long *tile_base, int *status) {
  chain_wait();  // vertices snapped, headers and grids zeroed
  chain_release();
  constexpr int SL = kSuSlicesSmall;
  extern __shared__ __align__(16) unsigned char su_dyn_smem[];
  SuSmem<SL> &sm = *reinterpret_cast<SuSmem<SL> *>(su_dyn_smem);
  __shared__ Params sp;
  __shared__ int job_s;
  // the current tile, the claim's end, and the current job's first tile and the one after its last
  __shared__ unsigned long long at, claim_end, job_first, job_end;
  const int tid = threadIdx.x;
  unsigned rows = 0;
  su_begin(sm, 0, kSuBlock);
  const int n = bh->n_jobs;
  const unsigned long long total = bh->total_tiles, chunk = bh->chunk;
  int cur = -1;
  bool again = false;
  if (tid == 0) {
    at = claim_end = job_first = job_end = 0;
    job_s = -1;
  }
  for (;;) {
    if (tid < 32) {
      unsigned long long tile = 0;
      int search = 0;
      if (tid == 0 && (!again || su_next_window(sm))) {
        if (++at >= claim_end) {
          at = atomicAdd(&bh->tile_counter, chunk);
          claim_end = at + chunk;
        }
        tile = at;
        if (tile >= total) job_s = -1;
        else search = 1 + (job_s >= 0 && tile < job_end && tile >= job_first);
        if (search == 2) sm.tile = (long long)(tile - job_first);
      }
      search = __shfl_sync(0xFFFFFFFFu, search, 0);
      if (search == 1) {
        tile = __shfl_sync(0xFFFFFFFFu, tile, 0);
        const int j = find_job_warp(tile_base, n, tile);
        if (tid == 0) {
          job_s = j;
          job_first = tile_base[j];
          job_end = tile_base[j + 1];
          sm.tile = (long long)(tile - job_first);
        }
      }
    }
    __syncthreads();
    const int j = job_s;
    if (j < 0) break;
    if (j != cur) {  // a new job: flush the previous job's counters, load its Params
      if (cur >= 0) su_flush(sp.hdr, sm, rows, status + cur);
      __syncthreads();
      if (tid < (int)(sizeof(Params) / sizeof(uint32_t)))
        reinterpret_cast<uint32_t *>(&sp)[tid] = reinterpret_cast<const uint32_t *>(&jobs[j].p)[tid];
      if (tid == 0) {  // a new job's tile is at its first window
        sm.lg = sm.tile_lg = jobs[j].p.lg;
        sm.tile_tets = jobs[j].p.tile_tets;
      }
      __syncthreads();
      cur = j;
    }
    again = su_pass<STRICT, CULL, false, true, false, true, SL>(sp, sp.n_tets, sm, rows);
  }
  if (cur >= 0) su_flush(sp.hdr, sm, rows, status + cur);
}

// ------------------------------------------------------------------ host side

typedef void (*SuKernel)(Params);

// Variant (list << 2) | (strict << 1) | cull.
template <bool PAIRS, int SL>
static SuKernel su_kernel(int v) {
  switch (v) {
    case 0: return k_slices<false, false, PAIRS, false, SL>;
    case 1: return k_slices<false, true, PAIRS, false, SL>;
    case 2: return k_slices<true, false, PAIRS, false, SL>;
    case 3: return k_slices<true, true, PAIRS, false, SL>;
    case 4: return k_slices<false, false, PAIRS, true, SL>;
    case 5: return k_slices<false, true, PAIRS, true, SL>;
    case 6: return k_slices<true, false, PAIRS, true, SL>;
    default: return k_slices<true, true, PAIRS, true, SL>;
  }
}

constexpr int kSuMaxDevices = 64;
static int g_su_occ[kSuMaxDevices][3][8];  // resident blocks per SM per form and variant, 0 = not yet queried
static std::atomic<int> g_su_lock{0};

size_t slices_smem_bytes(int slices) {
  return slices <= kSuSlicesSmall ? sizeof(SuSmem<kSuSlicesSmall>) : sizeof(SuSmem<kSuSlices>);
}

int su_group_log2(long long n_tets, int side, int ry, int slab, int slices, long long blocks) {
  if (n_tets < 1) return 0;
  const double cells = std::cbrt((double)n_tets / 6.0);
  const double w = (double)side / cells, span = w < slab ? w : slab;  // slices a tet spans, about
  int lg = 0;
  while (lg < kSuMaxGroup && (double)(slices << lg) < span) ++lg;
  while (lg < kSuMaxGroup && (double)(1 << lg) < span && ((n_tets << lg) / kSuBlock) * 2 < blocks) ++lg;
  // a guess of the rows, too high for a mesh that fills only part of its grid: it counts for half,
  // and for up to two tiles a block
  const float rows = (float)(0.25 * (double)ry / cells * span);
  while (lg < kSuMaxGroup && (double)(1 << lg) < span && su_share_more(2 * ((n_tets << lg) / kSuBlock), blocks, rows, lg))
    ++lg;
  return lg;
}

typedef void (*SuBatchKernel)(BatchHeader *, const JobDesc *, const unsigned long long *, int *);

static SuBatchKernel su_batch_kernel(bool strict, bool cull) {
  if (strict) return cull ? k_slices_batched<true, true> : k_slices_batched<true, false>;
  return cull ? k_slices_batched<false, true> : k_slices_batched<false, false>;
}

static int g_su_batch_occ[kSuMaxDevices][4];

int slices_batched_blocks(bool strict, bool cull) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kSuMaxDevices) return 0;
  int &slot = g_su_batch_occ[dev][(strict ? 2 : 0) | (cull ? 1 : 0)];
  if (slot == 0) {
    while (g_su_lock.exchange(1)) {
    }
    const SuBatchKernel kern = su_batch_kernel(strict, cull);
    const size_t smem = slices_smem_bytes(kSuSlicesSmall);
    int occ = 0;
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(kern),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kSuBlock, smem);
    if (e == cudaSuccess) slot = occ > 0 ? occ : 1;
    g_su_lock.store(0);
  }
  return slot;
}

int launch_slices_batched(BatchHeader *bh, const JobDesc *jobs, const unsigned long long *tile_base, int *status,
                          bool strict, bool cull, int sms, cudaStream_t stream) {
  const int occ = slices_batched_blocks(strict, cull);
  if (occ < 1) return VOXTET_ERR_CUDA;
  const cudaError_t e = launch_chained(su_batch_kernel(strict, cull), (unsigned)(sms * occ), kSuBlock,
                                       slices_smem_bytes(kSuSlicesSmall), stream, bh, jobs, tile_base, status);
  return e == cudaSuccess ? VOXTET_OK : VOXTET_ERR_CUDA;
}

int launch_slices(const Params &p_in, int variant, int slices, bool spread, int sms, cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kSuMaxDevices) return VOXTET_ERR_CUDA;
  // Pairs of words where the ORs are the bound (32-slice windows: grids above 512 per side) and every
  // row starts on an 8-byte boundary.  Measured on GB300: sliver mesh at 1024^3 1018 -> 996 us,
  // 162,000 tets at 1024^3 656 -> 606, 1.3 M at 2048^3 4.77 -> 4.40 ms, 4096^3 torus in slabs 4.22 ->
  // 3.89 ms; at 512^3, bound by issue, the longer masks cost more than they save.  They also do where a
  // mesh on a lattice puts the same rows of many tets side by side: 1.3 M tets of 6 x 9 x 15 voxels at
  // 1024^3 543 -> 577 us, of 17 x 17 x 17 839 -> 981.
  const int c = slices <= kSuSlicesSmall ? 0 : (p_in.W & 1) != 0 || (reinterpret_cast<uintptr_t>(p_in.out) & 7) != 0 ? 1 : 2;
  const SuKernel kern = c == 0   ? su_kernel<false, kSuSlicesSmall>(variant & 7)
                        : c == 1 ? su_kernel<false, kSuSlices>(variant & 7)
                                 : su_kernel<true, kSuSlices>(variant & 7);
  const size_t smem = slices_smem_bytes(slices);
  int occ = g_su_occ[dev][c][variant & 7];
  if (occ == 0) {
    while (g_su_lock.exchange(1)) {
    }
    cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(kern),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kSuBlock, smem);
    if (e == cudaSuccess && occ < 1) occ = 1;
    if (e == cudaSuccess) g_su_occ[dev][c][variant & 7] = occ;
    g_su_lock.store(0);
    if (e != cudaSuccess) return VOXTET_ERR_CUDA;
  }
  Params p = p_in;
  const bool list = (variant & 4) != 0;
  long long grid = (long long)sms * occ;
  // a list's length is known on the device only: the kernel shares its tets among more threads
  const int side = 1 << (kLatticeBits - p.sh);
  p.lg = list ? 0 : su_group_log2(p.n_tets, side, p.ry, p.z1 - p.z0, slices, grid);
  p.tile_tets = spread ? su_tile_tets(p.n_tets, p.lg, grid) : kSuBlock >> p.lg;
  const long long tiles = list ? grid : (p.n_tets + p.tile_tets - 1) / p.tile_tets;
  if (grid > tiles) grid = tiles;
  if (grid < 1) grid = 1;
  return launch_chained(kern, (unsigned)grid, kSuBlock, smem, stream, p) == cudaSuccess ? VOXTET_OK : VOXTET_ERR_CUDA;
}

}  // namespace voxtet
