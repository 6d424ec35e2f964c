// Pair search by tensor-core filter: the warp-level core of the tiled force
// kernels (forces_tiles.cu).
//
// A tile is a set of at most 32 cell-sorted particles from a bundle of
// neighbouring cell rows (ry x rz rows, cut along x where 32 particles are
// full), one per lane of a warp.  The warp
//   1. stages every particle j of the cells that the tile's spheres can reach
//      in shared memory (one copy per tile instead of one load per particle
//      and candidate);
//   2. asks the tensor cores which of them lie near: with coordinates taken
//      about the tile's centre, scaled by a power of two and rounded to FP16,
//      D = |x_j|^2 - 2 x_i x_j + (|x_i|^2 - rc_i^2 - slack) is one
//      m16n8k8 product per 16 x 8 pairs with FP32 accumulation, and the sign
//      bit of D says whether j may be within rc_i.  The slack covers the
//      rounding of the coordinates, so no pair within rc_i is lost; the bits of
//      32 candidates are collected with one funnel shift per pair and handed
//      to the lane that owns i;
//   3. leaves each lane a list of 32-bit masks, over which the caller
//      evaluates the marked pairs exactly (the FP32 or FP64 test r < rc_i and the
//      pair terms see the untouched coordinates).
//
// Why: walking cell rows per particle tests 2.1-2.5 candidates per accepted
// pair at about 32 instructions each, and a warp waits for the fullest window
// of every row (64% of the lanes active).  Here a candidate costs about two
// instructions (one row of the product, one shift, its share of the staging),
// only marked pairs pay for the pair arithmetic (1-2% of them are then rejected),
// and a lane runs through its pairs of all rows without meeting the other
// lanes in between.
//
// Why warp-wide products: the filter's product is private to 32 particles.  A
// tcgen05 product has at least 64 rows for one set of columns (128 to use every
// lane of the tensor memory), so the candidate columns per row would double, and
// the shifts that read the signs, not the products (a ninth of the
// tensor pipe), are what the filter costs.
//
// Periodic images keep the exact arithmetic of the row walk: an image at -L is
// staged as x_j - L; a tile whose cells reach past +L moves its whole frame by
// -L (x_i - L and, inside the box, x_j - L, both exact because the tile and
// everything within its cutoffs lie in the upper half).  A tile that reaches
// past both ends of an axis is left to the per-particle row walk, and so is
// every tile that may meet a coordinate outside the box (or a NaN): binning puts
// such particles into the boundary cells, where the kernel that cuts the tiles
// looks for them and marks their bundles.
#pragma once

#include <cuda_fp16.h>

#include "forces_core.cuh"

namespace dcm {

// Candidates staged at a time (a bulk tile at rc = 3 meets about 640): 16 warps
// of 16-byte positions, or 12 of 32-byte records, fit an SM.
template <typename E>
constexpr int tile_cand() { return sizeof(E) == 16 ? 512 : 384; }
constexpr int kTileEnd = 4;                  // candidates a list may be read past its end

// Shared memory of one warp.  E: what is staged per candidate, a position
// (x, y, z first) with whatever else the caller's pairs need.
template <typename E>
struct TileSmem {
  static constexpr int kCand = tile_cand<E>();
  E pos[kCand + kTileEnd];          // staged candidates; the last ones are far away and never accepted
  uint2 list[kCand / 32 + 2][32];     // per lane: mask of a group, shared address of its first candidate
  uint4 frag[32 * (sizeof(E) == sizeof(float4) ? 1 : 2)];  // the filter's operands of the group at work
};

// Counters of a launch.
enum { kTileFirst = 0, kTileLater = 1, kTileQueue = 2, kTileRest = 3, kTileOutside = 4, kTileCounters = 8 };

// The tiles of a launch (forces_tiles.cu): the slots in use are list[0 ..
// counters[kTileFirst]) and list[nslot - counters[kTileLater] .. nslot) from its
// end, slot s holds particles idx[32 s .. 32 s + 31], rest takes the slots that a
// kernel leaves to the row walk, outside says which bundles' pieces hold a
// coordinate outside the box (counters[kTileOutside]: whether any does).
struct TileTable {
  int32_t *counters, *list, *rest, *outside, *idx;
};
template <typename R>
int tile_cut(dcm_ctx* ctx, const TilePlan& tp, const typename RT<R>::R4* pos, const R* rc, const int32_t* cell_start,
             const Grid<R>& g, TileTable& t, int warps, cudaStream_t st);

// First bit (from the most significant) of a nonzero word.
__device__ __forceinline__ int first_bit(uint32_t w) {
  int b;
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(b) : "r"(w));
  return b;
}

__device__ __forceinline__ uint32_t pack_half(float lo, float hi) {
  uint32_t v;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(hi), "f"(lo));
  return v;
}
__device__ __forceinline__ float2 unpack_half(uint32_t v) {
  return __half22float2(*reinterpret_cast<const __half2*>(&v));
}

__device__ __forceinline__ void mma_16n8k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b, float c0, float c1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, {%7, %7, %8, %8};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(b), "f"(c0), "f"(c1));
}

__device__ __forceinline__ uint32_t shared_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Copy element `at` (of BYTES bytes, counted from dst and src) to shared memory
// if at < n: predicated, with the element's offset in the instruction.
template <int AT, typename E>
__device__ __forceinline__ void copy_if(uint32_t dst, const E* src, int n) {
  constexpr int BYTES = sizeof(E);
  if constexpr (BYTES == 16)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\t@p cp.async.cg.shared.global [%0 + %4], [%1 + %4], 16;\n\t}"
                 ::"r"(dst), "l"(src), "r"(n), "n"(AT), "n"(BYTES * AT)
                 : "memory");
  else
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %2, %3;\n\t@p cp.async.cg.shared.global [%0 + %4], [%1 + %4], 16;\n\t"
                 "@p cp.async.cg.shared.global [%0 + %5], [%1 + %5], 16;\n\t}"
                 ::"r"(dst), "l"(src), "r"(n), "n"(AT), "n"(BYTES * AT), "n"(BYTES * AT + 16)
                 : "memory");
}
// The same for elements whose two halves come from two arrays.
struct HalvesSource {
  const float4 *first, *second;
  __device__ __forceinline__ HalvesSource operator+(int k) const { return {first + k, second + k}; }
};
template <int AT>
__device__ __forceinline__ void copy_if(uint32_t dst, const HalvesSource& src, int n) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %3, %4;\n\t@p cp.async.cg.shared.global [%0 + %5], [%1 + %7], 16;\n\t"
               "@p cp.async.cg.shared.global [%0 + %6], [%2 + %7], 16;\n\t}"
               ::"r"(dst), "l"(src.first), "l"(src.second), "r"(n), "n"(AT), "n"(32 * AT), "n"(32 * AT + 16), "n"(16 * AT)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The filter's view of one tile: the frame (origin and scale) and the operand
// fragments of its 32 rows.  Row g + 8 s belongs to lane 4 g + s, so that a
// quad of lanes holds the fragments of its own particles.
struct TileFilter {
  float s, ox, oy, oz;  // x' = x s + o
  uint32_t a[4];        // rows g, g + 8, g + 16, g + 24: two of the eight k slots
  float c[4];           // |x_i'|^2 - rc_i'^2 - slack of those rows
  float c2[4];          // |x_i'|^2 - slack, for candidates with a cutoff of their own (filter_group2)
  uint32_t wr, rd[4];   // shared addresses: where the lane stores its candidate's operand, and its fragments
};

constexpr float kNever = 120000.f;   // a row's constant where there is no particle: nothing comes near
constexpr float kPadAt = 200.f;      // scaled distance at which the last group is padded (norm 40000)

// Set up the filter for a tile whose lanes hold particles at (x, y, z) (in the
// tile's frame) with cutoffs rc (negative: no particle), the box of the tile's
// particles [lo, hi] and their largest cutoff rmax.
__device__ __forceinline__ void filter_begin(TileFilter& f, uint4* frag, float x, float y, float z, float rc,
                                             const float (&lo)[3], const float (&hi)[3], float rmax, float scale,
                                             float lmax) {
  const int lane = threadIdx.x & 31, t = lane & 3;
  f.s = scale;
  f.ox = -0.5f * (lo[0] + hi[0]) * scale;
  f.oy = -0.5f * (lo[1] + hi[1]) * scale;
  f.oz = -0.5f * (lo[2] + hi[2]) * scale;
  // rounding of the coordinates: at most 2^-11 of their magnitude each, so the
  // distance is off by at most e (with the rounding of FP64 coordinates to
  // FP32); the norms and the sum by a few 2^-22 of q
  float qi = 0.f, qj = 0.f;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float h = 0.5f * (hi[d] - lo[d]) * scale, w = h + rmax * scale;
    qi += h * h;
    qj += w * w;
  }
  const float e = (sqrtf(qi) + sqrtf(qj)) * 0x1.04p-11f + lmax * scale * 0x1p-22f, r = fmaxf(rc, 0.f) * scale;
  const float slack = fmaf(2.f * r, e, e * e) + qj * 0x1p-16f + 0x1p-10f;
  const uint32_t xy = pack_half(fmaf(x, f.s, f.ox), fmaf(y, f.s, f.oy)), zz = pack_half(fmaf(z, f.s, f.oz), 0.f);
  const float2 hxy = unpack_half(xy), hz = unpack_half(zz);
  float ni = fmaf(hxy.x, hxy.x, fmaf(hxy.y, hxy.y, hz.x * hz.x)) - r * r - slack;
  const float nn2 = fmaf(hxy.x, hxy.x, fmaf(hxy.y, hxy.y, hz.x * hz.x)) -
                    (fmaf(2.f * rmax * scale, e, e * e) + qj * 0x1p-16f + 0x1p-10f);
  const bool none = !(rc >= 0.f);
  if (none) ni = kNever;
  const __half2 m2 = __floats2half2_rn(-2.f, -2.f);
  const __half2 axy = __hmul2(*reinterpret_cast<const __half2*>(&xy), m2);
  uint4 w;
  w.x = *reinterpret_cast<const uint32_t*>(&axy);
  w.y = pack_half(-2.f * hz.x, 1.f);
  w.z = pack_half(1.f, 0.f);
  w.w = __float_as_uint(ni);
  __syncwarp();
  frag[lane] = w;
  __syncwarp();
  const uint32_t* q = reinterpret_cast<const uint32_t*>(frag);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int owner = (lane & ~3) + k;
    f.a[k] = t < 3 ? q[owner * 4 + t] : 0u;
    f.c[k] = __uint_as_float(q[owner * 4 + 3]);
    f.c2[k] = __shfl_sync(0xffffffffu, none ? kNever : nn2, owner);
  }
  // candidate 8 t' + 2 k + e of a group is column 2 t' + e of product k, so that
  // the bits arrive in candidate order; the slot order keeps stores and loads
  // free of bank conflicts
  const int kk = (lane >> 1) & 3, nn = 2 * (lane >> 3) + (lane & 1), g = lane >> 2;
  f.wr = shared_addr(frag + 8 * kk + (nn ^ (2 * kk)));
#pragma unroll
  for (int k = 0; k < 4; ++k) f.rd[k] = shared_addr(q + (8 * k + (g ^ (2 * k))) * 4 + t);
}

// The signs of one product of the group's operand (at byte `at` behind the
// first) with the tile's rows: the mask of this lane's particle.
__device__ __forceinline__ uint32_t filter_signs(const TileFilter& f, const float (&c)[4], uint32_t at) {
  const int t = threadIdx.x & 3;
  float d[2][4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    uint32_t b;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b) : "r"(f.rd[k] + at) : "memory");
    mma_16n8k8(d[0][k], f.a[0], f.a[1], b, c[0], c[1]);
    mma_16n8k8(d[1][k], f.a[2], f.a[3], b, c[2], c[3]);
  }
  // the signs of rows g, g + 8 and of rows g + 16, g + 24, in two chains
  uint32_t h[2] = {0u, 0u};
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        h[0] = __funnelshift_l(__float_as_uint(d[0][k][2 * s + e]), h[0], 1);
        h[1] = __funnelshift_l(__float_as_uint(d[1][k][2 * s + e]), h[1], 1);
      }
  uint32_t m = __byte_perm(h[0], h[1], 0x1054);  // bytes of rows g, g + 8, g + 16, g + 24 from the top
  // transpose the 4 x 4 bytes of the quad: lane t keeps row g + 8 t
  uint32_t p = __shfl_xor_sync(0xffffffffu, m, 1);
  m = __byte_perm(m, p, t & 1 ? 0x6240 : 0x3715);
  p = __shfl_xor_sync(0xffffffffu, m, 2);
  return __byte_perm(m, p, t & 2 ? 0x5410 : 0x3276);
}

__device__ __forceinline__ void filter_store(uint32_t at, uint32_t xy, float z, float n) {
  const uint32_t zn = pack_half(z, n), rest = pack_half(n - unpack_half(zn).y, 0.f);
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(xy), "r"(zn), "r"(rest), "r"(0u) : "memory");
}

// One group of 32 candidates, candidate `lane` at (x, y, z): the mask of this
// lane's particle, bit 31 - k for candidate k.  TWO: also the candidates whose own
// cutoff rc reaches the particle, by a second product with |x_j|^2 - rc_j^2.
template <bool TWO>
__device__ __forceinline__ uint32_t filter_group(const TileFilter& f, float x, float y, float z, float rc) {
  const uint32_t xy = pack_half(fmaf(x, f.s, f.ox), fmaf(y, f.s, f.oy)), zz = pack_half(fmaf(z, f.s, f.oz), 0.f);
  const float2 hxy = unpack_half(xy), hz = unpack_half(zz);
  const float n = fmaf(hxy.x, hxy.x, fmaf(hxy.y, hxy.y, hz.x * hz.x));
  __syncwarp();
  filter_store(f.wr, xy, hz.x, n);
  if constexpr (TWO) filter_store(f.wr + 512u, xy, hz.x, n - (rc * f.s) * (rc * f.s));
  __syncwarp();
  uint32_t m = filter_signs(f, f.c, 0u);
  if constexpr (TWO) m |= filter_signs(f, f.c2, 512u);
  return m;
}

// Append a mask and its group's address to a lane's list if any bit is set.
__device__ __forceinline__ void list_push(uint32_t& ls, uint32_t m, uint32_t addr) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %1, 0;\n\t@q st.shared.v2.u32 [%0], {%1, %2};\n\t"
               "@q add.u32 %0, %0, 256;\n\t}"
               : "+r"(ls)
               : "r"(m), "r"(addr)
               : "memory");
}

// Coordinates of nonnegative floats reduced over the warp by their bits.
__device__ __forceinline__ float warp_min_nonneg(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ float warp_max_nonneg(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ int warp_incl_sum(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += u;
  }
  return v;
}

// A warp's first tile; it asks the queue, which starts behind them, for the others.  Neighbours in the list
// go to different SMs: a launch of few tiles took them on the SMs whose warps asked
// first, two per warp (FP64 forces of 6,451 particles 1150 - 1550 us from run to run,
// 760 so; mixed, 47,455 particles with cells of 3: 311 -> 171 us).
__device__ __forceinline__ int first_tile() { return (threadIdx.x >> 5) * gridDim.x + blockIdx.x; }

// Whether a tile may meet a coordinate outside the box: whether its own bundle
// or one of those within its largest reach holds any (y, z, reach: of the lanes'
// particles, which are one bundle's; lane 0 always holds one).  Called by whole warps,
// and only where some bundle does.
template <typename R>
static __device__ __noinline__ bool tile_meets_outside(const TileCfg& cfg, const int32_t* __restrict__ outside,
                                                       const Grid<R>& g, bool active, R y, R z, float reach) {
  const float most = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(active ? reach : 0.f)));
  const int h = (int)(most * (float)g.inv_edge + 0.05f) + 1, ny = g.n[1], nz = g.n[2];  // rows, with room for rounding
  const int by = __shfl_sync(0xffffffffu, cell_coord<R>(y, g.edge, g.inv_edge, ny), 0) / cfg.ry,
            bz = __shfl_sync(0xffffffffu, cell_coord<R>(z, g.edge, g.inv_edge, nz), 0) / cfg.rz;
  const int ry = cfg.ry + 2 * h, n = ry * (cfg.rz + 2 * h);
  bool any = false;
  for (int k = threadIdx.x & 31; k < n; k += 32) {
    const int v = ((by * cfg.ry - h + k % ry) % ny + ny) % ny, w = ((bz * cfg.rz - h + k / ry) % nz + nz) % nz;
    for (int p = 0; p < cfg.np; ++p)
      any = any || __ldg(outside + (v / cfg.ry + cfg.nby * (w / cfg.rz)) * cfg.np + p) != 0;
  }
  return __any_sync(0xffffffffu, any);
}

// Visits the candidates of one pass of a tile (at most 32 particles): stages
// them chunk by chunk, builds the lanes' mask lists and calls consume(last):
// each lane then walks its list up to (excluding) list[last].  Returns false
// (after possibly some chunks) if the tile cannot be evaluated this way; the
// caller then discards what it summed.
//
//   pos    where the elements come from: const E*, or HalvesSource
//   i      the lane's particle (ignored where !active), xi its position (out:
//          in the tile's frame), ri its cutoff (clamped)
//   ahead  called once, when the tile's own loads are done with
//   reach  radius within which the lane may need candidates: ri, or more where
//          own_cutoff(candidate) gives the candidates a cutoff of their own, which
//          then counts too (NoCutoff: it does not)
struct NoCutoff {};
template <typename R, typename E, typename Src, typename Own, typename A, typename F>
__device__ __forceinline__ bool tile_candidates(TileSmem<E>& sm, const Src pos,
                                                const int32_t* __restrict__ start, const Grid<R>& g,
                                                const TileCfg& cfg, bool active, int i, R (&xi)[3], float ri,
                                                float reach, Own own_cutoff, A&& ahead, F&& consume) {
  constexpr int kTileCand = TileSmem<E>::kCand;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const float Lf[3] = {(float)g.L[0], (float)g.L[1], (float)g.L[2]};
  float lo[3], hi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    // -0 becomes +0: it lies in the box, and its bits are the largest of all
    const float v = (float)xi[d] + 0.f;
    lo[d] = active ? v : Lf[d];
    hi[d] = active ? v : 0.f;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    lo[d] = warp_min_nonneg(lo[d]);
    hi[d] = warp_max_nonneg(hi[d]);
  }
  const float rmax = warp_max_nonneg(active ? reach : 0.f);
  const bool two = __any_sync(full, active && reach > ri);
  // cells that the spheres can reach, unwrapped, with the row walk's slack;
  // FP64 coordinates are rounded to FP32 here, a few 1e-7 of the box
  const float ed[3] = {(float)g.edge_x, (float)g.edge, (float)g.edge};
  const float ie[3] = {(float)g.inv_edge_x, (float)g.inv_edge, (float)g.inv_edge};
  const float rs = rmax * 1.000004f;
  int u0[3], u1[3];
  bool upper[3], cross[3], ok = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float eps = 5e-4f + 4e-7f * Lf[d] * ie[d];
    u0[d] = (int)floorf((lo[d] - rs) * ie[d] - eps);
    u1[d] = (int)floorf((hi[d] + rs) * ie[d] + eps);
    upper[d] = u1[d] >= g.n[d];
    cross[d] = upper[d] || u0[d] < 0;
    // one image per axis, and a frame moved by -L only where that is exact
    ok = ok && !(upper[d] && u0[d] < 0) && !(upper[d] && !(lo[d] - rs >= 0.5f * Lf[d])) && u0[d] >= -g.n[d] &&
         u1[d] < 2 * g.n[d];
  }
  if (!ok) return false;
  const int row_y = cell_coord<R>(xi[1], g.edge, g.inv_edge, g.n[1]);
  const int row_z = cell_coord<R>(xi[2], g.edge, g.inv_edge, g.n[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (upper[d]) {
      xi[d] -= g.L[d];
      lo[d] -= Lf[d];
      hi[d] -= Lf[d];
    }
  TileFilter f;
  filter_begin(f, sm.frag, (float)xi[0], (float)xi[1], (float)xi[2], active ? ri : -1.f, lo, hi, rmax, cfg.scale,
               fmaxf(Lf[0], fmaxf(Lf[1], Lf[2])));
  // The rows are visited in two halves like the squares of a chess board, so
  // that the pairs of every lane are spread evenly over the chunks (a lane waits
  // for the fullest list of each chunk).
  const int nyr = u1[1] - u0[1] + 1, nzr = u1[2] - u0[2] + 1, nseg = cross[0] ? 2 : 1;
  const int nyh = (nyr + 1) >> 1, nhalf = nyh * nzr * nseg;
  const bool images = cross[0] || cross[1] || cross[2];
  // the lane's own row among the items, on the side inside the box
  int own = -1, own_half = 0;
  if (active && row_y >= u0[1] && row_y <= u1[1] && row_z >= u0[2] && row_z <= u1[2]) {
    const int ry = row_y - u0[1], rz = row_z - u0[2];
    own = (rz * nyh + (ry >> 1)) * nseg + (nseg == 2 && !upper[0] ? 1 : 0);
    own_half = (ry + rz) & 1;
  }
  const uint32_t pos_s = shared_addr(sm.pos), list_s = shared_addr(&sm.list[0][lane]);
  const float rs2 = rs * rs;
  // a place that no particle of the tile reaches
  const R pad[3] = {(R)(-f.ox / f.s), (R)((kPadAt - f.oy) / f.s), (R)(-f.oz / f.s)};
  if (lane < kTileEnd) {
    E far{};  // what lists may be read past their end
    far.x = pad[0];
    far.y = pad[1];
    far.z = pad[2];
    sm.pos[kTileCand + lane] = far;
  }
  ahead();
  int staged = 0, selfcol = -1;  // candidates in shared memory, the lane's own particle among them
  int half = 0;
  for (int it0 = 0;;) {
    // one row segment per lane
    const int it = it0 + lane;
    int j0 = 0, cnt = 0;
    uint32_t im = 0;  // bit d: taken at x_j - L along d
    const int side = nseg == 2 ? it & 1 : 0, row = nseg == 2 ? it >> 1 : it;
    const int rz = (int)(((float)row + 0.5f) * __frcp_rn((float)nyh)), ry = 2 * (row - rz * nyh) + ((rz + half) & 1);
    if (it < nhalf && ry < nyr) {
      const int uy = u0[1] + ry, uz = u0[2] + rz;
      // gap between the tile's particles and the row, in the moved frame
      const float ya = (float)uy * ed[1] - (upper[1] ? Lf[1] : 0.f), za = (float)uz * ed[2] - (upper[2] ? Lf[2] : 0.f);
      const float gy = fmaxf(fmaxf(ya - hi[1], lo[1] - (ya + ed[1])), 0.f);
      const float gz = fmaxf(fmaxf(za - hi[2], lo[2] - (za + ed[2])), 0.f);
      // rows are dropped only if they are out of reach by more than the
      // rounding of their coordinates
      const float g2 = fmaf(gy, gy, gz * gz), tol = 4e-6f * fmaxf(Lf[1], Lf[2]) * (gy + gz);
      if (g2 - tol < rs2) {
        const int wy = uy < 0 ? uy + g.n[1] : (uy >= g.n[1] ? uy - g.n[1] : uy);
        const int wz = uz < 0 ? uz + g.n[2] : (uz >= g.n[2] ? uz - g.n[2] : uz);
        const float wx = window_half_width(fmaxf(rs2 - g2 + tol, 0.f));
        const float sx = upper[0] ? Lf[0] : 0.f, eps = 5e-4f + 4e-7f * Lf[0] * ie[0];
        int a = max((int)floorf((lo[0] + sx - wx) * ie[0] - eps), u0[0]);
        int b = min((int)floorf((hi[0] + sx + wx) * ie[0] + eps), u1[0]);
        // image shifts: below 0 the image, below n in a frame moved by -L
        im = ((upper[1] ? uy < g.n[1] : uy < 0) ? 2u : 0u) | ((upper[2] ? uz < g.n[2] : uz < 0) ? 4u : 0u);
        if (nseg == 2) {  // side 0: the cells that are shifted, side 1: the others
          const int split = upper[0] ? g.n[0] : 0;
          if (side == 0) {
            b = min(b, split - 1);
            im |= 1u;
          } else {
            a = max(a, split);
          }
          const int w = a < 0 ? g.n[0] : (a >= g.n[0] ? -g.n[0] : 0);  // all of [a, b] wraps alike
          a += w;
          b += w;
        }
        if (a <= b) {
          const int base = g.n[0] * (wy + g.n[1] * wz);  // 32-bit: fewer than 2^31 cells
          j0 = __ldg(start + base + a);
          cnt = max(__ldg(start + base + b + 1) - j0, 0);
        }
      }
    }
    const unsigned held = __ballot_sync(full, cnt > 0);
    const int incl = warp_incl_sum(cnt), off = incl - cnt, total = __shfl_sync(full, incl, 31);
    // where the lane's own particle comes in this batch
    int selfq = -1;
    {
      const int src = own - it0;
      const int o = __shfl_sync(full, off, src & 31), b = __shfl_sync(full, j0, src & 31),
                c = __shfl_sync(full, cnt, src & 31);
      if (own >= 0 && own_half == half && src >= 0 && src < 32 && i >= b && i < b + c) selfq = o + i - b;
    }
    it0 += 32;
    const bool end_half = it0 >= nhalf, final = end_half && half == 1;
    int done = 0;
    do {
      // stage what fits: four segments at a time, eight lanes each
      const int take = min(total - done, kTileCand - staged);
      const int k0 = max(done - off, 0), len = min(done + take - off, cnt) - k0, to = staged + off - done + k0;
      const int from = j0 + k0, sub = lane & 7;
      const int most = __reduce_max_sync(full, len);
#pragma unroll
      for (int r = 0; r < 32; r += 4) {
        if (!(held >> r & 15u)) continue;
        const int src = r + (lane >> 3);
        const int nn = __shfl_sync(full, len, src) - sub, jj = __shfl_sync(full, from, src) + sub;
        const uint32_t dst = pos_s + (uint32_t)((__shfl_sync(full, to, src) + sub) * (int)sizeof(E));
        const Src p = pos + jj;
        copy_if<0>(dst, p, nn);
        copy_if<8>(dst, p, nn);
        copy_if<16>(dst, p, nn);
        if (most > 24)
          for (int q = 24; q < most; q += 8) copy_if<0>(dst + (uint32_t)(q * sizeof(E)), p + q, nn - q);
      }
      if (images) {  // shift the image rows in place
        copy_async_wait();
        __syncwarp();
        for (unsigned rows = __ballot_sync(full, im != 0 && len > 0); rows; rows &= rows - 1) {
          const int src = __ffs(rows) - 1;
          const int nn = __shfl_sync(full, len, src), tt = __shfl_sync(full, to, src);
          const uint32_t code = __shfl_sync(full, im, src);
          for (int q = lane; q < nn; q += 32) {
            E p = sm.pos[tt + q];
            if (code & 1u) p.x -= g.L[0];
            if (code & 2u) p.y -= g.L[1];
            if (code & 4u) p.z -= g.L[2];
            sm.pos[tt + q] = p;
          }
        }
      }
      if (selfq >= done && selfq < done + take) selfcol = staged + selfq - done;
      staged += take;
      done += take;
      // a chunk is full, or ends with its half where the other one would not fit
      if (staged == kTileCand || (staged && done == total && (final || (end_half && 2 * staged > kTileCand)))) {
        if (staged + lane < (staged + 31 & ~31)) {  // fill the last group up
          E p{};
          p.x = pad[0];
          p.y = pad[1];
          p.z = pad[2];
          sm.pos[staged + lane] = p;
        }
        copy_async_wait();
        __syncwarp();
        uint32_t ls = list_s, ad = pos_s;
        const uint32_t end = pos_s + (uint32_t)(staged * (int)sizeof(E));
        const uint32_t own_ad = pos_s + (uint32_t)((selfcol & ~31) * (int)sizeof(E)), own_bit = ~(0x80000000u >> (selfcol & 31));
        do {
          const E p = *reinterpret_cast<const E*>(reinterpret_cast<const char*>(sm.pos) + (ad - pos_s) + lane * sizeof(E));
          uint32_t m;
          if constexpr (std::is_same_v<Own, NoCutoff>) {
            m = filter_group<false>(f, (float)p.x, (float)p.y, (float)p.z, 0.f);
          } else {
            m = two ? filter_group<true>(f, (float)p.x, (float)p.y, (float)p.z, own_cutoff(p))
                    : filter_group<false>(f, (float)p.x, (float)p.y, (float)p.z, 0.f);
          }
          if (ad == own_ad) m &= own_bit;
          list_push(ls, m, ad);
          ad += 32u * (uint32_t)sizeof(E);
        } while (ad < end);
        const int last = (int)(ls - list_s) >> 8;
        sm.list[last][lane] = make_uint2(0xf0000000u, pos_s + kTileCand * (uint32_t)sizeof(E));
        consume(last);
        __syncwarp();
        staged = 0;
        selfcol = -1;
      }
    } while (done < total);
    if (final) break;
    if (end_half) {
      half = 1;
      it0 = 0;
    }
  }
  return true;
}

// A lane's way through its list: the shared address of the next marked
// candidate.  Loads and the step are predicated, not branched around: nearly
// every step some lane of the warp moves on to its next word.
struct ListWalk {
  uint32_t w, ad, wn, adn, lp, end;  // current word and address, the next ones (loaded early), list position and end
  __device__ __forceinline__ void begin(uint32_t list_s, int last) {
    w = ad = 0;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(wn), "=r"(adn) : "r"(list_s) : "memory");
    lp = list_s + 256u;
    end = list_s + 256u * (uint32_t)last;
  }
  // whether marked candidates remain (before the ones past the end)
  __device__ __forceinline__ bool more() const { return lp - (w ? 512u : 256u) < end; }
  __device__ __forceinline__ uint32_t next(int log_size) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.eq.u32 q, %0, 0;\n\t@q mov.u32 %0, %2;\n\t@q mov.u32 %1, %3;\n\t"
        "@q ld.shared.v2.u32 {%2, %3}, [%4];\n\t@q add.u32 %4, %4, 256;\n\t}"
        : "+r"(w), "+r"(ad), "+r"(wn), "+r"(adn), "+r"(lp)
        :
        : "memory");
    const int b = first_bit(w);
    w ^= 0x80000000u >> b;
    return ad + ((uint32_t)b << log_size);
  }
};

__device__ __forceinline__ float4 lds4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ dvec4 lds4d(uint32_t addr) {
  dvec4 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%4];\n\tld.shared.v2.f64 {%2, %3}, [%4 + 16];"
      : "=d"(v.x), "=d"(v.y), "=d"(v.z), "=d"(v.w)
      : "r"(addr));
  return v;
}

}  // namespace dcm
