// Lennard-Jones forces with per-particle cutoffs over tiles of 32 particles
// (pair_tiles.cuh): the same pairs and the same per-pair arithmetic as the row
// walk of forces.cu, with the candidates found by the tensor-core filter.
//
// A small kernel cuts every bundle of cell rows into tiles; the force kernel
// keeps a fixed number of warps per SM, each of which takes tile after tile from
// a device queue.  Warps share nothing, so a long tile (at an interface the
// spheres hold eight times the bulk's volume) holds up one warp only.
//
// Bound by instruction issue: 64% of the issue slots at 16 warps per SM, the
// tensor pipe 11% busy, HBM nearly idle.  Sixteen warps of 512 staged
// candidates fill the SM's shared memory; 13 of 640 and 20 of 384 (at 96
// registers) were slower.  Kernel times against the row walk, energies included:
// 15.5M particles 6140 -> 4498 us, 1.0M 525 -> 380 (cells of 0.5 x 1.5 x 1.5; cubic
// ones 410), 260K in FP64 6000 -> 1725.
#include <algorithm>
#include <climits>
#include <cmath>

#include "pair_tiles.cuh"

namespace dcm {

// ---------------------------------------------------------------------------
// tiles
// ---------------------------------------------------------------------------

// One warp per piece of a bundle: deals its particles, in the order of their
// cell step along x, into tiles of 32 (a tile ends early only where it would
// grow longer than cfg.cap cells, and at the piece's end).  The particles of the
// tile in slot s are idx[32 s .. 32 s + 31] (-1: none).  Slots follow the
// particles (those before the piece / 32, plus cmax per piece, which covers the
// tiles that are not full), so sums kept per slot do not depend on timing; the
// list of the slots in use does (pieces append to it as they finish).  Tiles
// whose first or 16th particle has a cutoff above `wide` are listed from the
// front, the others from the back: the costly ones start first, so that a launch
// of few tiles per warp does not end on them (300K particles, a cylinder of
// liquid: 259 -> 246 us against full tiles alone first).  Coordinates
// outside the box are looked for in the boundary cells, the only ones that may
// hold them; the piece's flag says whether there are any.  queue: tiles that the warps
// of the next launch take by their number (first_tile), before they ask.  NR: cell rows of a bundle, at most; the starts of the next 32
// steps are loaded while these are dealt.
template <typename R, int NR>
__global__ void __launch_bounds__(128) k_tile_cut(const int32_t* __restrict__ start,
                                                  const typename RT<R>::R4* __restrict__ pos,
                                                  const R* __restrict__ rc, R wide, Grid<R> g, TileCfg cfg,
                                                  int32_t* __restrict__ idx, int32_t* __restrict__ list,
                                                  int32_t* __restrict__ counters, int32_t* __restrict__ flag,
                                                  int64_t nslot, int queue) {
  const int nx = g.n[0], ny = g.n[1], nz = g.n[2];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int piece = blockIdx.x * 4 + (threadIdx.x >> 5), b = piece / cfg.np;
  if (b >= cfg.nby * cfg.nbz) return;
  if (piece == 0 && lane == 0) counters[kTileQueue] = queue;
  const int by = b % cfg.nby, bz = b / cfg.nby;
  const int xs = (piece - b * cfg.np) * cfg.px, xe = min(xs + cfg.px, nx);
  const int y0 = by * cfg.ry, z0 = bz * cfg.rz, nr_y = min(cfg.ry, ny - y0), nr_z = min(cfg.rz, nz - z0);
  const int nr = nr_y * nr_z;
  // particles in the bundles before this one, and in the pieces before in it
  int before = 0;
  if (lane < nr_z) {
    const int z = nx * ny * (z0 + lane);
    before = __ldg(start + z + nx * y0) - __ldg(start + z);
  }
  if (xs > 0 && lane < nr) {
    const int c = nx * (y0 + lane % nr_y + ny * (z0 + lane / nr_y));
    before += __ldg(start + c + xs) - __ldg(start + c);
  }
  const int plane = __ldg(start + nx * ny * z0);
  int row[NR];
  unsigned outer = 0;  // rows of boundary cells
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    const int y = y0 + r % nr_y, z = z0 + r / nr_y;
    row[r] = nx * (y + ny * z);
    if (y == 0 || y == ny - 1 || z == 0 || z == nz - 1) outer |= 1u << r;
  }
  bool outside = false;
  int from[NR], to[NR];  // the particles of the lane's cells
  auto load = [&](int x) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const bool in = r < nr && x < xe;
      from[r] = in ? __ldg(start + row[r] + x) : 0;
      to[r] = in ? __ldg(start + row[r] + x + 1) : 0;
    }
  };
  load(xs + lane);
  before = __reduce_add_sync(full, before) + plane;
  const int64_t slot0 = (before >> 5) + (int64_t)piece * cfg.cmax;
  idx += 32 * slot0;
  const int lim = (int)min(32 * (nslot - slot0), (int64_t)INT_MAX);  // never reached (see above)
  int S = 0, B = 0, x0 = xs;  // next place, end of the open tile, its first cell step
  for (int xb = xs; xb < xe; xb += 32) {
    const int x = xb + lane;
    int k0[NR], k1[NR], c = 0;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      k0[r] = from[r];
      k1[r] = max(to[r], from[r]);
      c += k1[r] - k0[r];
    }
    if (xb + 32 < xe) load(x + 32);
    const int s = warp_incl_sum(c);
    int place = S + s - c, at = 0;  // where the lane's particles go; lanes settled
    for (;;) {
      const unsigned over = __ballot_sync(full, lane >= at && c > 0 && place + c > B);
      const unsigned longer = __ballot_sync(full, lane >= at && c > 0 && place < B && x - x0 >= cfg.cap);
      if (longer && (!over || __ffs(longer) <= __ffs(over))) {  // end the tile here, leave the rest of it empty
        const int q = __ffs(longer) - 1, gap = B - __shfl_sync(full, place, q), first = B - gap;
        if (lane < gap && first + lane < lim) idx[first + lane] = -1;
        if (lane >= q) place += gap;
        S += gap;
        at = q;
      } else if (over) {  // the tile is full: the next one begins in this step
        at = __ffs(over) - 1;
        x0 = xb + at;
        B += 32;
      } else {
        break;
      }
    }
    S += __shfl_sync(full, s, 31);
#pragma unroll
    for (int r = 0; r < NR; ++r)
      for (int k = k0[r]; k < k1[r]; ++k, ++place) {
        if (place < lim) idx[place] = k;
        if ((outer >> r & 1u) || x == 0 || x == nx - 1) {
          const auto q = ldg4(pos + k);
          outside = outside || !(q.x >= (R)0 && q.x < g.L[0] && q.y >= (R)0 && q.y < g.L[1] && q.z >= (R)0 &&
                                 q.z < g.L[2]);
        }
      }
  }
  outside = __any_sync(full, outside);
  if (lane == 0) {
    flag[piece] = outside;
    if (outside) counters[kTileOutside] = 1;
  }
  if (S + lane < B && S + lane < lim) idx[S + lane] = -1;
  __syncwarp();
  const int nt = min(B, lim) >> 5;
  for (int t0 = 0; t0 < nt; t0 += 32) {
    const int t = t0 + lane;
    bool is_wide = false;
    if (t < nt) {
      const volatile int32_t* m = idx + 32 * t;  // written by other lanes of this warp
      const int i0 = m[0], i1 = m[15];
      is_wide = rc[max(i0, 0)] > wide || rc[max(i1, 0)] > wide;
    }
    const unsigned w = __ballot_sync(full, t < nt && is_wide), v = __ballot_sync(full, t < nt && !is_wide);
    int at = 0;
    if (lane == 0 && w) at = atomicAdd(counters + kTileFirst, __popc(w));
    if (lane == 1 && v) at = atomicAdd(counters + kTileLater, __popc(v));
    const int aw = __shfl_sync(full, at, 0), av = __shfl_sync(full, at, 1);
    const unsigned below = (1u << lane) - 1u;
    if (t < nt) {
      if (is_wide)
        list[aw + __popc(w & below)] = (int32_t)(slot0 + t);
      else
        list[nslot - 1 - (av + __popc(v & below))] = (int32_t)(slot0 + t);
    }
  }
}

// ---------------------------------------------------------------------------
// forces
// ---------------------------------------------------------------------------

// One packed step of the pair loop: the arithmetic of pair_x2_d / pair_x2_dt
// (forces_core.cuh) on -1/r^2 in place of 1/r^2, which takes the sign changes
// out of the instruction stream: every product and sum is that of the row walk or
// its exact negative, the force sums come out as +F (not -F), and a packed
// FP32x2 operand never has to be negated.
template <bool TYPED, bool EW>
__device__ __forceinline__ void tile_pair(const float4& p0, const float4& p1, float xi, float yi, float zi, float rc2,
                                          const float* k8, Acc2& c) {
  const float2 one = make_float2(1.f, 1.f), two = make_float2(2.f, 2.f);
  const float2 dx = make_float2(p0.x - xi, p1.x - xi), dy = make_float2(p0.y - yi, p1.y - yi),
               dz = make_float2(p0.z - zi, p1.z - zi);
  const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
  float y0, y1;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(-r2.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y1) : "f"(-r2.y));
  float2 y = make_float2(y0, y1);
  const float2 e = __ffma2_rn(r2, y, one);
  y = __ffma2_rn(y, e, y);
  const bool a0 = r2.x < rc2, a1 = r2.y < rc2;
  y = make_float2(a0 ? y.x : 0.f, a1 ? y.y : 0.f);  // -1/r^2
  if constexpr (TYPED) {
    const bool t0 = p0.w >= 1.f, t1 = p1.w >= 1.f;
    const float2 sg = make_float2(t0 ? k8[3] : k8[2], t1 ? k8[3] : k8[2]),
                 e24 = make_float2(t0 ? k8[5] : k8[4], t1 ? k8[5] : k8[4]);
    const float2 s2 = __fmul2_rn(sg, y);
    const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);  // -(sigma/r)^6
    const float2 pv = __fmul2_rn(e24, __fmul2_rn(s6, __ffma2_rn(s6, two, one)));
    const float2 q = __fmul2_rn(pv, y);
    c.fx = __ffma2_rn(q, dx, c.fx);
    c.fy = __ffma2_rn(q, dy, c.fy);
    c.fz = __ffma2_rn(q, dz, c.fz);
    if constexpr (EW) {
      const float2 e4 = make_float2(t0 ? k8[7] : k8[6], t1 ? k8[7] : k8[6]),
                   us = make_float2(a0 ? (t0 ? -k8[1] : -k8[0]) : 0.f, a1 ? (t1 ? -k8[1] : -k8[0]) : 0.f);
      c.en = __fadd2_rn(c.en, __ffma2_rn(e4, __fmul2_rn(s6, __fadd2_rn(s6, one)), us));
      c.vir = __fadd2_rn(c.vir, pv);
    }
  } else {
    const float2 s6 = __fmul2_rn(__fmul2_rn(y, y), y);  // -1/r^6
    const float2 pv = __fmul2_rn(s6, __ffma2_rn(s6, two, one));
    const float2 q = __fmul2_rn(pv, y);
    c.fx = __ffma2_rn(q, dx, c.fx);
    c.fy = __ffma2_rn(q, dy, c.fy);
    c.fz = __ffma2_rn(q, dz, c.fz);
    if constexpr (EW) {
      c.en = __ffma2_rn(s6, __fadd2_rn(s6, one), c.en);
      c.vir = __fadd2_rn(c.vir, pv);
    }
  }
  if constexpr (EW) c.np += (int)a0 + (int)a1;
}

// Packed steps per turn of the pair loop (they hide each other's latency) and
// turns between two flushes of the running sums: at most 16 terms per packed
// lane, as many as the fullest z-plane of the row walk sums at rc = 3.
constexpr int kTurnSteps = 2, kFlushTurns = 8;
static_assert(2 * kTurnSteps <= kTileEnd, "a turn may read that far past a list's end");

// Pairs of the lane's list, two per packed step (steps past its end take the far particle).
template <bool TYPED, bool EW>
__device__ __forceinline__ void sum_list(ListWalk& l, float xi, float yi, float zi, float rc2, const float* k8,
                                         Acc<float>& c, Acc2& c2, Sums<Accum::kPlaneKahan>& S) {
  while (l.more()) {
    for (int s = 0; s < kFlushTurns; ++s) {
      float4 p[2 * kTurnSteps];
#pragma unroll
      for (int q = 0; q < 2 * kTurnSteps; ++q) p[q] = lds4(l.next(4));
#pragma unroll
      for (int q = 0; q < 2 * kTurnSteps; q += 2) tile_pair<TYPED, EW>(p[q], p[q + 1], xi, yi, zi, rc2, k8, c2);
      if (!l.more()) break;
    }
    flush_partials<Accum::kPlaneKahan, float, true, EW>(c, c2, S);
  }
}

// FP64: one pair at a time, the scalar loop's arithmetic.
template <bool TYPED>
__device__ __forceinline__ void sum_list(ListWalk& l, double xi, double yi, double zi, double rc2, int ti,
                                         const ForceArgs<double>& a, const double* ushift, Acc<double>& c) {
  while (l.more()) {
    const dvec4 p = lds4d(l.next(5));
    pair_one<double, TYPED>(xi - p.x, yi - p.y, zi - p.z, p.w, rc2, ti, a, ushift, c);
  }
}

// A tile's energy, virial and pair count: summed across the warp in FP64 into
// the tile's slot.
__device__ __forceinline__ void tile_partials(double e, double w, int np, double* __restrict__ part, int64_t nslot,
                                              uint32_t slot) {
  for (int o = 16; o > 0; o >>= 1) {
    e += __shfl_xor_sync(0xffffffffu, e, o);
    w += __shfl_xor_sync(0xffffffffu, w, o);
    np += __shfl_xor_sync(0xffffffffu, np, o);
  }
  if ((threadIdx.x & 31) == 0 && slot < nslot) {
    part[slot] = e;
    part[nslot + slot] = w;
    part[2 * nslot + slot] = (double)np;
  }
}

// Warps per block (nothing is shared between them): as many as the SM's shared
// memory holds, one block per SM.
template <typename R>
constexpr int tile_warps() {
  constexpr int fit = 227 * 1024 / (int)sizeof(TileSmem<typename RT<R>::R4>);
  constexpr int most = sizeof(R) == 4 ? 16 : 8;
  return fit < most ? fit : most;
}

template <typename R, bool TYPED, bool EW>
__global__ void __launch_bounds__(32 * tile_warps<R>(), 1) k_forces_tiles(
    const typename RT<R>::R4* __restrict__ pos, const R* __restrict__ rc, const int32_t* __restrict__ start,
    const __grid_constant__ ForceArgs<R> a, TileCfg cfg, const __grid_constant__ TileTable tt,
    typename RT<R>::R4* __restrict__ force, double* __restrict__ part, int64_t nslot) {
  using R4 = typename RT<R>::R4;
  constexpr bool kX2 = sizeof(R) == 4;
  constexpr Accum M = kX2 ? Accum::kPlaneKahan : Accum::kPlain;
  const unsigned full = 0xffffffffu;
  extern __shared__ __align__(32) unsigned char smem_raw[];
  TileSmem<R4>& sm = reinterpret_cast<TileSmem<R4>*>(smem_raw)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const Grid<R>& g = a.g;
  const int32_t *idx = tt.idx, *list = tt.list;
  int32_t* counters = tt.counters;
  const int nfirst = __ldg(counters + kTileFirst), ntile = nfirst + __ldg(counters + kTileLater);
  const bool outside = __ldg(counters + kTileOutside) != 0;
  auto take = [&]() {
    int t = 0;
    if (lane == 0) t = atomicAdd(counters + kTileQueue, 1);
    return t;  // in lane 0
  };
  // The loads that lead to a tile's particles (queue, slot, index, position)
  // each depend on the one before, so they run ahead: while one tile is
  // evaluated the next one's particles are loaded and the one after that is taken.
  auto slot_of = [&](int t0) {
    const int t = __shfl_sync(full, t0, 0);
    return t < ntile ? __ldg(t < nfirst ? list + t : list + (nslot - 1 - (t - nfirst))) : -1;
  };
  int slot = slot_of(first_tile()), slot1 = slot_of(take());
  int i = slot >= 0 ? __ldg(idx + 32 * (int64_t)slot + lane) : -1;
  R4 pi = ldg4(pos + max(i, 0));
  R ri = rc[max(i, 0)];
  while (slot >= 0) {
    const int t2 = take();
    const int i1 = slot1 >= 0 ? __ldg(idx + 32 * (int64_t)slot1 + lane) : -1;
    R4 p1 = pi;
    R r1 = ri;
    auto ahead = [&]() {
      p1 = ldg4(pos + max(i1, 0));
      r1 = rc[max(i1, 0)];
    };
    const bool active = i >= 0;
    const R rci = active ? clamp_cutoff<R>(ri, a.rc_max) : (R)0;
    const R rc2 = rci * rci;
    const int ti = TYPED ? type_of(pi.w, a.ntypes) : 0;
    R k8[8];
    row_constants<R, TYPED, kX2>(a, ti, rc2, k8);
    Acc<R> c;
    Acc2 c2;
    Sums<M> S;
    R xi[3] = {pi.x, pi.y, pi.z};
    // the FP64 cutoff rounded up
    const float rf = sizeof(R) == 4 ? (float)rci : __double2float_ru((double)rci);
    const bool met = outside && tile_meets_outside<R>(cfg, tt.outside, g, active, pi.y, pi.z, rf);
    const bool done = !met && tile_candidates<R, R4>(sm, pos, start, g, cfg, active, i, xi, rf, rf, NoCutoff{}, ahead, [&](int last) {
      ListWalk l;
      l.begin(shared_addr(&sm.list[0][lane]), last);
      if constexpr (kX2)
        sum_list<TYPED, EW>(l, xi[0], xi[1], xi[2], rc2, k8, c, c2, S);
      else
        sum_list<TYPED>(l, xi[0], xi[1], xi[2], rc2, ti, a, k8, c);
    });
    if (done) {
      double e = 0, w = 0;
      int np = 0;
      if constexpr (kX2) {  // finish_sums expects the sums of -F
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          S.s[q] = -S.s[q];
          S.k[q] = -S.k[q];
        }
      }
      if (active) force[i] = finish_sums<R, TYPED, kX2, M, EW || !kX2>(c, c2, S, k8, e, w, np);
      if (EW && part) tile_partials(e, w, np, part, nslot, (uint32_t)slot);
    } else {
      if (lane == 0) tt.rest[atomicAdd(counters + kTileRest, 1)] = slot;
      ahead();
    }
    slot = slot1;
    slot1 = slot_of(t2);
    i = i1;
    pi = p1;
    ri = r1;
  }
}

// The tiles that the filter does not serve, by the row walk.  Few of them: a
// block per tile, 16 lanes per particle (force_planes), because such a launch lasts
// as long as its longest walk (FP64 forces of 7,738 particles in a box of 4.25 rc_max,
// a quarter left over: 2480 us with a thread per particle, 1430 so).  Many of them
// (coordinates outside the box all over it): a warp per tile, a thread per particle,
// which keeps more lanes busy (all 8,900 tiles of 260K particles: 680 us with 16 lanes,
// 260 with one; the call with 2,000 tiles in FP64: 3430 and 2770).
constexpr int kRestBlock = 32 * kPlaneLanes;
template <typename R>
constexpr int rest_many() { return sizeof(R) == 4 ? 1500 : 600; }

template <typename R, bool TYPED, bool EW>
__global__ void __launch_bounds__(kRestBlock, sizeof(R) == 4 ? 2 : 1) k_forces_rest(const typename RT<R>::R4* __restrict__ pos,
                                                               const R* __restrict__ rc,
                                                               const int32_t* __restrict__ start, ForceArgs<R> a,
                                                               TileTable t, typename RT<R>::R4* __restrict__ force,
                                                               double* __restrict__ part, int64_t nslot) {
  constexpr bool kX2 = sizeof(R) == 4, kEW = EW || !kX2;
  __shared__ double sh[3][32];
  const int n = __ldg(t.counters + kTileRest);
  if (n >= rest_many<R>()) {
    constexpr int kWarps = kRestBlock / 32;
    for (int k = first_tile(); k < n; k += gridDim.x * kWarps) {
      const int slot = __ldg(t.rest + k);
      const int i = __ldg(t.idx + 32 * (int64_t)slot + (threadIdx.x & 31));
      double e = 0, w = 0;
      int np = 0;
      if (i >= 0)
        force[i] = force_one<R, TYPED, kX2, kX2 ? Accum::kPlaneKahan : Accum::kPlain, true, kEW>(
            pos, start, a.g, a, i, ldg4(pos + i), rc[i], e, w, np);
      __syncwarp();
      if (EW && part) tile_partials(e, w, np, part, nslot, (uint32_t)slot);
    }
    return;
  }
  const int q = threadIdx.x / kPlaneLanes;
  for (int k = blockIdx.x; k < n; k += gridDim.x) {
    const int slot = __ldg(t.rest + k);
    const int i = __ldg(t.idx + 32 * (int64_t)slot + q);
    double e = 0, w = 0;
    int np = 0;
    const auto f = force_planes<R, TYPED, kEW>(pos, start, a, i >= 0, max(i, 0), rc, e, w, np);
    const bool own = threadIdx.x % kPlaneLanes == 0;
    if (own && i >= 0) force[i] = f;
    if (EW && part) {  // summed in the order of the particles
      __syncthreads();
      if (own) {
        sh[0][q] = e;
        sh[1][q] = w;
        sh[2][q] = (double)np;
      }
      __syncthreads();
      if (threadIdx.x < 3) {
        double v = 0;
        for (int p = 0; p < 32; ++p) v += sh[threadIdx.x][p];
        part[threadIdx.x * nslot + slot] = v;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------

TilePlan tile_plan(const dcm_params& p, const int64_t* nc, int64_t n) {
  TilePlan t{};
  auto rows = [&](int64_t cells) {
    const int r = (int)std::lround(p.rc_min / p.l);
    return (int)std::min<int64_t>(std::max(1, std::min(r, 4)), cells);
  };
  t.cfg.ry = rows(nc[1]);
  t.cfg.rz = rows(nc[2]);
  t.cfg.nby = (int)((nc[1] + t.cfg.ry - 1) / t.cfg.ry);
  t.cfg.nbz = (int)((nc[2] + t.cfg.rz - 1) / t.cfg.rz);
  const double lx = p.lx > 0.0 ? p.lx : p.l, Lx = (double)nc[0] * lx;
  // Longest tile.  A launch of few tiles per warp (up to 16 on average) ends on its
  // longest ones, in the vapor beside an interface along x: 260K particles, 164 x 41 x 41
  // density boxes, 24 / 12 / 8 rc_max: 291 / 251 / 245 us.  A long launch wants them as
  // full as they get: a step of 15.5M particles 5430 / 5487 / 5588 us.
  auto longest = [&](double reach) {
    const double cap = std::min(reach * p.rc_max, 0.5 * Lx - 2.0 * p.rc_max);
    return (int)std::max(1.0, std::min(std::floor(cap / lx), 65535.0));
  };
  const int full = longest(24.0);
  t.cfg.cap = p.n_max < (int64_t)32 * 16 * 152 * 16 ? longest(12.0) : full;
  int k;
  std::frexp(p.rc_max, &k);  // rc_max = f 2^k, f in [0.5, 1)
  t.cfg.scale = std::ldexp(1.0f, 3 - k);
  const int64_t nb = (int64_t)t.cfg.nby * t.cfg.nbz;
  // Few bundles are cut into pieces along x, a warp each, because one warp takes
  // about 1.2 us per 32 cell steps (a box of 4800 x 16 x 16 cells: 372 us in 64
  // warps), and a launch of 8 warps per SM hides most of that.  Pieces of at least 16
  // rc_max and of 8 tiles at the mean density (for n_max particles, so that the
  // table of n never outgrows that of n_max): every piece ends on a tile that is not full.
  const double dense = (double)p.n_max / ((double)nc[0] * (double)nc[1] * (double)nc[2]) * t.cfg.ry * t.cfg.rz;
  const double least = std::max(16.0 * p.rc_max / lx, 8.0 * 32.0 / std::max(dense, 1e-9));  // cells
  const int64_t most = (int64_t)std::max(1.0, std::min((double)nc[0] / least, 65536.0));
  const int64_t pieces = std::max<int64_t>(1, std::min(most, (152 * 8 + nb - 1) / nb));
  t.cfg.px = (int)((nc[0] + pieces - 1) / pieces);
  t.cfg.np = (int)((nc[0] + t.cfg.px - 1) / t.cfg.px);
  auto spare = [&](int64_t cells, int cap) { return 2 + (int)((cells + cap - 1) / cap); };
  t.cfg.cmax = spare(t.cfg.px, t.cfg.cap);
  t.slots = n / 32 + nb * t.cfg.np * t.cfg.cmax + 1;
  // A box of at least 4 rc_max (in a smaller one most tiles at an interface
  // reach past both ends of an axis), cells no wider than the cutoff sphere
  // (FP16 range of the staged coordinates) and a table that stays in proportion
  // to the particles.
  const double Lmin = std::min(Lx, std::min((double)nc[1], (double)nc[2]) * p.l);
  t.usable = Lmin >= 4.0 * p.rc_max && p.l <= 2.0 * p.rc_max && lx <= 2.0 * p.rc_max &&
             8 * nb * spare(nc[0], full) <= n + 65536 && 32 * t.slots < (int64_t)1 << 31;
  return t;
}

// Launches below this many particles keep the row walk: that few leave most
// SMs without a tile, and a launch lasts as long as its longest tile (FP64:
// 4,838 particles 1594 us by the row walk, 618 over tiles; the mixed form takes
// 16 lanes per particle up to planes_max_n).
constexpr int64_t kTilesMinN = 4000;

bool tiles_serve(const dcm_ctx* ctx, int64_t n) {
  // A thin gas in cells of rc_min to 1.5 rc_min stays with the row walk in the mixed
  // form (fewer than 3 particles per sphere of rc_min on average): its tiles, one
  // cell across, end at their longest, half empty, and the walk meets few candidates.
  // 117K particles at density 0.02, rc 6, cells of 1.5 / 3 / 6: row walk 130 / 83 / 86
  // us, tiles 134 / 109 / 71; at 0.04 148 / 115 and 138 / 120.
  const dcm_params& p = ctx->p;
  if (p.precision == DCM_PREC_MIXED && p.l >= p.rc_min && p.l < 1.5 * p.rc_min &&
      (double)n * 4.19 * p.rc_min * p.rc_min * p.rc_min < 3.0 * p.box[0] * p.box[1] * p.box[2])
    return false;
  return ctx->tiles && n >= kTilesMinN && tile_plan(p, ctx->nc, n).usable;
}

template <typename R>
int tile_cut(dcm_ctx* ctx, const TilePlan& tp, const typename RT<R>::R4* pos, const R* rc, const int32_t* cell_start,
             const Grid<R>& g, TileTable& t, int warps, cudaStream_t st) {
  t.counters = ctx->tiles;
  t.list = t.counters + kTileCounters;
  t.rest = t.list + tp.slots;
  t.outside = t.rest + tp.slots;  // one per piece of a bundle, each of which has slots of its own
  t.idx = t.outside + tp.slots;
  const int64_t nb = (int64_t)tp.cfg.nby * tp.cfg.nbz * tp.cfg.np;
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(t.counters, 0, kTileCounters * sizeof(int32_t), st));
  auto kc = tp.cfg.ry * tp.cfg.rz <= 4 ? k_tile_cut<R, 4> : k_tile_cut<R, 16>;
  DCM_LAUNCH(ctx, kc, (unsigned)((nb + 3) / 4), 128, 0, st, cell_start, pos, rc, (R)(1.2 * ctx->p.rc_min), g, tp.cfg,
             t.idx, t.list, t.counters, t.outside, tp.slots, warps);
  return DCM_OK;
}
template int tile_cut<float>(dcm_ctx*, const TilePlan&, const float4*, const float*, const int32_t*,
                             const Grid<float>&, TileTable&, int, cudaStream_t);

template <typename R>
int tile_forces(dcm_ctx* ctx, bool typed, bool ew, int64_t n, const typename RT<R>::R4* pos, const R* rc,
                const int32_t* cell_start, const ForceArgs<R>& a, typename RT<R>::R4* force, double* part,
                cudaStream_t st) {
  const TilePlan tp = tile_plan(ctx->p, ctx->nc, n);
  if (part) DCM_CUDA_TRY(ctx, cudaMemsetAsync(part, 0, 3 * sizeof(double) * (size_t)tp.slots, st));
  int sms = 0;
  DCM_CUDA_TRY(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  constexpr int warps = tile_warps<R>(), smem = warps * (int)sizeof(TileSmem<typename RT<R>::R4>);
  const int grid = (int)std::min<int64_t>(tp.slots, sms);
  TileTable t;
  int r = tile_cut<R>(ctx, tp, pos, rc, cell_start, a.g, t, grid * warps, st);
  if (r) return r;
  auto k = typed ? (ew ? k_forces_tiles<R, true, true> : k_forces_tiles<R, true, false>)
                 : (ew ? k_forces_tiles<R, false, true> : k_forces_tiles<R, false, false>);
  auto kr = typed ? (ew ? k_forces_rest<R, true, true> : k_forces_rest<R, true, false>)
                  : (ew ? k_forces_rest<R, false, true> : k_forces_rest<R, false, false>);
  DCM_CUDA_TRY(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  DCM_LAUNCH(ctx, k, grid, 32 * warps, smem, st, pos, rc, cell_start, a, tp.cfg, t, force, part, tp.slots);
  DCM_LAUNCH(ctx, kr, (unsigned)std::min<int64_t>(tp.slots, 2 * sms), kRestBlock, 0, st, pos, rc, cell_start, a, t,
             force, part, tp.slots);
  return check_launch(ctx, "tile_forces");
}

template int tile_forces<float>(dcm_ctx*, bool, bool, int64_t, const float4*, const float*, const int32_t*,
                                const ForceArgs<float>&, float4*, double*, cudaStream_t);
template int tile_forces<double>(dcm_ctx*, bool, bool, int64_t, const dvec4*, const double*, const int32_t*,
                                 const ForceArgs<double>&, dvec4*, double*, cudaStream_t);

}  // namespace dcm
