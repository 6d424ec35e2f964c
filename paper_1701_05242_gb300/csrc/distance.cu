// Box-interface distances (Section 2.2, Algorithm 2.1): cutoff-based fast
// sweeping on the density-box grid.
//
// Algorithm 2.1 processes a queue of boxes breadth-first and keeps going
// until the largest change of a pass is below epsilon; its result is the
// fixed point of the local fast-sweeping update restricted to distances
// <= r_grid, whatever the visiting order.  On the GPU the same fixed point is
// reached by Jacobi sweeps (double buffered, so the result is deterministic):
// sweep 0 re-solves every box of the high-density phase; every later sweep
// re-solves only the boxes of its queue — the boxes that changed in the
// previous sweep and their six neighbours — which are exactly the boxes
// whose update can differ from the previous sweep's, so the iterates are
// those of full Jacobi sweeps while the work follows the moving front (the
// paper's queue Q); the MPI_Allreduce of the paper's version becomes the
// queue length in device memory.  The initial values and sweep 0 are one pass
// over the grid, the later sweeps one cooperative launch with a grid barrier
// between them, until a sweep changes nothing or iter_max sweeps have run;
// dcm_distance then reads the outcome on the host, the timestep does not.
#include <algorithm>

#include "dcm_internal.cuh"
#include "grid_sync.cuh"

namespace dcm {

// Godunov upwind update of |grad d| = 1 with spacing h from the three axis
// minima a (any order).  Returns +inf if all are +inf.
template <typename R>
__device__ __forceinline__ R godunov3(R a0, R a1, R a2, R h) {
  // sort ascending
  R t;
  if (a0 > a1) { t = a0; a0 = a1; a1 = t; }
  if (a1 > a2) { t = a1; a1 = a2; a2 = t; }
  if (a0 > a1) { t = a0; a0 = a1; a1 = t; }
  R d = a0 + h;
  if (d > a1) {
    R df = a0 - a1;
    d = (R)0.5 * (a0 + a1 + sqrt((R)2 * h * h - df * df));
    if (d > a2) {
      R sa = a0 + a1 + a2;
      R sq = a0 * a0 + a1 * a1 + a2 * a2;
      R disc = sa * sa - (R)3 * (sq - h * h);
      d = (sa + sqrt(disc > (R)0 ? disc : (R)0)) / (R)3;
    }
  }
  return d;
}

// Queue the high-density boxes among b and its six neighbours for sweep it+1
// (each box once: stamp holds the last sweep a box was queued for).  Called by
// every lane of a warp (push: whether this lane's box
// changed): the lanes take their queue places together, one atomic per warp and
// neighbour (the queue of a 51,200-box front takes about 200,000 entries per
// sweep, each of which was an atomic on the queue's length).
__device__ __forceinline__ void dist_push(bool push, int b, int x, int y, int z, int nx, int ny, int nz,
                                          const uint8_t* __restrict__ fixed0, int32_t* __restrict__ stamp,
                                          int32_t* __restrict__ qout, int32_t* __restrict__ qlen, int it) {
  const unsigned warp = 0xffffffffu;
  if (!__any_sync(warp, push)) return;
  const int nxy = nx * ny;  // fewer than 2^31 boxes in all
  const int nb[7] = {b,
                     x == 0 ? b + nx - 1 : b - 1,
                     x == nx - 1 ? b - x : b + 1,
                     y == 0 ? b + (ny - 1) * nx : b - nx,
                     y == ny - 1 ? b - y * nx : b + nx,
                     z == 0 ? b + (nz - 1) * nxy : b - nxy,
                     z == nz - 1 ? b - z * nxy : b + nxy};
  bool take[7];
#pragma unroll
  for (int k = 0; k < 7; ++k) take[k] = push && !fixed0[nb[k]];
#pragma unroll
  for (int k = 0; k < 7; ++k)
    if (take[k]) take[k] = atomicExch(stamp + nb[k], it + 1) != it + 1;
  const int lane = threadIdx.x & 31;
  unsigned m[7];
  int total = 0;
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    m[k] = __ballot_sync(warp, take[k]);
    total += __popc(m[k]);
  }
  if (!total) return;
  int at = 0;
  if (lane == 0) at = atomicAdd(qlen + it + 1, total);
  at = __shfl_sync(warp, at, 0);
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    if (take[k]) qout[at + __popc(m[k] & ((1u << lane) - 1u))] = nb[k];
    at += __popc(m[k]);
  }
}

// Update of one box from the previous iterate; true if it changed.  The
// iterates are read through L2 (__ldcg): other blocks wrote them earlier in the same
// launch, behind a grid barrier.
template <typename R>
__device__ __forceinline__ bool dist_update(const R* Din, R* Dout, int64_t b, int x, int y, int z, int nx, int ny,
                                            int nz, R h, R r_grid) {
  R cur = __ldcg(Din + b);
  int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
  int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
  int64_t row = (int64_t)nx * (y + (int64_t)ny * z);
  R a0 = fmin(__ldcg(Din + row + xm), __ldcg(Din + row + xp));
  R a1 = fmin(__ldcg(Din + x + nx * (ym + (int64_t)ny * z)), __ldcg(Din + x + nx * (yp + (int64_t)ny * z)));
  R a2 = fmin(__ldcg(Din + x + nx * (y + (int64_t)ny * zm)), __ldcg(Din + x + nx * (y + (int64_t)ny * zp)));
  R d = godunov3<R>(a0, a1, a2, h);
  bool ch = d < cur && d <= r_grid;
  Dout[b] = ch ? d : cur;
  return ch;
}

// Initial values and sweep 0 in one pass: before sweep 0 a box is 0 (low
// density or interface) or +inf, so the sweep reads the bytes of s and iface
// instead of the first iterate.  A thread marches along z.  HBM-bound: 33 MB read,
// 148 MB written for 16.4M boxes, 104 us (60 + 122 us as two passes); taken where
// rows are no multiple of four boxes, k_dist_first4 (43 us) where they are.
template <typename R>
__global__ void __launch_bounds__(256) k_dist_first(const uint8_t* __restrict__ s, const uint8_t* __restrict__ iface,
                                                    R* __restrict__ D0, R* __restrict__ D1, int nx, int ny, int nz,
                                                    int zc, R h, R r_grid, uint8_t* __restrict__ fixed0) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= nx || y >= ny) return;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  const int nxy = nx * ny, col = x + nx * y;
  auto zero = [&](int b) { return __ldg(s + b) == 0 || __ldg(iface + b) != 0; };
  const int xm = x == 0 ? nx - 1 : -1, xp = x == nx - 1 ? 1 - nx : 1;
  const int ym = y == 0 ? (ny - 1) * nx : -nx, yp = y == ny - 1 ? -(ny - 1) * nx : nx;
  bool below = zero(col + nxy * (z0 == 0 ? nz - 1 : z0 - 1)), here = zero(col + nxy * z0);
  for (int z = z0; z < z1; ++z) {
    const int b = col + nxy * z;
    const bool above = zero(col + nxy * (z == nz - 1 ? 0 : z + 1));
    const R inf = RT<R>::inf(), cur = here ? (R)0 : inf;
    R v = cur;
    if (!here) {
      const R a0 = zero(b + xm) || zero(b + xp) ? (R)0 : inf, a1 = zero(b + ym) || zero(b + yp) ? (R)0 : inf,
              a2 = below || above ? (R)0 : inf;
      const R d = godunov3<R>(a0, a1, a2, h);
      v = d < cur && d <= r_grid ? d : cur;
    }
    D0[b] = cur;
    D1[b] = v;
    fixed0[b] = (uint8_t)here;
    below = here;
    here = above;
  }
}

// Four boxes of a row per thread (nx a multiple of 4, flags 4-byte and
// distances 16-byte aligned): the flags of a box and its row neighbours come
// with one word and two bytes.
__device__ __forceinline__ uint32_t zero_bytes(uint32_t s, uint32_t f) {  // 0xff where s == 0 or f != 0
  return __vcmpeq4(s, 0u) | __vcmpne4(f, 0u);
}
__global__ void __launch_bounds__(256) k_dist_first4(const uint8_t* __restrict__ s, const uint8_t* __restrict__ iface,
                                                     float* __restrict__ D0, float* __restrict__ D1, int nx, int ny,
                                                     int nz, int zc, float h, float r_grid,
                                                     uint8_t* __restrict__ fixed0) {
  const int x = 4 * (blockIdx.x * 32 + (threadIdx.x & 31)), y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= nx || y >= ny) return;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  const int nxy = nx * ny, col = x + nx * y;
  auto word = [&](int b) {
    return zero_bytes(__ldg(reinterpret_cast<const uint32_t*>(s + b)), __ldg(reinterpret_cast<const uint32_t*>(iface + b)));
  };
  auto zero = [&](int b) { return __ldg(s + b) == 0 || __ldg(iface + b) != 0; };
  const int xm = x == 0 ? nx - 1 : -1, xp = x == nx - 4 ? 4 - nx : 4;
  const int ym = y == 0 ? (ny - 1) * nx : -nx, yp = y == ny - 1 ? -(ny - 1) * nx : nx;
  const float inf = RT<float>::inf();
  // sweep 0 knows three values per axis pair: 0 or +inf
  uint32_t below = word(col + nxy * (z0 == 0 ? nz - 1 : z0 - 1)), here = word(col + nxy * z0);
  for (int z = z0; z < z1; ++z) {
    const int b = col + nxy * z;
    const uint32_t above = word(col + nxy * (z == nz - 1 ? 0 : z + 1));
    float4 cur, v;
    if (here == 0xffffffffu) {
      cur = v = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      const uint32_t ax = (here << 8 | (zero(b + xm) ? 0xffu : 0u)) | (here >> 8 | (zero(b + xp) ? 0xff000000u : 0u));
      const uint32_t ay = word(b + ym) | word(b + yp), az = below | above;
      float* pc = &cur.x;
      float* pv = &v.x;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t bit = 1u << (8 * q);
        pc[q] = here & bit ? 0.f : inf;
        pv[q] = pc[q];
        if (!(here & bit)) {
          const float d = godunov3<float>(ax & bit ? 0.f : inf, ay & bit ? 0.f : inf, az & bit ? 0.f : inf, h);
          pv[q] = d < inf && d <= r_grid ? d : inf;
        }
      }
    }
    *reinterpret_cast<float4*>(D0 + b) = cur;
    *reinterpret_cast<float4*>(D1 + b) = v;
    *reinterpret_cast<uint32_t*>(fixed0 + b) = here & 0x01010101u;
    below = here;
    here = above;
  }
}

// The queue of sweep 1: the boxes that sweep 0 changed and their neighbours.
// Apart from the pass above, whose warps it would hold up at every front box.
template <typename R>
__global__ void __launch_bounds__(256) k_dist_queue0(const R* __restrict__ D1, int64_t nbox, int nx, int ny, int nz,
                                                     const uint8_t* __restrict__ fixed0, int32_t* __restrict__ stamp,
                                                     int32_t* __restrict__ qout, int32_t* __restrict__ qlen,
                                                     int32_t* __restrict__ flags) {
  const int64_t gs = (int64_t)gridDim.x * blockDim.x;
  for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < nbox; b0 += gs) {
    const int64_t b = b0 + threadIdx.x;
    // changed from +inf: finite and not fixed at 0
    const bool changed = b < nbox && D1[b] > (R)0 && D1[b] < RT<R>::inf();
    if (!__any_sync(0xffffffffu, changed)) continue;
    const int x = (int)(b % nx), y = (int)((b / nx) % ny), z = (int)(b / ((int64_t)nx * ny));
    dist_push(changed, (int)b, x, y, z, nx, ny, nz, fixed0, stamp, qout, qlen, 0);
    if ((threadIdx.x & 31) == 0) flags[0] = 1;
  }
}

// One large block per SM: the barrier between sweeps costs by the block.
constexpr int kCoopBlock = 1024;

// The sweeps after sweep 0 in one cooperative launch (every block resident):
// each over its queue, a bounded grid barrier after it, until a sweep changes
// nothing or `budget` sweeps have run.  The loop needs no host check and
// launches nothing per sweep.  A barrier wait that runs past budget_ns records
// DCM_ERR_TIMEOUT and ends the launch.
template <typename R>
__global__ void __launch_bounds__(kCoopBlock) k_dist_coop(R* D0, R* D1, int nx, int ny, int nz, R h, R r_grid,
                                                   const uint8_t* __restrict__ fixed0, int32_t* stamp, int32_t* q0,
                                                   int32_t* q1, int32_t* qlen, int32_t* flags, int budget,
                                                   uint32_t* sync, int64_t budget_ns, int32_t* status) {
  const unsigned full = 0xffffffffu;
  const uint32_t expected = gridDim.x;
  // neighbouring warps of the queue on different SMs: a sweep's queue fills a part
  // of the launch only, and the FP64 form needs every SM's units (64^3 boxes, 17
  // sweeps of two flat interfaces: 262 us with whole blocks in turn)
  const int64_t gt = ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31),
                gs = (int64_t)gridDim.x * blockDim.x;
  for (int it = 1; it < budget; ++it) {
    if (((volatile int32_t*)flags)[it - 1] == 0) break;  // the previous sweep changed nothing
    const R* Din = (it & 1) ? D1 : D0;
    R* Dout = (it & 1) ? D0 : D1;
    const int32_t* qin = (it & 1) ? q1 : q0;
    int32_t* qout = (it & 1) ? q0 : q1;
    const int32_t n = ((volatile int32_t*)qlen)[it];
    bool any = false;
    for (int64_t k = gt; k - (threadIdx.x & 31) < n; k += gs) {  // whole warps
      bool changed = false;
      int b = 0, x = 0, y = 0, z = 0;
      if (k < n) {
        b = __ldcg(qin + k);
        const int yz = b / nx;
        x = b - yz * nx;
        z = yz / ny;
        y = yz - z * ny;
        changed = dist_update<R>(Din, Dout, b, x, y, z, nx, ny, nz, h, r_grid);
      }
      any |= changed;
      dist_push(changed, b, x, y, z, nx, ny, nz, fixed0, stamp, qout, qlen, it);
    }
    if (__any_sync(full, any) && (threadIdx.x & 31) == 0) flags[it] = 1;
    if (!grid_sync(sync, expected, budget_ns, status)) return;
  }
}

// iters = 1 + index of the first sweep that changed nothing (or -1), and a
// device status if the budget ran out.  One warp; result (device, nullable)
// gets the same number as iters, or kSweepsAborted where a barrier wait ran out
// (sync[2], with DCM_ERR_TIMEOUT in the status already): the flags of the
// sweeps that did not run are zero then too, and mean nothing.
constexpr int kSweepsAborted = -2;
__global__ void k_dist_finish(const int32_t* flags, int sweeps, const uint32_t* sync, int32_t* iters, int32_t* result,
                              int32_t* status) {
  const int lane = threadIdx.x;
  const bool aborted = sync[2] != 0;
  int first = -1;
  for (int k0 = 0; k0 < sweeps && first < 0; k0 += 32) {
    const unsigned m = __ballot_sync(0xffffffffu, k0 + lane < sweeps && flags[k0 + lane] == 0);
    if (m) first = k0 + __ffs(m) - 1;
  }
  if (lane == 0) {
    const int v = first >= 0 && !aborted ? first + 1 : -1;
    if (iters) *iters = v;
    if (result) *result = aborted ? kSweepsAborted : v;
    if (first < 0 && !aborted) raise_status(status, DCM_ERR_NOT_CONVERGED);
  }
}

template <typename R>
int distance_sweeps(dcm_ctx* ctx, const uint8_t* s, const uint8_t* iface, R* D, int32_t* iters, bool host_check,
                    cudaStream_t st) {
  int nx = (int)ctx->nh[0], ny = (int)ctx->nh[1], nz = (int)ctx->nh[2];
  int64_t nbox = ctx->nbox;
  R h = (R)ctx->p.h, rg = (R)ctx->p.r_grid;
  R* buf[2] = {D, (R*)ctx->D[1]};
  int32_t* q[2] = {ctx->dq[0], ctx->dq[1]};
  const int iter_max = ctx->p.iter_max;
  // without a host check the budget is rounded up to an even number of sweeps,
  // so that the last iterate is in D wherever the sweeps end
  const int budget = host_check ? iter_max : iter_max + (iter_max & 1);
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->flags, 0, sizeof(int32_t) * (size_t)(iter_max + 2), st));
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->dqlen, 0, sizeof(int32_t) * (size_t)(iter_max + 2), st));
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->dstamp, 0xff, sizeof(int32_t) * (size_t)nbox, st));
  const int64_t cols = (int64_t)((nx + 31) / 32) * ((ny + 7) / 8);
  const int zc = (int)std::max<int64_t>(1, std::min<int64_t>(64, (int64_t)nz * cols / (152 * 8)));
  bool four = false;
  if constexpr (sizeof(R) == 4) {
    four = nx % 4 == 0 && (((uintptr_t)s | (uintptr_t)iface) & 3) == 0 && ((uintptr_t)D & 15) == 0;
    if (four) {
      const int64_t cols4 = (int64_t)((nx / 4 + 31) / 32) * ((ny + 7) / 8);
      const int zc4 = (int)std::max<int64_t>(1, std::min<int64_t>(64, (int64_t)nz * cols4 / (152 * 8)));
      DCM_LAUNCH(ctx, k_dist_first4, dim3((nx / 4 + 31) / 32, (ny + 7) / 8, (nz + zc4 - 1) / zc4), 256, 0, st, s, iface,
                 buf[0], buf[1], nx, ny, nz, zc4, h, rg, ctx->dfixed);
    }
  }
  if (!four)
    DCM_LAUNCH(ctx, k_dist_first<R>, dim3((nx + 31) / 32, (ny + 7) / 8, (nz + zc - 1) / zc), 256, 0, st, s, iface,
               buf[0], buf[1], nx, ny, nz, zc, h, rg, ctx->dfixed);
  DCM_LAUNCH(ctx, k_dist_queue0<R>, (unsigned)std::min<int64_t>((nbox + 255) / 256, 152 * 8), 256, 0, st, buf[1], nbox,
             nx, ny, nz, ctx->dfixed, ctx->dstamp, q[1], ctx->dqlen, ctx->flags);
  auto kern = k_dist_coop<R>;
  int per_sm = 0, sms = 0, dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCoopBlock, 0) != cudaSuccess || per_sm < 1)
    return set_error(ctx, DCM_ERR_CUDA, "distance sweeps: occupancy query failed");
  cudaLaunchConfig_t cfg = {};
  // no more blocks than boxes to sweep
  cfg.gridDim = dim3((unsigned)std::min<int64_t>((nbox + kCoopBlock - 1) / kCoopBlock, sms));
  cfg.blockDim = dim3(kCoopBlock);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->coop_sync, 0, 4 * sizeof(uint32_t), st));
  ++ctx->launches;
  cudaError_t e = cudaLaunchKernelEx(&cfg, kern, buf[0], buf[1], nx, ny, nz, h, rg, (const uint8_t*)ctx->dfixed,
                                     ctx->dstamp, q[0], q[1], ctx->dqlen, ctx->flags, budget, ctx->coop_sync,
                                     ctx->wait_budget, ctx->status);
  if (e != cudaSuccess) return set_error(ctx, DCM_ERR_CUDA, "distance sweeps: %s", cudaGetErrorString(e));
  DCM_LAUNCH(ctx, k_dist_finish, 1, 32, 0, st, ctx->flags, budget, (const uint32_t*)ctx->coop_sync, iters,
             host_check ? ctx->thr + 3 : nullptr, ctx->status);
  if (host_check) {
    DCM_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->host_status, ctx->thr + 3, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    DCM_CUDA_TRY(ctx, cudaStreamSynchronize(st));
    if (ctx->host_status[0] == kSweepsAborted)
      return set_error(ctx, DCM_ERR_TIMEOUT, "distance sweeps: a grid barrier's wait ran out");
    if (ctx->host_status[0] < 0) {
      if (iter_max & 1) DCM_CUDA_TRY(ctx, cudaMemcpyAsync(D, buf[1], sizeof(R) * nbox, cudaMemcpyDeviceToDevice, st));
      check_launch(ctx, "distance_sweeps");
      return set_error(ctx, DCM_ERR_NOT_CONVERGED, "fast sweeping did not converge in %d sweeps", iter_max);
    }
  }
  return check_launch(ctx, "distance_sweeps");
}

template int distance_sweeps<float>(dcm_ctx*, const uint8_t*, const uint8_t*, float*, int32_t*, bool, cudaStream_t);
template int distance_sweeps<double>(dcm_ctx*, const uint8_t*, const uint8_t*, double*, int32_t*, bool,
                                     cudaStream_t);

}  // namespace dcm
