// Regularised two-phase segmentation of the box counts (Section 2.1: the
// piecewise constant Mumford-Shah functional for two-phase segmentation,
// refs. [1, 18]), selected by params.segmentation = 1.
//
// The functional of a binary volume s with phase values c0, c1 is
//   E(s) = sum_b [ s_b (g_b - c1)^2 + (1 - s_b) (g_b - c0)^2 ] + nu sum_faces |s_b - s_b'|
// on the periodic grid of box counts g.  Starting from the threshold
// segmentation, each outer iteration sets c0, c1 to the means of g over the
// two phases (exact integer sums), then minimises the convex relaxation
//   min over u in [0,1]: sum_b w_b u_b + nu sum_faces |u_b - u_b'|,
//   w_b = (g_b - c1)^2 - (g_b - c0)^2,
// by the primal-dual iteration of Chambolle and Pock (one dual value per
// face, a stencil on the grid), and thresholds u at 1/2.  The loop stops
// after params.ms_outer iterations or when s no longer changes; the later
// launches of a finished loop exit at once (a device flag per iteration), so
// the host never waits.  Additions and products are rounded one by one
// (no fused multiply-add), in the order of the plain definition, so the FP64
// form reproduces an FP64 evaluation of the same steps.
#include "dcm_internal.cuh"

namespace dcm {

namespace {

constexpr double kMsTau = 0.28, kMsSigma = 0.28;  // tau sigma ||D||^2 < 1 with ||D||^2 <= 12

__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float r_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double r_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }

// Whether outer iteration o still runs: the earlier ones changed s, and both
// phases were present when it started (flags[0] is the stop mark).
__device__ __forceinline__ bool ms_active(const int32_t* flags, int o) {
  return flags[0] == 0 && (o == 0 || flags[o] != 0);
}

// Integer sums of the counts over the two phases: sums = {n0, S0, n1, S1}.
__global__ void k_ms_sums(const int32_t* __restrict__ g, const uint8_t* __restrict__ s, int64_t nbox,
                          unsigned long long* sums, const int32_t* flags, int o) {
  if (!ms_active(flags, o)) return;
  long long n1 = 0, s0 = 0, s1 = 0, n0 = 0;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    const int v = g[b];
    if (s[b]) {
      ++n1;
      s1 += v;
    } else {
      ++n0;
      s0 += v;
    }
  }
  for (int k = 16; k > 0; k >>= 1) {
    n0 += __shfl_xor_sync(0xffffffffu, n0, k);
    s0 += __shfl_xor_sync(0xffffffffu, s0, k);
    n1 += __shfl_xor_sync(0xffffffffu, n1, k);
    s1 += __shfl_xor_sync(0xffffffffu, s1, k);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(sums + 4 * o + 0, (unsigned long long)n0);
    atomicAdd(sums + 4 * o + 1, (unsigned long long)s0);
    atomicAdd(sums + 4 * o + 2, (unsigned long long)n1);
    atomicAdd(sums + 4 * o + 3, (unsigned long long)s1);
  }
}

// Phase values, data weights, and the start of the inner iteration (u = s, p = 0).
template <typename R>
__global__ void k_ms_start(const int32_t* __restrict__ g, const uint8_t* __restrict__ s, int64_t nbox,
                           const unsigned long long* sums, int32_t* flags, double* c, int o, R* __restrict__ w,
                           R* __restrict__ u, R* __restrict__ ub, R* __restrict__ p) {  // p: px, py, pz
  if (!ms_active(flags, o)) return;
  const unsigned long long n0 = sums[4 * o], n1 = sums[4 * o + 2];
  if (n0 == 0 || n1 == 0) {  // one phase is empty: s stays as it is
    if (blockIdx.x == 0 && threadIdx.x == 0) flags[0] = 1;
    return;
  }
  const double c0 = (double)(long long)sums[4 * o + 1] / (double)n0;
  const double c1 = (double)(long long)sums[4 * o + 3] / (double)n1;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    c[0] = c0;
    c[1] = c1;
  }
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    const double gv = (double)g[b];
    const double d1 = __dsub_rn(gv, c1), d0 = __dsub_rn(gv, c0);
    w[b] = (R)__dsub_rn(__dmul_rn(d1, d1), __dmul_rn(d0, d0));
    const R v = s[b] ? (R)1 : (R)0;
    u[b] = v;
    ub[b] = v;
    p[b] = p[nbox + b] = p[2 * nbox + b] = (R)0;
  }
}

// One inner iteration, from (ub, p) into (ub1, p1): the dual step
//   p_f <- clip(p_f + sigma (ubar_{b+e} - ubar_b), -nu, nu)
// for the three faces (b, b + e) of every box b, and the primal step
//   u' = clip(u - tau ((D^T p)_b + w_b), 0, 1), ubar = 2 u' - u
// in one pass: a thread forms the new duals of all six faces of its box (those
// it shares with the boxes below along x and y again, the one along z is carried
// from the box before as the thread marches along z), so nothing waits for
// another box.  44 B per box and iteration through HBM (two kernels: 68 B), and
// half the launches, which is what counts for grids that stay in L2: 1.05M
// boxes, 800 iterations, 11.7 -> 5.95 ms (7.4 us per iteration, of which the
// launch and the drain of one wave of blocks are most).
//
// The FP64 form is bound by the FP64 units: its blocks take 64 columns in a row,
// whatever the shape (blocks of 32 x 8 left 36% to 71% of their lanes idle in planes of
// 41 x 41, 33 x 9 and 16 x 16 boxes), and above kMsFused boxes the duals are not formed
// twice: two kernels, 17 FP64 operations per box instead of 26.  800 iterations, FP64,
// 32 x 8 / 64 in a row / two kernels: 41 x 41 x 164 boxes 22.3 / 13.2 / 14.1 ms, 1.05M
// 37.1 / 37.1 / 30.6, 4.1M 131 / 131 / 101.
constexpr int64_t kMsFused = 600000;
template <typename R>
constexpr int ms_block() { return sizeof(R) == 8 ? 64 : 256; }

template <typename R>
__global__ void __launch_bounds__(ms_block<R>()) k_ms_step(const R* __restrict__ ub, const R* __restrict__ p,
                                                 const R* __restrict__ w, R* __restrict__ u, R* __restrict__ ub1,
                                                 R* __restrict__ p1, int nx, int ny, int nz, int zc, R sigma, R tau,
                                                 R nu, const int32_t* flags, int o) {
  if (!ms_active(flags, o)) return;
  const int nxy = nx * ny;  // fewer than 2^31 boxes
  int x, y;
  if constexpr (sizeof(R) == 8) {
    const int c = blockIdx.x * ms_block<R>() + threadIdx.x;
    y = c / nx;
    x = c - nx * y;
  } else {
    x = blockIdx.x * 32 + (threadIdx.x & 31);
    y = blockIdx.y * 8 + (threadIdx.x >> 5);
  }
  if (x >= nx || y >= ny) return;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  const int col = x + nx * y;
  const int64_t nbox = (int64_t)nxy * nz;
  const R *px = p, *py = p + nbox, *pz = p + 2 * nbox;
  R *qx = p1, *qy = p1 + nbox, *qz = p1 + 2 * nbox;
  const int xm = x == 0 ? nx - 1 : -1, xp = x == nx - 1 ? 1 - nx : 1;
  const int ym = y == 0 ? (ny - 1) * nx : -nx, yp = y == ny - 1 ? -(ny - 1) * nx : nx;
  auto dual = [&](R pf, R ahead, R here) {
    const R q = r_add(pf, r_mul(sigma, r_sub(ahead, here)));
    return q < -nu ? -nu : (q > nu ? nu : q);
  };
  R here = __ldg(ub + col + nxy * z0);
  R dz;  // the dual of the face below along z
  {
    const int b = col + nxy * (z0 == 0 ? nz - 1 : z0 - 1);
    dz = dual(__ldg(pz + b), here, __ldg(ub + b));
  }
  for (int z = z0; z < z1; ++z) {
    const int b = col + nxy * z;
    const R above = __ldg(ub + (z == nz - 1 ? col : b + nxy));
    const R ux = __ldg(ub + b + xp), vx = __ldg(ub + b + xm), uy = __ldg(ub + b + yp), vy = __ldg(ub + b + ym);
    const R fx = dual(__ldg(px + b), ux, here), gx = dual(__ldg(px + b + xm), here, vx);
    const R fy = dual(__ldg(py + b), uy, here), gy = dual(__ldg(py + b + ym), here, vy);
    const R fz = dual(__ldg(pz + b), above, here);
    R dtp = r_add((R)0, r_sub(gx, fx));
    dtp = r_add(dtp, r_sub(gy, fy));
    dtp = r_add(dtp, r_sub(dz, fz));
    const R u0 = u[b];
    R v = r_sub(u0, r_mul(tau, r_add(dtp, __ldg(w + b))));
    v = v < (R)0 ? (R)0 : (v > (R)1 ? (R)1 : v);
    qx[b] = fx;
    qy[b] = fy;
    qz[b] = fz;
    ub1[b] = r_sub(r_mul((R)2, v), u0);
    u[b] = v;
    here = above;
    dz = fz;
  }
}

// The two steps of an iteration apart, in place (p: px, py, pz).
template <typename R>
__global__ void __launch_bounds__(256) k_ms_dual(const R* __restrict__ ub, R* __restrict__ p, int nx, int ny, int nz,
                                                 R sigma, R nu, const int32_t* flags, int o) {
  if (!ms_active(flags, o)) return;
  const int64_t nxy = (int64_t)nx * ny, nbox = nxy * nz;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(b % nx), y = (int)((b / nx) % ny), z = (int)(b / nxy);
    const int64_t ahead[3] = {x == nx - 1 ? b - x : b + 1, y == ny - 1 ? b - (int64_t)y * nx : b + nx,
                              z == nz - 1 ? b - z * nxy : b + nxy};
    const R here = ub[b];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const R q = r_add(p[e * nbox + b], r_mul(sigma, r_sub(ub[ahead[e]], here)));
      p[e * nbox + b] = q < -nu ? -nu : (q > nu ? nu : q);
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(256) k_ms_primal(const R* __restrict__ p, const R* __restrict__ w, R* __restrict__ u,
                                                   R* __restrict__ ub, int nx, int ny, int nz, R tau,
                                                   const int32_t* flags, int o) {
  if (!ms_active(flags, o)) return;
  const int64_t nxy = (int64_t)nx * ny, nbox = nxy * nz;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(b % nx), y = (int)((b / nx) % ny), z = (int)(b / nxy);
    const int64_t behind[3] = {x == 0 ? b + nx - 1 : b - 1, y == 0 ? b + (int64_t)(ny - 1) * nx : b - nx,
                               z == 0 ? b + (nz - 1) * nxy : b - nxy};
    R dtp = (R)0;
#pragma unroll
    for (int e = 0; e < 3; ++e) dtp = r_add(dtp, r_sub(p[e * nbox + behind[e]], p[e * nbox + b]));
    const R u0 = u[b];
    R v = r_sub(u0, r_mul(tau, r_add(dtp, w[b])));
    v = v < (R)0 ? (R)0 : (v > (R)1 ? (R)1 : v);
    ub[b] = r_sub(r_mul((R)2, v), u0);
    u[b] = v;
  }
}

// s = (u >= 1/2); flags[o + 1] = 1 if any box changed.
template <typename R>
__global__ void k_ms_threshold(const R* __restrict__ u, uint8_t* __restrict__ s, int64_t nbox, int32_t* flags,
                               int o) {
  if (!ms_active(flags, o)) return;
  bool changed = false;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t t = u[b] >= (R)0.5 ? 1 : 0;
    changed |= t != s[b];
    s[b] = t;
  }
  if (__any_sync(0xffffffffu, changed) && (threadIdx.x & 31) == 0) flags[o + 1] = 1;
}

template <typename R>
int ms_run(dcm_ctx* ctx, const int32_t* count, uint8_t* s, cudaStream_t st) {
  const int nx = (int)ctx->nh[0], ny = (int)ctx->nh[1], nz = (int)ctx->nh[2];
  const int64_t nbox = ctx->nbox;
  const int outer = ctx->p.ms_outer, inner = ctx->p.ms_inner;
  const unsigned grid = (unsigned)std::min<int64_t>((nbox + 255) / 256, 152 * 8);
  R* u = (R*)ctx->ms_u;
  R* ub[2] = {(R*)ctx->ms_ub, (R*)ctx->ms_ub + nbox};
  R* p[2] = {(R*)ctx->ms_p, (R*)ctx->ms_p + 3 * nbox};
  R* w = (R*)ctx->ms_w;
  // columns of boxes, cut along z so that small grids fill the chip
  constexpr bool kRow = sizeof(R) == 8;
  constexpr int kBlock = ms_block<R>();
  const int cx = kRow ? (int)(((int64_t)nx * ny + kBlock - 1) / kBlock) : (nx + 31) / 32, cy = kRow ? 1 : (ny + 7) / 8;
  const int zc = (int)std::max<int64_t>(4, std::min<int64_t>(32, (int64_t)nz * cx * cy / (152 * 6 * (256 / kBlock))));
  const dim3 blocks(cx, cy, (nz + zc - 1) / zc);
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->ms_flags, 0, sizeof(int32_t) * (size_t)(outer + 2), st));
  DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->ms_sums, 0, sizeof(unsigned long long) * 4 * (size_t)outer, st));
  for (int o = 0; o < outer; ++o) {
    DCM_LAUNCH(ctx, k_ms_sums, grid, 256, 0, st, count, s, nbox, ctx->ms_sums, ctx->ms_flags, o);
    DCM_LAUNCH(ctx, k_ms_start<R>, grid, 256, 0, st, count, s, nbox, ctx->ms_sums, ctx->ms_flags, ctx->ms_c, o, w, u,
               ub[0], p[0]);
    for (int it = 0; it < inner; ++it) {
      if (kRow && nbox >= kMsFused) {
        DCM_LAUNCH(ctx, k_ms_dual<R>, grid, 256, 0, st, ub[0], p[0], nx, ny, nz, (R)kMsSigma, (R)ctx->p.ms_nu,
                   ctx->ms_flags, o);
        DCM_LAUNCH(ctx, k_ms_primal<R>, grid, 256, 0, st, p[0], w, u, ub[0], nx, ny, nz, (R)kMsTau, ctx->ms_flags, o);
      } else {
        DCM_LAUNCH(ctx, k_ms_step<R>, blocks, kBlock, 0, st, ub[it & 1], p[it & 1], w, u, ub[(it + 1) & 1],
                   p[(it + 1) & 1], nx, ny, nz, zc, (R)kMsSigma, (R)kMsTau, (R)ctx->p.ms_nu, ctx->ms_flags, o);
      }
    }
    DCM_LAUNCH(ctx, k_ms_threshold<R>, grid, 256, 0, st, u, s, nbox, ctx->ms_flags, o);
  }
  return check_launch(ctx, "ms_segment");
}

}  // namespace

int ms_segment(dcm_ctx* ctx, const int32_t* count, uint8_t* s, cudaStream_t st) {
  if (ctx->precision == DCM_PREC_FP64) return ms_run<double>(ctx, count, s, st);
  return ms_run<float>(ctx, count, s, st);
}

}  // namespace dcm
