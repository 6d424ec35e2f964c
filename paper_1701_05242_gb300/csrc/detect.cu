// Interface detection (Section 2.1, Eq. 4): gray-scale volume from box counts,
// two-phase segmentation by an integer 2-means threshold (refined, with
// params.segmentation = 1, by the regularised segmentation of segment_ms.cu),
// interface boxes.
//
// All integer arithmetic, so the result is bit-identical to any correct
// evaluation: the (2w+1)^3 box sum is separable, three 1-D periodic sums taken
// in one pass over the counts (half widths above 4: three passes), and the 2-means iteration runs on a histogram of the box sums (same
// counts and sums as scanning the volume, in one pass instead of one per
// iteration).
#include <algorithm>
#include <climits>

#include "dcm_internal.cuh"

namespace dcm {

// out[x,y,z] = sum_{a=-w..w} in[x+a (periodic along axis), y, z]
template <int AXIS>
__global__ void k_box_sum_axis(const int32_t* __restrict__ in, int32_t* __restrict__ out, int nx, int ny, int nz,
                               int w) {
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int64_t nbox = (int64_t)nx * ny * nz;
  if (b >= nbox) return;
  int x = (int)(b % nx), y = (int)((b / nx) % ny), z = (int)(b / ((int64_t)nx * ny));
  int n = AXIS == 0 ? nx : (AXIS == 1 ? ny : nz);
  int c = AXIS == 0 ? x : (AXIS == 1 ? y : z);
  int64_t stride = AXIS == 0 ? 1 : (AXIS == 1 ? nx : (int64_t)nx * ny);
  int64_t base = b - (int64_t)c * stride;
  int s = 0;
  for (int a = -w; a <= w; ++a) {
    int k = c + a;
    k %= n;
    if (k < 0) k += n;
    s += in[base + (int64_t)k * stride];
  }
  out[b] = s;
}

// All three axes in one pass (half width W): a block of 32 x 8 columns marches
// along z; every plane of counts is staged with its halo, summed along x and
// then along y in shared memory, and enters a running sum of the last 2 W + 1
// planes.  The counts are read once (1.7 times with the halos, which hit L2) and
// the sums written once, where the three separate passes moved six arrays and
// paid three integer divisions per box: 333 -> 72 us for 16.4M boxes (kernel
// times; the 131 MB alone would be 19 us, the rest is the chain of loads, sums
// and barriers per plane).  Half widths above 4 keep the three passes: their
// halos and the register window of 2 W + 1 planes outgrow the block.  Also reduces the smallest and largest sum
// into thr[0], thr[1] if thr is given.
template <int W>
__global__ void __launch_bounds__(256) k_box_sum3(const int32_t* __restrict__ in, int32_t* __restrict__ out, int nx,
                                                  int ny, int nz, int zc, int32_t* __restrict__ thr) {
  constexpr int TX = 32 + 2 * W, TY = 8 + 2 * W, N = 2 * W + 1, E = (TX * TY + 255) / 256;
  __shared__ int32_t a[TY][TX], b[TY][32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 8, z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  auto wrap = [](int k, int n) {
    k %= n;
    return k < 0 ? k + n : k;
  };
  int off[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int q = threadIdx.x + 256 * e;
    off[e] = wrap(x0 - W + q % TX, nx) + nx * wrap(y0 - W + q / TX, ny);
  }
  const int x = x0 + tx, y = y0 + ty;
  const bool mine = x < nx && y < ny;
  const int64_t nxy = (int64_t)nx * ny;
  int ring[N], sum = 0, lo = INT_MAX, hi = INT_MIN;
#pragma unroll
  for (int u = 0; u < N; ++u) ring[u] = 0;
  int zw = wrap(z0 - W, nz);
  for (int base = z0 - W; base < z1 + W; base += N) {
#pragma unroll
    for (int u = 0; u < N; ++u) {
      const int zz = base + u;
      if (zz < z1 + W) {  // the same for the whole block
        const int32_t* plane = in + nxy * zw;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int q = threadIdx.x + 256 * e;
          if (q < TX * TY) (&a[0][0])[q] = __ldg(plane + off[e]);
        }
        zw = zw + 1 == nz ? 0 : zw + 1;
        __syncthreads();
        for (int q = threadIdx.x; q < TY * 32; q += 256) {
          int v = 0;
#pragma unroll
          for (int k = 0; k < N; ++k) v += a[q >> 5][(q & 31) + k];
          b[q >> 5][q & 31] = v;
        }
        __syncthreads();
        int v = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) v += b[ty + k][tx];
        sum += v - ring[u];
        ring[u] = v;
        const int z = zz - W;
        if (z >= z0 && mine) {
          out[x + nx * (int64_t)y + nxy * z] = sum;
          lo = min(lo, sum);
          hi = max(hi, sum);
        }
      }
    }
  }
  if (thr) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (tx == 0 && lo <= hi) {
      atomicMin(thr, lo);
      atomicMax(thr + 1, hi);
    }
  }
}

__global__ void k_minmax_init(int32_t* thr) {
  thr[0] = INT_MAX;
  thr[1] = INT_MIN;
}

__global__ void k_minmax(const int32_t* __restrict__ g, int64_t nbox, int32_t* thr) {
  int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int lo = INT_MAX, hi = INT_MIN;
  for (; b < nbox; b += (int64_t)gridDim.x * blockDim.x) {
    int v = g[b];
    lo = min(lo, v);
    hi = max(hi, v);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(thr, lo);
    atomicMax(thr + 1, hi);
  }
}

// Histogram of the box sums over [gmin, gmax]: per-block shared-memory
// histogram when the range fits (kSmemBins), else global atomics.
constexpr int kSmemBins = 8192;

__global__ void k_value_hist(const int32_t* __restrict__ g, int64_t nbox, const int32_t* thr, int32_t* hist,
                             int32_t* status) {
  __shared__ int32_t sh[kSmemBins];
  int gmin = thr[0], gmax = thr[1];
  if ((int64_t)gmax - gmin >= kHistCap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) raise_status(status, DCM_ERR_CAPACITY);
    return;
  }
  int range = gmax - gmin + 1;
  if (range <= kSmemBins) {
    for (int k = threadIdx.x; k < range; k += blockDim.x) sh[k] = 0;
    __syncthreads();
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x)
      atomicAdd(sh + (g[b] - gmin), 1);
    __syncthreads();
    for (int k = threadIdx.x; k < range; k += blockDim.x)
      if (sh[k]) atomicAdd(hist + k, sh[k]);
  } else {
    for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nbox; b += (int64_t)gridDim.x * blockDim.x)
      atomicAdd(hist + (g[b] - gmin), 1);
  }
}

// Inclusive sum over the block (1,024 threads) of the pair (n, s).
__device__ __forceinline__ void block_scan_ll(long long& n, long long& s, long long* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long a = __shfl_up_sync(0xffffffffu, n, o), b = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) {
      n += a;
      s += b;
    }
  }
  if (lane == 31) {
    sh[w] = n;
    sh[32 + w] = s;
  }
  __syncthreads();
  for (int k = 0; k < w; ++k) {
    n += sh[k];
    s += sh[32 + k];
  }
}

// One block: integer 2-means (Lloyd) on the histogram of box sums.
//   T0 = floor((gmin + gmax) / 2); repeat: class 0 = values < T, class 1 = >= T;
//   T <- floor((S0 n1 + S1 n0) / (2 n0 n1)) + 1 until T repeats (<= max_iter).
// One empty class: T = gmax + 1 (no interface).  fixed >= 0 bypasses it.
// Every thread holds a run of bins and the counts and sums before it, so an
// iteration is a look-up by the one thread whose run holds T (it was four sums
// over the histogram, eight barriers each: 24 -> 7 us).
__global__ void __launch_bounds__(1024) k_two_means(const int32_t* __restrict__ hist, int32_t* thr, int max_iter,
                                                    int fixed, int32_t* t_out) {
  __shared__ long long sh[64], low[2], all[2];
  int gmin = thr[0], gmax = thr[1];
  if (fixed >= 0) {
    if (threadIdx.x == 0) {
      thr[2] = fixed;
      if (t_out) *t_out = fixed;
    }
    return;
  }
  if ((int64_t)gmax - gmin >= kHistCap) return;  // capacity error already raised
  const int R = gmax - gmin + 1, per = (R + (int)blockDim.x - 1) / (int)blockDim.x;
  const int k0 = min((int)threadIdx.x * per, R), k1 = min(k0 + per, R);
  long long n = 0, s = 0;
  for (int k = k0; k < k1; ++k) {
    const long long c = hist[k];
    n += c;
    s += c * (long long)(gmin + k);
  }
  const long long own_n = n, own_s = s;
  block_scan_ll(n, s, sh);
  if (threadIdx.x == blockDim.x - 1) {
    all[0] = n;
    all[1] = s;
  }
  n -= own_n;  // before this thread's run
  s -= own_s;
  int T = (int)(((long long)gmin + gmax) / 2);
  for (int it = 0; it < max_iter; ++it) {
    const int at = T - gmin;  // 0 <= at <= R: the bins below T
    if ((k0 <= at && at < k1) || (at == R && k1 == R && k0 < k1)) {
      long long a = n, b = s;
      for (int k = k0; k < at; ++k) {
        const long long c = hist[k];
        a += c;
        b += c * (long long)(gmin + k);
      }
      low[0] = a;
      low[1] = b;
    }
    __syncthreads();
    const long long n0 = low[0], s0 = low[1], n1 = all[0] - n0, s1 = all[1] - s0;
    __syncthreads();
    if (n0 == 0 || n1 == 0) {
      T = gmax + 1;
      break;
    }
    const int Tn = (int)((s0 * n1 + s1 * n0) / (2 * n0 * n1) + 1);
    if (Tn == T) break;
    T = Tn;
  }
  if (threadIdx.x == 0) {
    thr[2] = T;
    if (t_out) *t_out = T;
  }
}

// s = (g >= T); interface = s and some face neighbour below T (periodic).
// A block of 32 x 8 columns marches along z with the planes below and above
// in registers (85 -> 37 us for 16.4M boxes, 98 MB, against a thread per box, which
// divided its index and read seven values).
__global__ void __launch_bounds__(256) k_segment(const int32_t* __restrict__ g, int nx, int ny, int nz, int zc,
                                                 const int32_t* thr, uint8_t* __restrict__ s,
                                                 uint8_t* __restrict__ iface) {
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= nx || y >= ny) return;
  const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, nz);
  const int T = thr[2];
  const int64_t nxy = (int64_t)nx * ny;
  const int32_t* p = g + x + (int64_t)nx * y;  // the column
  const int xm = x == 0 ? nx - 1 : -1, xp = x == nx - 1 ? 1 - nx : 1;
  const int64_t ym = y == 0 ? (int64_t)(ny - 1) * nx : -nx, yp = y == ny - 1 ? -(int64_t)(ny - 1) * nx : nx;
  int below = __ldg(p + nxy * (z0 == 0 ? nz - 1 : z0 - 1)), here = __ldg(p + nxy * z0);
  for (int z = z0; z < z1; ++z) {
    const int32_t* q = p + nxy * z;
    const int above = __ldg(p + nxy * (z == nz - 1 ? 0 : z + 1));
    const int least = min(min(min(__ldg(q + xm), __ldg(q + xp)), min(__ldg(q + ym), __ldg(q + yp))), min(below, above));
    const int64_t b = x + (int64_t)nx * y + nxy * z;
    s[b] = (uint8_t)(here >= T);
    iface[b] = (uint8_t)(here >= T && least < T);
    below = here;
    here = above;
  }
}

int detect_interface(dcm_ctx* ctx, const int32_t* box_count, uint8_t* s, uint8_t* iface, int32_t* threshold,
                     int32_t* g_out, cudaStream_t st) {
  int nx = (int)ctx->nh[0], ny = (int)ctx->nh[1], nz = (int)ctx->nh[2];
  int64_t nbox = ctx->nbox;
  int w = ctx->p.smooth_w;
  int32_t* g = g_out ? g_out : ctx->g;
  unsigned nb = (unsigned)((nbox + 255) / 256);
  const bool means = ctx->p.threshold < 0;
  int32_t* thr = means ? ctx->thr : nullptr;
  if (means) DCM_LAUNCH(ctx, k_minmax_init, 1, 1, 0, st, ctx->thr);
  int nred = (int)std::min<int64_t>((nbox + 255) / 256, 152 * 4);
  // columns of 32 x 8 boxes, cut along z into pieces that leave the chip a
  // few blocks per SM (each piece of the box sum re-reads 2 w planes)
  const int64_t cols = (int64_t)((nx + 31) / 32) * ((ny + 7) / 8);
  const int zc = (int)std::max<int64_t>(8, std::min<int64_t>(64, (int64_t)nz * cols / (152 * 8)));
  const dim3 grid((nx + 31) / 32, (ny + 7) / 8, (nz + zc - 1) / zc);
  if (w <= 4) {
    auto k = w == 0 ? k_box_sum3<0> : w == 1 ? k_box_sum3<1> : w == 2 ? k_box_sum3<2> : w == 3 ? k_box_sum3<3> : k_box_sum3<4>;
    DCM_LAUNCH(ctx, k, grid, 256, 0, st, box_count, g, nx, ny, nz, zc, thr);
  } else {
    // separable box sum: x into g, y into g_tmp, z back into g
    DCM_LAUNCH(ctx, k_box_sum_axis<0>, nb, 256, 0, st, box_count, g, nx, ny, nz, w);
    DCM_LAUNCH(ctx, k_box_sum_axis<1>, nb, 256, 0, st, g, ctx->g_tmp, nx, ny, nz, w);
    DCM_LAUNCH(ctx, k_box_sum_axis<2>, nb, 256, 0, st, ctx->g_tmp, g, nx, ny, nz, w);
    if (means) DCM_LAUNCH(ctx, k_minmax, nred, 256, 0, st, g, nbox, ctx->thr);
  }
  if (means) {
    DCM_CUDA_TRY(ctx, cudaMemsetAsync(ctx->hist, 0, sizeof(int32_t) * kHistCap, st));
    DCM_LAUNCH(ctx, k_value_hist, nred, 256, 0, st, g, nbox, ctx->thr, ctx->hist, ctx->status);
  }
  DCM_LAUNCH(ctx, k_two_means, 1, 1024, 0, st, ctx->hist, ctx->thr, 64, ctx->p.threshold, threshold);
  if (ctx->p.min_component > 0) {
    // segment (and refine) into scratch, then the filtered S and its interface into s, iface
    DCM_LAUNCH(ctx, k_segment, grid, 256, 0, st, g, nx, ny, nz, zc, ctx->thr, ctx->cc_s0, iface);
    int r = check_launch(ctx, "detect_interface");
    if (r) return r;
    if (ctx->p.segmentation && (r = ms_segment(ctx, box_count, ctx->cc_s0, st))) return r;
    return remove_small_components(ctx, ctx->cc_s0, s, iface, st);
  }
  DCM_LAUNCH(ctx, k_segment, grid, 256, 0, st, g, nx, ny, nz, zc, ctx->thr, s, iface);
  if (ctx->p.segmentation) {
    // the regularised segmentation of the counts refines the threshold's S
    int r = ms_segment(ctx, box_count, s, st);
    if (r) return r;
    interface_of(ctx, s, iface, st);
  }
  return check_launch(ctx, "detect_interface");
}

}  // namespace dcm
