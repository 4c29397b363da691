// Device side of the warm start (include/lbm_warm.h): the droplet-field fill and the
// phase-averaged density sums.
#include <cuda_runtime.h>

#include "lbm_internal.h"

namespace lbm {

namespace {

// Both field kernels work on tiles of kTileX x kTileY nodes, four to a thread.
constexpr int kTileX = 64, kTileY = 16, kFillThreads = 256;
constexpr int kTileNodes = kTileX * kTileY / kFillThreads;
constexpr int kDropTile = 256;  // droplets staged in shared memory per pass

// First node of this block's tile (tiles are numbered along x, then y).
__device__ __forceinline__ void tile_origin(int nx, int& x0, int& y0) {
  const unsigned across = (unsigned)((nx + kTileX - 1) / kTileX);
  x0 = (int)(blockIdx.x % across) * kTileX;
  y0 = (int)(blockIdx.x / across) * kTileY;
}

// Smallest periodic distance (as the kernel below forms it) of a coordinate to the integers
// lo .. hi: on either side of c it rises to half the period and falls again, so it is
// smallest at an end unless c lies between them.  Only for c in [0, n].
__device__ __forceinline__ double range_distance(double c, int lo, int hi, int n) {
  if (c >= (double)lo && c <= (double)hi) return 0.0;
  const double a = fabs((double)lo - c), b = fabs((double)hi - c);
  return fmin(fmin(a, (double)n - a), fmin(b, (double)n - b));
}

// The largest tanh profile over the droplets within reach (8 widths beyond the half-density
// circle), else rho_v.  A droplet is staged for a tile only if it reaches it (with a node to
// spare), so a node looks at the few droplets near it instead of all: with 64 droplets on
// 4096^2 the FP64 distances to all of them took 36 ms, this takes 1.  Inside a
// droplet, where tanh rounds to -1, it is not evaluated.  The order of the staged droplets
// varies from run to run; their maximum does not.
__global__ void __launch_bounds__(kFillThreads) fill_droplets_kernel(
    double* __restrict__ rho, int nx, int ny, const DropRec* __restrict__ drops, int n,
    double rho_v, double width) {
  __shared__ DropRec sd[kDropTile];
  __shared__ int count;
  int x0, y0;
  tile_origin(nx, x0, y0);
  const int x1 = min(x0 + kTileX, nx) - 1, y1 = min(y0 + kTileY, ny) - 1;
  const int x = x0 + (int)threadIdx.x % kTileX, yt = y0 + (int)threadIdx.x / kTileX;
  const double reach = 8.0 * width;
  double best[kTileNodes];
#pragma unroll
  for (int j = 0; j < kTileNodes; ++j) best[j] = rho_v;
  for (int base = 0; base < n; base += kDropTile) {
    const int k0 = base + (int)threadIdx.x;
    __syncthreads();
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    if (k0 < n) {
      const DropRec d = drops[k0];
      bool near = true;
      if (d.cx >= 0.0 && d.cx <= (double)nx && d.cy >= 0.0 && d.cy <= (double)ny) {
        const double dx = range_distance(d.cx, x0, x1, nx), dy = range_distance(d.cy, y0, y1, ny);
        near = sqrt(dx * dx + dy * dy) <= d.r_half + reach + 1.0;
      }
      if (near) sd[atomicAdd(&count, 1)] = d;
    }
    __syncthreads();
    const int m = count;
    for (int k = 0; k < m; ++k) {
      const DropRec d = sd[k];
      double dx = fabs((double)x - d.cx);
      dx = fmin(dx, (double)nx - dx);
#pragma unroll
      for (int j = 0; j < kTileNodes; ++j) {
        double dy = fabs((double)(yt + j * (kTileY / kTileNodes)) - d.cy);
        dy = fmin(dy, (double)ny - dy);
        const double s = sqrt(::fma(dx, dx, dy * dy)) - d.r_half;
        if (s > reach) continue;
        const double t = 2.0 * s / width;
        // rounded before it is subtracted, whatever the compiler contracts around it
        const double fall = __dmul_rn(0.5 * (d.rho_in - rho_v), t < -20.0 ? -1.0 : tanh(t));
        const double v = 0.5 * (d.rho_in + rho_v) - fall;
        best[j] = fmax(best[j], v);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kTileNodes; ++j) {
    const int y = yt + j * (kTileY / kTileNodes);
    if (x < nx && y < ny) rho[(long long)y * nx + x] = best[j];
  }
}

// u0 = -F / (2 rho) with F of Eq. 7 from psi of Eq. 24 of the density field: the initial
// velocity for which the force-corrected velocity of Eq. 6, (sum e f + F/2) / rho, is zero
// when f is the equilibrium at (rho, u0).  psi beyond a wall is that of the adjacent row.
// FP64-bound: psi (a division and a square root) is evaluated once per node of the tile and
// its one-node border into shared memory, 1.16 times per node, instead of nine times
// (4096^2: 9.9 ms before, 2.4 now).
__global__ void __launch_bounds__(kFillThreads) balanced_velocity_kernel(
    const double* __restrict__ rho, InstParams P, double* __restrict__ ux,
    double* __restrict__ uy) {
  constexpr int W = kTileX + 2, H = kTileY + 2;
  __shared__ double psi[H][W];
  const int nx = P.nx, ny = P.ny;
  int x0, y0;
  tile_origin(nx, x0, y0);
  for (int i = threadIdx.x; i < W * H; i += kFillThreads) {
    const int r = i / W, c = i - r * W;
    const int xx = wrapi(x0 + c - 1, nx);
    const int yr = y0 + r - 1;
    const int yy = P.walls ? (yr < 0 ? 0 : (yr >= ny ? ny - 1 : yr)) : wrapi(yr, ny);
    psi[r][c] = psi_eval_f64(rho[(long long)yy * nx + xx], P.b4, P.RT, P.a, P.two_over_G);
  }
  __syncthreads();
  const int cx = (int)threadIdx.x % kTileX, x = x0 + cx;
#pragma unroll
  for (int j = 0; j < kTileNodes; ++j) {
    const int cy = (int)threadIdx.x / kTileX + j * (kTileY / kTileNodes), y = y0 + cy;
    if (x >= nx || y >= ny) continue;
    double gx = 0.0, gy = 0.0;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
      const double w = (q <= 4) ? (1.0 / 3.0) : (1.0 / 12.0);
      const double wp = w * psi[1 + cy + ey_of(q)][1 + cx + ex_of(q)];
      gx += wp * ex_of(q);
      gy += wp * ey_of(q);
    }
    const double f = -P.G * psi[1 + cy][1 + cx];  // F = -G psi(x) sum w psi(x + e) e
    const long long i = (long long)y * nx + x;
    const double r = rho[i];
    ux[i] = -0.5 * f * gx / r;
    uy[i] = -0.5 * f * gy / r;
  }
}

template <typename S>
__global__ void __launch_bounds__(256) phase_sums_kernel(const S* __restrict__ rho, long long n,
                                                         double vmax, double lmin,
                                                         double* __restrict__ part) {
  __shared__ double red[4][256];
  double sv = 0.0, cv = 0.0, sl = 0.0, cl = 0.0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < n;
       i += (long long)gridDim.x * 256) {
    const double r = (double)rho[i];
    if (r < vmax) {
      sv += r;
      cv += 1.0;
    }
    if (r > lmin) {
      sl += r;
      cl += 1.0;
    }
  }
  const int t = threadIdx.x;
  red[0][t] = sv;
  red[1][t] = cv;
  red[2][t] = sl;
  red[3][t] = cl;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (t < h)
      for (int k = 0; k < 4; ++k) red[k][t] += red[k][t + h];
    __syncthreads();
  }
  if (t < 4) part[4 * blockIdx.x + t] = red[t][0];
}

}  // namespace

// Blocks of the field kernels: one per tile.
static unsigned tiles(int nx, int ny) {
  return (unsigned)((nx + kTileX - 1) / kTileX) * (unsigned)((ny + kTileY - 1) / kTileY);
}

cudaError_t launch_fill_droplets(double* rho, int nx, int ny, const DropRec* drops, int n,
                                 double rho_v, double width, cudaStream_t st) {
  fill_droplets_kernel<<<tiles(nx, ny), kFillThreads, 0, st>>>(rho, nx, ny, drops, n, rho_v,
                                                               width);
  return cudaGetLastError();
}

cudaError_t launch_balanced_velocity(const double* rho, const InstParams& P, double* ux,
                                    double* uy, cudaStream_t st) {
  balanced_velocity_kernel<<<tiles(P.nx, P.ny), kFillThreads, 0, st>>>(rho, P, ux, uy);
  return cudaGetLastError();
}

template <typename S>
cudaError_t launch_phase_sums(const S* rho, long long n, double vmax, double lmin, double* part,
                              cudaStream_t st) {
  phase_sums_kernel<S><<<kPhaseBlocks, 256, 0, st>>>(rho, n, vmax, lmin, part);
  return cudaGetLastError();
}

template cudaError_t launch_phase_sums<float>(const float*, long long, double, double, double*,
                                              cudaStream_t);
template cudaError_t launch_phase_sums<double>(const double*, long long, double, double, double*,
                                               cudaStream_t);

}  // namespace lbm
