// Device passes of the spectral diagnostics around the FFTs (lbm_spectral.h). FP64
// throughput is 1/64 of FP32's on this part, so the FP64 instructions of a pass, not its
// bytes, bound it at these sizes; each pass reads its inputs once and keeps no
// intermediate field.
#include <cmath>

#include "api_common.h"
#include "lbm_spectral.h"

using namespace lbm;

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 1216;
constexpr int kMaxShells = 6000;  // shared-memory histogram of at most 48 KB

// Integer wavenumber of index j on an axis of n points (fftfreq's order).
__device__ __forceinline__ int wavenumber(int j, int n) { return j < (n + 1) / 2 ? j : j - n; }

struct Grid {
  int nx, ny, nz, nxh;
  unsigned modes;  // of a half spectrum
};

__device__ __forceinline__ void mode_of(const Grid& g, unsigned m, int& x, int& y, int& z) {
  const unsigned row = m / (unsigned)g.nxh;
  x = (int)(m - row * (unsigned)g.nxh);
  const unsigned zz = row / (unsigned)g.ny;
  y = (int)(row - zz * (unsigned)g.ny);
  z = (int)zz;
}

// (a + ib) of i (p q - r s): the derivative's factor i turns (re, im) into (-im, re).
__global__ void __launch_bounds__(kThreads) k_curl_div(const Grid g, const double2* __restrict__ u,
                                                       double2* __restrict__ w, double scale) {
  const unsigned n = g.modes;
  for (unsigned m = blockIdx.x * kThreads + threadIdx.x; m < n; m += gridDim.x * kThreads) {
    int x, y, z;
    mode_of(g, m, x, y, z);
    // an even axis has no derivative of its Nyquist mode
    const double kx = 2 * x == g.nx ? 0.0 : scale * x;
    const double ky = 2 * y == g.ny ? 0.0 : scale * wavenumber(y, g.ny);
    const double kz = 2 * z == g.nz ? 0.0 : scale * wavenumber(z, g.nz);
    const size_t N = n;
    const double2 a = u[m], b = u[N + m], c = u[2 * N + m];
    w[m] = make_double2(kz * b.y - ky * c.y, ky * c.x - kz * b.x);
    w[N + m] = make_double2(kx * c.y - kz * a.y, kz * a.x - kx * c.x);
    w[2 * N + m] = make_double2(ky * a.y - kx * b.y, kx * b.x - ky * a.x);
    w[3 * N + m] = make_double2(-(kx * a.y + ky * b.y + kz * c.y), kx * a.x + ky * b.x + kz * c.x);
  }
}

// Block sums of m |w|^2 and m d^2 (fixed order), then one block adds the partials.
__global__ void __launch_bounds__(kThreads) k_dissipation(const double* __restrict__ w,
                                                          const double* __restrict__ T, long long n,
                                                          double mu, double inv_T_ref, int sutherland,
                                                          double* __restrict__ partials) {
  __shared__ double sh[2][kThreads];
  double s = 0.0, d = 0.0;
  for (long long i = blockIdx.x * (long long)kThreads + threadIdx.x; i < n;
       i += (long long)gridDim.x * kThreads) {
    double m = mu;
    if (sutherland) {
      const double t = T[i] * inv_T_ref;
      m = mu * ((1.0 + 0.4042) * (t * sqrt(t)) / (t + 0.4042));
    }
    const double wx = w[i], wy = w[n + i], wz = w[2 * n + i], dv = w[3 * n + i];
    s += m * (wx * wx + wy * wy + wz * wz);
    d += m * (dv * dv);
  }
  sh[0][threadIdx.x] = s;
  sh[1][threadIdx.x] = d;
  __syncthreads();
  for (int half = kThreads / 2; half > 0; half >>= 1) {
    if ((int)threadIdx.x < half) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + half];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + half];
    }
    __syncthreads();
  }
  if (threadIdx.x < 2) partials[2 * blockIdx.x + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void __launch_bounds__(kThreads) k_dissipation_final(const double* __restrict__ partials,
                                                                int blocks, double inv_n,
                                                                double* __restrict__ out) {
  __shared__ double sh[2][kThreads / 2];
  const int j = threadIdx.x & 1, t = threadIdx.x >> 1;
  double r = 0.0;
  for (int b = t; b < blocks; b += kThreads / 2) r += partials[2 * b + j];
  sh[j][t] = r;
  __syncthreads();
  for (int half = kThreads / 4; half > 0; half >>= 1) {
    if (t < half) sh[j][t] += sh[j][t + half];
    __syncthreads();
  }
  if (threadIdx.x < 2) out[threadIdx.x] = sh[threadIdx.x][0] * inv_n;
}

// Shell sums: 32 consecutive modes of a warp mostly share their shell with their
// neighbours (|m| changes slowly along x), so runs of equal shells are summed by shuffles
// and the first lane of each run adds to the block's histogram in shared memory. (One
// global FP64 atomic per mode took 425 us per component at 128^3: 2 M of them on 112
// addresses.) Modes with 0 < x < nx/2 stand for their conjugates too.
__global__ void __launch_bounds__(kThreads) k_shells(const Grid g, const double2* __restrict__ u,
                                                     double half_inv_n2, double* __restrict__ e,
                                                     int nshell) {
  extern __shared__ double hist[];
  for (int s = threadIdx.x; s < nshell; s += kThreads) hist[s] = 0.0;
  __syncthreads();
  const unsigned n = g.modes, lane = threadIdx.x & 31;
  const size_t N = n;
  const unsigned stride = gridDim.x * kThreads;
  // whole warps stay in the loop together
  for (unsigned long long w0 = blockIdx.x * kThreads + (threadIdx.x & ~31u); w0 < n; w0 += stride) {
    const unsigned long long m = w0 + lane;
    int shell = -1;
    double v = 0.0;
    if (m < n) {
      int x, y, z;
      mode_of(g, (unsigned)m, x, y, z);
      const long long ky = wavenumber(y, g.ny), kz = wavenumber(z, g.nz);
      const long long k2 = (long long)x * x + ky * ky + kz * kz;
      // round(sqrt(k2)): s with s^2 - s < k2 <= s^2 + s (k2 is an integer, no ties)
      long long s = (long long)(sqrtf((float)k2) + 0.5f);
      while (s * s - s >= k2 && s > 0) --s;
      while (s * s + s < k2) ++s;
      shell = (int)s;
      const double2 a = u[m], b = u[N + m], c = u[2 * N + m];
      v = a.x * a.x + a.y * a.y + b.x * b.x + b.y * b.y + c.x * c.x + c.y * c.y;
      v *= (x > 0 && 2 * x != g.nx) ? 2.0 * half_inv_n2 : half_inv_n2;
    }
    const int before = __shfl_up_sync(0xffffffffu, shell, 1);
    const bool head = lane == 0 || before != shell;
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    const unsigned after = lane == 31 ? 0u : heads >> (lane + 1);
    const unsigned end = after ? lane + __ffs(after) - 1 : 31;  // last lane of this run
    for (unsigned o = 1; o < 32; o <<= 1) {
      const double t = __shfl_down_sync(0xffffffffu, v, o);
      if (lane + o <= end) v += t;
    }
    if (head && shell >= 0) atomicAdd(&hist[shell], v);
  }
  __syncthreads();
  for (int s = threadIdx.x; s < nshell; s += kThreads)
    if (hist[s] != 0.0) atomicAdd(&e[s], hist[s]);
}

bool make_grid(int nx, int ny, int nz, Grid* g) {
  if (nx < 1 || ny < 1 || nz < 1) return false;
  const long long nxh = nx / 2 + 1;
  if ((long long)nx * ny >= (1LL << 31) || (long long)nx * ny * nz >= (1LL << 31) ||
      nxh * ny * nz >= (1LL << 31))
    return false;
  *g = Grid{nx, ny, nz, (int)nxh, (unsigned)(nxh * ny * nz)};
  return true;
}

unsigned blocks_for(long long n) {
  const long long b = (n + kThreads - 1) / kThreads;
  return (unsigned)(b < kMaxBlocks ? (b < 1 ? 1 : b) : kMaxBlocks);
}

lbm_status launched(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(LBM_E_CUDA, "%s failed: %s", what, cudaGetErrorString(e));
  return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_spectral_curl_div(const void* uh, void* wh, int nx, int ny, int nz, double k0,
                                 void* cuda_stream) {
  Grid g;
  if (!uh || !wh || !make_grid(nx, ny, nz, &g)) return fail(LBM_E_INVAL, "NULL pointer or bad grid size");
  const double scale = k0 / ((double)nx * ny * nz);
  k_curl_div<<<blocks_for(g.modes), kThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      g, static_cast<const double2*>(uh), static_cast<double2*>(wh), scale);
  return launched("curl and divergence pass");
}

lbm_status lbm_spectral_dissipation(const double* w, const double* T, long long n, double mu,
                                    double T_ref, int sutherland, double* out, void* cuda_stream) {
  if (!w || !T || !out || n < 1 || n >= (1LL << 31))
    return fail(LBM_E_INVAL, "NULL pointer or bad number of points");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const unsigned blocks = blocks_for(n);
  k_dissipation<<<blocks, kThreads, 0, s>>>(w, T, n, mu, 1.0 / T_ref, sutherland, out + 2);
  k_dissipation_final<<<1, kThreads, 0, s>>>(out + 2, (int)blocks, 1.0 / (double)n, out);
  return launched("dissipation pass");
}

int lbm_spectral_shell_count(int nx, int ny, int nz) {
  const double x = nx / 2, y = ny / 2, z = nz / 2;
  return (int)std::floor(std::sqrt(x * x + y * y + z * z) + 0.5) + 1;
}

lbm_status lbm_spectral_shells(const void* uh, int nx, int ny, int nz, double* e, int nshell,
                               void* cuda_stream) {
  Grid g;
  if (!uh || !e || !make_grid(nx, ny, nz, &g)) return fail(LBM_E_INVAL, "NULL pointer or bad grid size");
  if (nshell != lbm_spectral_shell_count(nx, ny, nz) || nshell > kMaxShells)
    return fail(LBM_E_INVAL, "%d shells for this grid, at most %d", nshell, kMaxShells);
  const double n = (double)nx * ny * nz;
  unsigned blocks = blocks_for(g.modes);
  if (blocks > 608) blocks = 608;  // every block adds its histogram to e once
  k_shells<<<blocks, kThreads, sizeof(double) * nshell, static_cast<cudaStream_t>(cuda_stream)>>>(
      g, static_cast<const double2*>(uh), 0.5 / (n * n), e, nshell);
  return launched("shell sums");
}

}  // extern "C"
