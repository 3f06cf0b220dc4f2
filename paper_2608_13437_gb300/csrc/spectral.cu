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

__device__ __forceinline__ void mode_of(int nx, int ny, unsigned m, int& x, int& y, int& z) {
  const unsigned row = m / (unsigned)nx;
  x = (int)(m - row * (unsigned)nx);
  const unsigned zz = row / (unsigned)ny;
  y = (int)(row - zz * (unsigned)ny);
  z = (int)zz;
}

// Curl and divergence of u = (a, b, c) from z = FFT(a + ib) over the whole grid and the
// half spectrum of c; out as the spectra of w_x + i w_y and w_z + i div, so each complex
// transform carries two real fields. One thread per mode of the half spectrum: it takes a
// and b apart with z(-k), and writes the modes k and -k (conjugate spectra), except on the
// planes x = 0 and Nyquist, which hold both.
__global__ void __launch_bounds__(kThreads) k_curl_div(const Grid g, const double2* __restrict__ z,
                                                       const double2* __restrict__ ch,
                                                       double2* __restrict__ w, double scale) {
  const unsigned n = g.modes;
  const size_t N = (size_t)g.nx * g.ny * g.nz;
  const double half = 0.5 * scale;
  for (unsigned m = blockIdx.x * kThreads + threadIdx.x; m < n; m += gridDim.x * kThreads) {
    int x, y, zz;
    mode_of(g.nxh, g.ny, m, x, y, zz);
    // an even axis has no derivative of its Nyquist mode
    const double kx = 2 * x == g.nx ? 0.0 : (double)x;
    const double ky = 2 * y == g.ny ? 0.0 : (double)wavenumber(y, g.ny);
    const double kz = 2 * zz == g.nz ? 0.0 : (double)wavenumber(zz, g.nz);
    const int xm = x ? g.nx - x : 0, ym = y ? g.ny - y : 0, zm = zz ? g.nz - zz : 0;
    const size_t at = (size_t)x + (size_t)g.nx * ((size_t)y + (size_t)g.ny * zz);
    const size_t mirror = (size_t)xm + (size_t)g.nx * ((size_t)ym + (size_t)g.ny * zm);
    const double2 p = z[at], q = z[mirror];
    // a = (p + conj q) / 2, b = (p - conj q) / 2i, c; all times scale
    const double2 a = make_double2(half * (p.x + q.x), half * (p.y - q.y));
    const double2 b = make_double2(half * (p.y + q.y), half * (q.x - p.x));
    const double2 c0 = ch[m], c = make_double2(scale * c0.x, scale * c0.y);
    // the derivative's factor i turns (re, im) into (-im, re)
    const double2 wx = make_double2(kz * b.y - ky * c.y, ky * c.x - kz * b.x);
    const double2 wy = make_double2(kx * c.y - kz * a.y, kz * a.x - kx * c.x);
    const double2 wz = make_double2(ky * a.y - kx * b.y, kx * b.x - ky * a.x);
    const double2 dv = make_double2(-(kx * a.y + ky * b.y + kz * c.y), kx * a.x + ky * b.x + kz * c.x);
    w[at] = make_double2(wx.x - wy.y, wx.y + wy.x);
    w[N + at] = make_double2(wz.x - dv.y, wz.y + dv.x);
    if (x > 0 && 2 * x != g.nx) {
      w[mirror] = make_double2(wx.x + wy.y, wy.x - wx.y);
      w[N + mirror] = make_double2(wz.x + dv.y, dv.x - wz.y);
    }
  }
}

// Block sums of m |w|^2 and m d^2 (fixed order), then one block adds the partials.
__global__ void __launch_bounds__(kThreads) k_dissipation(const double2* __restrict__ w,
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
    const double2 p = w[i], q = w[n + i];  // (w_x, w_y), (w_z, div)
    s += m * (p.x * p.x + p.y * p.y + q.x * q.x);
    d += m * (q.y * q.y);
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

// Shell sums of |z|^2 over rows of nx modes (kFull: the whole grid, for z = FFT(a + ib):
// a shell holds k and -k, over which |z|^2 sums to |a|^2 + |b|^2) or of a half spectrum
// (modes with 0 < x < nx/2 stand for their conjugates too). 32 consecutive modes of a warp
// mostly share their shell with their neighbours (|m| changes slowly along x), so runs of
// equal shells are summed by shuffles and the first lane of each run adds to the block's
// histogram in shared memory. (One global FP64 atomic per mode took 425 us per component
// at 128^3: 2 M of them on 112 addresses.)
template <bool kFull>
__device__ void shell_sums(const Grid& g, const double2* __restrict__ u, double half_inv_n2,
                           double* __restrict__ hist) {
  const int row = kFull ? g.nx : g.nxh;
  const unsigned n = (unsigned)row * (unsigned)g.ny * (unsigned)g.nz, lane = threadIdx.x & 31;
  const unsigned stride = gridDim.x * kThreads;
  // whole warps stay in the loop together
  for (unsigned long long w0 = blockIdx.x * kThreads + (threadIdx.x & ~31u); w0 < n; w0 += stride) {
    const unsigned long long m = w0 + lane;
    int shell = -1;
    double v = 0.0;
    if (m < n) {
      int x, y, z;
      mode_of(row, g.ny, (unsigned)m, x, y, z);
      const long long kx = wavenumber(x, g.nx), ky = wavenumber(y, g.ny), kz = wavenumber(z, g.nz);
      const long long k2 = kx * kx + ky * ky + kz * kz;
      // round(sqrt(k2)): s with s^2 - s < k2 <= s^2 + s (k2 is an integer, no ties)
      long long s = (long long)(sqrtf((float)k2) + 0.5f);
      while (s > 0 && s * s - s >= k2) --s;
      while (s * s + s < k2) ++s;
      shell = (int)s;
      const double2 a = u[m];
      v = a.x * a.x + a.y * a.y;
      v *= (!kFull && x > 0 && 2 * x != g.nx) ? 2.0 * half_inv_n2 : half_inv_n2;
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
}

__global__ void __launch_bounds__(kThreads) k_shells(const Grid g, const double2* __restrict__ z,
                                                     const double2* __restrict__ ch,
                                                     double half_inv_n2, double* __restrict__ e,
                                                     int nshell) {
  extern __shared__ double hist[];
  for (int s = threadIdx.x; s < nshell; s += kThreads) hist[s] = 0.0;
  __syncthreads();
  shell_sums<true>(g, z, half_inv_n2, hist);
  shell_sums<false>(g, ch, half_inv_n2, hist);
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

lbm_status lbm_spectral_curl_div(const void* zh, const void* ch, void* wh, int nx, int ny, int nz,
                                 double k0, void* cuda_stream) {
  Grid g;
  if (!zh || !ch || !wh || !make_grid(nx, ny, nz, &g)) return fail(LBM_E_INVAL, "NULL pointer or bad grid size");
  const double scale = k0 / ((double)nx * ny * nz);
  k_curl_div<<<blocks_for(g.modes), kThreads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      g, static_cast<const double2*>(zh), static_cast<const double2*>(ch), static_cast<double2*>(wh),
      scale);
  return launched("curl and divergence pass");
}

lbm_status lbm_spectral_dissipation(const void* w, const double* T, long long n, double mu,
                                    double T_ref, int sutherland, double* out, void* cuda_stream) {
  if (!w || !T || !out || n < 1 || n >= (1LL << 31))
    return fail(LBM_E_INVAL, "NULL pointer or bad number of points");
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const unsigned blocks = blocks_for(n);
  k_dissipation<<<blocks, kThreads, 0, s>>>(static_cast<const double2*>(w), T, n, mu, 1.0 / T_ref, sutherland, out + 2);
  k_dissipation_final<<<1, kThreads, 0, s>>>(out + 2, (int)blocks, 1.0 / (double)n, out);
  return launched("dissipation pass");
}

int lbm_spectral_shell_count(int nx, int ny, int nz) {
  const double x = nx / 2, y = ny / 2, z = nz / 2;
  return (int)std::floor(std::sqrt(x * x + y * y + z * z) + 0.5) + 1;
}

lbm_status lbm_spectral_shells(const void* zh, const void* ch, int nx, int ny, int nz, double* e,
                               int nshell, void* cuda_stream) {
  Grid g;
  if (!zh || !ch || !e || !make_grid(nx, ny, nz, &g)) return fail(LBM_E_INVAL, "NULL pointer or bad grid size");
  if (nshell != lbm_spectral_shell_count(nx, ny, nz) || nshell > kMaxShells)
    return fail(LBM_E_INVAL, "%d shells for this grid, at most %d", nshell, kMaxShells);
  const double n = (double)nx * ny * nz;
  unsigned blocks = blocks_for((long long)nx * ny * nz);
  if (blocks > 608) blocks = 608;  // every block adds its histogram to e once
  k_shells<<<blocks, kThreads, sizeof(double) * nshell, static_cast<cudaStream_t>(cuda_stream)>>>(
      g, static_cast<const double2*>(zh), static_cast<const double2*>(ch), 0.5 / (n * n), e, nshell);
  return launched("shell sums");
}

}  // extern "C"
