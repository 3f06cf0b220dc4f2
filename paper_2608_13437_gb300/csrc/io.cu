// Outputs of the current state through the AA read map of its parity: per-cell
// moments (float-float sums) and primitives as the step computes them, the sensor
// exactly as the next step computes it, canonical population arrays in and out, and
// raw slot planes.
#include <type_traits>

#include "diag_device.cuh"
#include "lbm_internal.h"
#include "step_impl.cuh"

namespace lbm {

namespace {

__device__ __forceinline__ void decompose(const DomainConst& P, long long cell, int& x, int& y,
                                          int& z) {
  cell_xyz(P, cell, x, y, z);
}

// Moments of cells [c0, c0 + cnt) (c0 a multiple of 32) through the AA read map of the
// step's parity, from the step's own loads and FP32 decode. LBM_MOM_Q: per field a
// float-float sum of the seven populations and the reference (two-sum, about 48
// significant bits), widened to the output type. LBM_MOM_PRIM: the primitives exactly as
// the step computes them (its FP32 sums and closure). No FP64 arithmetic: FP64 here is
// only an output format.
// One warp per tile. 16-bit storage is bound by issue here as much as by HBM: the
// float-float sums go two fields at a time (packed), whole-tile rows take the step's
// warp-uniform addressing, and 128 registers leave 16 warps an SM (256^3 FP16, Q: 726 us at
// even and 890 at odd parity with the general index maps and 12 warps, 649 and 680 now;
// HBM's time for its 4.2 GB is 626. FP32 was at HBM's time and stays there). An L2 prefetch
// of the tile a warp takes next, with a grid of resident blocks, was slower (744-860).
// WHICH: the output, or -1 to choose at run time. Primitives need five fields only, two of the
// four groups of a slot. Behind one set of loads the other groups were fetched too where
// held x ends make the loads conditional, so these domains take a kernel for each output
// (256^3 primitives, odd parity: FP32 837 -> 637 us, FP16 486 -> 377; all moments FP16 787
// -> 704). Periodic ones share a kernel: there the loads stand together in front of the
// choice, and with one output alone they were spread out between the sums (256^3 FP16 all
// moments 631 -> 678 us).
constexpr int kMomThreads = 128, kMomBlocks = 4;  // 128 registers a thread
template <typename S, int PARITY, bool HELD, bool ROWS, bool ESO, int WHICH>
__global__ void __launch_bounds__(kMomThreads, kMomBlocks)
    k_moments(const DomainConst P, const S* __restrict__ pop, const float* __restrict__ ghost, int which,
              void* out, int out_f64, long long c0, long long cnt) {
  const int lane = threadIdx.x & (kTile - 1);
  const long long warps = (long long)gridDim.x * (kMomThreads / kTile);
  const long long tiles = (cnt + kTile - 1) / kTile, t0 = c0 / kTile;
  for (long long w = blockIdx.x * (long long)(kMomThreads / kTile) + threadIdx.x / kTile; w < tiles; w += warps) {
    const long long r = w * kTile + lane;
    if (r >= cnt) continue;
    float d[kF][kQ];
    load_tile_cell<PARITY, HELD, ROWS, ESO, S>(P, pop, ghost, t0 + w, lane, d);
    if (WHICH < 0 ? which == 1 : WHICH == 1) {
      float Q[kF];
#pragma unroll
      for (int k = 0; k < kF; ++k) {
        float t = d[k][0];
#pragma unroll
        for (int i = 1; i < kQ; ++i) t = add(t, d[k][i]);
        Q[k] = t;
      }
      Q[0] = add(Q[0], P.rho_ref);
      Q[4] = add(Q[4], P.E_ref);
      Prim<float> s;
      closure<float>(Q, P.gm1, P.mu, P.visc0, P.heat0, P.inv_T_ref, P.sutherland, s);
      const float v[6] = {s.rho, s.u[0], s.u[1], s.u[2], s.T, s.p};
#pragma unroll
      for (int j = 0; j < 6; ++j) {
        if (out_f64) static_cast<double*>(out)[(long long)j * cnt + r] = (double)v[j];
        else static_cast<float*>(out)[(long long)j * cnt + r] = v[j];
      }
    } else {
#pragma unroll
      for (int k = 0; k < kF; k += 2) {
        FF2 a = {pack2(d[k][0], d[k + 1][0]), pack2(0.0f, 0.0f)};
#pragma unroll
        for (int i = 1; i < kQ; ++i) ff_add2(a, pack2(d[k][i], d[k + 1][i]));
        if (k == 0) ff_add2(a, pack2(P.rho_ref, -0.0f));
        if (k == 4) ff_add2(a, pack2(P.E_ref, -0.0f));
        FF v[2];
        unpack2(a.hi, v[0].hi, v[1].hi);
        unpack2(a.lo, v[0].lo, v[1].lo);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const long long at = (long long)(k + j) * cnt + r;
          if (out_f64) static_cast<double*>(out)[at] = ff_value(v[j]);
          else static_cast<float*>(out)[at] = add(v[j].hi, v[j].lo);
        }
      }
    }
  }
}

template <typename S>
void launch_moments_t(const DomainConst& P, int parity, const S* pop, const float* ghost, int which,
                      void* out, int out_f64, long long c0, long long cnt, cudaStream_t s) {
  const int block = kMomThreads;
  const long long need = (cnt + kMomThreads - 1) / kMomThreads;
  const long long most = (long long)sm_count() * 32;
  const unsigned grid = (unsigned)(need < most ? need : most);
  with_tile_form(P, parity, [&](auto f) {
    using F = decltype(f);
    auto launch = [&](auto w) {
      k_moments<S, F::parity, F::held, F::rows, F::eso, decltype(w)::value>
          <<<grid, block, 0, s>>>(P, pop, ghost, which, out, out_f64, c0, cnt);
    };
    if constexpr (!F::held) launch(std::integral_constant<int, -1>{});
    else if (which == 1) launch(std::integral_constant<int, 1>{});
    else launch(std::integral_constant<int, 0>{});
  });
}

template <typename S>
__global__ void k_sensor(const DomainConst P, int parity, const S* __restrict__ pop,
                         const float* __restrict__ ghost, void* out, int out_f64, long long c0,
                         long long cnt) {
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < cnt;
       r += (long long)gridDim.x * blockDim.x) {
    const long long cell = c0 + r;
    int x, y, z;
    decompose(P, cell, x, y, z);
    const CellIndex c = make_index(P, x, y, z);
    float d[kF][kQ];
    if (parity) {
      if (P.bc_x) load_cell<1, true, S>(P, pop, ghost, c, d);
      else load_cell<1, false, S>(P, pop, ghost, c, d);
    } else {
      if (P.bc_x) load_cell<0, true, S>(P, pop, ghost, c, d);
      else load_cell<0, false, S>(P, pop, ghost, c, d);
    }
    SensorOut so;
    collide_cell<true>(P, d, &so);
    const double v[3] = {(double)so.theta_dt / (double)P.dt, (double)so.chi, (double)so.omega_h};
    for (int j = 0; j < 3; ++j) {
      if (out_f64) static_cast<double*>(out)[(long long)j * cnt + r] = v[j];
      else static_cast<float*>(out)[(long long)j * cnt + r] = (float)v[j];
    }
  }
}

__device__ __forceinline__ double weight(int i) { return i == 0 ? 0.25 : 0.125; }

__device__ __forceinline__ double ref_of(const DomainConst& P, int k) {
  return k == 0 ? (double)P.rho_ref : (k == 4 ? (double)P.E_ref : 0.0);
}

// Canonical populations of cells [c0, c0 + cnt) (c0 a multiple of 32), buf[(k, i)][cnt],
// decoded (dtype F32/F64) or native, out of the state (SET = 0) or into it. One warp per
// tile moves all 98 arrays: a direction's 14 fields by the layout's vector accesses, the
// arrays in runs of 32 cells. (One launch per array read or wrote 4 of every 16 bytes of
// the layout and took 98 x 6 us at 64^3; this is bound by the link or by HBM.)
// S: storage type, T: the arrays' element type; NATIVE moves the stored bits (S == T), the
// ghost value encoded like a stored one.
template <typename S, typename T, bool NATIVE, bool SET>
__global__ void __launch_bounds__(kMomThreads, kMomBlocks) k_populations(const DomainConst P, int parity,
                                                             S* __restrict__ pop,
                                                             const float* __restrict__ ghost,
                                                             T* __restrict__ buf, long long c0,
                                                             long long cnt) {
  using V4 = typename Codec<S>::V4;
  using V2 = typename Codec<S>::V2;
  union Fields {  // a direction's 14 fields as the layout's groups
    struct {
      V4 v4[3];
      V2 v2;
    };
    S f[kF];
    __device__ Fields() {}
  };
  const int lane = threadIdx.x & (kTile - 1);
  const long long warps = (long long)gridDim.x * (kMomThreads / kTile);
  const long long tiles = (cnt + kTile - 1) / kTile, t0 = c0 / kTile;
  for (long long w = blockIdx.x * (long long)(kMomThreads / kTile) + threadIdx.x / kTile; w < tiles; w += warps) {
    const long long r = w * kTile + lane;
    if (r >= cnt) continue;
    int x, y, z;
    tile_xyz(P, t0 + w, lane, x, y, z);
    const CellIndex c = make_index(P, x, y, z);
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const bool held = from_ghost(P, c, i);
      if (SET && held) continue;  // held ends keep the ghost inflow
      const long long cell = src_cell(P, c, parity, i);
      if (!LBM_CHECK(P, cell >= 0 && cell < P.ntile * kTile)) continue;
      S* const base = pop + tile_start(cell);
      const int slot = parity ? opp(i) : i, ln = (int)(cell & (kTile - 1));
      Fields u;
      if (!SET && !held) {
#pragma unroll
        for (int g = 0; g < 3; ++g) u.v4[g] = *reinterpret_cast<const V4*>(base + group_offset(slot, g, ln));
        u.v2 = *reinterpret_cast<const V2*>(base + group_offset(slot, 3, ln));
      }
#pragma unroll
      for (int k = 0; k < kF; ++k) {
        T* const at = buf + (long long)(k * kQ + i) * cnt + r;
        if constexpr (SET) {
          if constexpr (NATIVE) u.f[k] = *at;
          else u.f[k] = Codec<S>::enc((float)((double)*at - weight(i) * ref_of(P, k)), P.inv_scale[k]);
        } else if constexpr (NATIVE) {
          *at = held ? Codec<S>::enc(ghost_value(P, ghost, c, k, i), P.inv_scale[k]) : u.f[k];
        } else {
          const double dev = held ? (double)ghost_value(P, ghost, c, k, i)
                                  : Codec<S>::dec64(u.f[k], (double)P.scale[k]);
          *at = (T)(weight(i) * ref_of(P, k) + dev);
        }
      }
      if constexpr (SET) {
#pragma unroll
        for (int g = 0; g < 3; ++g) *reinterpret_cast<V4*>(base + group_offset(slot, g, ln)) = u.v4[g];
        *reinterpret_cast<V2*>(base + group_offset(slot, 3, ln)) = u.v2;
      }
    }
  }
}

template <typename S, bool SET>
void launch_populations_t(const DomainConst& P, int parity, void* pop, const float* ghost, void* buf,
                          int dtype, long long c0, long long cnt, cudaStream_t s) {
  const long long need = (cnt + kMomThreads - 1) / kMomThreads, most = (long long)sm_count() * 32;
  const unsigned grid = (unsigned)(need < most ? need : most);
  S* p = static_cast<S*>(pop);
  if (dtype == 2)
    k_populations<S, S, true, SET><<<grid, kMomThreads, 0, s>>>(P, parity, p, ghost, static_cast<S*>(buf), c0, cnt);
  else if (dtype == 1)
    k_populations<S, double, false, SET><<<grid, kMomThreads, 0, s>>>(P, parity, p, ghost, static_cast<double*>(buf), c0, cnt);
  else
    k_populations<S, float, false, SET><<<grid, kMomThreads, 0, s>>>(P, parity, p, ghost, static_cast<float*>(buf), c0, cnt);
}

// Raw stored values of storage slot `slot` of all fields on plane z, [k][y][x]; T is an
// unsigned integer of the element's size, so the bits move unchanged.
template <typename T>
__global__ void k_plane(const DomainConst P, T* __restrict__ pop, int z, int slot,
                        T* __restrict__ buf, int set) {
  const long long plane = (long long)P.nx * P.ny;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < plane * kF;
       r += (long long)gridDim.x * blockDim.x) {
    const int k = (int)(r / plane);
    const long long cell = r - k * plane + plane * z;
    if (!LBM_CHECK(P, cell >= 0 && cell < P.ncell)) continue;
    const long long at = pop_index(cell, k, slot);
    if (set) pop[at] = buf[r];
    else buf[r] = pop[at];
  }
}

int grid_for(long long n, int block) {
  long long g = (n + block - 1) / block;
  const long long most = (long long)sm_count() * 32;
  if (g > most) g = most;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace


cudaError_t launch_moments(const DomainConst& P, int store, int parity, const void* pop,
                           const float* ghost, int which, void* out, int out_f64, long long c0,
                           long long cnt, cudaStream_t s) {
  switch (store) {
    case 0: launch_moments_t(P, parity, (const float*)pop, ghost, which, out, out_f64, c0, cnt, s); break;
    case 1: launch_moments_t(P, parity, (const __half*)pop, ghost, which, out, out_f64, c0, cnt, s); break;
    default: launch_moments_t(P, parity, (const __nv_bfloat16*)pop, ghost, which, out, out_f64, c0, cnt, s); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_sensor(const DomainConst& P, int store, int parity, const void* pop,
                          const float* ghost, void* out, int out_f64, long long c0, long long cnt,
                          cudaStream_t s) {
  const int block = 128, grid = grid_for(cnt, block);
  switch (store) {
    case 0: k_sensor<float><<<grid, block, 0, s>>>(P, parity, (const float*)pop, ghost, out, out_f64, c0, cnt); break;
    case 1: k_sensor<__half><<<grid, block, 0, s>>>(P, parity, (const __half*)pop, ghost, out, out_f64, c0, cnt); break;
    default: k_sensor<__nv_bfloat16><<<grid, block, 0, s>>>(P, parity, (const __nv_bfloat16*)pop, ghost, out, out_f64, c0, cnt); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_populations(const DomainConst& P, int store, int parity, void* pop,
                               const float* ghost, void* buf, int dtype, int set, long long c0,
                               long long cnt, cudaStream_t s) {
  switch (store * 2 + set) {
    case 0: launch_populations_t<float, false>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
    case 1: launch_populations_t<float, true>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
    case 2: launch_populations_t<__half, false>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
    case 3: launch_populations_t<__half, true>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
    case 4: launch_populations_t<__nv_bfloat16, false>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
    default: launch_populations_t<__nv_bfloat16, true>(P, parity, pop, ghost, buf, dtype, c0, cnt, s); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_plane(const DomainConst& P, int store, void* pop, int z, int slot, void* buf,
                         int set, cudaStream_t s) {
  const int block = 256, grid = grid_for((long long)P.nx * P.ny * kF, block);
  if (store == 0)
    k_plane<unsigned><<<grid, block, 0, s>>>(P, (unsigned*)pop, z, slot, (unsigned*)buf, set);
  else
    k_plane<unsigned short><<<grid, block, 0, s>>>(P, (unsigned short*)pop, z, slot,
                                                   (unsigned short*)buf, set);
  return cudaGetLastError();
}

}  // namespace lbm
