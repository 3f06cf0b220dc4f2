// Many steps of a small domain in one launch, with the populations held in registers.
//
// A grid of up to about 58 thousand cells (one brick of at most 384 cells per SM) is far
// too small to be bound by memory: a step moves its 98 populations per cell through the
// L2 for no reason but that launches end, and costs 3.3 us at 16 thousand cells, of which
// about 1 us is the gap between two launches and most of the rest one chain of dependent
// loads, arithmetic and stores. Here each block keeps a brick of cells for n steps, one
// thread per cell with its 14 x 7 populations in registers (255 of them for bricks of up to
// 256 cells, 168 above), and per step only what the lattice links carry moves: within the
// brick through shared memory, between bricks through inboxes in global memory (the L2).
//
//   * Every directional population leaves as the words of the storage type (rounded as a
//     plain step's store rounds it) and is decoded on arrival as a plain step's load does;
//     collide_cell is the same code. So the state after n steps is the plain kernel's, bit
//     for bit, for every storage type, rounding mode, streaming map and parity.
//   * An inbox holds 16-byte packets of three words and a tag, the number of the step that
//     sent them. Packets are written and read whole (128-bit scalar accesses), so a reader
//     polls the packet itself until the tag is the current step's: one trip through the
//     L2, no flags, no fences, no grid-wide barrier. A brick has two inboxes, for even and
//     odd tags. A neighbour overwrites an inbox two steps later; by then it has received
//     this brick's packets of the step between, which were sent after the inbox was read.
//   * The same dependence orders memory at both ends of the launch: a brick stores its
//     populations after the last step, when it has received packets from its neighbours,
//     which they send after they have loaded theirs, and a location is loaded and stored by
//     one brick and its direct neighbours along that population's axis alone.
//   * Launched cooperatively (every block resident, or the launch fails). A poll gives up
//     after a bounded number of tries, or soon after another block has; the block then sets
//     flag bit 2 and returns without storing, launches that find the bit set do nothing, and
//     the host reports LBM_E_TIMEOUT.
//   * Tags go on from each block's own step count in device memory, so a launch may be
//     repeated (also by a graph) without the host's knowledge of it. A block that gives up or
//     does nothing counts the launch's steps all the same, so the counts stay equal and
//     nothing that a failed launch leaves in an inbox passes for a later step's.
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

namespace {

template <typename S>
struct Words {
  static constexpr int n = std::is_same<S, float>::value ? kF : kF / 2;  // of one direction
  static constexpr int packets = (n + 2) / 3;
};

// The words of direction i's 14 fields, as store_dir stores them.
template <typename S, bool SR>
__device__ __forceinline__ void pack_dir(const DomainConst& P, const float (&d)[kF][kQ], int i,
                                         Dither* dz, unsigned (&w)[Words<S>::n]) {
  float v[kF];
#pragma unroll
  for (int k = 0; k < kF; ++k) v[k] = d[k][i];
  if constexpr (std::is_same<S, float>::value) {
#pragma unroll
    for (int k = 0; k < kF; ++k) w[k] = __float_as_uint(v[k]);
  } else {
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      uint2 e;
      if constexpr (SR) {
        const unsigned r0 = dz->next(), r1 = dz->next();
        e = Codec<S>::enc4_sr(v + 4 * g, P.inv_scale + 4 * g, r0, r1);
      } else {
        e = Codec<S>::enc4(v + 4 * g, P.inv_scale + 4 * g);
      }
      w[2 * g] = e.x;
      w[2 * g + 1] = e.y;
    }
    if constexpr (SR) w[6] = Codec<S>::enc2_sr(v + 12, P.inv_scale + 12, dz->next());
    else w[6] = Codec<S>::enc2(v + 12, P.inv_scale + 12);
  }
}

// Decodes direction i's words, as load_cell decodes what it loads.
template <typename S>
__device__ __forceinline__ void unpack_dir(const DomainConst& P, const unsigned (&w)[Words<S>::n],
                                           float (&d)[kF][kQ], int i) {
  float v[kF];
  if constexpr (std::is_same<S, float>::value) {
#pragma unroll
    for (int k = 0; k < kF; ++k) v[k] = __uint_as_float(w[k]);
  } else {
#pragma unroll
    for (int g = 0; g < 3; ++g)
      Codec<S>::dec4(make_uint2(w[2 * g], w[2 * g + 1]), P.scale + 4 * g, v + 4 * g);
    Codec<S>::dec2(w[6], P.scale + 12, v + 12);
  }
#pragma unroll
  for (int k = 0; k < kF; ++k) d[k][i] = v[k];
}

// A direction's words as the groups of 4 + 4 + 4 + 2 fields of the population layout
// and of the exchange through shared memory.
template <typename S>
__device__ __forceinline__ typename Codec<S>::V4 words4(const unsigned* w, int g) {
  if constexpr (std::is_same<S, float>::value)
    return make_float4(__uint_as_float(w[4 * g]), __uint_as_float(w[4 * g + 1]),
                       __uint_as_float(w[4 * g + 2]), __uint_as_float(w[4 * g + 3]));
  else
    return make_uint2(w[2 * g], w[2 * g + 1]);
}
template <typename S>
__device__ __forceinline__ typename Codec<S>::V2 words2(const unsigned* w) {
  if constexpr (std::is_same<S, float>::value)
    return make_float2(__uint_as_float(w[12]), __uint_as_float(w[13]));
  else
    return w[6];
}
template <typename S>
__device__ __forceinline__ void from_groups(const typename Codec<S>::V4 (&a)[3],
                                            typename Codec<S>::V2 b,
                                            unsigned (&w)[Words<S>::n]) {
  if constexpr (std::is_same<S, float>::value) {
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      w[4 * g] = __float_as_uint(a[g].x);
      w[4 * g + 1] = __float_as_uint(a[g].y);
      w[4 * g + 2] = __float_as_uint(a[g].z);
      w[4 * g + 3] = __float_as_uint(a[g].w);
    }
    w[12] = __float_as_uint(b.x);
    w[13] = __float_as_uint(b.y);
  } else {
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      w[2 * g] = a[g].x;
      w[2 * g + 1] = a[g].y;
    }
    w[6] = b;
  }
}

// Inbox packets: 128-bit scalar accesses, so the three words and the tag arrive together.
__device__ __forceinline__ void packet_store(uint4* p, unsigned a, unsigned b, unsigned c, unsigned tag) {
  const unsigned long long lo = a | ((unsigned long long)b << 32), hi = c | ((unsigned long long)tag << 32);
  asm volatile(
      "{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\t"
      "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(lo), "l"(hi)
      : "memory");
}
__device__ __forceinline__ uint4 packet_load(const uint4* p) {
  unsigned long long lo, hi;
  asm volatile(
      "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\t"
      "mov.b128 {%0, %1}, t;\n\t}"
      : "=l"(lo), "=l"(hi)
      : "l"(p)
      : "memory");
  return make_uint4((unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32));
}

__device__ __forceinline__ bool gave_up(const unsigned* flag) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
  return (v & 2u) != 0;
}

// Exchange buffers of a block: two where 200 KB of shared memory hold them, which saves a
// barrier per step.
template <typename S, int MAXT>
constexpr int exchange_buffers() {
  return (size_t)MAXT * 13 * kF * sizeof(S) <= 200 * 1024 ? 2 : 1;
}

// MAXT: threads of the largest block. 256 leave 255 registers a thread, which lets one warp
// per scheduler overlap more of its own latencies: 1024 x 4 x 4 FP32 2.13 -> 1.78 us a step,
// 256 x 4 x 3 1.94 -> 1.74, 32^3 3.21 -> 3.10; 384 leave 168. (The second exchange buffer
// and the last step's stores outside the loop: 1.68, 1.59 and 2.98.)
template <typename S, bool SR, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    k_resident(const DomainConst P, const ResidentPlan R, S* __restrict__ pop,
               const float* __restrict__ ghost, unsigned* __restrict__ flag,
               uint4* __restrict__ inbox, unsigned* __restrict__ epochs, int parity0,
               const ResidentRun run) {
  using V4 = typename Codec<S>::V4;
  using V2 = typename Codec<S>::V2;
  constexpr int NW = Words<S>::n, NP = Words<S>::packets;
  extern __shared__ __align__(16) unsigned char smem[];
  const int steps = run.steps;
  const unsigned epoch = epochs[blockIdx.x];
  // Nothing is done with the incomplete state that a launch before this one left, nor by a
  // block that is to fail: its neighbours wait in vain. (Both loads run beside the set-up.)
  const bool idle = threadIdx.x == 0 && (gave_up(flag) || (int)blockIdx.x == run.silent);
  const int T = blockDim.x, tid = threadIdx.x;
  // exchange buffers (one, or two for even and odd tags), the rest populations of the last
  // step, and the table of the packet sets that arrive from outside
  constexpr int kBuffers = exchange_buffers<S, MAXT>();
  V4* const x4 = reinterpret_cast<V4*>(smem);                  // [kBuffers][6][3][T], rest [3][T]
  V2* const x2 = reinterpret_cast<V2*>(x4 + (6 * kBuffers + 1) * 3 * T);  // [kBuffers][6][T], [T]
  uint2* const table = reinterpret_cast<uint2*>(x2 + (6 * kBuffers + 1) * T);
  // brick and cell
  const int bx = blockIdx.x % R.g[0], by = blockIdx.x / R.g[0] % R.g[1],
            bz = blockIdx.x / (R.g[0] * R.g[1]);
  const int lx = tid % R.b[0], ly = tid / R.b[0] % R.b[1], lz = tid / (R.b[0] * R.b[1]);
  const int x = bx * R.b[0] + lx, y = by * R.b[1] + ly, z = bz * R.b[2] + lz;
  const bool active = lz < R.b[2] && x < P.nx && y < P.ny && z < P.nz;
  // Per direction i = 1..6: where the population leaving along i goes: the thread of this
  // brick that owns the next cell, or kOut for the neighbouring brick.
  constexpr int kOut = 0xFFFF;
  int to[6];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int l = a == 0 ? lx : (a == 1 ? ly : lz);
    const int stride = a == 0 ? 1 : (a == 1 ? R.b[0] : R.b[0] * R.b[1]);
    const int first = (a == 0 ? bx : (a == 1 ? by : bz)) * R.b[a];
    const int n = a == 0 ? P.nx : (a == 1 ? P.ny : P.nz);
    const int width = min(R.b[a], n - first);  // of this brick
    const bool whole = R.g[a] == 1;            // the brick spans the axis: wrap inside
    to[2 * a] = l + 1 < width ? tid + stride : (whole ? tid - (width - 1) * stride : kOut);
    to[2 * a + 1] = l > 0 ? tid - stride : (whole ? tid + (width - 1) * stride : kOut);
  }
  // offset of packet 0 of direction i to the face cell f of brick b's inbox 0: an inbox
  // holds [packet][set], the sets of the axes that leave the brick one after the other
  auto slot = [&](int b, int i, int f) {
    const int a = (i - 1) >> 1;
    const int face = a == 0 ? R.b[1] * R.b[2] : (a == 1 ? R.b[0] * R.b[2] : R.b[0] * R.b[1]);
    return (unsigned)(b * 2 * NP * R.sets + R.first[a] + ((i - 1) & 1) * face + f);
  };
  auto neighbour = [&](int i) {  // the brick that direction i leads to
    const int a = (i - 1) >> 1, s = (i & 1) ? 1 : -1;
    const int c = a == 0 ? bx : (a == 1 ? by : bz);
    int m = c + s;
    if (m == R.g[a]) m = 0;
    if (m < 0) m = R.g[a] - 1;
    const int step = a == 0 ? 1 : (a == 1 ? R.g[0] : R.g[0] * R.g[1]);
    return (int)blockIdx.x + (m - c) * step;
  };

  // Table of the packet sets that arrive from outside: inbox offset, and direction (less
  // one) and thread of the receiving cell.
  int n_in = 0;
  {
    const int w[3] = {min(R.b[0], P.nx - bx * R.b[0]), min(R.b[1], P.ny - by * R.b[1]),
                      min(R.b[2], P.nz - bz * R.b[2])};
    const int s[3] = {1, R.b[0], R.b[0] * R.b[1]};  // thread strides
    for (int a = 0; a < 3; ++a) {
      if (R.g[a] == 1) continue;
      const int u = a == 0 ? 1 : 0, v = a == 2 ? 1 : 2;  // the face's axes
      for (int e = tid; e < w[u] * w[v]; e += T) {
        const int lu = e % w[u], lv = e / w[u], f = lu + R.b[u] * lv;
        const int at = lu * s[u] + lv * s[v];
        // along +a into the cells at the low end, along -a at the high end
        table[n_in + 2 * e] = make_uint2(slot(blockIdx.x, 2 * a + 1, f), (2u * a) << 16 | at);
        table[n_in + 2 * e + 1] =
            make_uint2(slot(blockIdx.x, 2 * a + 2, f), (2u * a + 1) << 16 | (at + (w[a] - 1) * s[a]));
      }
      n_in += 2 * w[u] * w[v];
    }
  }
  if (__syncthreads_or(idle)) {
    if (tid == 0) epochs[blockIdx.x] = epoch + (unsigned)steps;
    return;
  }

  float d[kF][kQ];
  const CellIndex c = make_index(P, x, y, z);
  if (active) {
    if (parity0) load_cell<1, false, S>(P, pop, nullptr, c, d);
    else load_cell<0, false, S>(P, pop, nullptr, c, d);
  }
  bool bad = false;
  // Where the state is stored after the last step: the read position of the new parity.
  const int parity1 = (parity0 + steps) & 1;
  auto store_groups = [&](int i, const V4* v4, const V2* v2) {
    const long long cell = src_cell(P, c, parity1, i);
    if (!LBM_CHECK(P, cell >= 0 && cell < P.ntile * kTile)) return;
    S* base = pop + tile_start(cell);
    const int lane = (int)(cell & (kTile - 1));
    const int sl = parity1 ? opp(i) : i;
#pragma unroll
    for (int g = 0; g < 3; ++g) *reinterpret_cast<V4*>(base + group_offset(sl, g, lane)) = v4[g * T + tid];
    *reinterpret_cast<V2*>(base + group_offset(sl, 3, lane)) = v2[tid];
  };
  V4* const rest4 = x4 + 6 * kBuffers * 3 * T;
  V2* const rest2 = x2 + 6 * kBuffers * T;
  V4* s4 = x4;
  V2* s2 = x2;

#pragma unroll 1
  for (int t = 0; t < steps; ++t) {
    const unsigned tag = epoch + (unsigned)t + 1u;
    if (kBuffers == 2) {
      s4 = x4 + (tag & 1u) * (6 * 3 * T);
      s2 = x2 + (tag & 1u) * (6 * T);
    }
    if (active) {
      if (P.bc_x) {  // held x ends: the inward populations come from the ghost layer
        if (x == 0) {
#pragma unroll
          for (int k = 0; k < kF; ++k) d[k][1] = ghost_value(P, ghost, c, k, 1);
        }
        if (x == P.nx - 1) {
#pragma unroll
          for (int k = 0; k < kF; ++k) d[k][2] = ghost_value(P, ghost, c, k, 2);
        }
      }
      const float probe = collide_cell<false>(P, d, nullptr);
      bad = bad || !isfinite(probe);
      [[maybe_unused]] Dither dz(0, 0.0f, 0.0f);
      if constexpr (SR) dz = Dither(c.own, d[0][0], d[4][0]);
#pragma unroll
      for (int i = 0; i < kQ; ++i) {
        unsigned w[NW];
        pack_dir<S, SR>(P, d, i, &dz, w);
        if (i == 0) {
          if (t + 1 == steps) {
#pragma unroll
            for (int g = 0; g < 3; ++g) rest4[g * T + tid] = words4<S>(w, g);
            rest2[tid] = words2<S>(w);
          }
          if constexpr (!std::is_same<S, float>::value) unpack_dir<S>(P, w, d, 0);
          continue;
        }
        const int dst = to[i - 1];
        if (dst == kOut) {
          // the destination cell has the same place on its brick's face
          const int f = i < 3 ? ly + R.b[1] * lz : (i < 5 ? lx + R.b[0] * lz : lx + R.b[0] * ly);
          uint4* p = inbox + slot(neighbour(i), i, f) + (tag & 1u) * (unsigned)(NP * R.sets);
#pragma unroll
          for (int q = 0; q < NP; ++q)
            packet_store(p + (size_t)q * R.sets, w[3 * q], 3 * q + 1 < NW ? w[3 * q + 1] : tag,
                         3 * q + 2 < NW ? w[3 * q + 2] : tag, tag);
        } else {
#pragma unroll
          for (int g = 0; g < 3; ++g) s4[((i - 1) * 3 + g) * T + dst] = words4<S>(w, g);
          s2[(i - 1) * T + dst] = words2<S>(w);
        }
      }
    }
    // What the neighbours send: thread tid fetches packet sets tid, tid + T, ... of the brick
    // (all packets of one cell and direction), so the polls of all faces are one trip
    // through the L2 instead of one per direction, and puts them where the exchange within
    // the brick would.
    bool dead = false;
    for (int e = tid; e < n_in; e += T) {
      const uint2 in = table[e];
      const uint4* p = inbox + in.x + (tag & 1u) * (unsigned)(NP * R.sets);
      unsigned w[3 * NP];
      for (int tries = 0;;) {
        uint4 m[NP];
#pragma unroll
        for (int q = 0; q < NP; ++q) m[q] = packet_load(p + (size_t)q * R.sets);
        bool ok = true;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          // every word of a packet is used, so that its load stays one access: with the
          // spare words of the last packet ignored the load was narrowed and the packet
          // could be read half old, half new
          ok = ok && m[q].w == tag;
          if (3 * q + 1 >= NW) ok = ok && m[q].y == tag;
          if (3 * q + 2 >= NW) ok = ok && m[q].z == tag;
        }
        if (ok || dead) {
          dead = dead || !ok;
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            w[3 * q] = m[q].x;
            w[3 * q + 1] = m[q].y;
            w[3 * q + 2] = m[q].z;
          }
          break;
        }
        if ((++tries & (kResidentPollsPerLook - 1)) == 0) dead = tries >= run.polls || gave_up(flag);
      }
#pragma unroll
      for (int g = 0; g < 3; ++g) s4[(in.y >> 16) * 3 * T + g * T + (in.y & 0xFFFFu)] = words4<S>(w, g);
      s2[(in.y >> 16) * T + (in.y & 0xFFFFu)] = words2<S>(w);
    }
    if (__syncthreads_or(dead)) {  // a block whose wait ran out stops here
      if (tid == 0) {
        atomicOr(flag, 2u);
        epochs[blockIdx.x] = epoch + (unsigned)steps;
      }
      return;
    }
    if (active) {
#pragma unroll
      for (int i = 1; i < kQ; ++i) {
        V4 a[3];
#pragma unroll
        for (int g = 0; g < 3; ++g) a[g] = s4[((i - 1) * 3 + g) * T + tid];
        unsigned w[NW];
        from_groups<S>(a, s2[(i - 1) * T + tid], w);
        unpack_dir<S>(P, w, d, i);
      }
    }
    // One buffer: everyone is done with it before the next step writes it. With two, the
    // next step's barrier separates this step's reads from the writes two steps on.
    if (kBuffers == 1) __syncthreads();
  }
  // the state as the last exchange left it, words as they are
  if (active) {
    store_groups(0, rest4, rest2);
#pragma unroll
    for (int i = 1; i < kQ; ++i) store_groups(i, s4 + (i - 1) * 3 * T, s2 + (i - 1) * T);
  }
  if (bad) atomicOr(flag, 1u);
  if (tid == 0) epochs[blockIdx.x] = epoch + (unsigned)steps;
}

// Shared memory of a block: the exchange buffers, the rest populations, and the table (at
// most six packet sets a cell).
template <typename S, int MAXT>
constexpr size_t smem_bytes(int threads) {
  return (size_t)threads * ((6 * exchange_buffers<S, MAXT>() + 1) * kF * sizeof(S) + 6 * sizeof(uint2));
}

template <typename S, bool SR, int MAXT>
cudaError_t launch_threads(const DomainConst& P, const ResidentPlan& R, void* pop, const float* ghost,
                     unsigned* flag, void* inbox, unsigned* epochs, int parity, const ResidentRun& run,
                     cudaStream_t s) {
  const size_t smem = smem_bytes<S, MAXT>(R.threads);
  cudaError_t e = cudaFuncSetAttribute(k_resident<S, SR, MAXT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem_bytes<S, MAXT>(MAXT));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(R.blocks());
  cfg.blockDim = dim3(R.threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_resident<S, SR, MAXT>, P, R, static_cast<S*>(pop), ghost, flag,
                            static_cast<uint4*>(inbox), epochs, parity, run);
}

template <typename S, bool SR>
cudaError_t launch_t(const DomainConst& P, const ResidentPlan& R, void* pop, const float* ghost,
                     unsigned* flag, void* inbox, unsigned* epochs, int parity, const ResidentRun& run,
                     cudaStream_t s) {
  if (R.threads <= 256)
    return launch_threads<S, SR, 256>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s);
  return launch_threads<S, SR, kResidentMaxThreads>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s);
}

}  // namespace

namespace {

// Nanoseconds of a plain step, of `streams` such domains at once: launches overlap, so only
// the part that follows the cells adds up. Fitted to 64 x 4 x 4 ... 38^3 on 1 to 12 streams;
// within 15 % while the L2 holds the states (beyond it plain steps take up to twice as long).
long long plain_cost(const DomainConst& P, int store, int streams) {
  return store == 0 ? 2050 + 52 * P.ncell * streams / 1000 : 2300 + 25 * P.ncell * streams / 1000;
}

}  // namespace

bool resident_plan(const DomainConst& P, int store, int sms, ResidentPlan* R, long long* plan_cost) {
  if (!P.collide || P.ncell > (long long)sms * kResidentMaxThreads) return false;
  const int n[3] = {P.nx, P.ny, P.nz};
  long long best = -1;
  // every number of bricks along an axis that its side can be cut into evenly (the smallest
  // brick for that number)
  auto side = [](int n, int g) { return (n + g - 1) / g; };
  for (int gx = 1; gx <= std::min(n[0], sms); ++gx) {
    const int bx = side(n[0], gx);
    if (side(n[0], bx) != gx || bx > kResidentMaxThreads) continue;
    for (int gy = 1; gy <= std::min(n[1], sms / gx); ++gy) {
      const int by = side(n[1], gy);
      if (side(n[1], by) != gy || bx * by > kResidentMaxThreads) continue;
      for (int gz = 1; gz <= std::min(n[2], sms / (gx * gy)); ++gz) {
        const int bz = side(n[2], gz);
        if (side(n[2], bz) != gz || bx * by * bz > kResidentMaxThreads) continue;
        const int face[3] = {gx > 1 ? by * bz : 0, gy > 1 ? bx * bz : 0, gz > 1 ? bx * by : 0};
        // Nanoseconds of a step, fitted to sweeps of 80 bricks of nine domains (FP32, within
        // about 15 %): one warp's latency (more with 168 registers), the issue of the brick's
        // warps, a trip to the neighbours along each axis that leaves the brick, the packets,
        // and one more poll for every further set of them that a thread fetches.
        const long long warps = (bx * by * bz + 31) / 32;
        const long long sets = 2LL * (face[0] + face[1] + face[2]), threads = 32 * warps;
        long long cost = (warps <= 8 ? 900 : 1300) + 150 * warps;
        for (int a = 0; a < 3; ++a) cost += face[a] ? 300 : 0;
        if (sets > 0) cost += 300 * ((sets + threads - 1) / threads - 1) + 100 * sets / threads;
        if (best < 0 || cost < best) {
          best = cost;
          *R = ResidentPlan{{bx, by, bz}, {gx, gy, gz}, (int)threads, (int)std::max(1LL, sets),
                            {0, 2 * face[0], 2 * (face[0] + face[1])}};
        }
      }
    }
  }
  // Against the plain kernel's nanoseconds at these sizes, fitted to the same domains (FP32);
  // with 16-bit storage the plain kernel was slower on all of them. Resident against plain,
  // 1000 steps a call, FP32: 1.66 us at 1024 x 4 x 4 (3.28), 3.28 at 32^3 (4.17), 3.95 at 38^3
  // (5.40), 2.05 at 24^3 (3.02), 2.30 at 20 x 12 x 9 (2.45); FP16 1.66 (3.48), 2.88 (3.66),
  // 3.67 (4.43), 2.02 (3.22), 2.30 (2.89) and 2.20 at 16^3 (3.02).
  if (best < 0) return false;
  *plan_cost = best;
  return store != 0 || best < plain_cost(P, store, 1);
}

// A launch holds its SMs for all its steps and starts only when all its blocks fit beside those
// of other launches, so domains on several streams take turns once the SMs are full, while
// plain launches interleave. Microseconds for one step of every domain, plain against
// resident: 32^3 FP32 on 1, 2, 4 streams 4.0/3.1, 5.5/6.1, 8.6/12.3, FP16 3.4/2.8, 4.5/5.4,
// 5.6/10.8; 1024 x 4 x 4 (two fit at once) FP32 on 1, 2, 4, 8 streams 3.2/1.8, 4.2/2.1, 5.5/4.0,
// 8.8/7.9, FP16 3.0/1.8, 3.6/2.2, 4.4/4.1, 5.8/8.1; 24^3 (two fit) FP32 on 2, 4, 6 streams
// 4.0/2.7, 5.3/5.3, 6.2/7.9; 256 x 4 x 3 (nine fit) FP16 on 8 and 12 streams 3.5/2.3, 4.1/3.1.
// Taking turns costs up to 1.3 times the plan's time each.
bool resident_pays(const DomainConst& P, int store, int sms, const ResidentPlan& R, long long cost,
                   int streams) {
  // blocks on an SM at once: registers and shared memory of up to 256 threads
  const int per_sm = R.threads <= 256 ? 256 / R.threads : 1;
  const int at_once = std::max(1, sms * per_sm / R.blocks());
  return streams <= at_once || cost * streams * 6 / (5 * at_once) < plain_cost(P, store, streams);
}

size_t resident_inbox_bytes(const ResidentPlan& R, int store) {
  const int packets = store == 0 ? Words<float>::packets : Words<__half>::packets;
  return (size_t)R.blocks() * 2 * packets * R.sets * sizeof(uint4);
}

cudaError_t launch_resident(const DomainConst& P, const ResidentPlan& R, int store, int parity,
                            void* pop, const float* ghost, unsigned* flag, void* inbox,
                            unsigned* epochs, const ResidentRun& run, cudaStream_t s) {
  cudaError_t e;
  if (store == 0) e = launch_t<float, false>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s);
  else if (store == 1)
    e = P.sround ? launch_t<__half, true>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s)
                 : launch_t<__half, false>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s);
  else
    e = P.sround ? launch_t<__nv_bfloat16, true>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s)
                 : launch_t<__nv_bfloat16, false>(P, R, pop, ghost, flag, inbox, epochs, parity, run, s);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

}  // namespace lbm
