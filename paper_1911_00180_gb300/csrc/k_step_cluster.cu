// Many time steps of a small grid in one launch: the state lives in the shared memory of one
// thread-block cluster.
//
// A small grid's step is over in microseconds, so launching it costs more than running it
// (64 x 64 x Q16: 14.5 us a step with one periodic and one step launch, of which the two
// kernels run 5).  Here a cluster of up to 16 blocks keeps all planes of the grid in shared
// memory, a band of rows or columns per block with a halo of one cell, and applies the update
// (Eq. lbm-energy with the due hop of each direction, Eq. worm-paths, Eq. algorithm) for a
// whole chunk of steps: the bands exchange their edge cells through distributed shared
// memory, one cluster barrier per step orders the exchange, and global memory is touched only
// at the first and the last step.
//   * A thread owns cells of the band and walks the step's directions in the kind-sorted
//     order of the other step kernels, with the same operations (bfloat16 values rounded
//     every step), so the results are theirs bit for bit.
//   * Two buffers of values and cell terms alternate; halo cells behind isothermal walls hold
//     the wall's values in both, cells outside the frame zeros.
//   * Diffuse walls (horizontal, specularity 0) collect and re-emit in shared memory between
//     two steps, with the sums in the wall pass's order.
// What bounds it: the latency of Q updates per cell with one block of threads an SM, the halo
// and the barrier; not bandwidth.  Cycles of a step on 16 blocks at 2.07 GHz, 64 x 64 x Q16:
// update 1340, table 260, halo 990, barrier 950, 3700 in all (1.8 us a step, 14.5 with
// launches); the 200 x 24 x Q32 film: 4140, 240, walls 1690, halo 880, barrier 1350, 8400 in all
// (4.0 us, 22 with launches).  A launch adds 10-20 us, with few directions half of it the state's
// reads and writes (cluster_min_steps has the rule that follows).  Halos filled by an
// element loop over (direction, cell) took 4900 cycles (the index divisions), halos across
// rows of the other axis 3100 (scattered remote stores), so a thread keeps its halo cell and
// lines run along the halo.
#include <algorithm>

#include "cluster_layout.hpp"
#include "elem.cuh"
#include "wlbm_internal.hpp"

namespace wlbm {

namespace {

constexpr int kClMaxThreads = 1024;
constexpr int kClFewThreads = 512;         // up to here a thread has 128 registers

__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
// Shared address `a` of this block's layout in the block of rank r.
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t r) {
  uint32_t d;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(r));
  return d;
}
__device__ __forceinline__ void cl_store(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, __nv_bfloat16 v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(__bfloat16_as_ushort(v))
               : "memory");
}

// Loads and stores of this block's shared memory by 32-bit address.
__device__ __forceinline__ uint4 cl_lds4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a));
  return v;
}
__device__ __forceinline__ float cl_lds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
template <typename T>
__device__ __forceinline__ float cl_lds_val(uint32_t a) {
  if constexpr (sizeof(T) == 4) return cl_lds(a);
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return __uint_as_float(uint32_t(v) << 16);
}
// Store a new value; returns it as stored.
__device__ __forceinline__ float cl_sts(uint32_t a, float v, float) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
  return v;
}
__device__ __forceinline__ float cl_sts(uint32_t a, float v, __nv_bfloat16) {
  const unsigned short b = __bfloat16_as_ushort(__float2bfloat16_rn(v));
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(b) : "memory");
  return __uint_as_float(uint32_t(b) << 16);
}

__device__ __forceinline__ float cl_elem(float v, float) { return v; }
__device__ __forceinline__ __nv_bfloat16 cl_elem(float v, __nv_bfloat16) {   // exact here
  return __float2bfloat16_rn(v);
}

__device__ __forceinline__ int cl_mod(int v, int n) {
  const int r = v % n;
  return r < 0 ? r + n : r;
}

// Groups of threads that share the directions of `cells` cells, where a block has threads for
// more than one: group g takes the eights g, g + groups, ...
__device__ __forceinline__ int cl_groups(int cells, int q) {
  return max(1, min(int(blockDim.x) / cells, q / 8));
}

// What a cell of the frame is.
enum : int { kClVoid, kClIso, kClGhost, kClIn };   // outside, isothermal, diffuse ghost, interior

__device__ __forceinline__ int cl_kind(const ClusterArgs& a, int x, int y, float* iso) {
  *iso = 0.f;
  if ((!a.xper && (x < -1 || x > a.nx)) || (!a.yper && (y < -1 || y > a.ny))) return kClVoid;
  if (!a.xper && (x == -1 || x == a.nx)) {
    *iso = a.iso[x < 0 ? 0 : 1];
    return kClIso;
  }
  if (!a.yper && (y == -1 || y == a.ny)) {
    *iso = a.iso[y < 0 ? 2 : 3];
    return a.row_kind[y < 0 ? 0 : 1] == WLBM_BC_ISOTHERMAL ? kClIso : kClGhost;
  }
  return kClIn;
}

// One entry of a step's table: byte offsets, from the cell, of the value read and of the
// source terms (words times 4), w_i, and the offset of the direction's plane (paused: bit 31).
using ClEnt = uint4;

// All directions of one cell (shared addresses of the cell in buffer planes, terms and W);
// returns the sum of the new values.  As in the one-step kernels,
//   float32   g = 1 - W(s) (paused: of y), x = W E of s
//   bfloat16  x = X(s) - E_in / scale, paused (X - F)(y) + F(s) - E_in / scale
// UNI: 1 - W is g0 at every cell the directions come from.  B directions are in flight.
template <typename T, bool UNI, int B>
__device__ __forceinline__ float cl_cell(uint32_t cur, uint32_t nxt, uint32_t x, uint32_t f,
                                         uint32_t w, uint32_t tab, int q, float g0, float xf,
                                         float eins, float* accw) {
  constexpr bool BF = sizeof(T) == 2;
  float acc = 0.f, aw = 0.f;
  const uint32_t end = tab + 16u * uint32_t(q);
#pragma unroll 1
  for (; tab < end; tab += 16u * B) {
    ClEnt e[B];
    float v[B], xs[B], g[B];
#pragma unroll
    for (int d = 0; d < B; ++d) e[d] = cl_lds4(tab + 16u * d);
#pragma unroll
    for (int d = 0; d < B; ++d) {
      const bool paused = int32_t(e[d].w) < 0;
      v[d] = cl_lds_val<T>(cur + e[d].x);
      xs[d] = cl_lds((BF && paused ? f : x) + e[d].y);
      g[d] = UNI ? g0 : __fsub_rn(1.f, cl_lds(w + (paused ? 0u : e[d].y)));
    }
#pragma unroll
    for (int d = 0; d < B; ++d) {
      const float wi = __uint_as_float(e[d].z);
      if constexpr (BF) {
        if (int32_t(e[d].w) < 0) xs[d] = __fadd_rn(xf, xs[d]);
        xs[d] = __fsub_rn(xs[d], eins);
        aw += wi;
      }
      v[d] = fmaf(g[d], v[d], __fmul_rn(wi, xs[d]));
    }
#pragma unroll
    for (int d = 0; d < B; ++d) acc += cl_sts(nxt + (e[d].w & 0x7fffffffu), v[d], T());
  }
  *accw = aw;
  return acc;
}

// The ghost cells of periodic and isothermal sides, which the steps keep in shared memory only, as
// a caller may look for them: images of the new state, and walls' values (one value per thread of
// the cluster).  val, E, Ep: the band's cells; src, w: plane and weight of every direction.  0.8 us
// a launch of the 200 x 24 x Q32 film (1.8 with a wall's cell per thread), 3 of the 64 x 64 x Q16
// periodic grid; inlined, it cost that grid's 1000 steps 9 us (other registers in their loops).
template <typename T>
__device__ __noinline__ void cl_frame(const ClusterArgs& a, const unsigned char* val, uint32_t plane,
                                      const float* E, const float* Ep, const int* src,
                                      const float* w, int own, int minor) {
  constexpr bool BF = sizeof(T) == 2;
  const int q = a.q, ws = cl_line(minor), m0 = int(blockIdx.x) * a.per;
  T* const planes = static_cast<T*>(a.planes);
  const int col = a.ny + 2, row = a.xper ? a.nx + 2 : a.nx;   // cells of a column, of a row
  const int cols = a.xper ? 0 : 2 * col;
  const int low = !a.yper && a.row_kind[0] == WLBM_BC_ISOTHERMAL ? row : 0;
  const int high = !a.yper && a.row_kind[1] == WLBM_BC_ISOTHERMAL ? row : 0;
  const int n = cols + low + high;
  for (int k = int(blockIdx.x * blockDim.x + threadIdx.x); k < n * q;
       k += int(gridDim.x * blockDim.x)) {
    const int i = k / n, u = k - i * n;
    int x, y, side;
    if (u < cols) {
      side = u < col ? 0 : 1;
      x = side == 0 ? -1 : a.nx;
      y = u - side * col - 1;
    } else {
      side = u < cols + low ? 2 : 3;
      x = u - cols - (side == 3 ? low : 0) - (a.xper ? 1 : 0);
      y = side == 2 ? -1 : a.ny;
    }
    const int64_t o = int64_t(y + 2) * a.pitch + x + kX0;
    Elem<T>::st(planes + int64_t(src[i]) * a.plane + o, BF ? 0.f : __fmul_rn(w[i], a.iso[side]));
    if (BF && i == 0) a.e[o] = a.e_ref[o] = a.iso[side];
  }
  if (!a.xper && !a.yper) return;
  const int cells = own * minor, groups = cl_groups(cells, q);
  for (int k = int(threadIdx.x); k < cells * groups; k += int(blockDim.x)) {
    const int group = k / cells, M = (k - group * cells) / minor, m = k - group * cells - M * minor;
    const int at = (M + 1) * ws + m + 1;
    const int x = a.split_rows ? m : m0 + M, y = a.y_first + (a.split_rows ? m0 + M : m);
    const int right = a.xper && x == 0 ? a.nx : 0, left = a.xper && x == a.nx - 1 ? a.nx : 0;
    const int up = a.yper && y == 0 ? a.ny : 0, down = a.yper && y == a.ny - 1 ? a.ny : 0;
    if ((right | left | up | down) == 0) continue;
    const int64_t o = int64_t(y + 2) * a.pitch + x + kX0;
    auto images = [&](auto put) {   // in x, in y and in both
      for (int j = 1; j < 9; ++j) {
        const int jx = j % 3, jy = j / 3;
        const int dx = jx == 0 ? 0 : jx == 1 ? right : -left;
        const int dy = jy == 0 ? 0 : jy == 1 ? up : -down;
        if ((jx == 0 || dx != 0) && (jy == 0 || dy != 0)) put(o + int64_t(dy) * a.pitch + dx);
      }
    };
    for (int i = 8 * group; i < q; i += 8 * groups) {
      T v[8];
#pragma unroll
      for (int d = 0; d < 8; ++d) v[d] = reinterpret_cast<const T*>(val + uint32_t(i + d) * plane)[at];
      images([&](int64_t to) {
#pragma unroll
        for (int d = 0; d < 8; ++d) planes[int64_t(src[i + d]) * a.plane + to] = v[d];
      });
    }
    if (group != 0) continue;
    images([&](int64_t to) {
      a.e[to] = E[at];
      if (BF) a.e_ref[to] = Ep[at];
    });
  }
}

template <typename T, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    k_step_cluster(const __grid_constant__ ClusterArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr bool BF = sizeof(T) == 2;
  constexpr int ES = int(sizeof(T));
  constexpr int B = MAXT <= kClFewThreads ? 8 : 4;   // directions in flight (Q is a multiple of 8)
  const int q = a.q, tid = int(threadIdx.x), nthr = int(blockDim.x);
  const int rank = int(cl_rank()), nc = a.nc;
  // own cells: `per` rows or columns of the computed range, all of the other axis
  const int n_rows = a.y_last - a.y_first + 1;
  const int major = a.split_rows ? n_rows : a.nx;
  const int m0 = rank * a.per, m1 = min(m0 + a.per, major);
  const int own = m1 - m0;                                  // major extent (>= 1)
  const int minor = a.split_rows ? a.nx : n_rows;
  const int h = (a.split_rows ? own : minor) + 2, w = (a.split_rows ? minor : own) + 2;
  // offsets are those of the largest band, so that blocks can address one another's memory;
  // lines along the minor axis are contiguous, so that a halo is
  const int ws = cl_line(minor);
  const ClLayout<uint32_t> L = cl_layout<uint32_t>(q, a.per + 2, ws, ES);
  const int sr = a.split_rows ? ws : 1, sc = a.split_rows ? 1 : ws;   // strides of rows, columns
  const int xb = (a.split_rows ? 0 : m0) - 1, yb = a.y_first + (a.split_rows ? m0 : 0) - 1;
  const bool mper = a.split_rows ? a.yper : a.xper;         // major axis periodic
  const bool nper = a.split_rows ? a.xper : a.yper;         // minor axis periodic
  float* Wc = reinterpret_cast<float*>(smem + L.w);
  float* Ec = reinterpret_cast<float*>(smem + L.e);
  float* Ep = reinterpret_cast<float*>(smem + L.ep);
  ClEnt* tab = reinterpret_cast<ClEnt*>(smem + L.tab);
  float* rho = reinterpret_cast<float*>(smem + L.rho);      // [2][q]: y-, y+
  auto xbuf = [&](int b) { return reinterpret_cast<float*>(smem + L.x) + uint32_t(b) * L.cells; };
  auto fbuf = [&](int b) { return reinterpret_cast<float*>(smem + L.f) + uint32_t(b) * L.cells; };
  auto vbuf = [&](int b) { return smem + L.val + uint32_t(b) * uint32_t(q) * L.plane; };

  // directions of steps 0 and 1 for the table (one direction per thread; q <= nthr)
  int i1 = 0, c1 = 0, i2 = 0;
  if (tid < q) {
    i1 = a.order[tid];
    i2 = a.steps > 1 ? a.order[size_t(q + 17) + tid] : 0;
    c1 = a.codes[i1];
  }
  float* wsm = rho + 2 * q;
  for (int k = tid; k < 3 * q; k += nthr) rho[k] = k < 2 * q ? a.rho[2 * q + k] : a.w[k - 2 * q];
  int* src = reinterpret_cast<int*>(smem + L.src);
  for (int i = tid; i < q; i += nthr) src[i] = ((a.codes[i] >> 4) & 1) * q + i;
  __syncthreads();

  // ------------------------------------------------------------------- state read
  // Threads in turn along x, the axis that is contiguous in memory, whichever axis is split; a
  // cell's directions eight at a time, all loaded before the first is stored (one load, one store
  // left a latency per direction: one step of 11 x 11 x Q256 95 us, now 23).
  const int rgroups = cl_groups(h * w, q);
  for (int k = tid; k < h * w * rgroups; k += nthr) {
    const int group = k / (h * w), r = (k - group * h * w) / w, c = k - (group * h + r) * w;
    const int at = r * sr + c * sc;
    int x = xb + c, y = yb + r;
    float iso;
    const int kind = cl_kind(a, x, y, &iso);
    if (a.xper) x = cl_mod(x, a.nx);
    if (a.yper) y = cl_mod(y, a.ny);
    const int64_t o = int64_t(y + 2) * a.pitch + x + kX0;
    if (group == 0) {
      float e = 0.f, wv = 0.f, ref = 0.f;
      if (kind == kClIn || kind == kClGhost) {
        e = a.e[o];
        if (BF) ref = a.e_ref[o];
        if (kind == kClIn) wv = a.wfield ? a.wfield[o] : a.w0;
      } else if (kind == kClIso) {
        ref = iso;   // an isothermal cell's values refer to the wall's own equilibrium
      }
      Wc[at] = wv;
      Ec[at] = e;
      if (BF) Ep[at] = ref;
      const float fv = __fmul_rn(wv, e);
      for (int b = 0; b < 2; ++b) {
        if constexpr (BF) {
          xbuf(b)[at] = __fmul_rn(fmaf(__fsub_rn(1.f, wv), ref, fv), a.inv_scale);
          fbuf(b)[at] = __fmul_rn(fv, a.inv_scale);
        } else {
          xbuf(b)[at] = fv;
        }
      }
    }
    const T* p = static_cast<const T*>(a.planes) + o;
    const bool held = kind == kClIn || kind == kClGhost;
    for (int i = 8 * group; i < q; i += 8 * rgroups) {
      T v[8];
      if (held) {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = p[int64_t(src[i + u]) * a.plane];
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          Elem<T>::st(&v[u], kind == kClIso && !BF ? __fmul_rn(wsm[i + u], iso) : 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        reinterpret_cast<T*>(vbuf(0) + uint32_t(i + u) * L.plane)[at] = v[u];
        reinterpret_cast<T*>(vbuf(1) + uint32_t(i + u) * L.plane)[at] = v[u];
      }
    }
  }
  auto put_table = [&](int t) {   // entries of step t from (i1, c1)
    if (tid >= q) return;
    const int cx = c_hop_x[c1 & 7], cy = c_hop_y[c1 & 7];
    const int d = -(cy * sr + cx * sc);
    const bool paused = c1 & 8;
    tab[(t & 1) * q + tid] =
        make_uint4(uint32_t(i1) * L.plane + uint32_t((paused ? 0 : d) * ES), uint32_t(d * 4),
                   __float_as_uint(wsm[i1]), uint32_t(i1) * L.plane | (paused ? 1u << 31 : 0u));
  };
  // Diffuse wall pass on the values in buffer b: stored columns c_lo .. c_hi - 1 of the ghost
  // rows of the sides in `sides` (bit 0: y-, bit 1: y+).
  auto wall_rows = [&](int b, int sides, int c_lo, int c_hi) {
    float* part = reinterpret_cast<float*>(smem + L.part);
    const int n = c_hi - c_lo, two = sides == 3 ? 2 : 1;
    if (sides == 0 || n <= 0) return;   // the same for the whole block
    unsigned char* v = vbuf(b);
    auto side_of = [&](int s) { return sides == 3 ? s : sides - 1; };
    auto cell_of = [&](int s, int c) {
      return ((side_of(s) == 0 ? -1 : a.ny) - yb) * sr + c * sc;
    };
    auto value = [&](int i, int cell) {
      const float s = Elem<T>::ld_shared(reinterpret_cast<T*>(v + uint32_t(i) * L.plane) + cell);
      return BF ? fmaf(s, a.scale, __fmul_rn(wsm[i], Ep[cell])) : s;
    };
    const int stride = two * n;
    for (int k = tid; k < kClSums * stride; k += nthr) {
      const int gi = k / stride, u = k - gi * stride, s = u >= n ? 1 : 0;
      const int cell = cell_of(s, c_lo + u - s * n);
      const float* rh = rho + side_of(s) * q;
      float sum = 0.f;
#pragma unroll 4
      for (int i = gi; i < q; i += kClSums)
        if (rh[i] == 0.f) sum += value(i, cell);
      part[k] = sum;
    }
    __syncthreads();
    // every thread of a (side, column) adds the eight sums in turn, then takes its directions
    const int per = max(1, nthr / stride);
    for (int u = tid % stride; u < stride && tid < per * stride; u += stride) {
      const int s = u >= n ? 1 : 0, cell = cell_of(s, c_lo + u - s * n);
      const float* rh = rho + side_of(s) * q;
      float A = 0.f;
#pragma unroll
      for (int k = 0; k < kClSums; ++k) A += part[k * stride + u];
      const float R = BF ? Ep[cell] : 0.f;
#pragma unroll 4
      for (int i = tid / stride; i < q; i += per) {
        float d = rh[i] == 0.f ? 0.f : fmaf(A, rh[i], value(i, cell));
        if (BF) d = __fmul_rn(__fsub_rn(d, __fmul_rn(wsm[i], R)), a.inv_scale);
        Elem<T>::st(reinterpret_cast<T*>(v + uint32_t(i) * L.plane) + cell, d);
      }
    }
    if (stride > nthr)   // rows longer than the block
      for (int u = nthr + tid; u < stride; u += nthr) {
        const int s = u >= n ? 1 : 0, cell = cell_of(s, c_lo + u - s * n);
        const float* rh = rho + side_of(s) * q;
        float A = 0.f;
        for (int k = 0; k < kClSums; ++k) A += part[k * stride + u];
        for (int i = 0; i < q; ++i) {
          float d = rh[i] == 0.f ? 0.f : fmaf(A, rh[i], value(i, cell));
          if (BF) d = __fmul_rn(__fsub_rn(d, __fmul_rn(wsm[i], Ep[cell])), a.inv_scale);
          Elem<T>::st(reinterpret_cast<T*>(v + uint32_t(i) * L.plane) + cell, d);
        }
      }
    __syncthreads();
  };
  // columns of the stored rows that hold cells of a diffuse wall (not the isothermal corners)
  const int g_lo = a.xper ? 0 : max(0, -xb), g_hi = a.xper ? w : min(w, a.nx - xb);
  auto sides_in = [&](int lo, int hi) {   // diffuse walls among the stored rows lo .. hi - 1
    int m = 0;
    for (int side = 0; side < 2; ++side) {
      const int r = (side == 0 ? -1 : a.ny) - yb;
      if (!a.yper && a.row_kind[side] == WLBM_BC_ADIABATIC_DIFFUSE && r >= lo && r < hi)
        m |= 1 << side;
    }
    return m;
  };
  const int own_sides = sides_in(1, h - 1);
  put_table(0);
  __syncthreads();
  wall_rows(0, sides_in(0, h), g_lo, g_hi);   // the first step's walls, halo copies included
  cl_sync();

  // ------------------------------------------------------------------------ steps
  const uint32_t smem32 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  const bool to_prev = rank > 0 || mper, to_next = rank + 1 < nc || mper;
  const int prev = rank > 0 ? rank - 1 : nc - 1, next = rank + 1 < nc ? rank + 1 : 0;
  const int prev_own = min((prev + 1) * a.per, major) - prev * a.per;
  const uint32_t map_prev = cl_map(smem32, uint32_t(prev)), map_next = cl_map(smem32, uint32_t(next)),
                 map_own = cl_map(smem32, uint32_t(rank));
  const int cells = own * minor;
  const float g0 = __fsub_rn(1.f, a.w0);
  // The halo cells this block fills: its first line in the previous band, its last in the next
  // one, and, where the minor axis is periodic, its own ends.  A thread takes one of them (its
  // source, its place and the block it is in) for every `groups`-th direction.
  const int line = minor + 2, spots = 2 * line + (nper ? 2 * own : 0);
  const int groups = max(1, min(nthr / spots, 8));
  const int sgroup = tid / spots;
  int sat = -1, dat = 0;
  uint32_t dbase = smem32;
  auto spot = [&](int s) {
    sat = -1;
    if (s >= spots) return;
    int sm, sn, dm, dn;       // source and destination, stored (major, minor) coordinates
    if (s < 2 * line) {
      const bool down = s < line;
      if (!(down ? to_prev : to_next)) return;
      dn = sn = down ? s : s - line;
      if (dn == 0 || dn == line - 1) {
        if (!nper) return;
        sn = dn == 0 ? minor : 1;
      }
      sm = down ? 1 : own;
      dm = down ? prev_own + 1 : 0;
      dbase = down ? map_prev : map_next;
    } else {
      const int u = s - 2 * line;
      const bool left = u < own;
      sm = dm = 1 + (left ? u : u - own);
      sn = left ? minor : 1;
      dn = left ? 0 : minor + 1;
      dbase = map_own;
    }
    sat = sm * ws + sn;
    dat = dm * ws + dn;
  };
  if (sgroup < groups) spot(tid - sgroup * spots);
  int b = 0;
  for (int t = 0; t < a.steps; ++t, b ^= 1) {
    // the next step's directions: its table now, the schedule two steps ahead
    int in = 0;
    if (tid < q && t + 1 < a.steps) {
      i1 = i2;
      c1 = a.codes[size_t(t + 1) * q + i1];
      if (t + 2 < a.steps) in = a.order[size_t(t + 2) * (q + 17) + tid];
    }
    const float *xc = xbuf(b), *fc = fbuf(b);
    float *xn = xbuf(b ^ 1), *fn = fbuf(b ^ 1);
    for (int k = tid; k < cells; k += nthr) {
      const int M = 1 + k / minor, m = 1 + k - (M - 1) * minor, at = M * ws + m;
      const int x = xb + (a.split_rows ? m : M), y = yb + (a.split_rows ? M : m);
      const bool uni = !a.wfield && (a.xper || (x > 0 && x < a.nx - 1)) &&
                       (a.yper || (y > 0 && y < a.ny - 1));
      const float ein = Ec[at];
      float xf = 0.f, eins = 0.f, aw;
      if (BF) {
        xf = __fsub_rn(xc[at], fc[at]);
        eins = __fmul_rn(ein, a.inv_scale);
      }
      const uint32_t tb = smem32 + L.tab + uint32_t((t & 1) * q) * 16u;
      const uint32_t v0 = smem32 + L.val + uint32_t(b * q) * L.plane + uint32_t(at * ES),
                     v1 = smem32 + L.val + uint32_t((b ^ 1) * q) * L.plane + uint32_t(at * ES);
      const uint32_t xa = smem32 + L.x + (uint32_t(b) * L.cells + uint32_t(at)) * 4u,
                     fa = smem32 + L.f + (uint32_t(b) * L.cells + uint32_t(at)) * 4u,
                     wa = smem32 + L.w + uint32_t(at) * 4u;
      // (one form per warp: a warp with both would run one after the other)
      float e = __all_sync(__activemask(), uni)
                    ? cl_cell<T, true, B>(v0, v1, xa, fa, wa, tb, q, g0, xf, eins, &aw)
                    : cl_cell<T, false, B>(v0, v1, xa, fa, wa, tb, q, g0, xf, eins, &aw);
      if (BF) e = fmaf(e, a.scale, __fmul_rn(ein, aw));   // d' = scale v' + w_i E_in
      Ec[at] = e;
      const float wv = Wc[at], fv = __fmul_rn(wv, e);
      if (BF) {
        Ep[at] = ein;
        xn[at] = __fmul_rn(fmaf(__fsub_rn(1.f, wv), ein, fv), a.inv_scale);
        fn[at] = __fmul_rn(fv, a.inv_scale);
      } else {
        xn[at] = fv;
      }
    }
    if (t + 1 < a.steps) {
      put_table(t + 1);
      i2 = in;
      __syncthreads();
      wall_rows(b ^ 1, own_sides, max(g_lo, 1), min(g_hi, w - 1));   // the next step's walls
      // edge cells to the halos: the values of every direction, then the terms
      for (int p0 = 0; p0 < spots; p0 += nthr) {
        if (spots > nthr) spot(p0 + tid);
        if (sat < 0) continue;
        const uint32_t off = L.val + uint32_t((b ^ 1) * q) * L.plane;
        const uint32_t from = smem32 + off + uint32_t(sat * ES), to = dbase + off + uint32_t(dat * ES);
#pragma unroll 8
        for (int i = sgroup; i < q; i += groups) {
          const float v = cl_lds_val<T>(from + uint32_t(i) * L.plane);
          cl_store(to + uint32_t(i) * L.plane, cl_elem(v, T()));
        }
        if (sgroup == groups - 1) {
          const uint32_t xo = L.x + uint32_t(b ^ 1) * L.cells * 4u;
          cl_store(dbase + xo + uint32_t(dat * 4), cl_lds(smem32 + xo + uint32_t(sat * 4)));
          if (BF) {
            const uint32_t fo = L.f + uint32_t(b ^ 1) * L.cells * 4u;
            cl_store(dbase + fo + uint32_t(dat * 4), cl_lds(smem32 + fo + uint32_t(sat * 4)));
          }
        }
      }
      cl_sync();
    }
  }
  __syncthreads();

  // ---------------------------------------------------------------- state written
  for (int i = tid; i < q; i += nthr) {
    const int code = a.codes[size_t(a.steps - 1) * q + i];
    src[i] = (((code >> 4) & 1) ^ ((code & 8) ? 0 : 1)) * q + i;
  }
  __syncthreads();
  const int wgroups = cl_groups(cells, q);
  for (int k = tid; k < cells * wgroups; k += nthr) {
    const int group = k / cells, u = k - group * cells;
    const int r = 1 + u / (w - 2), c = 1 + u - (r - 1) * (w - 2), at = r * sr + c * sc;
    const int64_t o = int64_t(yb + r + 2) * a.pitch + xb + c + kX0;
    T* p = static_cast<T*>(a.planes) + o;
    for (int i = 8 * group; i < q; i += 8 * wgroups) {
      T v[8];
#pragma unroll
      for (int d = 0; d < 8; ++d)
        v[d] = reinterpret_cast<const T*>(vbuf(b) + uint32_t(i + d) * L.plane)[at];
#pragma unroll
      for (int d = 0; d < 8; ++d) p[int64_t(src[i + d]) * a.plane] = v[d];
    }
    if (group != 0) continue;
    a.e[o] = Ec[at];
    if (BF) a.e_ref[o] = Ep[at];
  }
  cl_frame<T>(a, vbuf(b), L.plane, Ec, Ep, src, wsm, own, minor);
}

template <typename T>
const void* cluster_fn_t(int threads) {
  return threads <= kClFewThreads ? (const void*)k_step_cluster<T, kClFewThreads>
                                  : (const void*)k_step_cluster<T, kClMaxThreads>;
}
const void* cluster_fn(int storage, int threads) {
  return storage == WLBM_STORE_BF16_DEV ? cluster_fn_t<__nv_bfloat16>(threads)
                                        : cluster_fn_t<float>(threads);
}

size_t cluster_bytes(const ClusterArgs& a, int es) {
  const int rows = a.y_last - a.y_first + 1;
  return size_t(cl_bytes(a.q, a.per, a.split_rows ? a.nx : rows, es));
}

void cluster_config(int storage, const ClusterArgs& a, cudaStream_t s, cudaLaunchConfig_t* c,
                    cudaLaunchAttribute* attr) {
  *c = cudaLaunchConfig_t{};
  c->gridDim = dim3(unsigned(a.nc));
  c->blockDim = dim3(unsigned(a.threads));
  c->dynamicSmemBytes = cluster_bytes(a, storage == WLBM_STORE_BF16_DEV ? 2 : 4);
  c->stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = unsigned(a.nc);
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  c->attrs = attr;
  c->numAttrs = 1;
}

}  // namespace

cudaError_t configure_step_cluster() {
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 4 && e == cudaSuccess; ++k) {
    const void* fn = cluster_fn(k & 1, k & 2 ? kClMaxThreads : kClFewThreads);
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kClSmem));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  return e;
}

// Steps a launch has to advance to pay for reading and writing the state through 16 SMs (0: none
// do).  The other side is one-step launches (k_step_direct and the boundary passes).  Microseconds
// of a call of n steps, calls in a row, cluster / one-step launches:
//   a cell per thread: n = 1 33 / 21, n = 3 39 / 35, n = 4 44 / 46, n = 64 276 / 535 (64 x 64 x
//     Q64); film 139 x 17 x Q32 20 / 20, 28 / 35, 33 / 46, 216 / 537; bfloat16 95 x 95 x Q64
//     42 / 21, 56 / 47, 60 / 61, 474 / 783.
//   few cells of 256 directions or more: n = 1 23 / 35, n = 64 437 / 1687 (film 11 x 11 x Q256).
//   more cells per thread: n = 16 91 / 96, n = 32 158 / 183, n = 64 288 / 349 (134 x 134 x Q16);
//     bfloat16 141 / 137, 238 / 267, 438 / 524 (1117 x 17 x Q32), 119 / 107, 201 / 198,
//     371 / 391 (512 x 64 x Q16).  With fewer than eight directions to each of a thread's cells
//     the one-step launches keep ahead: n = 64 394 / 342 (bfloat16 1878 x 29 x Q8), 426 / 390
//     (1448 x 23 x Q16), 467 / 370 (float32 film 1512 x 24 x Q8), though 289 / 320 for float32
//     189 x 189 x Q8.
static int cluster_min_steps(const ClusterArgs& c) {
  const int rows = c.y_last - c.y_first + 1;
  const int64_t cells = int64_t(c.per) * (c.split_rows ? c.nx : rows);
  const int64_t each = (cells + c.threads - 1) / c.threads;
  if (each > 1) return 8 * each <= c.q ? 32 : 0;
  return c.q >= 256 && cells * c.q <= 16384 ? 1 : 4;
}

bool cluster_plan(int storage, ClusterArgs* a) {
  const int es = storage == WLBM_STORE_BF16_DEV ? 2 : 4;
  const int rows = a->y_last - a->y_first + 1;
  if (a->q > 512) return false;
  double best = 0.0;
  ClusterArgs pick{};
  for (int nc = kClMax; nc >= 1; nc /= 2)
    for (int split = 1; split >= 0; --split) {
      const int major = split ? rows : a->nx, minor = split ? a->nx : rows;
      ClusterArgs c = *a;
      c.split_rows = split;
      c.per = (major + nc - 1) / nc;
      c.nc = (major + c.per - 1) / c.per;   // no empty band
      if (!cl_fits(c.q, c.per, minor, es)) continue;
      const int64_t cells = int64_t(c.per) * minor;
      c.threads = int(std::min<int64_t>(kClMaxThreads, (std::max<int64_t>(cells, c.q) + 31) / 32 * 32));
      // cycles of a step: the directions of a thread's cells in turn, the halo, the barrier
      const double waves = double((cells + c.threads - 1) / c.threads);
      const double cost = waves * c.q * (30.0 + c.threads / 32.0 * 3.0) +
                          2.0 * double(c.q) * (minor + c.per) / c.threads * 40.0 + 600.0;
      if (best != 0.0 && cost >= best) continue;
      cudaLaunchConfig_t cfg;
      cudaLaunchAttribute attr;
      cluster_config(storage, c, nullptr, &cfg, &attr);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, cluster_fn(storage, c.threads), &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        continue;
      }
      best = cost;
      pick = c;
    }
  if (best == 0.0) return false;
  pick.min_steps = cluster_min_steps(pick);
  *a = pick;
  return pick.min_steps > 0;
}

cudaError_t launch_step_cluster(int storage, const ClusterArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(storage, a, s, &cfg, &attr);
  ClusterArgs args = a;
  void* params[1] = {&args};
  const cudaError_t e = cudaLaunchKernelExC(&cfg, cluster_fn(storage, a.threads), params);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace wlbm
