// Step kernel for grids that leave the TMA tiles' blocks too few: one cell per thread, the
// directions read straight from L2.
//
// Same update as the other step kernels (Eq. lbm-energy with the due worm hop of each
// direction, Eq. worm-paths; E' = sum_i d_i', Eq. lbm-energy-density), the same rounded
// operations and the directions in the same kind-sorted order, so the same bits.
//
// A grid of 256 x 256 cells has 38 tiles of 128 x 14: a quarter of the SMs work, each waiting
// for a ring of copies one L2 latency deep.  Here a warp takes 32 columns of one row and a
// block kRows such rows, so the same grid has 256 blocks; the state of such grids sits in L2,
// and what bounds a step is its latency: launch, table and cell terms (two dependent loads),
// then kU directions' values in flight per thread while the previous kU are computed.  The
// cell terms (1 - W, W E and for bfloat16 the reference term) of the block's cells and their
// one-cell halo are in shared memory, where a direction's hop is one offset: no loop per kind,
// and nothing to wait for between kinds.
#include "elem.cuh"
#include "wlbm_internal.hpp"

namespace wlbm {

namespace {

constexpr int kRows = 8;             // rows (warps) per block
constexpr int kThreads = 32 * kRows;
constexpr int kSW = 34;              // staged row: 32 cells and one halo cell each side
constexpr int kTile = (kRows + 2) * kSW;
constexpr int kU = 8;                // directions in flight per thread (Q is a multiple of 8)

// Where the direct kernels are the faster ones, in blocks the TMA form would have (152 SMs; up
// to about one block an SM the TMA form leaves a ring's latency uncovered).  Microseconds a
// step, TMA / direct, both with ordinary launches (overlapping ones take 0.5-1.5 off either):
// float32 256^2 x Q32 (38 tiles) 16.1 / 9.7, 300 x 400 x Q64 (87) 20.8 /
// 14.5, 777 x 313 x Q40 (161) 22.9 / 18.0, 2048 x 128 x Q128 (160) 67.2 / 59.0, but 600^2 x Q64
// (215) 37.9 / 39.7 and 640 x 700 x Q128 (250) 85.3 / 90.1; bfloat16 256^2 x Q32 17.9 / 12.0,
// 400^2 x Q64 (116) 27.3 / 19.6, but 512^2 x Q64 (148) 23.2 / 28.2.  A backward pass with its
// recompute, reverse steps alone changed: 384 x 300 x Q64 (88 reverse tiles) 75.6 / 65.2 us a
// step, 450 x 400 x Q40 (116) 69.0 / 69.4, 512^2 x Q64 (185) 109.5 / 122.
constexpr int kDirectF32 = 176, kDirectBF16 = 128, kDirectAdj = 96;

// One direction of the step, relative to a cell's element in plane 0 and to its staged terms.
struct alignas(16) DirectDir {
  int32_t src, dst;   // source value (hop applied for a propagating direction), new value
  float w;
  int16_t own, from;  // staged terms: of the source value's cell, of the cell y - c
};

template <typename T, bool FIELD_W>
__global__ void __launch_bounds__(kThreads) k_step_direct(const StepArgs a) {
  constexpr bool REF = sizeof(T) == 2;
  __shared__ float sG[kTile], sX[kTile], sF[REF ? kTile : 1];
  extern __shared__ __align__(16) unsigned char smem[];
  DirectDir* table = reinterpret_cast<DirectDir*>(smem);
  const int tid = int(threadIdx.x), lane = tid & 31, ty = tid >> 5;
  const int col0 = a.cmin + 32 * int(blockIdx.x);
  const int row0 = a.rmin + kRows * int(blockIdx.y);
  for (int j = tid; j < a.q; j += kThreads) {
    const int i = a.order[j];
    const int code = a.codes[i];
    const int hop = code & 7, paused = (code >> 3) & 1, par = (code >> 4) & 1;
    const int cx = c_hop_x[hop], cy = c_hop_y[hop];
    DirectDir d;
    d.src = int((a.tape ? i : par * a.q + i) * a.plane) - (paused ? 0 : cy * a.pitch + cx);
    d.dst = int((a.tape ? i : (paused ? par : 1 - par) * a.q + i) * a.plane);
    d.w = a.w[i];
    d.from = int16_t(-(cy * kSW + cx));
    d.own = paused ? int16_t(0) : d.from;
    table[j] = d;
  }
  step_waits();
#pragma unroll
  for (int h = 0; h < (kTile + kThreads - 1) / kThreads; ++h) {
    const int idx = tid + h * kThreads;
    const int rr = idx / kSW, cc = idx - rr * kSW;
    const int row = row0 - 1 + rr, c = col0 - 1 + cc;
    if (idx >= kTile) break;
    float wv = 0.f, ev = 0.f, rv = 0.f;
    if (row < a.rows && c < a.pitch) {   // row0 - 1 >= 0, col0 - 1 >= kGhostCol - 1
      const int64_t o = int64_t(row) * a.pitch + c;
      ev = a.e_in[o];
      wv = FIELD_W ? a.wfield[o] : uniform_w(a, row, c);
      if (REF) rv = a.e_ref[o];
    }
    const float f = __fmul_rn(wv, ev), g = __fsub_rn(1.f, wv);
    sG[idx] = g;
    if (REF) {
      sX[idx] = __fmul_rn(fmaf(g, rv, f), a.inv_scale);
      sF[idx] = __fmul_rn(f, a.inv_scale);
    } else {
      sX[idx] = f;
    }
  }
  __syncthreads();
  const int row = row0 + ty, col = col0 + lane;
  if (row > a.rmax || col < a.cmin || col > a.cmax) return;
  const int64_t cell = int64_t(row) * a.pitch + col;
  const int at = (ty + 1) * kSW + lane + 1;
  const T* src = static_cast<const T*>(a.planes) + cell;
  T* dst = static_cast<T*>(a.tape ? a.tape_dst : a.planes) + cell;
  const float ein = REF ? a.e_in[cell] : 0.f;
  const float eins = REF ? __fmul_rn(ein, a.inv_scale) : 0.f;
  float acc = 0.f, accw = 0.f;
  float next[kU];
#pragma unroll
  for (int u = 0; u < kU; ++u) next[u] = Elem<T>::ld(src + table[u].src);
  for (int j = 0; j < a.q; j += kU) {
    float v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) v[u] = next[u];
    if (j + kU < a.q) {
#pragma unroll
      for (int u = 0; u < kU; ++u) next[u] = Elem<T>::ld(src + table[j + kU + u].src);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const DirectDir d = table[j + u];
      float x;
      if (REF) {
        // propagating: X(y - c); paused: (X(y) - F(y)) + F(y - c); less E_in(y) / scale
        const float t = d.own == 0 ? __fadd_rn(__fsub_rn(sX[at], sF[at]), sF[at + d.from])
                                   : sX[at + d.from];
        x = __fsub_rn(t, eins);
      } else {
        x = sX[at + d.from];
      }
      const float o = fmaf(sG[at + d.own], v[u], __fmul_rn(d.w, x));
      acc += Elem<T>::st(dst + d.dst, o);
      if (REF) accw += d.w;
    }
  }
  step_ends();
  a.e_out[cell] = REF ? fmaf(acc, a.scale, __fmul_rn(ein, accw)) : acc;
}

// One direction of a reverse step: its plane, the offset of x + c_k in the plane and in the
// staged s'.
struct alignas(16) DirectAdj {
  int32_t plane, hop;
  float w;
  int16_t from, paused;
};

// The transpose of a step (k_adjoint.cu has the algebra), cells and directions as above: the
// same operations in the order of k_adj_tma.  A block has the rows of k_adj_tma's tiles: its
// float32 harvest of an isothermal x wall adds the same cells.
constexpr int kAdjThreads = 32 * kAdjTmaRows;
constexpr int kAdjTile = (kAdjTmaRows + 2) * kSW;
constexpr int kAdjU = 4;
__global__ void __launch_bounds__(kAdjThreads, 2) k_adj_direct(const AdjArgs a,
                                                               const uint16_t* order) {
  __shared__ float sS[kAdjTile];
  // isothermal harvest of the block's rows at the x walls, added as k_adj_tma's warps of two
  // rows mostly do: each warp's first row, then each warp's second
  __shared__ float hrow[2][kAdjTmaRows];
  extern __shared__ __align__(16) unsigned char smem[];
  DirectAdj* table = reinterpret_cast<DirectAdj*>(smem);
  const int tid = int(threadIdx.x), lane = tid & 31, ty = tid >> 5;
  const int col0 = kGhostCol + 32 * int(blockIdx.x);
  const int row0 = 1 + kAdjTmaRows * int(blockIdx.y);
  for (int j = tid; j < a.q; j += kAdjThreads) {
    const int k = order[j];
    const int code = a.codes[k];
    const int cx = c_hop_x[code & 7], cy = c_hop_y[code & 7];
    table[j] = {int(k * a.plane), cy * a.pitch + cx, a.w[k], int16_t(cy * kSW + cx),
                int16_t(code & 8)};
  }
  if (tid < 2 * kAdjTmaRows) hrow[tid / kAdjTmaRows][tid % kAdjTmaRows] = 0.f;
  step_waits();
#pragma unroll
  for (int h = 0; h < (kAdjTile + kAdjThreads - 1) / kAdjThreads; ++h) {
    const int idx = tid + h * kAdjThreads;
    const int rr = idx / kSW, cc = idx - rr * kSW;
    const int row = row0 - 1 + rr, c = col0 - 1 + cc;
    if (idx >= kAdjTile) break;
    sS[idx] = row < a.ny + 4 && c < a.pitch ? a.s_in[int64_t(row) * a.pitch + c] : 0.f;
  }
  __syncthreads();
  const int row = row0 + ty, col = col0 + lane;
  bool harvest = false;
  if (row <= a.ny + 2 && col <= kX0 + a.nx) {
    const int64_t cell = int64_t(row) * a.pitch + col;
    const int at = (ty + 1) * kSW + lane + 1;
    const float* lam = a.lam_in + cell;
    const float* tape = a.dtil + cell;
    float* out = a.lam_out + cell;
    const float W = w_at(a, row, col), own = sS[at];
    const int iso = iso_wall_of(a, row, col);
    harvest = iso >= 0;
    const float keep = harvest ? 0.f : 1.f - W;
    float sigma = 0.f, a0 = 0.f, ed = 0.f, pd = 0.f, hs = 0.f;
    float nb[kAdjU], nd[kAdjU], np[kAdjU];
    auto fetch = [&](int j) {
#pragma unroll
      for (int u = 0; u < kAdjU; ++u) {
        const DirectAdj d = table[j + u];
        nb[u] = lam[d.plane + d.hop];
        nd[u] = tape[d.plane];
        np[u] = d.paused ? lam[d.plane] : 0.f;
      }
    };
    fetch(0);
    for (int j = 0; j < a.q; j += kAdjU) {
      float b[kAdjU], dv[kAdjU], p[kAdjU];
#pragma unroll
      for (int u = 0; u < kAdjU; ++u) {
        b[u] = nb[u];
        dv[u] = nd[u];
        p[u] = np[u];
      }
      if (j + kAdjU < a.q) fetch(j + kAdjU);
#pragma unroll
      for (int u = 0; u < kAdjU; ++u) {
        const DirectAdj d = table[j + u];
        const float bv = b[u] + sS[at + d.from];
        const float av = d.paused ? p[u] + own : bv;
        sigma = fmaf(d.w, bv, sigma);
        if (u == 0 && j == 0) a0 = av;
        ed += dv[u];
        pd = fmaf(dv[u], av - a0, pd);
        if (harvest) hs = fmaf(d.w, av, hs);
        out[d.plane] = keep * av;
      }
    }
    step_ends();
    a.s_out[cell] = W * sigma;
    a.gw[cell] += fmaf(sigma - a0, ed, -pd);
    if (harvest) hrow[col == kGhostCol ? 0 : 1][ty] = hs;
  }
  // one global atomic per wall and block
  if (__syncthreads_or(harvest) && tid < 2) {
    float sum = 0.f;
    for (int r = 0; r < kAdjTmaRows; r += 2) sum += hrow[tid][r];
    for (int r = 1; r < kAdjTmaRows; r += 2) sum += hrow[tid][r];
    const int iso = a.iso_side[tid];
    if (iso >= 0 && sum != 0.f) atomicAdd(a.gtw + iso, double(sum));
  }
}

template <typename T>
cudaError_t launch_direct_t(const StepArgs& a, cudaStream_t s) {
  const dim3 grid((a.cmax - a.cmin) / 32 + 1, (a.rmax - a.rmin) / kRows + 1);
  const size_t bytes = size_t(a.q) * sizeof(DirectDir);
  if (a.wfield) launch_dependent(k_step_direct<T, true>, grid, kThreads, bytes, s, a);
  else launch_dependent(k_step_direct<T, false>, grid, kThreads, bytes, s, a);
  return cudaGetLastError();
}

}  // namespace

bool step_is_direct(int storage, const StepArgs& a) {
  // an explicit ring depth, tile loop or 128-column bfloat16 form selects the TMA kernels
  if (a.ring_stages != 0 || a.loop_blocks != 0 ||
      (storage == WLBM_STORE_BF16_DEV && !a.tape && !a.wide))
    return false;
  const int w = tma_tile_width(), r = tma_tile_rows();
  const int tiles = ((a.cmax - a.cbase) / w + 1) * ((a.rmax - a.rmin) / r + 1);
  // (the table's element offsets are 32-bit)
  return tiles <= (storage == WLBM_STORE_BF16_DEV ? kDirectBF16 : kDirectF32) &&
         2 * int64_t(a.q) * a.plane <= INT32_MAX;
}

cudaError_t launch_step_direct(int storage, const StepArgs& a, cudaStream_t s) {
  return storage == WLBM_STORE_BF16_DEV ? launch_direct_t<__nv_bfloat16>(a, s)
                                        : launch_direct_t<float>(a, s);
}

bool adj_direct_ok(const AdjArgs& a, int tiles) {
  // (isothermal y walls: the float32 harvest of a block is that of 128 columns)
  return tiles <= kDirectAdj && a.iso_side[2] < 0 && a.iso_side[3] < 0 &&
         int64_t(a.q) * a.plane <= INT32_MAX;
}

cudaError_t launch_adj_direct(const AdjArgs& a, const uint16_t* order, cudaStream_t s) {
  const dim3 grid((a.nx + 2 + 31) / 32, (a.ny + 2 + kAdjTmaRows - 1) / kAdjTmaRows);
  launch_dependent(k_adj_direct, grid, kAdjThreads, size_t(a.q) * sizeof(DirectAdj), s, a, order);
  return cudaGetLastError();
}

}  // namespace wlbm
