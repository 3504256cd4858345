// Boundary, initialisation, moment and reduction kernels of libwlbm.
//
//  k_walls     ghost cells of non-periodic walls (Sec. 2.6): isotropic blackbody walls
//              overwrite d_i = w_i (e_eq(T_w) - e_ref) (Eq. isotropic); adiabatic diffuse
//              walls collect the components that do not point into the domain and
//              re-emit them into the inward ones with fractions w_i (s_i.n) / sum
//              (Eq. adiabatic-diffuse, normalised so that energy is conserved).
//  k_periodic  periodic links (Sec. 2.6): ghost rows copy the opposite interior rows,
//              then ghost columns copy the opposite columns (corners via the diagonal);
//              before a step, per plane only the side that step's hop pulls from.
//  k_sources   internal temperature / radiation sources (Sec. 2.6): listed cells take fixed
//              values every step.
//  k_range     smallest and largest value of a start field (the bfloat16 scale).
//  k_init      local equilibrium start e_i = w_i e_eq(T) (Sec. 2.4) in float64.
//  k_moments   T - T_ref by Eq. pseudo-T in a cancellation-free form, q by Eq. q_corr.
//  k_reduce    float64 sums: energy (interior, + adiabatic-wall ghost cells), heat flux
//              (all cells and the central band of columns), band energy moment for the
//              conductivity fit, and the largest temperature change since the previous
//              reduction (and between window means, for the steady-state run).
#include <algorithm>
#include <cstring>

#include "elem.cuh"
#include "round_product.cuh"
#include "walls.cuh"
#include "wlbm_internal.hpp"

namespace wlbm {

namespace {

// Single-grid wall pass: kStagedWarps(q) warps and staged values for q <= kStagedMaxQ,
// else the streaming path with kWallWarps warps.
constexpr int kStagedMaxQ = 256;
constexpr int kMaxWallWarps = 32;
inline int staged_warps(int q) { return std::min(kMaxWallWarps, std::max(kWallWarps, q / 4)); }

template <typename T, bool SPEC>
__global__ void __launch_bounds__(32 * kMaxWallWarps) k_walls(const WallArgs a) {
  __shared__ WallSmem sm;
  extern __shared__ float4 wall_vals[];
  walls_chunk<T, SPEC>(a, a.codes, a.e_ref, int(blockIdx.x), sm,
                       a.q <= kStagedMaxQ ? wall_vals : nullptr);
}

// Batched wall pass: block b belongs to instance block_inst[b] (a host-built table: one
// load instead of a search); the instance's wall arguments are copied to shared memory
// once, so the segment lookup and the per-direction staging read no global memory chain.
// Codes and the reference-energy plane of step t come from the instance record.
template <typename T, bool SPEC>
__global__ void __launch_bounds__(32 * kWallWarps) k_walls_batch(const BatchWalls* B,
                                                                  const int* block_inst, int t) {
  __shared__ WallSmem sm;
  __shared__ __align__(16) WallArgs wa;
  const int b = int(blockIdx.x);
  const BatchWalls& I = B[block_inst[b]];
  static_assert(sizeof(WallArgs) % 4 == 0, "copied as 32-bit words");
  const int* src = reinterpret_cast<const int*>(&I.w);
  int* dst = reinterpret_cast<int*>(&wa);
  for (int i = int(threadIdx.x); i < int(sizeof(WallArgs) / 4); i += int(blockDim.x))
    dst[i] = src[i];
  const int cur = (I.phase + t) % I.n_e;
  float* e_ref = I.n_e == 3 ? I.e[(cur + 2) % 3] : nullptr;
  const uint8_t* codes = I.codes + size_t(t) * I.w.q;
  const int chunk = b - I.first_block;
  __syncthreads();
  walls_chunk<T, SPEC>(wa, codes, e_ref, chunk, sm, nullptr);
}

// Internal sources / radiation cells: one warp per cell, lanes over the directions.  With
// bfloat16 storage the cell's reference energy becomes the imposed total, so the stored
// values are the imposed ones relative to it (as for isothermal walls).
template <typename T>
__global__ void __launch_bounds__(256) k_sources(const SourceArgs a) {
  step_waits();
  const int s = int(blockIdx.x) * 8 + (int(threadIdx.x) >> 5);
  const int lane = int(threadIdx.x) & 31;
  if (s >= a.n) return;
  const int64_t off = a.off[s];
  const float R = a.esum[s];
  T* planes = static_cast<T*>(a.planes);
  for (int i = lane; i < a.q; i += 32) {
    T* p = planes + int64_t(((a.codes[i] >> 4) & 1) * a.q + i) * a.plane + off;
    wall_store(p, a.val[int64_t(s) * a.q + i], a.w[i], a.e_ref != nullptr, R, a.inv_scale);
  }
  if (lane == 0) {
    a.e_cur[off] = R;
    if (a.e_ref) a.e_ref[off] = R;
  }
}

// Ghost cell t of plane p (planes q, q + 1: local and reference energy).
template <typename T>
__device__ __forceinline__ void periodic_cell(const PeriodicArgs& a, int t, int p) {
  const int ncy = a.yper ? (a.xper ? a.nx : a.nx + 2) : 0;
  const int cy0 = a.xper ? kX0 : kGhostCol;
  const int ncx = a.xper ? 2 * (a.ny + 2) : 0;
  if (t >= 2 * ncy + ncx) return;
  // Before a step with known codes, a direction plane gets only the ghost cells that step
  // pulls from: the bottom (top) ghost row if its hop has c_y = +1 (-1), the left (right)
  // ghost column if c_x = +1 (-1), nothing if it pauses.  Energy planes, the adjoint's tape
  // and refreshes outside the step loop (a parity mask, no codes) copy everything.
  const bool partial = p < a.q && !a.tape && !a.par && a.codes;
  int hx = 0, hy = 0;
  if (partial) {
    const int code = a.codes[p];
    if (code & 8) return;
    hx = c_hop_x[code & 7];
    hy = c_hop_y[code & 7];
  }
  int rd, cd, rs, cs;
  if (t < 2 * ncy) {
    const int side = t / ncy, k = t - side * ncy;
    if (partial && hy != (side == 0 ? 1 : -1)) return;
    cd = cs = cy0 + k;
    rd = side == 0 ? 1 : a.ny + 2;
    rs = side == 0 ? a.ny + 1 : 2;
  } else {
    const int k = t - 2 * ncy;
    const int side = k / (a.ny + 2);
    if (partial && hx != (side == 0 ? 1 : -1)) return;
    rd = 1 + (k - side * (a.ny + 2));
    rs = rd;
    if (a.yper) {
      if (rd == 1) rs = a.ny + 1;
      else if (rd == a.ny + 2) rs = 2;
    }
    cd = side == 0 ? kGhostCol : kX0 + a.nx;
    cs = side == 0 ? kX0 + a.nx - 1 : kX0;
  }
  const int64_t od = int64_t(rd) * a.pitch + cd, os = int64_t(rs) * a.pitch + cs;
  if (p == a.q) {
    a.e_cur[od] = a.e_cur[os];
  } else if (p == a.q + 1) {
    a.e_ref[od] = a.e_ref[os];
  } else {
    const int par = a.tape ? 0 : a.par ? parity_of(*a.par, p) : (a.codes[p] >> 4) & 1;
    T* base = static_cast<T*>(a.planes) + int64_t(par * a.q + p) * a.plane;
    base[od] = base[os];
  }
}

template <typename T>
__global__ void k_periodic(const PeriodicArgs a) {
  step_waits();
  periodic_cell<T>(a, int(blockIdx.x * blockDim.x + threadIdx.x), int(blockIdx.y));
}

// Batched periodic pass of step t: block column b serves instance blocks[b].x, whose first
// block column is blocks[b].y; plane pointers and energy roles come from the instance record.
// One launch for all instances where each had its own: eight 256^2 x Q32 grids step in 38.7 us
// instead of 71, which the host spent on nine launches (33 us with overlapping launches).
template <typename T>
__global__ void __launch_bounds__(256) k_periodic_batch(const BatchInst* insts, const int2* blocks,
                                                         int t) {
  const int2 at = blocks[blockIdx.x];
  const BatchInst& I = insts[at.x];
  const int p = int(blockIdx.y);
  if (p >= I.a.q + I.n_e - 1) return;   // float32: one energy plane, bfloat16: two
  const int cur = (I.phase + t) % I.n_e;
  PeriodicArgs a;
  a.planes = I.a.planes; a.plane = I.a.plane; a.pitch = I.a.pitch;
  a.nx = I.a.nx; a.ny = I.a.ny; a.q = I.a.q;
  a.codes = I.codes + size_t(t) * I.a.q;
  a.e_cur = I.e[cur];
  a.e_ref = I.n_e == 3 ? I.e[(cur + 2) % 3] : nullptr;
  a.xper = I.a.xper; a.yper = I.a.yper;
  a.tape = 0;
  a.par = nullptr;
  step_waits();
  periodic_cell<T>(a, (int(blockIdx.x) - at.y) * 256 + int(threadIdx.x), p);
}

// Order-preserving map of a float's bits to an unsigned (negative values reversed).
__device__ __forceinline__ unsigned ordered_bits(float v) {
  const unsigned u = __float_as_uint(v);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}

// Smallest and largest of n floats, NaN left out, as ordered bits combined into out[0] (from
// ~0u) and out[1] (from 0).  Bound by the one read of the field: 16-byte loads where the
// address allows, four in flight a thread.  It replaces a copy of the field to the host and an
// expm1 per cell there (2048^2 cells: a 480-step run 146.4 -> 95.9 ms).
__global__ void __launch_bounds__(256) k_range(const float* x, int64_t n, unsigned* out) {
  float lo = INFINITY, hi = -INFINITY;   // fminf and fmaxf drop a NaN
  bool any = false;
  auto take = [&](float v) {
    lo = fminf(lo, v);
    hi = fmaxf(hi, v);
    any = any || v == v;
  };
  const int64_t stride = int64_t(gridDim.x) * 256, first = int64_t(blockIdx.x) * 256 + threadIdx.x;
  const int64_t n4 = reinterpret_cast<uintptr_t>(x) % 16 == 0 ? n / 4 : 0;
  const float4* x4 = reinterpret_cast<const float4*>(x);
#pragma unroll 4
  for (int64_t k = first; k < n4; k += stride) {
    const float4 v = x4[k];
    take(v.x);
    take(v.y);
    take(v.z);
    take(v.w);
  }
  for (int64_t k = 4 * n4 + first; k < n; k += stride) take(x[k]);
  unsigned l = any ? ordered_bits(lo) : ~0u, h = any ? ordered_bits(hi) : 0u;
  l = __reduce_min_sync(0xffffffffu, l);
  h = __reduce_max_sync(0xffffffffu, h);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(out, l);
    atomicMax(out + 1, h);
  }
}

// Bound by the state's write and a cell's expm1 once the products leave the float64 pipe, which
// took three of its operations a value (bfloat16: six): 4096 x 256 x Q128 825 -> 160 us
// (bfloat16 1581 -> 176).
template <typename T>
__global__ void __launch_bounds__(256) k_init(const InitArgs a) {
  __shared__ float sw[kMaxQ];
  for (int i = int(threadIdx.x); i < a.q; i += 256) sw[i] = a.w[i];
  __syncthreads();
  const int fw = a.nx + 2, fh = a.ny + 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= fw * fh) return;
  const int fy = t / fw, fx = t - fy * fw;            // framed coordinates
  const int x = min(max(fx - 1, 0), a.nx - 1), y = min(max(fy - 1, 0), a.ny - 1);
  const double temp = a.t_ref + double(a.dT[int64_t(y) * a.nx + x]);
  const SplitDouble de = split_double(1.0 / expm1(a.theta / temp) - a.e_ref);
  const int64_t off = int64_t(fy + 1) * a.pitch + (kGhostCol + fx);
  T* planes = static_cast<T*>(a.planes);
  if (a.e_refp) {   // reference energy = the equilibrium energy of this cell
    float e0 = 0.f;
#pragma unroll 8
    for (int i = 0; i < a.q; ++i) e0 += round_product(sw[i], de);
    a.e_refp[off] = e0;
  }
  float e = 0.f;
#pragma unroll 8
  for (int i = 0; i < a.q; ++i)
    e += dev_store(planes + int64_t(i) * a.plane + off, round_product(sw[i], de), sw[i],
                   a.e_refp, off, a.scale, a.inv_scale);
  a.e_cur[off] = e;
}

// A pair of opposite directions i and j = i + Q/2 as the flux sums need it: the elements of
// their current planes relative to the buffer, w_i - w_j and s_i.  Staged once a block, so that a
// pair costs two loads and the arithmetic (parities, weights and plane offsets worked out per
// cell kept the warps issuing, not loading).
struct alignas(16) FluxPair {
  int64_t i, j;
  float dw, sx, sy, pad;
};
template <typename Par>
__device__ __forceinline__ void stage_pairs(FluxPair* tab, int64_t plane, int q, Par par,
                                            const float* w, const float* sx, const float* sy) {
  for (int i = int(threadIdx.x); i < q / 2; i += int(blockDim.x)) {
    const int j = i + q / 2;
    tab[i] = {int64_t(par(i) * q + i) * plane, int64_t(par(j) * q + j) * plane, w[i] - w[j],
              sx[i], sy[i], 0.f};
  }
}

// Heat flux of one cell, q = sum_i e_i s_i (Eq. heat-flux, v = 1 here), taken over the
// pairs of opposite directions i and i + Q/2 (the ring order puts them Q/2 apart, with
// s_{i+Q/2} = -s_i exactly): q = sum_{i < Q/2} (e_i - e_{i+Q/2}) s_i, summed with Kahan's
// compensation (the product's rounding folded into the compensated term by one fma).  So
// the float32 result is within a few roundings of |q| for any Q, where a plain float32 sum
// of Q products errs by about Q roundings of the summands' magnitude (at Q = 1024 more than
// 1e-5 of a direction's amplitude).
// The difference e_i - e_j of stored values: float32 deviations subtract directly; bfloat16 ones
// before the scaling, and the reference parts w R leave only (w_i - w_j) R.  at: the cell's
// element in the buffer; four pairs' values are loaded while the previous four are added.
template <typename T>
__device__ __forceinline__ void cell_flux(const T* at, const FluxPair* tab, int q, bool ref,
                                          float R, float scale, float& qx, float& qy) {
  const int h = q / 2;        // a multiple of 4
  float cx = 0.f, cy = 0.f;   // compensations: what the running sums lost
  qx = 0.f;
  qy = 0.f;
  float na[4], nb[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    na[u] = Elem<T>::ld(at + tab[u].i);
    nb[u] = Elem<T>::ld(at + tab[u].j);
  }
  for (int i = 0; i < h; i += 4) {
    float d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = na[u] - nb[u];
    if (i + 4 < h) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        na[u] = Elem<T>::ld(at + tab[i + 4 + u].i);
        nb[u] = Elem<T>::ld(at + tab[i + 4 + u].j);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const FluxPair p = tab[i + u];
      const float v = ref ? fmaf(d[u], scale, __fmul_rn(p.dw, R)) : d[u];
      const float yx = fmaf(v, p.sx, -cx), yy = fmaf(v, p.sy, -cy);
      const float tx = qx + yx, ty = qy + yy;
      cx = (tx - qx) - yx;
      cy = (ty - qy) - yy;
      qx = tx;
      qy = ty;
    }
  }
}

// Bound by the one read of the state: 4096 x 256 x Q128 91 us (126 with the per-direction data
// worked out per cell), the copy rate's floor 80.
template <typename T>
__global__ void __launch_bounds__(256) k_moments(const MomentArgs a) {
  extern __shared__ __align__(16) unsigned char pair_smem[];
  FluxPair* tab = reinterpret_cast<FluxPair*>(pair_smem);
  if (a.qx || a.qy) {
    stage_pairs(tab, a.plane, a.q, [&](int i) { return parity_of(a.par, i); }, a.w, a.sx, a.sy);
    __syncthreads();
  }
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.nx * a.ny) return;
  const int y = t / a.nx, x = t - y * a.nx;
  const int64_t off = int64_t(y + 2) * a.pitch + (x + kX0);
  if (a.dT) {
    // L = ln(1 + 1/e) = L_ref + log1p(dE/(e_ref+1)) - log1p(dE/e_ref);
    // T - T_ref = theta/L - theta/L_ref = -theta dL / (L_ref (L_ref + dL)).
    const float de = a.e_cur[off];
    const float dl = log1pf(de / a.e_ref1) - log1pf(de / a.e_ref);
    const float v = a.weight * (-a.theta * dl / (a.l_ref * (a.l_ref + dl)));
    a.dT[t] = a.accumulate ? a.dT[t] + v : v;
  }
  if (a.qx || a.qy) {
    float qx, qy;
    cell_flux(static_cast<const T*>(a.planes) + off, tab, a.q, a.e_refp != nullptr,
              a.e_refp ? a.e_refp[off] : 0.f, a.scale, qx, qy);
    const float wx = a.weight * (qx * a.vg), wy = a.weight * (qy * a.vg);
    if (a.qx) a.qx[t] = a.accumulate ? a.qx[t] + wx : wx;
    if (a.qy) a.qy[t] = a.accumulate ? a.qy[t] + wy : wy;
  }
}

// T - T_ref of a cell's float32 local-energy deviation (Eq. pseudo-T in the same
// cancellation-free float32 form as k_moments; float64 per cell would cost more than the
// rest of the reduction on this GPU's float64 rate).  The reductions over cells that use
// it stay in float64.
__device__ __forceinline__ float temperature_dev32(float de, float e_ref, float e_ref1,
                                                   float l_ref, float theta) {
  const float dl = log1pf(de / e_ref1) - log1pf(de / e_ref);
  return -theta * dl / (l_ref * (l_ref + dl));
}

// max that keeps NaN (a NaN temperature must show in the residual)
__device__ __forceinline__ double fmax_nan(double a, double b) {
  return (a != a || b != b) ? __longlong_as_double(0x7ff8000000000000ll) : (a > b ? a : b);
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  return v;
}

// Per-direction data of a reduction block, staged once in shared memory.
struct ReduceSmem {
  float w[kMaxQ];
  uint8_t par[kMaxQ];
};

// Per-cell contributions of k_reduce at framed index t: the sums v[] and the residual.
template <typename T>
__device__ __forceinline__ void reduce_cell(const ReduceArgs& a, const ReduceSmem& sm,
                                            const FluxPair* tab, int t, double* v, double* res,
                                            double* resw) {
  const int fw = a.nx + 2, fh = a.ny + 2;
  const int fy = t / fw, fx = t - fy * fw;
  const bool gx = fx == 0 || fx == fw - 1, gy = fy == 0 || fy == fh - 1;
  const int64_t off = int64_t(fy + 1) * a.pitch + (kGhostCol + fx);
  const T* planes = static_cast<const T*>(a.planes);
  if (!gx && !gy) {
    const double e = double(a.e_cur[off]);
    v[0] += e;
    v[1] += e;
    // a cell's flux over its Q directions in float32 (as in k_moments: the stored values
    // are float32 or coarser), the sums over cells in float64
    float qx, qy;
    cell_flux(planes + off, tab, a.q, a.e_refp != nullptr, a.e_refp ? a.e_refp[off] : 0.f,
              float(a.scale), qx, qy);
    v[2] += qx;
    v[3] += qy;
    const int x = fx - 1;
    if (x >= a.band_x0 && x < a.band_x0 + a.band_w) {
      v[4] += qx;
      v[5] += (double(x) - a.band_xbar) * e;
    }
    const int64_t c = int64_t(fy - 1) * a.nx + x;
    const double tn = double(temperature_dev32(a.e_cur[off], float(a.e_ref), float(a.e_ref1),
                                               float(a.l_ref), float(a.theta)));
    if (a.has_snap) *res = fmax_nan(*res, fabs(tn - a.snap[c]));
    a.snap[c] = tn;
    if (a.win) {
      const double acc = a.win_first ? tn : a.win[c] + tn;
      if (a.win_last) {
        const double mean = acc * a.win_inv;
        if (a.win_has_prev) *resw = fmax_nan(*resw, fabs(mean - a.win_prev[c]));
        a.win_prev[c] = mean;
      } else {
        a.win[c] = acc;
      }
    }
  } else if (wall_energy_cell(fx, fy, fw, fh, a.diff_mask)) {
    double e = 0.0;            // wall cells are few: float64 over the directions
    for (int i = 0; i < a.q; ++i)
      e += dev_load(planes + int64_t(sm.par[i] * a.q + i) * a.plane + off, sm.w[i], a.e_refp,
                    off, float(a.scale));
    v[1] += e;
  }
}

// Stage 2, by the block that ends last: the blocks' partials combined in a fixed order into
// a.out.
__device__ __forceinline__ void reduce_finish(const ReduceArgs& a, int nblocks) {
  double v[kReduceSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  unsigned long long m[2] = {0ull, 0ull};
  for (int b = int(threadIdx.x); b < nblocks; b += 256) {
    const double* p = a.part + int64_t(b) * kReduceOut;
#pragma unroll
    for (int k = 0; k < kReduceSums; ++k) v[k] += __ldcg(p + k);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const unsigned long long u =
          static_cast<unsigned long long>(__double_as_longlong(__ldcg(p + kReduceSums + k)));
      m[k] = u > m[k] ? u : m[k];
    }
  }
  __shared__ double red[kReduceSums][8];
  __shared__ unsigned long long redm[2][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kReduceSums; ++k) {
    const double s = warp_sum(v[k]);
    if (lane == 0) red[k][wid] = s;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const unsigned long long u = warp_max_u64(m[k]);
    if (lane == 0) redm[k][wid] = u;
  }
  __syncthreads();
  if (threadIdx.x < kReduceSums) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[threadIdx.x][w];
    a.out[threadIdx.x] = s;
  } else if (threadIdx.x < kReduceOut) {
    unsigned long long u = 0ull;
    for (int w = 0; w < 8; ++w) u = redm[threadIdx.x - kReduceSums][w] > u
                                        ? redm[threadIdx.x - kReduceSums][w] : u;
    a.out[threadIdx.x] = __longlong_as_double(static_cast<long long>(u));
  }
}

// A grid-stride pass of resident blocks (64 registers, four an SM; more of them in a second wave
// left most SMs idle at its end); block b writes its kReduceOut partial results to a.part[b],
// and the one that ends last combines them.  4096 x 256 x Q128 146 us in one launch (145 + 9 in
// two before; a reduction of the 200 x 24 film is mostly launches): the chain of each cell's
// float64 sums, snapshot and temperature between its loads keeps it from the 83 of one read.
template <typename T>
__global__ void __launch_bounds__(256, 4) k_reduce(const ReduceArgs a) {
  const int cells = (a.nx + 2) * (a.ny + 2);
  __shared__ ReduceSmem sm;
  for (int i = int(threadIdx.x); i < a.q; i += 256) {
    sm.w[i] = a.w[i];
    sm.par[i] = uint8_t(parity_of(a.par, i));
  }
  extern __shared__ __align__(16) unsigned char pair_smem[];
  FluxPair* tab = reinterpret_cast<FluxPair*>(pair_smem);
  stage_pairs(tab, a.plane, a.q, [&](int i) { return parity_of(a.par, i); }, a.w, a.sx, a.sy);
  __syncthreads();
  double v[kReduceSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  double res = 0.0, resw = 0.0;   // largest |T - T_snap| and window change (>= 0 or NaN)
  for (int t = int(blockIdx.x) * 256 + int(threadIdx.x); t < cells; t += int(gridDim.x) * 256)
    reduce_cell<T>(a, sm, tab, t, v, &res, &resw);
  __shared__ double red[kReduceSums][8];
  __shared__ unsigned long long redm[2][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kReduceSums; ++k) {
    const double s = warp_sum(v[k]);
    if (lane == 0) red[k][wid] = s;
  }
  // |.| is non-negative, so its bit pattern orders like its value (NaN above all)
  const unsigned long long m0 = warp_max_u64(static_cast<unsigned long long>(__double_as_longlong(res)));
  const unsigned long long m1 = warp_max_u64(static_cast<unsigned long long>(__double_as_longlong(resw)));
  if (lane == 0) {
    redm[0][wid] = m0;
    redm[1][wid] = m1;
  }
  __syncthreads();
  if (threadIdx.x < kReduceSums) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[threadIdx.x][w];
    a.part[int64_t(blockIdx.x) * kReduceOut + threadIdx.x] = s;
  } else if (threadIdx.x < kReduceOut) {
    unsigned long long m = 0ull;
    for (int w = 0; w < 8; ++w) m = redm[threadIdx.x - kReduceSums][w] > m
                                        ? redm[threadIdx.x - kReduceSums][w] : m;
    a.part[int64_t(blockIdx.x) * kReduceOut + threadIdx.x] = __longlong_as_double(
        static_cast<long long>(m));
  }
  // the count returns to 0 by itself
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(a.done, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  reduce_finish(a, int(gridDim.x));
}

template <typename T>
__global__ void k_get_state(const StateArgs a) {
  const int fw = a.nx + 2, fh = a.ny + 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (t >= fw * fh) return;
  const int fy = t / fw, fx = t - fy * fw;
  const int64_t off = int64_t(fy + 1) * a.pitch + (kGhostCol + fx);
  const T* p = static_cast<const T*>(a.planes) + int64_t(parity_of(a.par, i) * a.q + i) * a.plane;
  a.framed[int64_t(i) * fw * fh + t] = dev_load(p + off, a.w[i], a.e_refp, off, a.scale);
}

template <typename T>
__global__ void k_set_state(const StateArgs a) {
  const int fw = a.nx + 2, fh = a.ny + 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (t >= fw * fh) return;
  const int fy = t / fw, fx = t - fy * fw;
  const int64_t off = int64_t(fy + 1) * a.pitch + (kGhostCol + fx);
  T* p = static_cast<T*>(a.planes) + int64_t(parity_of(a.par, i) * a.q + i) * a.plane;
  dev_store(p + off, a.framed[int64_t(i) * fw * fh + t], a.w[i], a.e_refp, off, a.scale,
            a.inv_scale);
}

template <typename T>
__global__ void k_energy(const StateArgs a) {
  const int fw = a.nx + 2, fh = a.ny + 2;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= fw * fh) return;
  const int fy = t / fw, fx = t - fy * fw;
  const int64_t off = int64_t(fy + 1) * a.pitch + (kGhostCol + fx);
  const T* planes = static_cast<const T*>(a.planes);
  float e = 0.f;
  for (int i = 0; i < a.q; ++i)
    e += dev_load(planes + int64_t(parity_of(a.par, i) * a.q + i) * a.plane + off, a.w[i],
                  a.e_refp, off, a.scale);
  a.e_cur[off] = e;
}

inline unsigned blocks_for(int64_t n, int per) { return unsigned((n + per - 1) / per); }

template <typename T>
cudaError_t walls_t(const WallArgs& a, cudaStream_t s) {
  const int chunks = wall_chunk_count(a.nseg, a.seg);
  if (chunks == 0) return cudaSuccess;
  const bool staged = a.q <= kStagedMaxQ;
  const int warps = staged ? staged_warps(a.q) : kWallWarps;
  const size_t bytes = staged ? size_t(a.q) * 32 * sizeof(float4) : 0;
  if (a.any_spec)
    launch_dependent(k_walls<T, true>, chunks, 32 * warps, bytes, s, a);
  else
    launch_dependent(k_walls<T, false>, chunks, 32 * warps, bytes, s, a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t periodic_t(const PeriodicArgs& a, bool early, cudaStream_t s) {
  const int blocks = periodic_blocks(a.nx, a.ny, a.xper, a.yper);
  if (blocks == 0) return cudaSuccess;
  const dim3 grid(unsigned(blocks), a.q + (a.e_ref ? 2 : 1));
  if (early)
    launch_dependent(k_periodic<T>, grid, 256, 0, s, a);
  else
    k_periodic<T><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

int periodic_blocks(int nx, int ny, int xper, int yper) {
  const int ncy = yper ? (xper ? nx : nx + 2) : 0;
  const int ncx = xper ? 2 * (ny + 2) : 0;
  return int(blocks_for(2 * int64_t(ncy) + ncx, 256));
}

cudaError_t launch_periodic_batch(int storage, const BatchInst* insts, const int2* blocks,
                                  int total_blocks, int max_q, bool early, int t,
                                  cudaStream_t s) {
  if (total_blocks <= 0) return cudaSuccess;
  const bool bf = storage == WLBM_STORE_BF16_DEV;
  const dim3 grid(unsigned(total_blocks), unsigned(max_q) + (bf ? 2 : 1));
  const auto k = bf ? k_periodic_batch<__nv_bfloat16> : k_periodic_batch<float>;
  if (early) launch_dependent(k, grid, 256, 0, s, insts, blocks, t);
  else k<<<grid, 256, 0, s>>>(insts, blocks, t);
  return cudaGetLastError();
}

cudaError_t launch_walls_batch(int storage, const BatchWalls* b, const int* block_inst,
                               int total_blocks, int t, bool any_spec, cudaStream_t s) {
  if (total_blocks <= 0) return cudaSuccess;
  const dim3 g{unsigned(total_blocks)}, blk{32 * kWallWarps};
  if (storage == WLBM_STORE_BF16_DEV) {
    if (any_spec) launch_dependent(k_walls_batch<__nv_bfloat16, true>, g, blk, 0, s, b, block_inst, t);
    else launch_dependent(k_walls_batch<__nv_bfloat16, false>, g, blk, 0, s, b, block_inst, t);
  } else {
    if (any_spec) launch_dependent(k_walls_batch<float, true>, g, blk, 0, s, b, block_inst, t);
    else launch_dependent(k_walls_batch<float, false>, g, blk, 0, s, b, block_inst, t);
  }
  return cudaGetLastError();
}

int wall_blocks(const WallArgs& a) { return wall_chunk_count(a.nseg, a.seg); }

cudaError_t configure_walls() {
  const int bytes = kStagedMaxQ * 32 * int(sizeof(float4));
  const void* fns[4] = {(const void*)k_walls<float, false>, (const void*)k_walls<float, true>,
                        (const void*)k_walls<__nv_bfloat16, false>,
                        (const void*)k_walls<__nv_bfloat16, true>};
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 4 && e == cudaSuccess; ++k)
    e = cudaFuncSetAttribute(fns[k], cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}

cudaError_t launch_walls(int storage, const WallArgs& a, cudaStream_t s) {
  return storage == WLBM_STORE_BF16_DEV ? walls_t<__nv_bfloat16>(a, s) : walls_t<float>(a, s);
}

cudaError_t launch_periodic(int storage, const PeriodicArgs& a, bool early, cudaStream_t s) {
  return storage == WLBM_STORE_BF16_DEV ? periodic_t<__nv_bfloat16>(a, early, s)
                                        : periodic_t<float>(a, early, s);
}

cudaError_t launch_range(const float* x, int64_t n, unsigned* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0xff, 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(out + 1, 0, 4, s);
  if (e != cudaSuccess) return e;
  const unsigned g = unsigned(std::min<int64_t>((n + 1023) / 1024, 152 * 8));
  k_range<<<g, 256, 0, s>>>(x, n, out);
  return cudaGetLastError();
}

bool range_value(unsigned u, float* v) {
  const unsigned b = u & 0x80000000u ? u & 0x7fffffffu : ~u;
  std::memcpy(v, &b, sizeof(*v));
  return *v == *v;
}

cudaError_t launch_init(int storage, const InitArgs& a, cudaStream_t s) {
  const unsigned g = blocks_for(int64_t(a.nx + 2) * (a.ny + 2), 256);
  if (storage == WLBM_STORE_BF16_DEV)
    k_init<__nv_bfloat16><<<g, 256, 0, s>>>(a);
  else
    k_init<float><<<g, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_moments(int storage, const MomentArgs& a, cudaStream_t s) {
  const unsigned g = blocks_for(int64_t(a.nx) * a.ny, 256);
  const size_t bytes = a.qx || a.qy ? size_t(a.q / 2) * sizeof(FluxPair) : 0;
  if (storage == WLBM_STORE_BF16_DEV)
    k_moments<__nv_bfloat16><<<g, 256, bytes, s>>>(a);
  else
    k_moments<float><<<g, 256, bytes, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sources(int storage, const SourceArgs& a, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  const unsigned g = unsigned((a.n + 7) / 8);
  if (storage == WLBM_STORE_BF16_DEV)
    launch_dependent(k_sources<__nv_bfloat16>, g, 256, 0, s, a);
  else
    launch_dependent(k_sources<float>, g, 256, 0, s, a);
  return cudaGetLastError();
}

cudaError_t launch_reduce(int storage, const ReduceArgs& a, cudaStream_t s) {
  const int cells = (a.nx + 2) * (a.ny + 2);
  const int nb = std::max(1, std::min(kReduceBlocks, (cells + 255) / 256));
  const size_t bytes = size_t(a.q / 2) * sizeof(FluxPair);
  if (storage == WLBM_STORE_BF16_DEV)
    k_reduce<__nv_bfloat16><<<nb, 256, bytes, s>>>(a);
  else
    k_reduce<float><<<nb, 256, bytes, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_get_state(int storage, const StateArgs& a, cudaStream_t s) {
  const dim3 g(blocks_for(int64_t(a.nx + 2) * (a.ny + 2), 256), a.q);
  if (storage == WLBM_STORE_BF16_DEV)
    k_get_state<__nv_bfloat16><<<g, 256, 0, s>>>(a);
  else
    k_get_state<float><<<g, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_set_state(int storage, const StateArgs& a, cudaStream_t s) {
  const dim3 g(blocks_for(int64_t(a.nx + 2) * (a.ny + 2), 256), a.q);
  const unsigned g1 = blocks_for(int64_t(a.nx + 2) * (a.ny + 2), 256);
  if (storage == WLBM_STORE_BF16_DEV) {
    k_set_state<__nv_bfloat16><<<g, 256, 0, s>>>(a);
    k_energy<__nv_bfloat16><<<g1, 256, 0, s>>>(a);
  } else {
    k_set_state<float><<<g, 256, 0, s>>>(a);
    k_energy<float><<<g1, 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace wlbm
