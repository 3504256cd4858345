// Shared memory of a block of k_step_cluster: where its arrays lie, and which bands fit.
// Plain C++ besides the kernel, so that the host can check the arithmetic without a GPU.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define WLBM_HOST_DEVICE __host__ __device__
#else
#define WLBM_HOST_DEVICE
#endif

namespace wlbm {

constexpr int kClMax = 16;                 // blocks of a cluster (above 8: non-portable size)
constexpr int kClSmem = 227 * 1024;
constexpr int kClSums = 8;                 // partial sums of a wall's collected energy

// Row length, in cells, of a block's arrays: its lines along the minor axis, halo included.  Odd,
// so that lines next to one another start in different banks.
WLBM_HOST_DEVICE inline int cl_line(int minor) { return (minor + 2) | 1; }

// Shared memory of a block holding `lines` lines (halo included) of `line` cells.  U: 32 bits in
// the kernel, whose blocks fit; 64 for the question whether they do, which is asked of every
// grid (bfloat16 4416 x 532 x Q448 in one block takes 2^32 + 85520 bytes).
template <typename U>
struct ClLayout {
  U val, x, f, w, e, ep, tab, rho, part, src, total;
  U plane;   // bytes of one direction's cells
  U cells;
};

template <typename U>
WLBM_HOST_DEVICE inline ClLayout<U> cl_layout(int q, int lines, int line, int es) {
  ClLayout<U> L;
  L.cells = U(lines) * U(line);
  L.plane = (L.cells * U(es) + 15u) & ~U(15);
  U o = 0;
  auto take = [&](U bytes) {
    const U at = o;
    o += (bytes + 15u) & ~U(15);
    return at;
  };
  L.val = take(2u * U(q) * L.plane);
  L.x = take(2u * L.cells * 4u);                      // [2][cells] source terms
  L.f = es == 2 ? take(2u * L.cells * 4u) : L.x;      // bfloat16: W E / scale
  L.w = take(L.cells * 4u);                           // W_corr
  L.e = take(L.cells * 4u);                           // local energy, own cells
  L.ep = es == 2 ? take(L.cells * 4u) : L.e;          // and one step before
  L.tab = take(2u * U(q) * 16u);
  L.rho = take(3u * U(q) * 4u);                       // re-emission fractions of y-, y+; w
  L.src = take(U(q) * 4u);                            // plane of every direction
  L.part = take(kClSums * 2u * U(lines > line ? lines : line) * 4u);
  L.total = o;
  return L;
}

// Bytes of a block whose band is `per` lines of `minor` cells, and whether a block may have them.
inline uint64_t cl_bytes(int q, int per, int minor, int es) {
  return cl_layout<uint64_t>(q, per + 2, cl_line(minor), es).total;
}
inline bool cl_fits(int q, int per, int minor, int es) {
  return cl_bytes(q, per, minor, es) <= uint64_t(kClSmem);
}

}  // namespace wlbm
