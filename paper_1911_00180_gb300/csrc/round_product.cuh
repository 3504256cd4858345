// The start field's products w_i * dE, rounded as float64 and float32 round them in turn.  Device
// code of k_init (k_aux.cu); only rounded single operations and fmaf, so that the host can run
// it against the product itself.
#pragma once

namespace wlbm {

namespace {

// float(double(w) * de), the product rounded to float64 and then to float32, mostly without
// the float64 pipe (2 operations a cycle and SM): de = hi + lo, and ph + s with ph = w hi
// rounded and s its exact remainder + w lo is within |ph| 2^-44 of the float64 product
// (de - hi - lo <= 2^-48 |de|, s rounds to 2^-47 |ph|, the product itself to 2^-53).  Rounding
// is monotonic, so where both ends of that interval round to the same float32 it is the
// result; else (one value in some 2^19, and products too small to split) float64 decides.
struct SplitDouble {
  double d;
  float hi, lo;
  bool small;   // w hi 2^-44 could leave the normal float32 range
};
__device__ __forceinline__ SplitDouble split_double(double d) {
  const float hi = float(d);
  return {d, hi, float(d - double(hi)), !(fabsf(hi) > 1e-18f && fabsf(hi) < 1e30f)};
}
// a call, so that the float64 instructions are not issued under a false predicate
__device__ __noinline__ float product64(float w, double d) { return float(double(w) * d); }
__device__ __forceinline__ float round_product(float w, const SplitDouble& x) {
  const float ph = __fmul_rn(w, x.hi);
  const float s = fmaf(w, x.lo, fmaf(w, x.hi, -ph));
  const float tol = fabsf(ph) * 0x1p-44f;
  const float r0 = __fadd_rn(ph, __fsub_rn(s, tol)), r1 = __fadd_rn(ph, __fadd_rn(s, tol));
  return r0 == r1 && !x.small ? r0 : product64(w, x.d);
}

}  // namespace

}  // namespace wlbm
