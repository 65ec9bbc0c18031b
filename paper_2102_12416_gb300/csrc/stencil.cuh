// The stencil's arithmetic on 16-byte vectors, shared by the step kernels.
#pragma once

#include "common.cuh"

namespace jgb {

// ---- 16-byte vectors ---------------------------------------------------------
template <typename T> struct V16;
template <> struct V16<float> {
  static constexpr int N = 4;
  __device__ static __forceinline__ void load(const float* p, float (&v)[4]) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  }
  __device__ static __forceinline__ void store(float* p, const float (&v)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <> struct V16<double> {
  static constexpr int N = 2;
  __device__ static __forceinline__ void load(const double* p, double (&v)[2]) {
    const double2 x = *reinterpret_cast<const double2*>(p);
    v[0] = x.x; v[1] = x.y;
  }
  __device__ static __forceinline__ void store(double* p, const double (&v)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
};

// Sum of the six neighbours in the stencil's order.  With EMU (FP64 states
// inside the integer adder's domain) the three pair sums run on the integer
// pipe and the two outer additions on the FP64 pipe: both pipes share the
// work and the result is bit-identical (`third`: the sum of the first two pairs
// is an integer one too).
template <typename T, bool EMU>
__device__ __forceinline__ T nsum(T xm, T xp, T ym, T yp, T zm, T zp, bool third = false) {
  if (EMU) {
    const double sx = dadd_nn((double)xm, (double)xp), sy = dadd_nn((double)ym, (double)yp),
                 sz = dadd_nn((double)zm, (double)zp);
    return (T)__dadd_rn(third ? dadd_nn(sx, sy) : __dadd_rn(sx, sy), sz);
  }
  return radd(radd(radd(xm, xp), radd(ym, yp)), radd(zm, zp));
}

// nsum with the z pair on the FP64 pipe (bit-identical: both adders round
// to nearest-even).
template <typename T, bool EMU>
__device__ __forceinline__ T nsum_zn(T xm, T xp, T ym, T yp, T zm, T zp) {
  if (EMU) {
    const double sx = dadd_nn((double)xm, (double)xp), sy = dadd_nn((double)ym, (double)yp),
                 sz = __dadd_rn((double)zm, (double)zp);
    return (T)__dadd_rn(__dadd_rn(sx, sy), sz);
  }
  return radd(radd(radd(xm, xp), radd(ym, yp)), radd(zm, zp));
}

}  // namespace jgb
