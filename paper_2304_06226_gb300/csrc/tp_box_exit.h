// Distance to the face by which a ray leaves a box, by cross-multiplication.
// Plain C++ as well as CUDA, so that it can be run on the host.
#pragma once
#include <math.h>
#ifdef __CUDACC__
#define TP_HD __host__ __device__ __forceinline__
#else
#define TP_HD inline
#endif

namespace tp {

// d != 0 without the FP64 pipe, which bounds the FP64 kernels
TP_HD bool nonzero(double d) {
#ifdef __CUDA_ARCH__
  return ((__double2hiint(d) & 0x7fffffff) | __double2loint(d)) != 0;
#else
  return d != 0.0;
#endif
}

// Box of half extents p, ray q + t v in its frame: the nearest of the faces
// ahead (2 * axis, + 1 on the positive side) and the distance n / d to it, with
// one division (three reciprocals were a third of the FP64 instructions of a
// slab's flight).  An axis the ray is parallel to has no face ahead, wherever q
// lies.  Returns `none` (face -1) for no direction.
TP_HD double box_exit(const double p[3], const double q[3], const double v[3], double none, int* face) {
  double bn = 1.0, bd = 0.0;
  int bf = -1;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int a = 0; a < 3; ++a) {
    const bool neg = signbit(v[a]);
    const double n = p[a] + (neg ? q[a] : -q[a]), d = fabs(v[a]);
    if (nonzero(d) && n * bd < bn * d) { bn = n; bd = d; bf = 2 * a + (neg ? 0 : 1); }
  }
  *face = bf;
  return bf >= 0 ? bn / bd : none;
}

}  // namespace tp
