// Output jobs of the ring-synthesis kernels (ringfft.cu, ringsynth.cu).
#pragma once

#include "common.cuh"

namespace tl {

// One output map: its coefficient plane's first ring (T2 [ring][m], chosen on the
// host, so that the kernel indexes no parameter array at run time), phi-derivative
// order k, 1/sin(theta) weight and output scale (double, and rounded to float).
struct JobDev {
  const void *in;
  void *out;
  double scale;
  float scalef;
  int k, div_sint;
  long long tile;  // output layout: 0 plain, else the tile stride (see d3_pix)
  int il;          // input rows four-ring interleaved (element m at row[4 m])
};

// The ring's coefficient row in a plane and the element stride along m
template <typename T2>
__device__ __forceinline__ const T2 *job_row(const JobDev &J, int r, int mmax, int &fs) {
  fs = J.il ? 4 : 1;
  return J.il ? (const T2 *)J.in + (size_t)(r >> 2) * (size_t)(mmax + 1) * 4 + (r & 3)
              : (const T2 *)J.in + (size_t)r * (mmax + 1);
}
#define TL_MAX_JOBS 96
struct JobList {
  int n;
  JobDev job[TL_MAX_JOBS];
};

// (i)^k g
template <typename T2>
__device__ __forceinline__ T2 rot_ik(T2 a, int k) {
  T2 g;
  switch (k & 3) {
    case 0: g = a; break;
    case 1: g.x = -a.y; g.y = a.x; break;
    case 2: g.x = -a.x; g.y = -a.y; break;
    default: g.x = a.y; g.y = -a.x; break;
  }
  return g;
}

}  // namespace tl
