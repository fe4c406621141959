// Row pass of the complex constraint (constraint.cu), shared with the object step that precedes it
// (update.cu): row prefix sums of |ln a| and |phi| in 32.32 fixed point, P(y, x) = sum over x' < x of the
// value at (y, x'), obj_h x (obj_w + 1) each. v * 2^32 is exact in FP32, so llrintf of it is the nearest
// 32.32 value of v.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "engine.h"
#include "fft.cuh"

namespace ptycho {

__device__ __forceinline__ void cc_values(float2 o, long long& l, long long& p) {
  const float f = 4294967296.0f;
  l = llrintf(fabsf(logf(fmaxf(sqrtf(cabs2(o)), 1e-6f))) * f);
  p = llrintf(fabsf(atan2f(o.y, o.x)) * f);
}

// one block of 256 threads per object row y, pixel(x) giving its value (called once per pixel): warp w
// scans segment w of SEG pixels (32 per step, a carry between steps), then every segment adds the totals
// of the segments before it
template <class Pixel>
__device__ __forceinline__ void constraint_row(const ConstraintArgs& c, int y, Pixel pixel) {
  __shared__ long long s_tl[8], s_tp[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int W1 = c.obj_w + 1;
  const int SEG = ((c.obj_w + 7) / 8 + 31) / 32 * 32;
  const int x_lo = min(c.obj_w, w * SEG), x_hi = min(c.obj_w, x_lo + SEG);
  long long* pl = c.map_lna + (size_t)y * W1;
  long long* pp = c.map_phi + (size_t)y * W1;
  if (threadIdx.x == 0) {
    pl[0] = 0;
    pp[0] = 0;
  }
  long long cl = 0, cp = 0;  // this segment's sums so far
  for (int x0 = x_lo; x0 < x_hi; x0 += 32) {
    const int x = x0 + lane;
    long long vl = 0, vp = 0;
    if (x < x_hi) cc_values(pixel(x), vl, vp);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const long long ul = __shfl_up_sync(0xffffffffu, vl, d);
      const long long up = __shfl_up_sync(0xffffffffu, vp, d);
      if (lane >= d) {
        vl += ul;
        vp += up;
      }
    }
    if (x < x_hi) {
      pl[x + 1] = cl + vl;
      pp[x + 1] = cp + vp;
    }
    cl += __shfl_sync(0xffffffffu, vl, 31);
    cp += __shfl_sync(0xffffffffu, vp, 31);
  }
  if (lane == 0) {
    s_tl[w] = cl;
    s_tp[w] = cp;
  }
  __syncthreads();
  long long ol = 0, op = 0;
  for (int q = 0; q < w; ++q) {
    ol += s_tl[q];
    op += s_tp[q];
  }
  if (w > 0)
    for (int x = x_lo + lane; x < x_hi; x += 32) {
      pl[x + 1] += ol;
      pp[x + 1] += op;
    }
}

}  // namespace ptycho
