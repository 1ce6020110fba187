// Residual sums of a prior pass (the quantities of Eq. paramS): per-thread accumulation and the CTA's
// partial sums, added in a fixed order.
#pragma once
#include "kernels.h"

namespace cip {

template <typename T>
__device__ __forceinline__ void block_reduce_store(const T (&v)[kNPart], double* out) {
  __shared__ double red[32][kNPart];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double s[kNPart];
#pragma unroll
  for (int i = 0; i < kNPart; ++i) {
    double x = (double)v[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    s[i] = x;
  }
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < kNPart; ++i) red[warp][i] = s[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int i = 0; i < kNPart; ++i) {
      double acc = 0.0;
      for (int w = 0; w < nw; ++w) acc += red[w][i];
      out[i] = acc;
    }
  }
}

template <typename T>
__device__ __forceinline__ void acc_resid(T (&part)[kNPart], T w, T t, T un, const T* tprev, size_t g) {
  // a thread sums a few dozen terms at most, so the plan's precision suffices here; the
  // block and grid reductions run in double (FP64 issue is scarce on this part)
  const T r = w - t;
  part[0] = fma(r, r, part[0]);
  part[1] = fma(w, w, part[1]);
  part[2] = fma(t, t, part[2]);
  part[3] = fma(un, un, part[3]);
  if (tprev) {
    const T dt = t - tprev[g];
    part[4] = fma(dt, dt, part[4]);
  }
}

}  // namespace cip
