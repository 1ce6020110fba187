// Column-FFT teams shared by the column-pass kernels.
#pragma once
#include "fft.cuh"

namespace cip {

// FFT elements per thread of one column FFT: one warp per FFT of 256..1024
// points in complex64 (so that the stage barriers are warp barriers), two warps
// at 2048; complex128 keeps 16 elements (register budget).
template <typename T> constexpr int cp_elems(int N) {
  if (sizeof(T) == 4) return N <= 256 ? 8 : (N == 512 ? 16 : 32);
  return N <= 128 ? 8 : 16;
}
template <typename T> constexpr int cp_team(int N) { return N / cp_elems<T>(N); }

// Channel slot stride of the fused tile (complex elements): the padded FFT
// layout, rounded to 16 bytes.
template <typename T> constexpr int cp_slot(int N) {
  return sizeof(T) == 4 ? ((spad(N) + 1) & ~1) : spad(N);
}

// Team barrier: a masked warp barrier for teams inside one warp, a named
// barrier (id 1 + team) for teams of several warps.
struct ColSync {
  int id, n;
  unsigned mask;
  __device__ __forceinline__ void operator()() const {
    if (n > 32) asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
    else __syncwarp(mask);
  }
};
__device__ __forceinline__ ColSync col_sync(int team, int tt) {
  ColSync s;
  s.n = tt;
  s.id = 1 + team;
  if (tt >= 32) s.mask = 0xffffffffu;
  else s.mask = ((tt == 32) ? 0xffffffffu : ((1u << tt) - 1u)) << ((team * tt) & 31);
  return s;
}

}  // namespace cip
