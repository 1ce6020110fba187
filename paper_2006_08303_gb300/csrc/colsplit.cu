// Split form of the column pass (the x-update of Eq. solx_Trans_DFT, three
// kernels instead of one): a forward column DFT of q-hat into the column
// buffer, an element-wise per-frequency solve X = xb + Psi^{-1}/N^2 Q over
// that layout, and an inverse column DFT into x-hat.  It moves 16 more bytes
// per voxel than the fused kernel (colpass.cu) but needs no shared-memory tile
// of all channels; the plan's autotuner chooses between the two per shape.
#include "fft.cuh"
#include "kernels.h"

namespace cip {

namespace {

// X = xb + Pinv Q at every bin, in place on colbuf; thread = (k2, k1), k1 fastest.
// A bin's factor is read once, row by row of the packed triangle; each thread copies the rows ahead
// asynchronously into its own shared-memory slots (no barrier), kRowBufs rows deep, so the loads in
// flight are not bounded by its registers.  The first rows and the data term are requested before the
// grid dependency, since they do not depend on the forward column DFTs (lowcol does: no const
// __restrict__, whose read-only loads the wait does not order).  Plain loads (72
// registers of them in flight at most) ran at 2.5 TB/s; split column pass before and now: 1024^2 x 10
// 127.8 -> 106.8 us, 1024^2 x 16 384 -> 206, 512^2 x 10 43.9 -> 30.3, 256^2 x 5 13.1 -> 11.2 us.
constexpr int kSolveThreads = 128, kRowBufs = 3;
template <typename T, int MMAX> constexpr int solve_minblocks() {
  return sizeof(T) == 4 ? (MMAX <= 12 ? 7 : 4) : 3;
}
template <typename T, int MMAX> constexpr size_t solve_smem() {
  return (size_t)kRowBufs * MMAX * kSolveThreads * 2 * sizeof(T);
}

template <typename T, int MMAX>
__global__ void __launch_bounds__(kSolveThreads, solve_minblocks<T, MMAX>())
    solve_split_kernel(typename CT<T>::type* __restrict__ colbuf, const typename CT<T>::type* pinv,
                       const typename CT<T>::type* xb, int N, int M, int plain, const typename CT<T>::type* lowcol,
                       const typename CT<T>::type* __restrict__ tw, T rho) {
  using C = typename CT<T>::type;
  const int k1 = blockIdx.x * kSolveThreads + threadIdx.x;
  const int k2 = blockIdx.y;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw) + threadIdx.x;  // entry j of row buffer s at buf[(s MMAX + j) kSolveThreads]
  const int npk = M * (M + 1) / 2;
  const bool on = k1 < N;
  const C* prow = pinv + binp(k2, 0, on ? k1 : 0, npk, N);  // plane stride kBinBlock
  auto issue = [&](int i) {
    if (on) {
      for (int j = 0; j < M - i; ++j, prow += kBinBlock) {
        const unsigned dst = smem_addr(buf + ((i % kRowBufs) * MMAX + j) * kSolveThreads);
        if constexpr (sizeof(C) == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(prow) : "memory");
        else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(prow) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  C r[MMAX], x[MMAX];
#pragma unroll
  for (int i = 0; i < kRowBufs - 1; ++i) issue(i);
  if (on) {
    const C* xcol = xb + binp(k2, 0, k1, M, N);  // plane stride kBinBlock
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < M) x[i] = xcol[(size_t)i * kBinBlock];
  }
  grid_dep_wait();  // the forward column DFTs are complete from here on
  grid_dep_launch();
  if (!on) return;
  const int CP = col_pitch(N);
  C* col = colbuf + (size_t)k2 * M * CP + k1;
  // columns k2 < kLowK of a TV plan with the low-column correction: Q from the column DFTs of the
  // components of t - u, the differences applied as spectral products
  const bool low = lowcol && k2 < kLowK;
  C dh = mk<C>(0.0, 0.0), dv = dh;
  if (low) {
    const C wh = ldg_tw(&tw[k2 * (kTwN / N)]), wv = ldg_tw(&tw[k1 * (kTwN / N)]);
    dh = mk<C>(wh.x - 1.0, -wh.y);  // exp(+2 pi i k2 / N) - 1
    dv = mk<C>(wv.x - 1.0, -wv.y);
  }
#pragma unroll
  for (int i = 0; i < MMAX; ++i) {
    if (i < M) {
      if (low) {
        C q = mk<C>(0.0, 0.0);
        cfmac(q, dh, lowcol[((size_t)k2 * M + i) * CP + k1]);
        cfmac(q, dv, lowcol[((size_t)(kLowK + k2) * M + i) * CP + k1]);
        r[i] = mk<C>(rho * q.x, rho * q.y);
      } else {
        r[i] = col[(size_t)i * CP];
      }
      if (plain) {  // plain FP32 method: X = Pinv (b + Q)
        r[i] = cadd(r[i], x[i]);
        x[i] = mk<C>(0.0, 0.0);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < MMAX; ++i) {
    if (i < M) {
      issue(i + kRowBufs - 1);  // (past the last row: an empty group)
      asm volatile("cp.async.wait_group %0;" ::"n"(kRowBufs - 1) : "memory");
      const C* p = buf + (i % kRowBufs) * MMAX * kSolveThreads;
#pragma unroll
      for (int j = i; j < MMAX; ++j) {
        if (j < M) {
          const C pij = p[(j - i) * kSolveThreads];
          cfma(x[i], pij, r[j]);
          if (j != i) cfmac(x[j], pij, r[i]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < MMAX; ++i)
    if (i < M) col[(size_t)i * CP] = x[i];
}

template <typename T, int MMAX>
cudaError_t solve_launch(typename CT<T>::type* colbuf, const typename CT<T>::type* pinv, const typename CT<T>::type* xb,
                         int N, int M, int plain, const typename CT<T>::type* lowcol, const typename CT<T>::type* tw,
                         T rho, Chain s) {
  auto k = solve_split_kernel<T, MMAX>;
  constexpr size_t sm = solve_smem<T, MMAX>();
  static PerDeviceOnce once;
  cudaError_t e = once([&] {
    cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (r != cudaSuccess) return r;
    return cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3((N + kSolveThreads - 1) / kSolveThreads, N / 2 + 1), dim3(kSolveThreads), sm, s, 0, colbuf,
                    pinv, xb, N, M, plain, lowcol, tw, rho);
}

template <typename T>
cudaError_t solve_m(typename CT<T>::type* colbuf, const typename CT<T>::type* pinv, const typename CT<T>::type* xb,
                    int N, int M, int plain, const typename CT<T>::type* lowcol, const typename CT<T>::type* tw,
                    T rho, Chain s) {
#define CIP_SOLVE(MM) \
  return solve_launch<T, MM>(colbuf, pinv, xb, N, M, plain, lowcol, tw, rho, s)
  if (M <= 4) CIP_SOLVE(4);
  if (M <= 8) CIP_SOLVE(8);
  if (M <= 10) CIP_SOLVE(10);
  if (M <= 12) CIP_SOLVE(12);
  if (M <= 16) CIP_SOLVE(16);
#undef CIP_SOLVE
  return cudaErrorInvalidValue;
}

}  // namespace

template <typename T>
cudaError_t launch_passB_split(const PassBArgs<T>& a, typename CT<T>::type* colbuf, int N, Chain s,
                               int* launches, const typename CT<T>::type* lowbuf, typename CT<T>::type* lowcol,
                               T rho) {
  // q-hat and x-hat use the column layout already: the column DFTs need no transposition; the
  // low-column maps of the correction (2 kLowK M columns) ride along in the forward launch
  cudaError_t e = launch_cols_fft<T>(a.qh, colbuf, a.tw, N, a.M, -1, s, lowbuf, lowcol, lowbuf ? 2 * kLowK * a.M : 0);
  if (e != cudaSuccess) return e;
  e = solve_m<T>(colbuf, a.pinv, a.bhat, N, a.M, a.plain, lowbuf ? lowcol : nullptr, a.tw, rho, s);
  if (e != cudaSuccess) return e;
  e = launch_cols_fft<T>(colbuf, a.xh, a.tw, N, a.M, +1, s);
  if (launches) *launches += 3;
  return e;
}

template cudaError_t launch_passB_split<float>(const PassBArgs<float>&, float2*, int, Chain, int*,
                                               const float2*, float2*, float);
template cudaError_t launch_passB_split<double>(const PassBArgs<double>&, double2*, int, Chain, int*,
                                                const double2*, double2*, double);

}  // namespace cip
