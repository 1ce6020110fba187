// Fused column pass for few channels (the x-update of Eq. solx_Trans_DFT; complex64): one CTA per
// half-spectrum column k2, as colpass_fused_kernel, but without a ring of stages.
//   * one team per channel runs the forward column FFT, its first stage reading global memory, its last
//     leaving the channel's values in a shared-memory tile;
//   * every thread solves one bin at a time, X = xb + Psi^{-1} Q with the packed Hermitian factor, whose
//     M (M + 1) / 2 entries were copied asynchronously into the thread's own slots -- the first bin's,
//     and its data term, before the grid dependency (they do not depend on the preceding prior pass),
//     each following bin's row by row as the rows are used;
//   * one team per channel runs the inverse column FFT; its last stage writes global memory.
// Where the ring kernel's few stages serve few solving warps one after the other, here every bin is
// solved at once from data that is already in shared memory: the iteration alone on the device takes
// less time.  It issues more instructions (a copy and a load per entry), so iterations that share the
// device with other plans' (batches, the server) run the faster of the ring kernel and the split form
// instead (8 TV plans of 1024^2 x 3 in a batch: split 337 us an iteration of all, ring 369; of 1024^2 x 1
// 147 and 225).
// One TV iteration, the faster of ring and split -> this kernel: 64^2 x 3 5.97 (ring) -> 5.04 us, 256^2 x 3 8.92
// (ring) -> 7.93, 512^2 x 5 25.7 (ring) -> 22.9, 1024^2 x 3 57.4 (split) -> 46.7, 1024^2 x 1 26.8 (split) -> 22.6; 16
// plans of 128^2 .. 512^2 in a batch 8.38 -> 9.0 ms.  With 10 channels at 512^2 (whose slots leave room for three
// rows ahead) 37.1 -> 37.8: not offered.
#include "colteam.cuh"
#include "kernels.h"

namespace cip {

namespace {

constexpr int kDirectMaxM = 8;

struct DirectShape {
  int threads, solvers;
  size_t smem;
};
// a team per channel (at least two warps); as many solvers as threads, at most one per bin
DirectShape direct_shape(int N, int M) {
  DirectShape f{};
  const int fft = (M * cp_team<float>(N) + 31) / 32 * 32;
  f.threads = fft < 64 ? 64 : fft;
  f.solvers = f.threads < N ? f.threads : N;
  f.smem = ((size_t)M * cp_slot<float>(N) + (size_t)f.solvers * (M * (M + 1) / 2)) * sizeof(float2);
  return f;
}

struct DirectArgs {
  const float2* qh;    // [H][S][CP] q-hat row spectra (column layout)
  float2* xh;          // [H][S][CP] x-hat row spectra (column layout)
  const float2* pinv;  // packed Psi^{-1} / N^2, blocked by 32 bins (binp, npk planes)
  const float2* xb;    // data term / N^2 (or b for the plain FP32 method), blocked by 32 bins (M planes)
  const float2* tw;
  int M, S, solvers, plain;
};

template <int LOGN, int MMAX> constexpr int direct_threads() {
  const int t = 32 * ((MMAX * cp_team<float>(1 << LOGN) + 31) / 32);
  return t < 64 ? 64 : t;
}

template <int LOGN, int MMAX>
__global__ void __launch_bounds__(direct_threads<LOGN, MMAX>(), 2) coldirect_kernel(const DirectArgs a) {
  using C = float2;
  constexpr int N = 1 << LOGN, E = cp_elems<float>(N), TT = N / E;
  constexpr int CP = col_pitch(N), SLOT = cp_slot<float>(N);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int M = a.M, npk = M * (M + 1) / 2, NS = a.solvers;
  C* tile = reinterpret_cast<C*>(smem_raw);
  const int tid = threadIdx.x, k2 = blockIdx.x;
  const bool solver = tid < NS;
  C* buf = tile + (size_t)M * SLOT + tid;  // entry e of the packed triangle at buf[e NS]
  const int team = tid / TT, tt = tid % TT;
  const bool in_team = team < M;
  const ColSync cs = col_sync(team, TT);
  auto row0 = [&](int i) { return i * M - (i * (i - 1)) / 2; };  // first entry of row i
  auto copy_row = [&](int i, int k1) {  // row i of bin k1's packed triangle (nothing past the last row or bin)
    if (i < M && k1 < N) {
      const C* p = a.pinv + binp(k2, row0(i), k1, npk, N);
      unsigned dst = smem_addr(buf + (size_t)row0(i) * NS);
      for (int j = i; j < M; ++j, p += kBinBlock, dst += NS * (unsigned)sizeof(C))
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(p) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  C xn[MMAX];  // data term of the thread's next bin
  auto load_xb = [&](int k1) {
    const C* xbp = a.xb + binp(k2, 0, k1, M, N);
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < M) xn[i] = __ldg(xbp + (size_t)i * kBinBlock);
  };
  if (solver) {
#pragma unroll
    for (int i = 0; i < MMAX; ++i) copy_row(i, tid);
    load_xb(tid);
  }
  // the whole column's factor and data term into L2 (one contiguous run each in the blocked layout;
  // requests of at most 64 KB)
  if (tid < 2) {
    const int planes = tid == 0 ? npk : M;
    const C* base = (tid == 0 ? a.pinv : a.xb) + binp(k2, 0, 0, planes, N);
    const size_t n = (size_t)N * planes, step = 65536 / sizeof(C);
    for (size_t o = 0; o < n; o += step) prefetch_l2(base + o, (n - o < step ? n - o : step) * sizeof(C));
  }
  grid_dep_wait();
  grid_dep_launch();
  if (in_team) {
    C* slot = tile + (size_t)team * SLOT;
    const C* src = a.qh + ((size_t)k2 * a.S + team) * CP;
    auto in0 = [&](int i0, int off) { return src[i0 + off]; };
    auto outL = [&](int i0, int off, C v) { slot[i0 + off] = v; };
    fft_team_io<C, LOGN, E, -1, true>(slot, tt, a.tw, cs, in0, outL);
  }
  __syncthreads();
  for (int k1 = solver ? tid : N; k1 < N; k1 += NS) {
    C r[MMAX], x[MMAX];
#pragma unroll
    for (int i = 0; i < MMAX; ++i) {
      if (i < M) {
        r[i] = tile[(size_t)i * SLOT + k1];
        x[i] = xn[i];
        if (a.plain) {  // plain FP32 method: X = Pinv (b + Q)
          r[i] = cadd(r[i], x[i]);
          x[i] = mk<C>(0.0, 0.0);
        }
      }
    }
    if (k1 + NS < N) load_xb(k1 + NS);
    // MMAX groups are always in flight (one per row, empty past row M - 1), so row i's is complete when
    // all but the newest MMAX - 1 are
#pragma unroll
    for (int i = 0; i < MMAX; ++i) {
      asm volatile("cp.async.wait_group %0;" ::"n"(MMAX - 1) : "memory");
      if (i < M) {
        const C* p = buf + (size_t)row0(i) * NS;
#pragma unroll
        for (int j = i; j < MMAX; ++j) {
          if (j < M) {
            const C pij = p[(size_t)(j - i) * NS];
            cfma(x[i], pij, r[j]);
            if (j != i) cfmac(x[j], pij, r[i]);
          }
        }
      }
      copy_row(i, k1 + NS);
    }
#pragma unroll
    for (int i = 0; i < MMAX; ++i)
      if (i < M) tile[(size_t)i * SLOT + k1] = x[i];
  }
  __syncthreads();
  if (in_team) {
    C* slot = tile + (size_t)team * SLOT;
    C* dst = a.xh + ((size_t)k2 * a.S + team) * CP;
    auto in0 = [&](int i0, int off) { return slot[i0 + off]; };
    auto outL = [&](int i0, int off, C v) { dst[i0 + off] = v; };
    fft_team_io<C, LOGN, E, +1, false>(slot, tt, a.tw, cs, in0, outL);
  }
}

// two CTAs per SM
constexpr size_t kDirectSmem = (228 * 1024 - 2048) / 2;

template <int LOGN, int MMAX> cudaError_t launch_direct(const DirectArgs& a, const DirectShape& f, cudaStream_t s) {
  auto k = coldirect_kernel<LOGN, MMAX>;
  static PerDeviceOnce once;
  cudaError_t e = once(
      [&] { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDirectSmem); });
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3((1 << LOGN) / 2 + 1), dim3(f.threads), f.smem, s, 0, a);
}

}  // namespace

// complex64, up to 8 channels, N <= 1024, two CTAs per SM
bool coldirect_fits(int N, int M) { return N <= 1024 && M <= kDirectMaxM && direct_shape(N, M).smem <= kDirectSmem; }

cudaError_t launch_coldirect(const PassBArgs<float>& b, int S, cudaStream_t s) {
  if (!coldirect_fits(b.N, b.M)) return cudaErrorInvalidConfiguration;
  const DirectShape f = direct_shape(b.N, b.M);
  const DirectArgs a{b.qh, b.xh, b.pinv, b.bhat, b.tw, b.M, S, f.solvers, b.plain};
#define CIP_DIRECT(L) return b.M <= 4 ? launch_direct<L, 4>(a, f, s) : launch_direct<L, kDirectMaxM>(a, f, s)
  switch (b.N) {
    case 64: CIP_DIRECT(6);
    case 128: CIP_DIRECT(7);
    case 256: CIP_DIRECT(8);
    case 512: CIP_DIRECT(9);
    case 1024: CIP_DIRECT(10);
    default: return cudaErrorInvalidValue;
  }
#undef CIP_DIRECT
}

}  // namespace cip
