// Convolutional-dictionary synthesis prior (Alg. 2, 2D filters shared by all
// channels), the per-frequency part of one iteration:
//   x(w)   = xb(w) + Psi^{-1}(w)/N^2 p(w),  p_m = sum_l theta_l v_{l,m}      (Eq. solx_synt_DFT)
//   c_l    = conj(theta_l) x_m + rho G_{l,m},  G = F (t - u)                 (Eq. solz_DFT)
//   v_{.,m} = (c - conj(theta) (theta^T c) / (rho_w + ||theta||^2)) / rho_w  (Eq. solz_DFT_SM)
// with rho_w = rho, or rho + mu g(w) when the codes carry the gradient (Tikhonov) penalty of
// Eq. DL_PriorHP_conv (g = |r1^|^2 + |r2^|^2, the circular differences along both axes: the
// mu sum_i R_i^H R_i term of the note after Eq. solz keeps each bin's matrix diagonal + rank one)
// where theta_l is the DFT of filter l, Psi = I + beta Lambda^H Lambda (t = 1
// in Eq. solx_synt_DFT) and p is carried from the previous iteration's v.  One
// thread owns one (frequency, channel) pair; the L coefficient spectra of the
// channel are contiguous planes in the column layout [k2][m*L + l][k1].  The
// column DFTs around it and the element-wise shrinkage on the coefficient
// maps (the l1 prior pass over L*M maps) are the analysis path's kernels.
#include <algorithm>

#include <type_traits>

#include "fft.cuh"
#include "kernels.h"

namespace cip {

namespace {

template <typename T, int MMAX, int LMAX>
__global__ void __launch_bounds__(128) cd_solve_kernel(CDArgs<T> a) {
  using C = typename CT<T>::type;
  const int N = a.N, M = a.M, L = a.L;
  const int CP = col_pitch(N);
  const int k1 = blockIdx.x * blockDim.x + threadIdx.x;
  const int k2 = blockIdx.y;
  const int m = blockIdx.z;
  if (k1 >= N) return;
  const int npk = M * (M + 1) / 2;
  // All spectra here carry the inverse-DFT scale 1/N^2 (G, v, p, x, xb); the
  // stored factor is Psi^{-1}/N^2, so x = xb + N^2 (Psi^{-1}/N^2) p.
  // x_m = xb_m + sum_j P(m, j) p_j  (P Hermitian, packed upper triangle per bin)
  const C* pin = a.p_in + (size_t)k2 * M * CP + k1;
  const C* pcol = a.pinv + binp(k2, 0, k1, npk, N);  // plane stride kBinBlock
  C acc = mk<C>(0.0, 0.0);
#pragma unroll
  for (int j = 0; j < MMAX; ++j) {
    if (j < M) {
      const int i0 = min(m, j), j0 = max(m, j);
      const int pk = i0 * M - (i0 * (i0 - 1)) / 2 + (j0 - i0);
      const C pij = pcol[(size_t)pk * kBinBlock];
      const C pj = pin[(size_t)j * CP];
      if (m <= j) cfma(acc, pij, pj);
      else cfmac(acc, pij, pj);
    }
  }
  C x = a.xb[binp(k2, m, k1, M, N)];
  x.x += a.n2 * acc.x;
  x.y += a.n2 * acc.y;
  a.xcol[((size_t)k2 * M + m) * CP + k1] = x;
  // c_l = conj(theta_l) x + G_l ; s = theta^T c ; nrm = ||theta||^2
  C* g = a.colbuf + ((size_t)k2 * M * L + (size_t)m * L) * CP + k1;
  const C* th = a.theta + (size_t)k2 * a.th_planes * CP + k1;
  C c[LMAX];
  C s = mk<C>(0.0, 0.0);
  T nrm = T(0);
#pragma unroll
  for (int l = 0; l < LMAX; ++l) {
    if (l < L) {
      const C t = th[(size_t)l * CP];
      C cl = g[(size_t)l * CP];
      cfmac(cl, t, x);
      c[l] = cl;
      cfma(s, t, cl);
      nrm += t.x * t.x + t.y * t.y;
    }
  }
  const T rho_w = a.mu == T(0) ? a.rho : a.rho + a.mu * (T)(a.gs[k1] + a.gs[k2]);
  const T inv_rho = T(1) / rho_w;
  const T den = T(1) / (rho_w + nrm);
  const C coef = mk<C>(s.x * den, s.y * den);
  C pn = mk<C>(0.0, 0.0);
#pragma unroll
  for (int l = 0; l < LMAX; ++l) {
    if (l < L) {
      const C t = th[(size_t)l * CP];
      C v = c[l];
      // v = (c - conj(theta) coef) / rho
      v.x -= t.x * coef.x + t.y * coef.y;
      v.y -= t.x * coef.y - t.y * coef.x;
      v.x *= inv_rho;
      v.y *= inv_rho;
      g[(size_t)l * CP] = v;
      cfma(pn, t, v);
    }
  }
  a.p_out[((size_t)k2 * M + m) * CP + k1] = pn;
}

// The whole column pass of one (column k2, channel m) in one CTA: the forward column DFTs of the
// channel's L maps of G into a shared-memory tile, the x-update and the Sherman-Morrison z-update
// per bin on the tile, and the inverse column DFTs of v out of it.  The L maps are all a bin's
// z-update needs, so the code spectra are read once and written once (the three-kernel form, column
// DFT / cd_solve_kernel / column DFT, moves them six times).
// What bounds it: shared-memory traffic of the FFT stages (16 passes over the tile, ~20 us at 256^2 x 5
// with 32 filters); HBM needs 12 us for the two passes over the spectra.  Column pass there 95.7 ->
// 46.1 us (40 with the twiddles of each stage in a table of their own), 128^2 x 3 with 8 filters 16.9 ->
// 10.0, 512^2 x 3 with 16 filters 100 -> 54 us.
constexpr int kFuseThreads = 256;
template <typename T> constexpr int fuse_elems(int N) {  // FFT elements per thread: teams stay inside a warp
  if (sizeof(T) == 4) return N <= 256 ? 8 : (N == 512 ? 16 : 32);
  return N <= 128 ? 8 : 16;
}
template <typename T> constexpr int fuse_slot(int N) { return spad(N); }

template <typename T, int LOGN>
__global__ void __launch_bounds__(kFuseThreads) cd_fused_kernel(const CDArgs<T> a) {
  using C = typename CT<T>::type;
  constexpr int N = 1 << LOGN, E = fuse_elems<T>(N), TT = N / E, TEAMS = kFuseThreads / TT;
  constexpr int CP = col_pitch(N), ZS = fuse_slot<T>(N);
  static_assert(TT <= 32, "a team's barriers are warp barriers");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* tile = reinterpret_cast<C*>(smem_raw);  // [L][ZS]
  const int M = a.M, L = a.L;
  const int m = blockIdx.x, k2 = blockIdx.y, tid = threadIdx.x, team = tid / TT, tt = tid % TT;
  const unsigned mask = TT == 32 ? 0xffffffffu : (((1u << TT) - 1u) << ((team * TT) & 31));
  auto sync = [&]() { __syncwarp(mask); };
  const size_t map0 = ((size_t)k2 * M * L + (size_t)m * L) * CP;
  grid_dep_wait();
  grid_dep_launch();
  for (int l = team; l < L; l += TEAMS) {
    const C* src = a.qh + map0 + (size_t)l * CP;
    C* buf = tile + (size_t)l * ZS;
    auto in0 = [&](int i0, int off) { return src[i0 + off]; };
    auto outL = [&](int i0, int off, C v) { buf[spad(i0) + off + (off >> 4)] = v; };
    fft_team_io<C, LOGN, E, -1, true>(buf, tt, a.tw, sync, in0, outL);
  }
  __syncthreads();
  const int npk = M * (M + 1) / 2;
  const C* th0 = a.theta + (size_t)k2 * a.th_planes * CP;
  for (int k1 = tid; k1 < N; k1 += kFuseThreads) {
    // x_m = xb_m + N^2 sum_j (Psi^{-1} / N^2)(m, j) p_j, as in cd_solve_kernel
    const C* pin = a.p_in + (size_t)k2 * M * CP + k1;
    const C* pcol = a.pinv + binp(k2, 0, k1, npk, N);
    C acc = mk<C>(0.0, 0.0);
    for (int j = 0; j < M; ++j) {
      const int i0 = min(m, j), j0 = max(m, j);
      const C pij = pcol[(size_t)(i0 * M - (i0 * (i0 - 1)) / 2 + (j0 - i0)) * kBinBlock];
      const C pj = pin[(size_t)j * CP];
      if (m <= j) cfma(acc, pij, pj);
      else cfmac(acc, pij, pj);
    }
    C x = a.xb[binp(k2, m, k1, M, N)];
    x.x += a.n2 * acc.x;
    x.y += a.n2 * acc.y;
    a.xcol[((size_t)k2 * M + m) * CP + k1] = x;
    // c_l = conj(theta_l) x + G_l (formed again in the second loop: one shared-memory load and four
    // multiply-adds instead of 2 L registers), s = theta^T c, nrm = ||theta||^2
    const C* th = th0 + k1;
    C* g = tile + spad(k1);
    C s = mk<C>(0.0, 0.0);
    T nrm = T(0);
#pragma unroll 8
    for (int l = 0; l < L; ++l) {
      const C t = __ldg(th + (size_t)l * CP);
      C cl = g[(size_t)l * ZS];
      cfmac(cl, t, x);
      cfma(s, t, cl);
      nrm += t.x * t.x + t.y * t.y;
    }
    const T rho_w = a.mu == T(0) ? a.rho : a.rho + a.mu * (T)(a.gs[k1] + a.gs[k2]);
    const T inv_rho = T(1) / rho_w;
    const T den = T(1) / (rho_w + nrm);
    const C coef = mk<C>(s.x * den, s.y * den);
    C pn = mk<C>(0.0, 0.0);
#pragma unroll 8
    for (int l = 0; l < L; ++l) {
      const C t = __ldg(th + (size_t)l * CP);
      C v = g[(size_t)l * ZS];
      cfmac(v, t, x);
      v.x -= t.x * coef.x + t.y * coef.y;
      v.y -= t.x * coef.y - t.y * coef.x;
      v.x *= inv_rho;
      v.y *= inv_rho;
      g[(size_t)l * ZS] = v;
      if (a.colbuf) a.colbuf[map0 + (size_t)l * CP + k1] = v;  // kept for the dictionary update
      cfma(pn, t, v);
    }
    a.p_out[((size_t)k2 * M + m) * CP + k1] = pn;
  }
  __syncthreads();
  for (int l = team; l < L; l += TEAMS) {
    C* buf = tile + (size_t)l * ZS;
    C* dst = a.xh + map0 + (size_t)l * CP;
    auto in0 = [&](int i0, int off) { return buf[spad(i0) + off + (off >> 4)]; };
    auto outL = [&](int i0, int off, C v) { dst[i0 + off] = v; };
    fft_team_io<C, LOGN, E, +1, false>(buf, tt, a.tw, sync, in0, outL);
  }
}

// shared memory of the fused column pass; 0 where it does not run (a team wider than a warp, or a
// tile beyond one CTA's shared memory): the three-kernel form is used there
template <typename T> size_t fuse_smem(int N, int L) {
  if (N / fuse_elems<T>(N) > 32) return 0;
  const size_t sm = (size_t)L * fuse_slot<T>(N) * sizeof(typename CT<T>::type);
  return sm <= 224 * 1024 ? sm : 0;
}

template <typename T, int LOGN> cudaError_t launch_fused(const CDArgs<T>& a, Chain s) {
  if constexpr ((1 << LOGN) / fuse_elems<T>(1 << LOGN) > 32) {
    return cudaErrorInvalidValue;
  } else {
    auto k = cd_fused_kernel<T, LOGN>;
    static PerDeviceOnce once;
    cudaError_t e = once([&] { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024); });
    if (e != cudaSuccess) return e;
    return launch_pdl(k, dim3(a.M, a.N / 2 + 1), dim3(kFuseThreads), fuse_smem<T>(a.N, a.L), s, 0, a);
  }
}

// filters d[L][P][P] (centre P/2) placed on the N x N torus with the centre at (0,0)
template <typename Tin>
__global__ void embed_kernel(const Tin* __restrict__ d, double* __restrict__ out, int L, int P, int N) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= L * P * P) return;
  const int l = idx / (P * P), r = idx - l * P * P;
  const int i = r / P, j = r - i * P;
  const int c = P / 2;
  const int a = ((i - c) % N + N) % N, b = ((j - c) % N + N) % N;
  out[((size_t)l * N + a) * N + b] = (double)d[idx];
}

// theta from the half-pitch layout [L][N][P] (FP64) to the column layout [k2][L][CP]
template <typename T>
__global__ void theta_store_kernel(const SetupC<T>* __restrict__ th64, typename CT<T>::type* __restrict__ th, int L,
                                   int N) {
  using C = typename CT<T>::type;
  const int H = N / 2 + 1, P = half_pitch(N), CP = col_pitch(N);
  const size_t total = (size_t)L * N * H;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int k1 = (int)(i % N);
    const size_t r = i / N;
    const int l = (int)(r % L);
    const int k2 = (int)(r / L);
    th[((size_t)k2 * L + l) * CP + k1] = cconv<C>(th64[((size_t)l * N + k1) * P + k2]);
  }
}

// p_m = sum_l theta_l Z_{m,l} / N^2 from the column spectra Z of imported coefficient maps
template <typename T>
__global__ void p_from_z_kernel(const typename CT<T>::type* __restrict__ zcol, const typename CT<T>::type* __restrict__ th,
                                typename CT<T>::type* __restrict__ p, int N, int M, int L, int thp, T s) {
  using C = typename CT<T>::type;
  const int CP = col_pitch(N);
  const int k1 = blockIdx.x * blockDim.x + threadIdx.x;
  const int k2 = blockIdx.y, m = blockIdx.z;
  if (k1 >= N) return;
  C acc = mk<C>(0.0, 0.0);
  for (int l = 0; l < L; ++l)
    cfma(acc, th[((size_t)k2 * thp + l) * CP + k1], zcol[((size_t)k2 * M * L + (size_t)m * L + l) * CP + k1]);
  p[((size_t)k2 * M + m) * CP + k1] = mk<C>(acc.x * s, acc.y * s);
}

// ---- online dictionary update (Section IV-B, Eqs. d_admm, g_admm, h_admm, sold_3D) ----------
//
// State between steps: theta = F g and F(g - e) (spectra of the filters on the torus and of the
// filters minus the scaled dual), and g itself on its P x P support.  One step:
//   dl_solve  per bin: d-hat from the normal equation summed over the channels, w = d-hat + e-hat
//             with e-hat = theta - F(g - e); per column, Y(a, k2) = sum_k1 w exp(2 pi i k1 a / N)
//             for the P support rows a (so that d + e at the support points is a short sum over k2)
//   dl_filter per filter: v = d + e on the support, g = v / ||v|| (Eq. g_admm), the partial DFT
//             G(a, k2) = sum_b g(a, b) exp(-2 pi i k2 b / N)
//   dl_spec   per bin: g-hat = sum_a exp(-2 pi i k1 a / N) G(a, k2); e-hat <- w - g-hat (Eq.
//             h_admm, reading R22), so F(g - e) = 2 g-hat - w; theta = g-hat; p = sum_l theta_l z_l
// The spatial d and e off the support are never formed: g is zero there and e is only ever needed
// through its spectrum.

// exp(-2 pi i j / N) (SIGN < 0) or exp(+2 pi i j / N) (SIGN > 0) for any integer j (N a power of
// two: j mod N is j & (N - 1) in two's complement)
template <int SIGN, typename C>
__device__ __forceinline__ C tw_at(const C* __restrict__ tw, int j, int N) {
  const int r = j & (N - 1);
  C t = ldg_tw(&tw[r * (kTwN / N)]);
  if (SIGN > 0) t.y = -t.y;
  return t;
}

// Per frequency, one thread (k1 = block offset + thread, k2 = blockIdx.y, so that the warps read
// the column layout contiguously): the filter normal equation summed over the M channels,
// (sigma I + W W^H) d = b with W = [conj(zhat_{l,s})] (L x M) and b = W xhat + sigma F(g - e), by
// the Woodbury identity d = (b - W alpha) / sigma, (sigma I_M + W^H W) alpha = W^H b.  The L
// filters are streamed twice: once to accumulate W^H W and W^H b, once to form d; the M x M system
// is solved by Cholesky in registers.  Then w = d + e-hat is stored and its partial inverse DFT
// along k1 at the P support rows is summed over the CTA's bins: a small matrix product of the tile of
// w with the bins' exponentials, both in shared memory (62 shuffles per bin and filter as a
// reduce-scatter across each warp took more issue slots than the rest of the step); the last CTA of a column to finish adds the column's CTA sums in a fixed order, so the result
// does not depend on the order in which CTAs run.
// Two groups of kDLBlock threads share a bin: bound by the latency of the loads, one thread per bin left
// an SM seven warps to hide it behind.  They divide the entries of W^H b and W^H W (each sum still runs
// over all filters in order, so its rounding does not depend on the split); group 0 collects them in
// shared memory and solves the M x M system (both solving it cost 7% at M = 8, L = 9); then they divide
// the filters of the second pass.  Dividing
// the filters of the first pass as well was 4 us faster at 256^2 x 5, L = 32, but rounds differently, and
// the cancellation in b - W alpha turns that into 5e-5 of x at M = 8; four groups leave the 516 CTAs of
// N = 256 in two waves (146 us an iteration against 134).  dl_solve + dl_filter + dl_spec before and now,
// 256^2 x 5, L = 32, 11 x 11: 42 + 16 + 31 -> 36 + 14 + 18 us; an iteration 163 -> 136 us.
// Where there are CTAs enough without the second group, one group is the faster: the second adds barriers, and
// from M = 6 on no warps, since the registers of its threads leave half the CTAs on an SM.  Iterations, two groups
// and one: complex64 512^2 x 8 with 9 filters 334 and 305 us, 512^2 x 6 261 and 227, 512^2 x 1 32 filters 256 and
// 230, 256^2 x 8 93.2 and 81.5, but 256^2 x 7 32 filters 194 and 201, 512^2 x 3 428 and 439, 128^2 x 8 47.2 and 55.9;
// complex128 512^2 x 3 1860 and 1816, 256^2 x 5 793 and 763, 128^2 x 5 254 and 302, 256^2 x 8 1186 and 1220.
template <typename T> constexpr bool dl_one_group(int N, int M) {
  if (sizeof(T) == 8) return N >= 512 || (N == 256 && M < 8);
  return (N >= 512 && (M == 1 || M >= 6)) || (N == 256 && M == 8);
}
// resident CTAs the registers are held to: four keep the 516 CTAs of N = 256 in one wave
template <typename T> constexpr int dl_blocks(int M, int PM) { return sizeof(T) == 4 ? (M <= 5 && PM <= 16 ? 4 : 2) : 1; }
// filters whose operands a thread loads together (the registers of complex128 hold one, or two of one group)
template <typename T> constexpr int dl_unroll(int NG) { return sizeof(T) == 4 ? 4 : (NG == 1 ? 2 : 1); }
// entries of the triangle of W^H W that group 0 takes beside b (M products) and W^H b (M products)
constexpr int dl_first(int M, int NG) {
  const int e = M * (M + 1) / 2;
  return NG == 1 ? e : (e > 2 * M ? (e - 2 * M) / 2 : 0);
}
// elements of the region that holds the entries of group 1 and then the tile of w
template <int M, int NG> constexpr int dl_part() {
  constexpr int e = (M * (M + 1) / 2 - dl_first(M, NG)) * kDLBlock, t = 32 * (kDLBlock + 1);
  return e > t ? e : t;
}
// acc[j] = sum over 32 bins k of w[j WS + k] E[k ES]: pairs at distance 16 first, then 8, 4, 2, 1 (the
// order of a butterfly over a warp's lanes), the partial sums of the open levels held in registers
template <int ES, int WS, int NL, typename C>
__device__ __forceinline__ void dl_tree(const C* __restrict__ E, const C* __restrict__ w, C (&acc)[NL]) {
  C h4[NL], h2[NL], h1[NL];
#pragma unroll 1
  for (int t = 0; t < 8; ++t) {
    const int b = ((t & 1) << 2) | (t & 2) | (t >> 2);
    const C* e = E + b * ES;
    const C e0 = e[0], e1 = e[16 * ES], e2 = e[8 * ES], e3 = e[24 * ES];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      const C* v = w + j * WS + b;
      acc[j] = cadd(cadd(cmul(v[0], e0), cmul(v[16], e1)), cadd(cmul(v[8], e2), cmul(v[24], e3)));
    }
    auto level = [&](C (&h)[NL], bool open) {
#pragma unroll
      for (int j = 0; j < NL; ++j) {
        if (open) h[j] = acc[j];
        else acc[j] = cadd(h[j], acc[j]);
      }
    };
    level(h4, (t & 1) == 0);
    if (t & 1) level(h2, (t & 2) == 0);
    if ((t & 3) == 3) level(h1, (t & 4) == 0);
  }
}
template <typename T, int M, int PM, int NG>
__global__ void __launch_bounds__(NG * kDLBlock, dl_blocks<T>(M, PM)) dl_solve_kernel(const DLArgs<T> a) {
  using C = typename CT<T>::type;
  static_assert(kDLBlock == 64 && NG <= 2, "one or two groups of two warps");
  constexpr int NT = NG * kDLBlock;
  const int N = a.N, L = a.L, P = a.P;
  const int CP = col_pitch(N), H = N / 2 + 1;
  const int grp = threadIdx.x / kDLBlock, bt = threadIdx.x - grp * kDLBlock;
  const int tid = threadIdx.x;
  const int kb = blockIdx.x, nkb = gridDim.x;
  const int k1 = kb * kDLBlock + bt, k2 = blockIdx.y;
  const T n2 = (T)N * (T)N;
  const T sigma = a.sigma;
  extern __shared__ __align__(16) unsigned char dsm[];
  C* E = reinterpret_cast<C*>(dsm);                // [kDLBlock][PM]: exp(+2 pi i k1 (a - P/2) / N)
  C* part = E + kDLBlock * PM;                     // [entries of group 1][kDLBlock] of W^H W, then
  C* wt = part;                                    // [32][kDLBlock + 1]: w of this CTA's bins
  C* als = part + dl_part<M, NG>();                    // [M][kDLBlock]: alpha
  const C* zb = a.zcol + (size_t)k2 * M * L * CP + k1;  // z_{l,s} at zb[(s L + l) CP]
  const C* th = a.spec + (size_t)k2 * 2 * L * CP + k1;  // theta_l at th[l CP], F(g - e)_l at th[(L + l) CP]
  C x[M], c[M], G[M][M];
  for (int i = tid; i < kDLBlock * PM; i += NT) {
    const int ai = i % PM;
    E[i] = ai < P ? tw_at<+1>(a.tw, (kb * kDLBlock + i / PM) * (ai - P / 2), N) : mk<C>(0.0, 0.0);
  }
  grid_dep_wait();
  grid_dep_launch();
#pragma unroll
  for (int s = 0; s < M; ++s) {
    const C v = a.xcol[((size_t)k2 * M + s) * CP + k1];
    x[s] = mk<C>(v.x * n2, v.y * n2);
    c[s] = mk<C>(0.0, 0.0);
#pragma unroll
    for (int t = 0; t < M; ++t) G[s][t] = mk<C>(0.0, 0.0);
  }
  // group 0: b_l = sigma F(g - e)_l + sum_s conj(z_{l,s}) x_s, W^H b and the first E0 entries of the
  // triangle of W^H W; group 1: the others.  Each sum runs over all filters in order.
  constexpr int E0 = dl_first(M, NG);
  auto each = [&](auto f) {  // f(entry, s, t) over the triangle
#pragma unroll
    for (int s = 0; s < M; ++s)
#pragma unroll
      for (int t = 0; t <= s; ++t) f(s * (s + 1) / 2 + t, s, t);
  };
  auto load_z = [&](int l, C (&z)[M]) {
#pragma unroll
    for (int s = 0; s < M; ++s) {
      const C v = zb[((size_t)s * L + l) * CP];
      z[s] = mk<C>(v.x * n2, v.y * n2);
    }
  };
  if (NG == 1 || grp == 0) {
#pragma unroll 4
    for (int l = 0; l < L; ++l) {
      const C ge = th[(size_t)(L + l) * CP];
      C z[M], b = mk<C>(sigma * ge.x, sigma * ge.y);
      load_z(l, z);
#pragma unroll
      for (int s = 0; s < M; ++s) cfmac(b, z[s], x[s]);
#pragma unroll
      for (int s = 0; s < M; ++s) cfma(c[s], z[s], b);
      each([&](int e, int s, int t) {
        if (e < E0) cfmac(G[s][t], z[t], z[s]);  // z_s conj(z_t)
      });
    }
  } else {
#pragma unroll 4
    for (int l = 0; l < L; ++l) {
      C z[M];
      load_z(l, z);
      each([&](int e, int s, int t) {
        if (e >= E0) cfmac(G[s][t], z[t], z[s]);
      });
    }
  }
  if (NG > 1 && grp) {
    each([&](int e, int s, int t) {
      if (e >= E0) part[(e - E0) * kDLBlock + bt] = G[s][t];
    });
  }
  __syncthreads();
  C al[M];
  if (NG == 1 || grp == 0) {
    each([&](int e, int s, int t) {
      if (e >= E0) G[s][t] = part[(e - E0) * kDLBlock + bt];
    });
    // Cholesky of sigma I + G = R R^H (lower, in place), then R w = c and R^H alpha = w
#pragma unroll
    for (int j = 0; j < M; ++j) {
      T d = sigma + G[j][j].x;
#pragma unroll
      for (int k = 0; k < j; ++k) d -= G[j][k].x * G[j][k].x + G[j][k].y * G[j][k].y;
      const T r = sqrt(d > T(0) ? d : T(0)), inv = r > T(0) ? T(1) / r : T(0);
      G[j][j] = mk<C>(r, 0.0);
#pragma unroll
      for (int i = j + 1; i < M; ++i) {
        C acc = G[i][j];
#pragma unroll
        for (int k = 0; k < j; ++k) {  // acc -= G_ik conj(G_jk)
          const C u = G[i][k], v = G[j][k];
          acc.x -= u.x * v.x + u.y * v.y;
          acc.y -= u.y * v.x - u.x * v.y;
        }
        G[i][j] = mk<C>(acc.x * inv, acc.y * inv);
      }
    }
    C w[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
      C acc = c[i];
#pragma unroll
      for (int k = 0; k < i; ++k) {
        acc.x -= G[i][k].x * w[k].x - G[i][k].y * w[k].y;
        acc.y -= G[i][k].x * w[k].y + G[i][k].y * w[k].x;
      }
      const T inv = T(1) / G[i][i].x;
      w[i] = mk<C>(acc.x * inv, acc.y * inv);
    }
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
      C acc = w[i];
#pragma unroll
      for (int k = i + 1; k < M; ++k) {  // acc -= conj(G_ki) alpha_k
        acc.x -= G[k][i].x * al[k].x + G[k][i].y * al[k].y;
        acc.y -= G[k][i].x * al[k].y - G[k][i].y * al[k].x;
      }
      const T inv = T(1) / G[i][i].x;
      al[i] = mk<C>(acc.x * inv, acc.y * inv);
    }
#pragma unroll
    for (int s = 0; s < M; ++s) als[s * kDLBlock + bt] = al[s];
  }
  __syncthreads();  // part is free from here on (als is not part of it)
#pragma unroll
  for (int s = 0; s < M; ++s) al[s] = als[s * kDLBlock + bt];
  const T isg = T(1) / sigma;
  C* wb = a.wcol + (size_t)k2 * L * CP + k1;
  // the operands of U filters are loaded together
  constexpr int U = dl_unroll<T>(NG);
#pragma unroll 1
  for (int lb = grp; lb < L; lb += U * NG) {
    C z[U][M], ge[U], t[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int l = lb + u * NG;
      if (l < L) {
#pragma unroll
        for (int s = 0; s < M; ++s) z[u][s] = zb[((size_t)s * L + l) * CP];
        ge[u] = th[(size_t)(L + l) * CP];
        t[u] = th[(size_t)l * CP];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int l = lb + u * NG;
      if (l >= L) break;
      // b_l = sigma F(g - e)_l + sum_s conj(z_{l,s}) x_s, then d -= conj(z_s) alpha_s
      C d = mk<C>(sigma * ge[u].x, sigma * ge[u].y);
#pragma unroll
      for (int s = 0; s < M; ++s) {
        const C zs = mk<C>(z[u][s].x * n2, z[u][s].y * n2);
        cfmac(d, zs, x[s]);
        d.x -= zs.x * al[s].x + zs.y * al[s].y;
        d.y -= zs.x * al[s].y - zs.y * al[s].x;
      }
      // w = d-hat + e-hat, e-hat = theta - F(g - e)
      const C wl = mk<C>(fma(d.x, isg, t[u].x - ge[u].x), fma(d.y, isg, t[u].y - ge[u].y));
      wb[(size_t)l * CP] = wl;
      wt[l * (kDLBlock + 1) + bt] = wl;
    }
  }
  __syncthreads();
  // the support rows of the CTA's bins: thread = row a, filters l0, l0 + LSTEP, ...
  {
    constexpr int LSTEP = NT / PM;
    const int ai = tid % PM;
    C* yp = a.ypart + ((size_t)k2 * nkb + kb) * L * P;
    auto rows = [&](auto nl) {
      constexpr int NL = decltype(nl)::value;
#pragma unroll 1
      for (int l0 = tid / PM; l0 < L; l0 += NL * LSTEP) {
        const C* wr = wt + l0 * (kDLBlock + 1);
        C acc[2][NL];
        dl_tree<PM, LSTEP * (kDLBlock + 1)>(E + ai, wr, acc[0]);
        dl_tree<PM, LSTEP * (kDLBlock + 1)>(E + 32 * PM + ai, wr + 32, acc[1]);
#pragma unroll
        for (int j = 0; j < NL; ++j) {
          const int l = l0 + j * LSTEP;
          if (l < L && ai < P) yp[l * P + ai] = cadd(acc[0][j], acc[1][j]);
        }
      }
    };
    // as many at a time as few filters have (of the fixed four, L = 9 would compute 23 in vain); one in complex128,
    // where rows computed in vain cost FP64 issue and reading E again does not (256^2 x 1, 9 filters: 339 -> 293 us)
    if (sizeof(T) == 8 || L <= LSTEP) rows(std::integral_constant<int, 1>());
    else if (L <= 2 * LSTEP) rows(std::integral_constant<int, 2>());
    else rows(std::integral_constant<int, 4>());
  }
  __shared__ int last;
  __threadfence();  // this CTA's sums are visible device-wide before it is counted
  __syncthreads();
  if (tid == 0) last = atomicAdd(&a.cnt[k2], 1) == nkb - 1;
  __syncthreads();
  if (last) {
    __threadfence();
    const C* y0 = a.ypart + (size_t)k2 * nkb * L * P;
    for (int i = tid; i < L * P; i += NT) {
      C acc = mk<C>(0.0, 0.0);
      for (int b = 0; b < nkb; ++b) {
        const C v = __ldcg(y0 + (size_t)b * L * P + i);
        acc.x += v.x;
        acc.y += v.y;
      }
      const int l = i / P, ai = i - l * P;
      a.yfull[((size_t)l * P + ai) * H + k2] = acc;
    }
    if (tid == 0) a.cnt[k2] = 0;  // ready for the next step (stream order)
  }
}

// Per filter l = blockIdx.x: v = d + e at the P x P support points,
//   v(a, b) = N^-2 sum_k2 c_k2 Re[Y(a, k2) exp(2 pi i k2 (b - P/2) / N)]
// (c_k2 = 1 at k2 = 0 and N/2, 2 otherwise: the half spectrum of a real map); g = v / ||v||
// (Eq. g_admm: support and unit norm, reading R22); ||g - g_prev||^2 when a check follows; then the
// partial DFT G(a, k2) = sum_b g(a, b) exp(-2 pi i k2 (b - P/2) / N) for every k2.  Y of all
// support rows and the twiddles of every (k2, b) are staged in shared memory for `chunk` columns
// at a time (all H at once where they fit); kFiltSplit threads per output each take every
// kFiltSplit-th column, their partial sums added in a fixed order.
constexpr int kFiltThreads = 512, kFiltSplit = 4;
constexpr size_t kFiltSmem = 96 * 1024;
template <typename T> int filt_chunk(int N, int P) {
  const int H = N / 2 + 1;
  const int c = (int)(kFiltSmem / (2 * (size_t)P * sizeof(typename CT<T>::type)));
  return c < H ? c : H;
}
template <typename T>
__global__ void __launch_bounds__(kFiltThreads) dl_filter_kernel(const DLArgs<T> a, int chunk) {
  using C = typename CT<T>::type;
  const int N = a.N, L = a.L, P = a.P, H = N / 2 + 1, PP = P * P, cen = P / 2;
  const int l = blockIdx.x, tid = threadIdx.x;
  extern __shared__ __align__(16) unsigned char fsm[];
  C* ys = reinterpret_cast<C*>(fsm);  // [P][chunk]: Y(a, k2) of the chunk
  C* ws = ys + (size_t)P * chunk;       // [P][chunk]: exp(-2 pi i k2 (b - P/2) / N)
  __shared__ T vs[kDLMaxP * kDLMaxP];
  __shared__ T part[kFiltSplit][kFiltThreads / kFiltSplit];
  __shared__ T sinv;
  const T inv_n = T(1) / ((T)N * (T)N);
  const C* Y = a.yfull + (size_t)l * P * H;
  const int sub = tid % kFiltSplit, o0 = tid / kFiltSplit;
  constexpr int OSTEP = kFiltThreads / kFiltSplit;
  auto stage = [&](int c0, int nc, bool with_y, bool with_w) {
    __syncthreads();  // the previous chunk is consumed
    for (int i = tid; i < P * nc; i += kFiltThreads) {
      const int r = i / nc, c = i - r * nc;
      if (with_y) ys[(size_t)r * chunk + c] = Y[(size_t)r * H + c0 + c];
      if (with_w) ws[(size_t)r * chunk + c] = tw_at<-1>(a.tw, (c0 + c) * (r - cen), N);
    }
    __syncthreads();
  };
  if (chunk == H) stage(0, H, false, true);  // a single chunk's twiddles, while dl_solve finishes
  grid_dep_wait();
  grid_dep_launch();
  for (int ob = 0; ob < PP; ob += OSTEP) {  // outputs ob .. ob + OSTEP - 1 (one pass for P <= 11)
    const int o = ob + o0;
    const int ai = o < PP ? o / P : 0, bi = o < PP ? o - ai * P : 0;
    T acc = T(0);
    for (int c0 = 0; c0 < H; c0 += chunk) {
      const int nc = H - c0 < chunk ? H - c0 : chunk;
      if (ob == 0 || nc < H) stage(c0, nc, true, nc < H);  // a single chunk is staged once
      if (o < PP) {
        for (int c = sub; c < nc; c += kFiltSplit) {
          const C y = ys[(size_t)ai * chunk + c], t = ws[(size_t)bi * chunk + c];  // Re(y conj(t))
          const int k2 = c0 + c;
          const T w = (k2 == 0 || k2 == N / 2) ? T(1) : T(2);
          acc = fma(w, fma(y.x, t.x, y.y * t.y), acc);
        }
      }
    }
    if (o < PP) part[sub][o0] = acc;
    __syncthreads();
    if (sub == 0 && o < PP) {
      T v = part[0][o0];
#pragma unroll
      for (int i = 1; i < kFiltSplit; ++i) v += part[i][o0];
      vs[o] = v * inv_n;
    }
    __syncthreads();
  }
  // one warp takes the norm (and one lane its reciprocal): the FP64 units retire about two operations
  // per cycle and SM, so 512 threads summing in doubles cost more than the rest of the kernel
  T* g = a.gs + (size_t)l * PP;
  if (tid < 32) {
    double nn = 0.0;
    for (int o = tid; o < PP; o += 32) nn += (double)vs[o] * (double)vs[o];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
    if (tid == 0) sinv = nn > 0.0 ? (T)(1.0 / sqrt(nn)) : T(0);
  }
  __syncthreads();
  const T inv = sinv;
  if (a.check && tid < 32) {
    double ds = 0.0;
    for (int o = tid; o < PP; o += 32) {
      const double dg = (double)(T)(vs[o] * inv) - (double)g[o];
      ds += dg * dg;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ds += __shfl_xor_sync(0xffffffffu, ds, o);
    if (tid == 0) a.spart[l] = ds;
  }
  if (a.check) __syncthreads();  // g and vs are read above
  for (int o = tid; o < PP; o += kFiltThreads) {
    const T gn = vs[o] * inv;
    g[o] = gn;
    vs[o] = gn;
  }
  // G(a, k2) = sum_b g(a, b) ws[b][k2] over the same chunks (twiddles staged again when chunked)
  for (int c0 = 0; c0 < H; c0 += chunk) {
    const int nc = H - c0 < chunk ? H - c0 : chunk;
    if (nc < H) stage(c0, nc, false, true);
    else __syncthreads();  // vs is final
    for (int o = tid; o < P * nc; o += kFiltThreads) {
      const int ai = o / nc, c = o - ai * nc;
      C acc = mk<C>(0.0, 0.0);
      for (int bi = 0; bi < P; ++bi) {
        const T gv = vs[ai * P + bi];
        const C t = ws[(size_t)bi * chunk + c];
        acc.x = fma(gv, t.x, acc.x);
        acc.y = fma(gv, t.y, acc.y);
      }
      a.gfac[((size_t)(c0 + c) * L + l) * P + ai] = acc;
    }
  }
}

// Per frequency: g-hat_l = sum_a exp(-2 pi i k1 (a - P/2) / N) G_l(a, k2) = theta_l of the new
// filters; the dual update e-hat <- e-hat + d-hat - g-hat = w - g-hat (Eq. h_admm), stored as
// F(g - e) = 2 g-hat - w; p = sum_l theta_l z_l for the next x-update; and, before a check, the
// primal residual |F(d - g)|^2 = |w - e-hat_old - g-hat|^2 (Parseval on the half spectrum).
// The two groups divide the filters for g-hat, left in shared memory, and then the channels for p (each
// p still a sum over all filters in order): 31 -> 18 us at 256^2 x 5, L = 32.
template <typename T, int M, int PM, int NG>
__global__ void __launch_bounds__(NG * kDLBlock, dl_blocks<T>(M, PM)) dl_spec_kernel(const DLArgs<T> a) {
  constexpr int NT = NG * kDLBlock;
  using C = typename CT<T>::type;
  const int N = a.N, L = a.L, P = a.P, CP = col_pitch(N);
  const int tid = threadIdx.x, grp = tid / kDLBlock, bt = tid - grp * kDLBlock;
  const int k1 = blockIdx.x * kDLBlock + bt, k2 = blockIdx.y;
  extern __shared__ __align__(16) unsigned char dsm[];
  C* gk = reinterpret_cast<C*>(dsm);  // [32][PM]
  C* gs = gk + 32 * PM;               // [L][kDLBlock]: g-hat of this CTA's bins
  __shared__ double red[NT / 32];
  grid_dep_wait();
  grid_dep_launch();
  for (int i = tid; i < 32 * PM; i += NT) {
    const int l = i / PM, ai = i - l * PM;
    gk[i] = (l < L && ai < P) ? a.gfac[((size_t)k2 * L + l) * P + ai] : mk<C>(0.0, 0.0);
  }
  __syncthreads();
  const int cen = P / 2;
  C wa[PM];
#pragma unroll
  for (int i = 0; i < PM; ++i) wa[i] = i < P ? tw_at<-1>(a.tw, k1 * (i - cen), N) : mk<C>(0.0, 0.0);
  T r2 = T(0);
  C* th = a.spec + (size_t)k2 * 2 * L * CP + k1;
  const C* wb = a.wcol + (size_t)k2 * L * CP + k1;
  const C* zb = a.zcol + (size_t)k2 * M * L * CP + k1;
  constexpr int U = dl_unroll<T>(NG);
#pragma unroll 1
  for (int lb = grp; lb < L; lb += U * NG) {
    C wl[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (lb + u * NG < L) wl[u] = wb[(size_t)(lb + u * NG) * CP];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int l = lb + u * NG;
      if (l >= L) break;
      C gh = mk<C>(0.0, 0.0);
#pragma unroll
      for (int i = 0; i < PM; ++i) cfma(gh, wa[i], gk[l * PM + i]);
      const C w = wl[u];
      if (a.check) {
        const C t0 = th[(size_t)l * CP], ge0 = th[(size_t)(L + l) * CP];
        const T dx = w.x - t0.x + ge0.x - gh.x, dy = w.y - t0.y + ge0.y - gh.y;
        r2 = fma(dx, dx, fma(dy, dy, r2));
      }
      gs[l * kDLBlock + bt] = gh;
      th[(size_t)l * CP] = gh;
      th[(size_t)(L + l) * CP] = mk<C>(T(2) * gh.x - w.x, T(2) * gh.y - w.y);
    }
  }
  if (a.check) {
    const double wgt = (k2 == 0 || k2 == N / 2) ? 1.0 : 2.0;
    double v = wgt * (double)r2;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((tid & 31) == 0) red[tid >> 5] = v;
  }
  __syncthreads();
  // p of channels grp, grp + NG, ...: each sum runs over all filters in order
  constexpr int MG = (M + NG - 1) / NG;
  C pm[MG];
#pragma unroll
  for (int m = 0; m < MG; ++m) pm[m] = mk<C>(0.0, 0.0);
#pragma unroll 8
  for (int l = 0; l < L; ++l) {
    const C gh = gs[l * kDLBlock + bt];
#pragma unroll
    for (int m = 0; m < MG; ++m)
      if (grp + m * NG < M) cfma(pm[m], gh, zb[((size_t)(grp + m * NG) * L + l) * CP]);
  }
#pragma unroll
  for (int m = 0; m < MG; ++m)
    if (grp + m * NG < M) a.p_out[((size_t)k2 * M + grp + m * NG) * CP + k1] = pm[m];
  if (a.check && tid == 0) {
    double v = 0.0;
    for (int w = 0; w < NT / 32; ++w) v += red[w];
    a.rpart[(size_t)k2 * gridDim.x + blockIdx.x] = v;
  }
}

template <typename T>
__global__ void dl_rescale_kernel(typename CT<T>::type* __restrict__ spec, int L, int N, T f) {
  using C = typename CT<T>::type;
  const int CP = col_pitch(N), H = N / 2 + 1;
  const size_t total = (size_t)H * L * N;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const int k1 = (int)(i % N);
    const size_t r = i / N;
    const int l = (int)(r % L);
    const size_t k2 = r / L;
    C* th = spec + (k2 * 2 * L + l) * CP + k1;
    const C t = th[0], ge = th[(size_t)L * CP];
    th[(size_t)L * CP] = mk<C>(t.x - (t.x - ge.x) * f, t.y - (t.y - ge.y) * f);
  }
}

template <typename T, int M, int PM, int NG> cudaError_t dl_launch(const DLArgs<T>& a, bool spec, Chain s) {
  using C = typename CT<T>::type;
  const dim3 grid(a.N / kDLBlock, a.N / 2 + 1), block(NG * kDLBlock);
  constexpr size_t sm = (size_t)(kDLBlock * (PM + M) + dl_part<M, NG>()) * sizeof(C);
  constexpr size_t spec_max = (size_t)32 * (PM + kDLBlock) * sizeof(C);
  static PerDeviceOnce once;
  cudaError_t e = once([&] {
    cudaError_t r = cudaFuncSetAttribute(dl_solve_kernel<T, M, PM, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (r != cudaSuccess) return r;
    return cudaFuncSetAttribute(dl_spec_kernel<T, M, PM, NG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)spec_max);
  });
  if (e != cudaSuccess) return e;
  if (spec) return launch_pdl(dl_spec_kernel<T, M, PM, NG>, grid, block, (size_t)(32 * PM + a.L * kDLBlock) * sizeof(C), s, 0, a);
  return launch_pdl(dl_solve_kernel<T, M, PM, NG>, grid, block, sm, s, 0, a);
}
template <typename T, int PM> cudaError_t dl_by_m(const DLArgs<T>& a, bool spec, Chain s) {
  switch (a.M) {
#define DL_CASE(m) \
  case m:                                                                                               \
    if constexpr (dl_one_group<T>(256, m) || dl_one_group<T>(2048, m))                                   \
      if (dl_one_group<T>(a.N, m)) return dl_launch<T, m, PM, 1>(a, spec, s);                            \
    return dl_launch<T, m, PM, 2>(a, spec, s);
    DL_CASE(1) DL_CASE(2) DL_CASE(3) DL_CASE(4) DL_CASE(5) DL_CASE(6) DL_CASE(7) DL_CASE(8)
#undef DL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template <typename T> bool dl_args_ok(const DLArgs<T>& a) {
  return a.N % kDLBlock == 0 && a.N <= kTwN && a.L >= 1 && a.L <= 32 && a.P >= 1 && a.P <= kDLMaxP &&
         a.P <= a.N && a.M >= 1 && a.M <= 8;
}

}  // namespace

template <typename T> cudaError_t launch_dl_solve(const DLArgs<T>& a, Chain s) {
  if (!dl_args_ok(a)) return cudaErrorInvalidValue;
  return a.P <= 16 ? dl_by_m<T, 16>(a, false, s) : dl_by_m<T, 32>(a, false, s);
}
template <typename T> cudaError_t launch_dl_filter(const DLArgs<T>& a, Chain s) {
  if (!dl_args_ok(a)) return cudaErrorInvalidValue;
  const int chunk = filt_chunk<T>(a.N, a.P);
  const size_t sm = 2 * (size_t)a.P * chunk * sizeof(typename CT<T>::type);
  static PerDeviceOnce once;
  cudaError_t e = once([&] {
    return cudaFuncSetAttribute(dl_filter_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFiltSmem);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(dl_filter_kernel<T>, dim3(a.L), dim3(kFiltThreads), sm, s, 0, a, chunk);
}
template <typename T> cudaError_t launch_dl_spec(const DLArgs<T>& a, Chain s) {
  if (!dl_args_ok(a)) return cudaErrorInvalidValue;
  return a.P <= 16 ? dl_by_m<T, 16>(a, true, s) : dl_by_m<T, 32>(a, true, s);
}
template <typename T>
cudaError_t launch_dl_rescale(typename CT<T>::type* spec, int L, int N, T f, cudaStream_t s) {
  dl_rescale_kernel<T><<<4 * 152, 256, 0, s>>>(spec, L, N, f);
  return cudaGetLastError();
}
template cudaError_t launch_dl_solve<float>(const DLArgs<float>&, Chain);
template cudaError_t launch_dl_solve<double>(const DLArgs<double>&, Chain);
template cudaError_t launch_dl_filter<float>(const DLArgs<float>&, Chain);
template cudaError_t launch_dl_filter<double>(const DLArgs<double>&, Chain);
template cudaError_t launch_dl_spec<float>(const DLArgs<float>&, Chain);
template cudaError_t launch_dl_spec<double>(const DLArgs<double>&, Chain);
template cudaError_t launch_dl_rescale<float>(float2*, int, int, float, cudaStream_t);
template cudaError_t launch_dl_rescale<double>(double2*, int, int, double, cudaStream_t);

template <typename T>
cudaError_t launch_p_from_z(const typename CT<T>::type* zcol, const typename CT<T>::type* th,
                            typename CT<T>::type* p, int N, int M, int L, cudaStream_t s, double scale,
                            int th_planes) {
  dim3 grid((N + 127) / 128, N / 2 + 1, M);
  const T sc = scale > 0 ? (T)scale : T(1) / ((T)N * (T)N);
  p_from_z_kernel<T><<<grid, 128, 0, s>>>(zcol, th, p, N, M, L, th_planes > 0 ? th_planes : L, sc);
  return cudaGetLastError();
}
template cudaError_t launch_p_from_z<float>(const float2*, const float2*, float2*, int, int, int, cudaStream_t,
                                            double, int);
template cudaError_t launch_p_from_z<double>(const double2*, const double2*, double2*, int, int, int, cudaStream_t,
                                             double, int);

template <typename T> cudaError_t launch_cd_solve(const CDArgs<T>& a, cudaStream_t s) {
  dim3 grid((a.N + 127) / 128, a.N / 2 + 1, a.M);
  if (a.L > 32) return cudaErrorInvalidValue;
  if (a.M <= 4) {
    if (a.L <= 8) cd_solve_kernel<T, 4, 8><<<grid, 128, 0, s>>>(a);
    else cd_solve_kernel<T, 4, 32><<<grid, 128, 0, s>>>(a);
  } else if (a.M <= 16) {
    if (a.L <= 8) cd_solve_kernel<T, 16, 8><<<grid, 128, 0, s>>>(a);
    else cd_solve_kernel<T, 16, 32><<<grid, 128, 0, s>>>(a);
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

// Where it runs.  Fewer filters than FFT teams leave warps of a CTA idle for two whole FFTs, which costs most
// where a team's FFT is longest: complex64 at N = 1024 runs it from 8 filters (a team each) on; one channel,
// 7 filters 62.9 us against 49.1 in three kernels, 8 filters 47.1 against 56.2, three channels 1 filter
// 83.0 and 51.3, eight 209 and 189, but for 16 channels, where an iteration takes 629 and 670 us (below N = 1024
// it is the faster one from one filter on: 512^2 x 8 41.7 and 47.5).
// complex128 CTAs hold an SM each (registers), so that beyond one wave they queue while each waits for
// its few FP64 units: 256^2 x 8 with 1 filter 236 us against 138, 9 filters 433 and 373, 512^2 x 3 9 filters 787
// and 561; in one wave 256^2 x 1 9 filters 62.6 and 82.5; two waves with little work each 512^2 x 1 2 filters
// 87.7 and 94.2, 4 filters 108.7 and 100.5.  Up to N = 128 it is the faster one but for 12 and more filters in
// some waves (128^2 x 3: 1 filter 22.8 and 42.1, 32 filters 160 and 136).
template <typename T> bool cd_fused_fits(int N, int M, int L) {
  if (fuse_smem<T>(N, L) == 0) return false;
  if (sizeof(T) == 4) return N < 1024 || L >= kFuseThreads / (N / fuse_elems<T>(N)) || M >= 12;
  const int ctas = M * (N / 2 + 1), sms = 152;
  return N <= 128 || ctas <= sms || (ctas <= 2 * sms && L <= 3);
}
template <typename T> cudaError_t launch_cd_fused(const CDArgs<T>& a, Chain s) {
  if (a.L < 1 || a.L > 32 || !cd_fused_fits<T>(a.N, a.M, a.L)) return cudaErrorInvalidValue;
  switch (a.N) {
    case 64: return launch_fused<T, 6>(a, s);
    case 128: return launch_fused<T, 7>(a, s);
    case 256: return launch_fused<T, 8>(a, s);
    case 512: return launch_fused<T, 9>(a, s);
    case 1024: return launch_fused<T, 10>(a, s);
    default: return cudaErrorInvalidValue;
  }
}
template bool cd_fused_fits<float>(int, int, int);
template bool cd_fused_fits<double>(int, int, int);
template cudaError_t launch_cd_fused<float>(const CDArgs<float>&, Chain);
template cudaError_t launch_cd_fused<double>(const CDArgs<double>&, Chain);

template <typename Tin>
cudaError_t launch_embed_filters(const Tin* d, double* out, int L, int P, int N, cudaStream_t s) {
  const int n = L * P * P;
  embed_kernel<Tin><<<(n + 255) / 256, 256, 0, s>>>(d, out, L, P, N);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_theta_store(const SetupC<T>* th64, typename CT<T>::type* th, int L, int N, cudaStream_t s) {
  theta_store_kernel<T><<<512, 256, 0, s>>>(th64, th, L, N);
  return cudaGetLastError();
}

template cudaError_t launch_cd_solve<float>(const CDArgs<float>&, cudaStream_t);
template cudaError_t launch_cd_solve<double>(const CDArgs<double>&, cudaStream_t);
template cudaError_t launch_embed_filters<float>(const float*, double*, int, int, int, cudaStream_t);
template cudaError_t launch_embed_filters<double>(const double*, double*, int, int, int, cudaStream_t);
template cudaError_t launch_theta_store<float>(const cdf*, float2*, int, int, cudaStream_t);
template cudaError_t launch_theta_store<double>(const double2*, double2*, int, int, cudaStream_t);

}  // namespace cip
