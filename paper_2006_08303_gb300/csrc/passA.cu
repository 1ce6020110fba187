// Pass A: the fused prior pass of one ADMM iteration (Alg. 1 lines 5-6 and
// the T^H (t - u) term of the next x-update, Eq. solx_Trans_DFT).
//
// One CTA owns R consecutive image rows of one channel (plus one halo row on
// each side for TV).  It
//   1. loads the row half-spectra of x (written by pass B) and inverts the row
//      DFT two rows at a time (one complex FFT z = x_a + i x_b for two real
//      rows, so shared memory holds the tile as row pairs);
//   2. applies the analysis operator T (TV differences or the 8x8 orthonormal
//      block DCT; T = I is rowpass.cu), the soft-threshold t-update
//      (Eq. solt_trans) and the dual update (Eq. subu_trans), writing u; every
//      thread works on both rows of a pair, so shared-memory accesses are
//      whole 8- or 16-byte pairs;
//   3. forms q = (rho/2) T^T (t - u) and takes its forward row DFT, writing
//      the row half-spectra that pass B turns into the full 2D DFT.
// Optionally it stores t (for the next iteration's dual residual) and writes
// per-CTA partial sums of the residual norms (Eq. paramS quantities).
#include <type_traits>

#include "fft.cuh"
#include "kernels.h"
#include "reduce.cuh"

namespace cip {

namespace {

#ifndef PASSA_RT32
#define PASSA_RT32 48
#endif
#ifndef PASSA_TV_RT32
#define PASSA_TV_RT32 64
#endif

// FFT elements per thread: 8 for complex64 up to N = 1024 (more warps per
// tile), 16 otherwise (keeps the CTA within 1024 threads).
// (complex64 DCT tiles at N = 512 take 16: one warp per row-pair FFT, whose stage
// barriers are then warp syncs, while TV, which needs more registers for its halo rows,
// takes 8.)  Variant V = 1 of a complex64 iteration kernel at N = 256 .. 1024 takes the other
// of 8 and 16; the plan's autotuner times both inside whole iterations and keeps the faster.
template <typename T> constexpr int elems_a(int N, int prior, int V = 0) {
  const int e = (sizeof(T) == 4 && N <= 1024) ? ((N == 512 && !prior_is_tv(prior)) ? 16 : 8) : 16;
  return V == 1 ? 24 - e : e;
}
template <typename T> constexpr bool has_variant(int N, int prior) {
  return sizeof(T) == 4 && N >= 256 && N <= 1024 && (prior_is_tv(prior) || prior == PRIOR_DCT8);
}

// Pitch of the row-pair FFT buffers (complex elements): the padded FFT layout plus 4 slots from
// N = 256 on, so that the 4 or 5 buffers a warp writes at once (pair p, consecutive columns k,
// when the column-layout spectra are gathered or scattered) start in different bank groups.
constexpr int zs_of(int N) { return spad(N) + (N >= 256 ? 4 : 0); }

// rows per tile
template <typename T> constexpr int rows_for(int N, int prior) { return 8; }

// TV work split of the shrinkage phase.  A thread works on two adjacent columns and walks down
// rows, keeping the row above in registers, so the tile needs no shared-memory copy of the
// components of t - u: the phase costs 3 shared-memory loads per row pair and column pair, and the
// CTA's shared memory is the FFT buffers alone.  a_h of the column to the left comes from the next
// lane down; the values that cross a warp's 64 columns are formed once, ahead of the walk.
//   N <= 512: row groups of tv_rows() rows side by side, one column pair per thread; q stays in
//     registers until every thread has read the x tile (it is written in place).  A group recomputes
//     a_v of the row above it, so groups are as tall as they can be with most threads busy.
//   N >= 1024: every thread walks down all rows of its column pairs; q of a row pair is written over
//     the x rows that no later row needs, one barrier per row pair.
// Bound by the latency of its phases (long-scoreboard and barrier stalls; FFT shared-memory traffic
// 45-50% of the LSU pipe).  The prior pass alone, before (components of t - u in shared memory, 2 to
// 8-row tiles, u read where it is used) and now: 64^2 x 3 10.3 -> 8.0 us, 256^2 x 3 14.3 -> 9.8,
// 512^2 x 5 22.1 -> 17.5, 512^2 x 10 37.3 -> 26.5, 1024^2 x 10 125 -> 99, 2048^2 x 3 286 -> 168 us;
// isotropic 512^2 x 10 39.2 -> 30.2, 2048^2 x 3 302 -> 191 us.
constexpr int tv_rows(int N) { return N >= 512 ? 8 : (N >= 256 ? 4 : 2); }

// DCT tiles stage their R rows of u in shared memory with one TMA bulk
// copy issued before the grid dependency (u does not depend on the preceding
// column pass), when the staging area keeps the CTA within ~100 KB
template <typename T> constexpr bool u_staged(int N, int prior, int R) {
  using C = typename CT<T>::type;
  return !prior_is_tv(prior) &&
         (size_t)(R / 2) * zs_of(N) * sizeof(C) + (size_t)R * N * sizeof(T) <= 100 * 1024;
}

// TV tiles up to N = 512 stage theirs too: R + 1 rows (the row above included) of both components,
// so that the u reads, which every thread needs in one burst, cost no global latency after the FFTs
template <typename T> constexpr bool tv_staged(int N, int prior) {
  return sizeof(T) == 4 && prior_is_tv(prior) && N <= 512;
}

template <typename T> constexpr size_t smem_for(int N, int prior, int R) {
  using C = typename CT<T>::type;
  const int halo = prior_is_tv(prior) ? 1 : 0;
  size_t sm = (size_t)((R + 2 * halo) / 2) * zs_of(N) * sizeof(C);
  if (u_staged<T>(N, prior, R)) sm += (size_t)R * N * sizeof(T);
  if (tv_staged<T>(N, prior)) sm += 2 * (size_t)(R + 1) * N * sizeof(T);
  return sm;
}

// The TV CTAs of small images get threads beyond the FFT teams for the other phases (a row group's
// threads are then whole warps).
template <typename T> constexpr int threads_for(int N, int prior, int R, int V = 0) {
  const int npin = (R + (prior_is_tv(prior) ? 2 : 0)) / 2;
  const int n = ((npin * (N / elems_a<T>(N, prior, V)) + 31) / 32) * 32;
  return prior_is_tv(prior) && n < 256 ? 256 : n;
}

// CTAs per SM the register budget is cut for: as many as shared memory and the
// thread limit allow, at <= ~48 registers per thread for complex64 (so that a
// 10-channel 512 x 512 prior pass runs as one wave) and <= ~168 for complex128
// (whose 16-element FFT registers would otherwise spill).  The 256 threads of a complex128 TV tile
// take <= 128 from N = 128 on, two CTAs instead of one: 0 to 276 bytes of spills, but 128^2 x 8 74.5 -> 57.1 us an
// iteration, 256^2 x 8 178 -> 160, 512^2 x 8 472 -> 447 (at N = 64, 192 bytes, 70.2 -> 73.7 for 16 channels).
template <typename T> constexpr int minblocks_for(int nth, size_t smem, bool tv, int N) {
  const int by_regs =
      65536 / (nth * (sizeof(T) == 4 ? (tv ? PASSA_TV_RT32 : PASSA_RT32) : (tv && N >= 128 ? 128 : 168)));
  const int by_smem = (int)((227 * 1024) / (smem + 1024));
  const int by_thr = 2048 / nth;
  int b = by_regs < by_smem ? by_regs : by_smem;
  b = b < by_thr ? b : by_thr;
  b = b < 16 ? b : 16;  // small tiles (N <= 128): no point in squeezing registers further
  return b < 1 ? 1 : b;
}

// 8-point orthonormal DCT-II and its inverse through the even/odd split of
// the basis (row k of the matrix d[k*8+n] is symmetric in n <-> 7-n for even
// k and antisymmetric for odd k; rows 0, 4 are also symmetric and rows 2, 6
// antisymmetric in n <-> 3-n): 36 operations per transform instead of 64.
template <typename T>
__device__ __forceinline__ void dct8_fwd(const T* __restrict__ d, const T (&x)[8], T (&X)[8]) {
  T s[4], df[4];
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    s[n] = x[n] + x[7 - n];
    df[n] = x[n] - x[7 - n];
  }
  const T s03 = s[0] + s[3], s12 = s[1] + s[2], e0 = s[0] - s[3], e1 = s[1] - s[2];
  X[0] = d[0] * (s03 + s12);
  X[4] = d[32] * (s03 - s12);
  X[2] = fma(d[16], e0, d[17] * e1);
  X[6] = fma(d[48], e0, d[49] * e1);
#pragma unroll
  for (int k = 1; k < 8; k += 2) {
    T acc = d[k * 8] * df[0];
#pragma unroll
    for (int n = 1; n < 4; ++n) acc = fma(d[k * 8 + n], df[n], acc);
    X[k] = acc;
  }
}

template <typename T>
__device__ __forceinline__ void dct8_inv(const T* __restrict__ d, const T (&X)[8], T (&x)[8]) {
  const T a = d[0] * X[0], b = d[32] * X[4];
  const T A = a + b, B = a - b;
  const T C0 = fma(d[16], X[2], d[48] * X[6]), C1 = fma(d[17], X[2], d[49] * X[6]);
  const T e[4] = {A + C0, B + C1, B - C1, A - C0};
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    T o = d[8 + n] * X[1];
    o = fma(d[24 + n], X[3], o);
    o = fma(d[40 + n], X[5], o);
    o = fma(d[56 + n], X[7], o);
    x[n] = e[n] + o;
    x[7 - n] = e[n] - o;
  }
}

// the same on the two rows of a pair (real and imaginary parts)
template <typename T, bool FWD, typename C>
__device__ __forceinline__ void dct8_pair(const T* __restrict__ d, const C (&in)[8], C (&out)[8]) {
  T a[8], b[8], ra[8], rb[8];
#pragma unroll
  for (int n = 0; n < 8; ++n) {
    a[n] = in[n].x;
    b[n] = in[n].y;
  }
  if (FWD) {
    dct8_fwd(d, a, ra);
    dct8_fwd(d, b, rb);
  } else {
    dct8_inv(d, a, ra);
    dct8_inv(d, b, rb);
  }
#pragma unroll
  for (int n = 0; n < 8; ++n) out[n] = mk<C>(ra[n], rb[n]);
}

template <typename T>
__device__ __forceinline__ void shrink(T w, T u, T tau, T& t, T& un) {
  t = soft(w + u, tau);
  un = u + w - t;
}

// sums of 16 values per lane over the warp by recursive halving: at xor distance 16, 8, 4, 2 a lane
// keeps one half of its values (the upper half when that bit of the lane is set) and adds its
// partner's; then v[0] of lane l is the warp's sum of value l >> 1
template <typename T> __device__ __forceinline__ void reduce_scatter16(T* v, int lane) {
#pragma unroll
  for (int live = 16, o = 16; live > 1; live /= 2, o /= 2) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < live / 2; ++i) {
      const T keep = up ? v[i + live / 2] : v[i], send = up ? v[i] : v[i + live / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// products and differences that the compiler must not contract: the isotropic shrinkage spells its
// roundings out, so that every place that forms a pixel's components gets the same bits
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }

template <typename T, int LOGN, int PRIOR, int R, int V>
__global__ void __launch_bounds__(threads_for<T>(1 << LOGN, PRIOR, R, V),
                                  minblocks_for<T>(threads_for<T>(1 << LOGN, PRIOR, R, V),
                                                   smem_for<T>(1 << LOGN, PRIOR, R), prior_is_tv(PRIOR), 1 << LOGN))
    passA_kernel(const PassAArgs<T> a) {
  using C = typename CT<T>::type;
  constexpr int N = 1 << LOGN;
  constexpr int H = N / 2 + 1;
  constexpr int HALO = prior_is_tv(PRIOR) ? 1 : 0;
  constexpr int ROWS = R + 2 * HALO;
  constexpr int NPIN = ROWS / 2;
  constexpr int NPOUT = R / 2;
  constexpr int ZS = zs_of(N);
  constexpr int CP = col_pitch(N);
  constexpr int E = elems_a<T>(N, PRIOR, V);
  constexpr int TEAM = N / E;
  constexpr int NCOMP = prior_is_tv(PRIOR) ? 2 : 1;
  constexpr int NT = threads_for<T>(N, PRIOR, R, V);
  static_assert(kLowK == 2, "the TV walk forms k2 = 0 and 1");
  __shared__ T edge[R][prior_is_tv(PRIOR) ? N / 64 : 1];
  __shared__ T lows[2][prior_is_tv(PRIOR) && LOGN == 11 ? NT / 32 : 1][12];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* zb = reinterpret_cast<C*>(smem_raw);
  constexpr bool USTAGE = u_staged<T>(N, PRIOR, R);
  static_assert(!USTAGE || (NPIN * ZS * sizeof(C)) % 16 == 0, "the TMA destination must be 16-byte aligned");
  constexpr bool TVSTAGE = tv_staged<T>(N, PRIOR);
  static_assert(!TVSTAGE || (NPIN * ZS * sizeof(C)) % 16 == 0, "the TMA destination must be 16-byte aligned");
  // USTAGE (DCT): [R][N] rows r0 .. of u_in; TVSTAGE: [2][R + 1][N] rows r0 - 1 .. of both components
  T* us = reinterpret_cast<T*>(zb + NPIN * ZS);
  __shared__ unsigned long long ubar;

  const int tid = threadIdx.x;
  const int nth = blockDim.x;
  const int m = blockIdx.y;
  const int r0 = blockIdx.x * R;
  const bool import_mode = (a.flags & PA_IMPORT) != 0;
  const bool resid = (a.flags & PA_RESID) != 0;
  const bool store_t = (a.flags & PA_STORE_T) != 0;
  const T tau = a.tau;
  const size_t plane = (size_t)N * N;
  const T* u_in = a.u_in ? a.u_in + (size_t)m * NCOMP * plane : nullptr;
  T* u_out = a.u_out ? a.u_out + (size_t)m * NCOMP * plane : nullptr;
  T* tprev = a.tprev ? a.tprev + (size_t)m * NCOMP * plane : nullptr;
  const T* timp = a.t_imp ? a.t_imp + (size_t)m * NCOMP * plane : nullptr;
  const T* tprev_rd = resid ? tprev : nullptr;
  T part[kNPart] = {T(0), T(0), T(0), T(0), T(0)};
  // false when this thread's bounded wait for the staged u rows gave up: it then reads u from
  // global memory (the same values), never the shared-memory rows the copy may not have written
  bool u_ok = true;

  auto grow = [&](int j) { return (r0 - HALO + j) & (N - 1); };

  auto stage_tv = [&]() {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      T* dst = us + c * (R + 1) * N;
      bulk_copy_g2s(dst, u_in + c * plane + (size_t)grow(0) * N, (unsigned)(N * sizeof(T)), &ubar);
      bulk_copy_g2s(dst + N, u_in + c * plane + (size_t)r0 * N, (unsigned)(R * N * sizeof(T)), &ubar);
    }
  };
  if constexpr (USTAGE) {
    // u rows r0 .. r0+R-1 of this channel: one contiguous block (16-byte aligned: r0 is a
    // multiple of 8 and N >= 64), fetched by the TMA unit while the previous kernel drains
    if (tid == 0) {
      constexpr unsigned bytes = (unsigned)(R * N * sizeof(T));
      if (a.test_fault == 1) {
        // test of the bounded wait: two arrivals expected, one given, no copy issued, so the
        // phase never completes and nothing is in flight when the wait gives up
        mbar_init(&ubar, 2);
        mbar_arrive(&ubar);
      } else {
        mbar_init(&ubar, 1);
        mbar_arrive_expect_tx(&ubar, bytes);
        if (!import_mode) bulk_copy_g2s(us, u_in + (size_t)r0 * N, bytes, &ubar);
      }
    }
    __syncthreads();  // the barrier is initialised before anyone waits on it
  }
  if constexpr (TVSTAGE) {
    // per component the row above the tile (wraps to the last row) and the tile's R rows
    if (tid == 0) {
      if (a.test_fault == 1) {  // as for the DCT tile above
        mbar_init(&ubar, 2);
        mbar_arrive(&ubar);
      } else {
        mbar_init(&ubar, 1);
        mbar_arrive_expect_tx(&ubar, (unsigned)(2 * (R + 1) * N * sizeof(T)));
        if (!import_mode) stage_tv();
      }
    }
    __syncthreads();  // the barrier is initialised before anyone waits on it
  }
  // L2 prefetch of the u rows (and t_prev rows) read after the inverse FFT
  if (tid < 2 * NCOMP && !((USTAGE || TVSTAGE) && (tid & 1) == 0)) {
    const T* src = (tid & 1) ? tprev_rd : u_in;
    if (src) {
      const size_t comp = (size_t)(tid >> 1) * plane;
      prefetch_l2(src + comp + (size_t)r0 * N, (size_t)R * N * sizeof(T));
      if (HALO) prefetch_l2(src + comp + (size_t)grow(0) * N, (size_t)N * sizeof(T));
    }
  }

  grid_dep_wait();  // x (and u, t) of the previous kernels are complete from here on
  grid_dep_launch();
  // an import follows whatever wrote u (a copy or the rescaling of u), so its rows are fetched only now
  if (import_mode && tid == 0) {
    if constexpr (USTAGE) {
      if (a.test_fault != 1) bulk_copy_g2s(us, u_in + (size_t)r0 * N, (unsigned)(R * N * sizeof(T)), &ubar);
    }
    if constexpr (TVSTAGE) {
      if (a.test_fault != 1) stage_tv();
    }
  }
  if (!import_mode) {
    // 1. gather the row half-spectra of the tile (two rows per complex FFT) from the column
    //    layout and invert the row DFT; thread = (pair p, column k) with p fastest, so that a warp
    //    reads the contiguous row segments of a few columns
    const C* xh = a.xh + (size_t)m * CP;
    const size_t kstride = (size_t)a.M * CP;
    // (kGather loads in flight per thread before the first use)
    constexpr int ITEMS = NPIN * H, kGather = sizeof(T) == 4 ? 4 : 2;
    for (int base = tid; base < ITEMS; base += kGather * NT) {
      C xa[kGather], xb[kGather];
#pragma unroll
      for (int i = 0; i < kGather; ++i) {
        const int idx = base + i * NT;
        if (idx >= ITEMS) continue;
        const int p = idx % NPIN, k = idx / NPIN;
        const C* col = xh + (size_t)k * kstride;
        if constexpr (sizeof(C) == 8 && !HALO) {
          // rows r0 + 2p, r0 + 2p + 1: adjacent, 16-byte aligned (r0 even, CP even)
          const float4 v = *reinterpret_cast<const float4*>(col + r0 + 2 * p);
          xa[i] = mk<C>(v.x, v.y);
          xb[i] = mk<C>(v.z, v.w);
        } else {
          xa[i] = col[grow(2 * p)];
          xb[i] = col[grow(2 * p + 1)];
        }
      }
#pragma unroll
      for (int i = 0; i < kGather; ++i) {
        const int idx = base + i * NT;
        if (idx >= ITEMS) continue;
        const int p = idx % NPIN, k = idx / NPIN;
        pair_spectrum_put(zb + p * ZS, N, k, xa[i], xb[i]);
      }
    }
    __syncthreads();
    {
      const int team = tid / TEAM;
      const TeamSync ts = make_team_sync(team, TEAM);
      if (ts.cta || team < NPIN)
        fft_team<C, LOGN, 1, E, +1>(zb + (team < NPIN ? team : 0) * ZS, tid % TEAM, a.tw, ts, team < NPIN);
    }
    __syncthreads();
  }
  // 2. analysis operator, shrinkage, dual update; 3. q = qscale T^T (t - u')
  if constexpr (prior_is_tv(PRIOR)) {
    constexpr bool WALK = N >= 1024, LOW = LOGN == 11;
    // MODE 0: plain; 1: with residual sums and / or t stored; 2: import (t given, x unused)
    // u of component `comp` at tile row j, columns c0, c0 + 1
    auto ldu = [&](int comp, int j, int c0) -> C {
      if constexpr (TVSTAGE) return *reinterpret_cast<const C*>(us + (comp * (R + 1) + j) * N + c0);
      else return __ldg(reinterpret_cast<const C*>(u_in + comp * plane + (size_t)grow(j) * N + c0));
    };
    auto ldu1 = [&](int comp, int j, int c) -> T {
      if constexpr (TVSTAGE) return us[(comp * (R + 1) + j) * N + c];
      else return __ldg(u_in + comp * plane + (size_t)grow(j) * N + c);
    };
    constexpr bool ISO = PRIOR == PRIOR_TV_ISO;
    const C czero = mk<C>(0.0, 0.0);
    if constexpr (TVSTAGE) {
      // a warp whose wait gave up (the plan is flagged) copies the rows itself: whoever else writes them,
      // a late bulk copy included, writes the same values
      u_ok = mbar_wait_bounded(&ubar, 0, a.err, a.test_fault ? 64 : (1 << 22));
      if (__any_sync(0xffffffffu, !u_ok)) {
        for (int i = tid & 31; i < 2 * (R + 1) * N; i += 32) {
          const int comp = i / ((R + 1) * N), r = i - comp * (R + 1) * N;
          us[i] = u_in[comp * plane + (size_t)grow(r / N) * N + (r & (N - 1))];
        }
        __syncwarp();
      }
    }
    // isotropic TV: the pixel's two components shrink together (group soft threshold)
    auto group = [&](T wh, T uh, T wv, T uv, T& th, T& uhn, T& ah, T& tv, T& uvn, T& av) {
      const T vh = wh + uh, vv = wv + uv;
      const T nrm = sqrt(fma(vh, vh, mul_rn(vv, vv)));
      const T f = nrm > tau ? T(1) - tau / nrm : T(0);
      th = mul_rn(vh, f);
      tv = mul_rn(vv, f);
      uhn = sub_rn(vh, th);
      uvn = sub_rn(vv, tv);
      ah = sub_rn(th, uhn);
      av = sub_rn(tv, uvn);
    };
    // a_h of the output rows at the columns 64 b - 1, one thread each: what lane 0 of the warp that
    // works on the columns 64 b .. 64 b + 63 needs
    auto edges = [&](auto mode) {
      constexpr int MODE = decltype(mode)::value, NB = N / 64;
      if (tid < R * NB) {
        const int j = 1 + tid / NB, b = tid & (NB - 1), c = (64 * b - 1) & (N - 1), cr = 64 * b;
        const size_t g = (size_t)grow(j) * N + c;
        T t = T(0), un = T(0), ah;
        if constexpr (MODE == 2) {
          ah = timp[g] - u_in[g];
        } else {
          auto X = [&](int jj, int cc) {
            const C z = zb[(jj >> 1) * ZS + spad(cc)];
            return (jj & 1) ? z.y : z.x;
          };
          const T x = X(j, c);
          if constexpr (PRIOR == PRIOR_TV_ISO) {
            T t2, un2, av2;
            group(X(j, cr) - x, ldu1(0, j, c), X(j + 1, c) - x, ldu1(1, j, c), t, un, ah, t2, un2, av2);
          } else {
            shrink(X(j, cr) - x, ldu1(0, j, c), tau, t, un);
            ah = t - un;
          }
        }
        edge[tid / NB][b] = ah;
      }
      __syncthreads();
    };
    // One tile row j at the columns c0, c0 + 1: x of the row at c0 .. c0 + 2 and of the next row at
    // c0, c0 + 1, a_v of the row above in avp (replaced by this row's).  FULL: the row is one of the
    // tile's output rows (u, t and the residual sums are its own, q is formed).
    auto row = [&](auto mode, auto full, int j, int c0, const T(&x)[3], const T(&xn)[3], C uh, C uv, T(&avp)[2],
                   T(&q)[2], T(&ah)[2]) {
      constexpr int MODE = decltype(mode)::value;
      constexpr bool FULL = decltype(full)::value;
      const size_t g = (size_t)grow(j) * N + c0;
      T tv[2], uvn[2], th[2], uhn[2], av[2], wh[2] = {T(0), T(0)}, wv[2] = {T(0), T(0)};
      if constexpr (MODE == 2) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          tv[e] = timp[plane + g + e];
          uvn[e] = u_in[plane + g + e];
          if constexpr (FULL) {
            th[e] = timp[g + e];
            uhn[e] = u_in[g + e];
          }
        }
      } else {
        wv[0] = xn[0] - x[0];
        wv[1] = xn[1] - x[1];
        if constexpr (PRIOR == PRIOR_TV_ISO) {
          wh[0] = x[1] - x[0];
          wh[1] = x[2] - x[1];
          group(wh[0], uh.x, wv[0], uv.x, th[0], uhn[0], ah[0], tv[0], uvn[0], av[0]);
          group(wh[1], uh.y, wv[1], uv.y, th[1], uhn[1], ah[1], tv[1], uvn[1], av[1]);
        } else {
          shrink(wv[0], uv.x, tau, tv[0], uvn[0]);
          shrink(wv[1], uv.y, tau, tv[1], uvn[1]);
          if constexpr (FULL) {
            wh[0] = x[1] - x[0];
            wh[1] = x[2] - x[1];
            shrink(wh[0], uh.x, tau, th[0], uhn[0]);
            shrink(wh[1], uh.y, tau, th[1], uhn[1]);
          }
        }
      }
      if constexpr (PRIOR != PRIOR_TV_ISO || MODE == 2) {
        av[0] = tv[0] - uvn[0];
        av[1] = tv[1] - uvn[1];
        if constexpr (FULL) {
          ah[0] = th[0] - uhn[0];
          ah[1] = th[1] - uhn[1];
        }
      }
      if constexpr (FULL) {
        T ahm = __shfl_up_sync(0xffffffffu, ah[1], 1);
        if ((tid & 31) == 0) ahm = edge[j - 1][c0 / 64];
        *reinterpret_cast<C*>(u_out + plane + g) = cpack<C>(uvn[0], uvn[1]);
        *reinterpret_cast<C*>(u_out + g) = cpack<C>(uhn[0], uhn[1]);
        if constexpr (MODE == 1) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (resid) {
              acc_resid(part, wh[e], th[e], uhn[e], tprev_rd, g + e);
              acc_resid(part, wv[e], tv[e], uvn[e], tprev_rd ? tprev_rd + plane : nullptr, g + e);
            }
            if (store_t) {
              tprev[g + e] = th[e];
              tprev[plane + g + e] = tv[e];
            }
          }
        }
        q[0] = (ahm - ah[0] + avp[0] - av[0]) * a.qscale;
        q[1] = (ah[0] - ah[1] + avp[1] - av[1]) * a.qscale;
      }
      avp[0] = av[0];
      avp[1] = av[1];
    };
    // x of tile rows 2p, 2p + 1 at the columns c0 .. c0 + 2
    auto load_pair = [&](auto mode, int p, int c0, T(&xa)[3], T(&xb)[3]) {
      if constexpr (decltype(mode)::value != 2) {
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const C z = zb[p * ZS + spad((c0 + e) & (N - 1))];
          xa[e] = z.x;
          xb[e] = z.y;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 3; ++e) xa[e] = xb[e] = T(0);
      }
    };
    constexpr std::true_type full{};
    constexpr std::false_type halo{};
    auto phase = [&](auto mode) {
      edges(mode);
      if constexpr (!WALK) {
        constexpr int RG = tv_rows(N), NG = R / RG, TG = NT / NG;
        static_assert(TG >= N / 2 && TG % 32 == 0, "one column pair per thread, whole warps per row group");
        const int rg = tid / TG, cp = tid - rg * TG, c0 = 2 * cp;
        const bool on = rg < NG && cp < N / 2;
        const int p0 = rg * (RG / 2);  // output rows: tile rows 2 p0 + 1 .. 2 p0 + RG
        T qv[RG][2];
        if (on) {
          T xa[3], xb[3], avp[2], ah[2];
          load_pair(mode, p0, c0, xa, xb);
          row(mode, halo, 2 * p0, c0, xa, xb, ISO ? ldu(0, 2 * p0, c0) : czero, ldu(1, 2 * p0, c0), avp, qv[0], ah);
#pragma unroll
          for (int i = 0; i < RG / 2; ++i) {
            T ya[3], yb[3];
            load_pair(mode, p0 + i + 1, c0, ya, yb);
            const int j = 2 * (p0 + i) + 1;
            row(mode, full, j, c0, xb, ya, ldu(0, j, c0), ldu(1, j, c0), avp, qv[2 * i], ah);
            row(mode, full, j + 1, c0, ya, yb, ldu(0, j + 1, c0), ldu(1, j + 1, c0), avp, qv[2 * i + 1], ah);
#pragma unroll
            for (int e = 0; e < 3; ++e) xb[e] = yb[e];
          }
        }
        __syncthreads();  // every thread has read the x tile: q takes its place, as row pairs
        if (on) {
#pragma unroll
          for (int i = 0; i < RG / 2; ++i)
#pragma unroll
            for (int e = 0; e < 2; ++e) zb[(p0 + i) * ZS + spad(c0 + e)] = cpack<C>(qv[2 * i][e], qv[2 * i + 1][e]);
        }
      } else {
        constexpr int NIT = (N / 2 + NT - 1) / NT;
        T xb[NIT][3], avp[NIT][2], q[NIT][2][2];
        C un[NIT][2][2];  // u of the next two rows, [row][component], loaded one row pair ahead
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
          const int cp = tid + it * NT;
          if (cp < N / 2) {
            T xa[3], ah[2];
            load_pair(mode, 0, 2 * cp, xa, xb[it]);
            row(mode, halo, 0, 2 * cp, xa, xb[it], ISO ? ldu(0, 0, 2 * cp) : czero, ldu(1, 0, 2 * cp), avp[it],
                q[it][0], ah);
#pragma unroll
            for (int e = 0; e < 4; ++e) un[it][e >> 1][e & 1] = ldu(e & 1, 1 + (e >> 1), 2 * cp);
          }
        }
#pragma unroll 1
        for (int i = 0; i < R / 2; ++i) {
          // Row frequencies k2 = 0 and 1 (kLowK = 2) of the two components of a = t - u' on the
          // output rows, as direct sums with the exact table twiddle exp(-2 pi i c / N), for the
          // low-column correction of the x-update (launch_passB_split): near DC the FP32 transforms
          // of q = D^T a carry a uniform rounding error that Psi^{-1} amplifies by ~1/g, while
          // transforms of a itself do not.  Value 6 r + 3 comp + {0, 1, 2}: row r of the pair, sum a,
          // Re and Im of sum a exp(-2 pi i c / N)
          T low[LOW ? 16 : 1];
#pragma unroll
          for (int e = 0; e < (LOW ? 16 : 1); ++e) low[e] = T(0);
#pragma unroll
          for (int it = 0; it < NIT; ++it) {
            const int cp = tid + it * NT, c0 = 2 * cp;
            if (cp < N / 2) {
              T ya[3], yb[3], ah[2];
              load_pair(mode, i + 1, c0, ya, yb);
              auto add_low = [&](int r) {
                if constexpr (LOW) {
                  const C w0 = ldg_tw(&a.tw[c0 * (kTwN / N)]), w1 = ldg_tw(&a.tw[(c0 + 1) * (kTwN / N)]);
#pragma unroll
                  for (int s = 0; s < 2; ++s) {
                    const T v0 = s ? avp[it][0] : ah[0], v1 = s ? avp[it][1] : ah[1];
                    T* l = &low[6 * r + 3 * s];
                    l[0] += v0 + v1;
                    l[1] = fma(v1, (T)w1.x, fma(v0, (T)w0.x, l[1]));
                    l[2] = fma(v1, (T)w1.y, fma(v0, (T)w0.y, l[2]));
                  }
                }
              };
              C uc[2][2];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                uc[e >> 1][e & 1] = un[it][e >> 1][e & 1];
                if (i + 1 < R / 2) un[it][e >> 1][e & 1] = ldu(e & 1, 2 * i + 3 + (e >> 1), c0);
              }
              row(mode, full, 2 * i + 1, c0, xb[it], ya, uc[0][0], uc[0][1], avp[it], q[it][0], ah);
              add_low(0);
              row(mode, full, 2 * i + 2, c0, ya, yb, uc[1][0], uc[1][1], avp[it], q[it][1], ah);
              add_low(1);
#pragma unroll
              for (int e = 0; e < 3; ++e) xb[it][e] = yb[e];
            }
          }
          if constexpr (LOW) {
            // warp sums of the 12 values by recursive halving: lane l ends with value l >> 1
            reduce_scatter16(low, tid & 31);
            if ((tid & 1) == 0 && (tid & 31) < 24) lows[i & 1][tid >> 5][(tid & 31) >> 1] = low[0];
          }
          __syncthreads();  // every thread has read x rows 2i, 2i + 1: q rows 2i, 2i + 1 take their place
#pragma unroll
          for (int it = 0; it < NIT; ++it) {
            const int cp = tid + it * NT;
            if (cp < N / 2) {
#pragma unroll
              for (int e = 0; e < 2; ++e) zb[i * ZS + spad(2 * cp + e)] = cpack<C>(q[it][0][e], q[it][1][e]);
            }
          }
          if constexpr (LOW) {
            if (a.lowbuf && tid < 12) {  // value tid of rows 2i, 2i + 1: the warps' sums in order
              static_assert(NT % 128 == 0, "");
              T s4[NT / 128];  // four warps' sums at a time, then theirs: shorter chain, smaller rounding error
#pragma unroll
              for (int w4 = 0; w4 < NT / 128; ++w4) {
                const T(*l)[12] = &lows[i & 1][4 * w4];
                s4[w4] = (l[0][tid] + l[1][tid]) + (l[2][tid] + l[3][tid]);
              }
              T s = s4[0];
#pragma unroll
              for (int w4 = 1; w4 < NT / 128; ++w4) s += s4[w4];
              const int r = tid / 6, comp = (tid / 3) & 1, e = tid % 3;
              T* dst = reinterpret_cast<T*>(a.lowbuf + ((size_t)(comp * kLowK + (e > 0)) * a.M + m) * CP + r0 + 2 * i + r);
              if (e == 0) {
                dst[0] = s;
                dst[1] = T(0);
              } else {
                dst[e - 1] = s;
              }
            }
          }
        }
      }
    };
    if (import_mode) phase(std::integral_constant<int, 2>{});
    else if (resid || store_t) phase(std::integral_constant<int, 1>{});
    else phase(std::integral_constant<int, 0>{});
  } else if constexpr (PRIOR == PRIOR_DCT8) {
    if (!import_mode) {
      // row DCT of every 8-sample segment of both rows of a pair, in place
      for (int idx = tid; idx < NPOUT * (N / 8); idx += nth) {
        const int p = idx / (N / 8), c0 = (idx - p * (N / 8)) * 8;
        C v[8], o[8];
#pragma unroll
        for (int n = 0; n < 8; ++n) v[n] = zb[p * ZS + spad(c0 + n)];
        dct8_pair<T, true>(a.dct, v, o);
#pragma unroll
        for (int n = 0; n < 8; ++n) zb[p * ZS + spad(c0 + n)] = o[n];
      }
      __syncthreads();
    }
    if constexpr (USTAGE) u_ok = mbar_wait_bounded(&ubar, 0, a.err, a.test_fault ? 64 : (1 << 22));
    // column DCT -> coefficients w; shrink; dual; inverse column DCT of (t - u')
    for (int idx = tid; idx < (R / 8) * N; idx += nth) {
      const int br = idx / N, c = idx - br * N;
      T v[8], w[8], d[8];
      if (!import_mode) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const C z = zb[(br * 4 + q) * ZS + spad(c)];
          v[2 * q] = z.x;
          v[2 * q + 1] = z.y;
        }
        dct8_fwd(a.dct, v, w);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const size_t g = (size_t)(r0 + br * 8 + k) * N + c;
        const T uo = (USTAGE && u_ok) ? us[(br * 8 + k) * N + c] : u_in[g];
        T t, un;
        if (import_mode) {
          t = timp[g];
          un = uo;
          w[k] = T(0);
        } else {
          shrink(w[k], uo, tau, t, un);
        }
        u_out[g] = un;
        d[k] = t - un;
        if (resid) acc_resid(part, w[k], t, un, tprev_rd, g);
        if (store_t) tprev[g] = t;
      }
      dct8_inv(a.dct, d, v);
#pragma unroll
      for (int q = 0; q < 4; ++q) zb[(br * 4 + q) * ZS + spad(c)] = mk<C>(v[2 * q], v[2 * q + 1]);
    }
    __syncthreads();
    for (int idx = tid; idx < NPOUT * (N / 8); idx += nth) {
      const int p = idx / (N / 8), c0 = (idx - p * (N / 8)) * 8;
      C v[8], o[8];
#pragma unroll
      for (int n = 0; n < 8; ++n) v[n] = zb[p * ZS + spad(c0 + n)];
      dct8_pair<T, false>(a.dct, v, o);
#pragma unroll
      for (int n = 0; n < 8; ++n) zb[p * ZS + spad(c0 + n)] = mk<C>(o[n].x * a.qscale, o[n].y * a.qscale);
    }
  }
  __syncthreads();

  // 4. forward row DFT of q (two rows per FFT), 5. store row half-spectra
  {
    const int team = tid / TEAM;
    const TeamSync ts = make_team_sync(team, TEAM);
    if (ts.cta || team < NPOUT)
      fft_team<C, LOGN, 1, E, -1>(zb + (team < NPOUT ? team : 0) * ZS, tid % TEAM, a.tw, ts, team < NPOUT);
  }
  __syncthreads();
  // 5. scatter the row half-spectra of q into the column layout: rows r0 + 2p, r0 + 2p + 1 of
  //    column k are adjacent (one 16-byte store for complex64)
  C* qh = a.qh + (size_t)m * CP;
  const size_t qstride = (size_t)a.M * CP;
  for (int idx = tid; idx < NPOUT * H; idx += nth) {
    const int p = idx % NPOUT, k = idx / NPOUT;
    C qa, qb;
    pair_spectrum_get(zb + p * ZS, N, k, qa, qb);
    C* col = qh + (size_t)k * qstride + r0 + 2 * p;
    if constexpr (sizeof(C) == 8) {
      *reinterpret_cast<float4*>(col) = make_float4(qa.x, qa.y, qb.x, qb.y);
    } else {
      col[0] = qa;
      col[1] = qb;
    }
  }
  if (resid) block_reduce_store<T>(part, a.partials + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kNPart);
  if constexpr (USTAGE || TVSTAGE) {
    // a copy that was only late must not write this CTA's shared memory after the CTA ends
    if (tid == 0 && !u_ok && a.test_fault == 0) mbar_wait_bounded(&ubar, 0, a.err);
  }
}

template <typename T, int LOGN, int PRIOR, int V>
cudaError_t launchA(const PassAArgs<T>& a, Chain s) {
  constexpr int N = 1 << LOGN;
  constexpr int R = rows_for<T>(N, PRIOR);
  constexpr int nth = threads_for<T>(N, PRIOR, R, V);
  constexpr size_t sm = smem_for<T>(N, PRIOR, R);
  auto kern = passA_kernel<T, LOGN, PRIOR, R, V>;
  static PerDeviceOnce once;
  cudaError_t e = once([&] {
    if (sm > 48 * 1024) {
      cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (r != cudaSuccess) return r;
    }
    // the largest shared-memory carveout, so that the register-bound CTA count is reached
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                (int)cudaSharedmemCarveoutMaxShared);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(N / R, a.M), dim3(nth), sm, s, 0, a);
}

template <typename T, int PRIOR>
cudaError_t dispatchA(const PassAArgs<T>& a, int N, Chain s) {
  if constexpr (has_variant<T>(256, PRIOR)) {
    if (a.variant == 1) {
      switch (N) {
        case 256: return launchA<T, 8, PRIOR, 1>(a, s);
        case 512: return launchA<T, 9, PRIOR, 1>(a, s);
        case 1024: return launchA<T, 10, PRIOR, 1>(a, s);
        default: break;
      }
    }
  }
  switch (N) {
    case 64: return launchA<T, 6, PRIOR, 0>(a, s);
    case 128: return launchA<T, 7, PRIOR, 0>(a, s);
    case 256: return launchA<T, 8, PRIOR, 0>(a, s);
    case 512: return launchA<T, 9, PRIOR, 0>(a, s);
    case 1024: return launchA<T, 10, PRIOR, 0>(a, s);
    case 2048: return launchA<T, 11, PRIOR, 0>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

template <typename T> int passA_rows(int N, int prior) { return rows_for<T>(N, prior); }
template <typename T> size_t passA_smem(int N, int prior) { return smem_for<T>(N, prior, rows_for<T>(N, prior)); }

template <typename T> cudaError_t launch_passA(const PassAArgs<T>& a, int N, int prior, Chain s) {
  switch (prior) {
    case PRIOR_TV: return dispatchA<T, PRIOR_TV>(a, N, s);
    case PRIOR_TV_ISO: return dispatchA<T, PRIOR_TV_ISO>(a, N, s);
    case PRIOR_DCT8: return dispatchA<T, PRIOR_DCT8>(a, N, s);
    case PRIOR_L1: return launch_rowpass<T>(a, N, PRIOR_L1, s);
    default: return cudaErrorInvalidValue;
  }
}

template int passA_rows<float>(int, int);
template int passA_rows<double>(int, int);
template size_t passA_smem<float>(int, int);
template size_t passA_smem<double>(int, int);
template cudaError_t launch_passA<float>(const PassAArgs<float>&, int, int, Chain);
template cudaError_t launch_passA<double>(const PassAArgs<double>&, int, int, Chain);

}  // namespace cip
