// Row pass without exchange between neighbouring pixels: the prior pass of the l1 prior (T = I: the
// l1 analysis prior and the coefficient maps of the dictionaries), and the row transforms alone
// (read-back, wavelet chain).
//
// The inverse row FFT leaves thread tt of a team with the positions n = tt mod TT of its row pair, and
// the forward FFT starts from exactly these positions (fft.cuh: the last stage writes j + LS r, the
// first reads t + r N/8), so shrinkage, dual update and q happen in registers between the two FFTs and
// the rows themselves never go through shared memory.  What goes through it: the spectra (gathered
// from and scattered to the column layout, where a CTA's rows are contiguous per column) and one or
// two exchanges per FFT (stage merging of fft_last_merged where E allows it).
// Bound by shared-memory wavefronts (the general kernel ran its LSU pipe at 80% here): 12 accesses per
// complex value at N = 256, E = 32, against 21 with the rows in shared memory and unmerged stages.
// The l1 pass before (rows through shared memory) and now: 160 maps of 256^2 66.9 -> 57.9 us, 96 maps
// 44.0 -> 37.5, 512^2 x 10 22.0 -> 19.4 us; with the per-stage twiddle tables of common.cuh 39.9, 26.9
// and 16.6 us.
#include "fft.cuh"
#include "kernels.h"
#include "reduce.cuh"

namespace cip {

namespace {

// FFT elements per thread.  complex128 takes 8 up to N = 256: its tiles wait for the latency of their few
// FP64 units, and twice the threads halve the serial chain (with 8-row tiles, see row_rows: the l1 pass of
// 64^2 42.4 -> 21.9 us, 128^2 46.3 -> 25.0, 256^2 53.7 -> 43.0).  V is the plan's prior-pass variant: complex64 at N = 256 .. 1024 has 8, 16
// and (N = 256, where 32 merges the last two stages) 32 to choose from, timed by the autotuner.
template <typename T> constexpr int row_elems(int N, int V) {
  if (sizeof(T) == 8) return N <= 256 ? 8 : 16;
  if (N == 64) return 8;
  if (N == 128) return 8;
  if (N == 2048) return 32;
  const int e = N == 512 ? 16 : 8;  // the width the plan reports for V = 0 (prior_fft_default)
  return V == 0 ? e : (V == 1 ? 24 - e : 32);
}
// rows per CTA: 16 give whole 128-byte lines of the column layout; 8 from N = 512 on, where the
// tile has threads enough, and at N = 128, where 16 would halve the few CTAs of small problems; 8 in
// complex128, where a row pair is 32 bytes and the time is that of the SM with the most rows
template <typename T> constexpr int row_rows(int N) { return sizeof(T) == 4 && (N == 64 || N == 256) ? 16 : 8; }
constexpr int row_slot(int N) { return spad(N) + (N >= 256 ? 4 : 0); }
template <typename T> constexpr int row_threads(int N, int V) { return row_rows<T>(N) / 2 * (N / row_elems<T>(N, V)); }
template <typename T> constexpr int row_minblocks(int N, int V) {
  const int e = row_elems<T>(N, V);
  const int regs = sizeof(T) == 8 ? 168 : (e == 32 ? 128 : (e == 16 ? 80 : 56));
  const int b = 65536 / (row_threads<T>(N, V) * regs);
  return b < 1 ? 1 : (b > 16 ? 16 : b);
}

template <typename T, int LOGN, int KIND, int V>
__global__ void __launch_bounds__(row_threads<T>(1 << LOGN, V), row_minblocks<T>(1 << LOGN, V))
    row_kernel(const PassAArgs<T> a) {
  using C = typename CT<T>::type;
  constexpr int N = 1 << LOGN, H = N / 2 + 1, E = row_elems<T>(N, V), TT = N / E, R = row_rows<T>(N), NP = R / 2;
  constexpr int ZS = row_slot(N), CP = col_pitch(N), NT = row_threads<T>(N, V);
  constexpr int S8 = LOGN / 3, REM = LOGN % 3;
  constexpr bool MERGE = fft_merges<C, LOGN, E>();
  constexpr int RL = REM == 0 ? 8 : (REM == 1 ? 2 : 4), LSL = REM == 0 ? (1 << (3 * (S8 - 1))) : (1 << (3 * S8));
  // radix-8 stages between the first and the last (a merged last stage takes one of them in)
  constexpr int MID = S8 - 1 - (REM == 0 ? 1 : 0) - (MERGE ? 1 : 0);
  static_assert(NT % 32 == 0 && MID >= 0 && MID <= 2, "");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* zb = reinterpret_cast<C*>(smem_raw);  // [NP][ZS]
  const int tid = threadIdx.x, m = blockIdx.y, r0 = blockIdx.x * R;
  const int team = tid / TT, tt = tid % TT;
  const bool resid = KIND == PRIOR_L1 && (a.flags & PA_RESID) != 0;
  const bool store_t = KIND == PRIOR_L1 && (a.flags & PA_STORE_T) != 0;
  const bool import_mode = KIND == PRIOR_L1 && (a.flags & PA_IMPORT) != 0;
  const size_t plane = (size_t)N * N;
  const T* u_in = a.u_in ? a.u_in + (size_t)m * plane : nullptr;
  T* u_out = a.u_out ? a.u_out + (size_t)m * plane : nullptr;
  const TeamSync ts = make_team_sync(team, TT);
  auto sync = [&]() { ts.sync(); };
  auto none = [&]() {};
  C* buf = zb + team * ZS;
  auto pin = [&](int i0, int off) { return buf[spad(i0) + off + (off >> 4)]; };
  auto pout = [&](int i0, int off, C v) { buf[spad(i0) + off + (off >> 4)] = v; };
  C z[E];  // element i: position tt + TT i

  if constexpr (KIND == PRIOR_L1) {
    // u (and t_prev) rows into L2 while the preceding kernel drains; an import's u is not final yet
    if (tid == 0 && !import_mode) prefetch_l2(u_in + (size_t)r0 * N, (size_t)R * N * sizeof(T));
    if (tid == 32 % NT && resid) prefetch_l2(a.tprev + (size_t)m * plane + (size_t)r0 * N, (size_t)R * N * sizeof(T));
  }
  grid_dep_wait();
  grid_dep_launch();
  if (KIND != ROWS_IN && !import_mode) {
    // gather the row half-spectra of the tile (two rows per complex FFT) from the column layout:
    // thread = (pair p, column k), p fastest
    const C* xh = a.xh + (size_t)m * CP + r0;
    const size_t kstride = (size_t)a.M * CP;
    constexpr int ITEMS = NP * H, G = sizeof(T) == 4 ? 4 : 2;
    for (int base = tid; base < ITEMS; base += G * NT) {
      C xa[G], xb[G];
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const int idx = base + i * NT;
        if (idx >= ITEMS) continue;
        const C* col = xh + (size_t)(idx / NP) * kstride + 2 * (idx % NP);
        if constexpr (sizeof(C) == 8) {  // rows 2p, 2p + 1: 16-byte aligned (r0 and CP even)
          const float4 v = *reinterpret_cast<const float4*>(col);
          xa[i] = mk<C>(v.x, v.y);
          xb[i] = mk<C>(v.z, v.w);
        } else {
          xa[i] = col[0];
          xb[i] = col[1];
        }
      }
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const int idx = base + i * NT;
        if (idx < ITEMS) pair_spectrum_put(zb + (idx % NP) * ZS, N, idx / NP, xa[i], xb[i]);
      }
    }
    __syncthreads();
    fft_stage_io<C, LOGN, E, +1, 8, 1>(tt, a.tw, pin, sync, pout);
    sync();
    if constexpr (MID >= 1) {
      fft_stage_io<C, LOGN, E, +1, 8, 8>(tt, a.tw, pin, sync, pout);
      sync();
    }
    if constexpr (MID >= 2) {
      fft_stage_io<C, LOGN, E, +1, 8, 64>(tt, a.tw, pin, sync, pout);
      sync();
    }
    auto keep = [&](int i0, int off, C v) { z[(i0 - tt + off) / TT] = v; };
    if constexpr (MERGE) fft_last_merged<C, LOGN, E, +1>(tt, a.tw, pin, none, keep);
    else fft_stage_io<C, LOGN, E, +1, RL, LSL>(tt, a.tw, pin, none, keep);
  }
  const size_t g0 = (size_t)(r0 + 2 * team) * N + tt;  // row 2 team of the tile, position tt
  if constexpr (KIND == ROWS_OUT) {
#pragma unroll
    for (int i = 0; i < E; ++i) {
      u_out[g0 + TT * i] = z[i].x;
      u_out[g0 + N + TT * i] = z[i].y;
    }
    return;
  }
  T part[kNPart] = {T(0), T(0), T(0), T(0), T(0)};
  if constexpr (KIND == ROWS_IN) {
#pragma unroll
    for (int i = 0; i < E; ++i) z[i] = cpack<C>(u_in[g0 + TT * i] * a.qscale, u_in[g0 + N + TT * i] * a.qscale);
  } else {
    T* tprev = a.tprev + (size_t)m * plane;
    const T* timp = a.t_imp ? a.t_imp + (size_t)m * plane : nullptr;
    const T tau = a.tau;
#pragma unroll
    for (int c = 0; c < E; c += 8) {
      T uo[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int s = 0; s < 2; ++s) uo[i][s] = __ldg(u_in + g0 + s * N + TT * (c + i));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        T q[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const size_t g = g0 + s * N + TT * (c + i);
          const T w = import_mode ? T(0) : (s ? z[c + i].y : z[c + i].x);
          T t, un;
          if (import_mode) {
            t = timp[g];
            un = uo[i][s];
          } else {
            t = soft(w + uo[i][s], tau);
            un = uo[i][s] + w - t;
          }
          u_out[g] = un;
          if (resid) acc_resid(part, w, t, un, tprev, g);
          if (store_t) tprev[g] = t;
          q[s] = (t - un) * a.qscale;
        }
        z[c + i] = cpack<C>(q[0], q[1]);
      }
    }
    sync();  // every thread of the team has read the last stage's inputs
  }
  auto held = [&](int i0, int off) { return z[(i0 - tt + off) / TT]; };
  fft_stage_io<C, LOGN, E, -1, 8, 1>(tt, a.tw, held, none, pout);
  sync();
  if constexpr (MID >= 1) {
    fft_stage_io<C, LOGN, E, -1, 8, 8>(tt, a.tw, pin, sync, pout);
    sync();
  }
  if constexpr (MID >= 2) {
    fft_stage_io<C, LOGN, E, -1, 8, 64>(tt, a.tw, pin, sync, pout);
    sync();
  }
  if constexpr (MERGE) fft_last_merged<C, LOGN, E, -1>(tt, a.tw, pin, sync, pout);
  else fft_stage_io<C, LOGN, E, -1, RL, LSL>(tt, a.tw, pin, sync, pout);
  __syncthreads();
  // scatter the row half-spectra of q into the column layout
  C* qh = a.qh + (size_t)m * CP + r0;
  const size_t qstride = (size_t)a.M * CP;
  for (int idx = tid; idx < NP * H; idx += NT) {
    const int p = idx % NP, k = idx / NP;
    C qa, qb;
    pair_spectrum_get(zb + p * ZS, N, k, qa, qb);
    C* col = qh + (size_t)k * qstride + 2 * p;
    if constexpr (sizeof(C) == 8) {
      *reinterpret_cast<float4*>(col) = make_float4(qa.x, qa.y, qb.x, qb.y);
    } else {
      col[0] = qa;
      col[1] = qb;
    }
  }
  if (resid) block_reduce_store<T>(part, a.partials + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kNPart);
}

template <typename T, int LOGN, int KIND, int V> cudaError_t launch_row(const PassAArgs<T>& a, Chain s) {
  using C = typename CT<T>::type;
  constexpr int N = 1 << LOGN;
  constexpr size_t sm = (size_t)row_rows<T>(N) / 2 * row_slot(N) * sizeof(C);
  auto k = row_kernel<T, LOGN, KIND, V>;
  static PerDeviceOnce once;
  cudaError_t e = once([&] {
    if (sm > 48 * 1024) {
      cudaError_t r = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
      if (r != cudaSuccess) return r;
    }
    return cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3(N / row_rows<T>(N), a.M), dim3(row_threads<T>(N, V)), sm, s, 0, a);
}

template <typename T, int KIND> cudaError_t dispatch_row(const PassAArgs<T>& a, int N, Chain s) {
  // the row transforms alone take the variant that was fastest for them at every size (V below)
  if constexpr (sizeof(T) == 4) {
    const int v = KIND == PRIOR_L1 ? a.variant : (N == 256 ? 2 : (N == 1024 ? 1 : 0));
    switch (N) {
      case 256:
        if (KIND != PRIOR_L1 || v == 2) return launch_row<T, 8, KIND, 2>(a, s);
        if constexpr (KIND == PRIOR_L1) return v == 1 ? launch_row<T, 8, KIND, 1>(a, s) : launch_row<T, 8, KIND, 0>(a, s);
        break;
      case 512:
        if (KIND != PRIOR_L1 || v != 1) return launch_row<T, 9, KIND, 0>(a, s);
        if constexpr (KIND == PRIOR_L1) return launch_row<T, 9, KIND, 1>(a, s);
        break;
      case 1024:
        if (KIND != PRIOR_L1 || v == 1) return launch_row<T, 10, KIND, 1>(a, s);
        if constexpr (KIND == PRIOR_L1) return launch_row<T, 10, KIND, 0>(a, s);
        break;
      default: break;
    }
  }
  switch (N) {
    case 64: return launch_row<T, 6, KIND, 0>(a, s);
    case 128: return launch_row<T, 7, KIND, 0>(a, s);
    case 2048: return launch_row<T, 11, KIND, 0>(a, s);
    default: break;
  }
  if constexpr (sizeof(T) == 8) {
    switch (N) {
      case 256: return launch_row<T, 8, KIND, 0>(a, s);
      case 512: return launch_row<T, 9, KIND, 0>(a, s);
      case 1024: return launch_row<T, 10, KIND, 0>(a, s);
      default: break;
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace

template <typename T> int rowpass_rows(int N) { return row_rows<T>(N); }
template int rowpass_rows<float>(int);
template int rowpass_rows<double>(int);
template <typename T> int rowpass_elems(int N, int variant) { return row_elems<T>(N, variant); }
template int rowpass_elems<float>(int, int);
template int rowpass_elems<double>(int, int);

template <typename T> cudaError_t launch_rowpass(const PassAArgs<T>& a, int N, int kind, Chain s) {
  switch (kind) {
    case PRIOR_L1: return dispatch_row<T, PRIOR_L1>(a, N, s);
    case ROWS_OUT: return dispatch_row<T, ROWS_OUT>(a, N, s);
    case ROWS_IN: return dispatch_row<T, ROWS_IN>(a, N, s);
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_rowpass<float>(const PassAArgs<float>&, int, int, Chain);
template cudaError_t launch_rowpass<double>(const PassAArgs<double>&, int, int, Chain);

}  // namespace cip
