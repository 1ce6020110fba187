// C ABI of the library (declared in include/cip.h): plan lifetime, setup
// (Alg. 1 lines 1-2), the iteration loop (Alg. 1 lines 3-8), read-back,
// state import/export and per-kernel timing.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <tuple>
#include <string>
#include <vector>

#include "../../include/cip.h"
#include "kernels.h"

using namespace cip;

namespace {

constexpr int kPinvListCap = 64;
constexpr int kMaxTimed = 4096;

std::string g_create_error;

struct Staging {
  void* p = nullptr;
  cudaStream_t s = nullptr;
  ~Staging() {
    if (p) cudaFreeAsync(p, s);
  }
};

bool is_device_ptr(const void* p) {
  cudaPointerAttributes at;
  cudaError_t e = cudaPointerGetAttributes(&at, p);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

struct cip_plan {
  int N = 0, K = 0, M = 0, P = 0;
  cip_dtype dtype = CIP_F32;
  cip_options opt{};
  int prior = -1;
  double lam = 0, rho = 0, beta = 0;
  double mu = 0;  // dictionary: gradient (Tikhonov) weight on the codes
  double adapt_tau = 0, adapt_mu = 0;  // adaptive penalty (Eq. paramS); tau = 0: off
  void* yhat_keep = nullptr;           // measurement spectra kept for re-forming the data term
  bool have_psfs = false, have_y = false;
  int iteration = 0;
  int cur = 0;  // index of the u buffer holding the current u
  size_t esz = 4;
  int rowsA = 8, cc = 1, blocksA = 0, blocksB = 0;
  int colmode = 1;  // column pass: 1 fused kernel, 2 split (FFT / solve / FFT), 3 fused without the ring
  int recmode = 1;  // with colmode 3: the form of recorded iterations (batch, server), 1 or 2
  int avar = 0;     // prior-pass kernel variant (1: the other FFT width, 2: 32; complex64, N = 256 .. 1024)
  int test_fault = 0;  // test-only fault switch (cip_set_test_fault)
  // TV at N >= kLowFixMinN: low-column correction of the x-update (launch_passB_split)
  void* lowbuf = nullptr;  // [2][kLowK][M][CP] low-frequency row DFTs of the components of t - u
  void* lowq = nullptr;    // [2][kLowK][M][CP] their column DFTs
  // convolutional dictionary (prior CIP_PRIOR_CONVDICT): L filters of P x P, or of Q x P x P
  // (3D dictionary, Q >= 1; Q = 0 for the 2D dictionary)
  int L = 0, Pf = 0, Q = 0;
  void* w3 = nullptr;                   // 3D dictionary: exp(-2 pi i j / M), j < M, FP64 (setup)
  void* theta = nullptr;                // [H][L][CP] DFT of the embedded filters
  void* pbuf[2] = {nullptr, nullptr};   // [H][M][CP] p = sum_l theta_l v_l (ping-pong)
  int pcur = 0;
  void* xcol = nullptr;                 // [H][M][CP] x-hat of the last x-update
  // Kronecker wavelet (x) DCT prior (CIP_PRIOR_WDCT): two [M][N][N] work planes, the channel DCT
  // matrix [M][M] and the Symmlet-8 lowpass
  void* wbuf[3] = {nullptr, nullptr, nullptr};
  void* wcos = nullptr;
  double wcos_h[256] = {};  // the same matrix on the host (passed to the shrinkage kernel by value)
  double wfilt[16] = {};
  // online dictionary update (Section IV-B): sigma = 0 off.  While on, theta lives in the first L
  // planes of dl_spec and F(g - e) in the last L; the filters g on their P x P support in dl_gs.
  double dl_sigma = 0;
  double dl_tau = 0, dl_mu = 0;  // adaptation of sigma by the rule of Eq. paramS; tau = 0: off
  int dl_L = 0, dl_P = 0;   // L and P the buffers below were sized for
  void* filt = nullptr;     // [L][P][P] the filters given to cip_set_dictionary (2D; plan dtype)
  void* dl_spec = nullptr;  // [H][2L][CP]: theta = F g, F(g - e)
  void* dl_col = nullptr;   // [H][L][CP]: w = F(d + e) of the current step
  void* dl_ypart = nullptr; // [H][N/kDLBlock][L][P] per-CTA partial inverse DFTs at the support rows
  void* dl_yfull = nullptr; // [L][P][H] the same per column
  int* dl_cnt = nullptr;    // [H] CTA counters of the column sums
  void* dl_gfac = nullptr;  // [H][L][P] partial DFTs of the support rows of g
  void* dl_gs = nullptr;    // [L][P][P] g on the support
  double* dl_part = nullptr;  // [H N/kDLBlock + L] residual sums of the last check
  double* dl_host = nullptr;  // pinned copy of dl_part
  const cip_plan* factor_src = nullptr;  // plan whose factor this plan adopted (serving factor cache)
  // device buffers
  void* xh = nullptr;
  void* qh = nullptr;
  void* u[2] = {nullptr, nullptr};
  void* tprev = nullptr;
  void* pinv = nullptr;
  void* bhat = nullptr;       // data term xb = Psi^{-1} beta Lambda^H F y / N^2
  void* colbuf = nullptr;     // split column pass: column-contiguous spectra [N/2+1][M][N]
  void* pinv64 = nullptr;     // setup-precision copy of the packed factor (SetupC<T>)
  void* lam64 = nullptr;      // setup-precision PSF spectra [K*M][N][P] (SetupC<T>)
  void* tw = nullptr;        // plan-precision twiddles
  void* tw64 = nullptr;       // setup-precision twiddles (SetupC<T>)
  double* gs = nullptr;      // 4 sin^2(pi k / N)
  double* partials = nullptr;
  double* resid = nullptr;   // [kNPart + 2]
  int* conv = nullptr;
  int* pinv_list = nullptr;
  double* resid_host = nullptr;  // pinned
  bool resid_valid = false;
  // timing
  bool timing = false;
  std::vector<cudaEvent_t> evA, evB;
  int nA = 0, nB = 0;
  unsigned long long launches = 0;  // kernels launched by this plan
  cudaStream_t ast = nullptr;        // stream of the current call: buffers are allocated and freed on it
  std::string err;
};

namespace {

cip_status fail(cip_plan* p, cip_status s, const std::string& msg) {
  if (p) p->err = msg;
  else g_create_error = msg;
  return s;
}

#define CIP_LAUNCH(plan, call)                                                                        \
  do {                                                                                                \
    cudaError_t e_ = (call);                                                                          \
    if (e_ != cudaSuccess)                                                                            \
      return fail(plan, CIP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));          \
    (plan)->launches++;                                                                               \
  } while (0)

#define CIP_CUDA(plan, call)                                                                          \
  do {                                                                                                \
    cudaError_t e_ = (call);                                                                          \
    if (e_ != cudaSuccess)                                                                            \
      return fail(plan, e_ == cudaErrorMemoryAllocation ? CIP_ERR_OOM : CIP_ERR_CUDA,                 \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                              \
  } while (0)

size_t ncomp_of(int prior) { return prior_is_tv(prior) ? 2 : 1; }

bool is_cd(const cip_plan* p) { return p->prior == CIP_PRIOR_CONVDICT; }
// kind of prior pass: the dictionary's shrinkage acts on the coefficient maps with T = I
int prior_pass_kind(const cip_plan* p) { return is_cd(p) ? (int)PRIOR_L1 : p->prior; }
// row tile of the prior pass's work split (the wavelet prior shares the l1 split for its partials)
int tile_kind(int prior) { return (prior == CIP_PRIOR_CONVDICT || prior == CIP_PRIOR_WDCT) ? (int)PRIOR_L1 : prior; }
// maps the prior pass works on: image channels, or the L*M coefficient maps of the dictionary
int smaps(const cip_plan* p) { return is_cd(p) ? p->M * p->L : p->M; }

bool valid_n(int N) { return N >= 64 && N <= 2048 && (N & (N - 1)) == 0; }

// TV plans from this size on take Q of the columns k2 < kLowK from the transforms of the
// components of t - u (launch_passB_split): below it the FP32 rounding that Psi^{-1} amplifies
// near DC stays within the per-step tolerance
constexpr int kLowFixMinN = 2048;
bool low_fix(const cip_plan* p) { return !is_cd(p) && prior_is_tv(p->prior) && p->N >= kLowFixMinN; }
size_t low_elems(const cip_plan* p) { return (size_t)kLowK * p->M * col_pitch(p->N); }

// sizes in elements
size_t half_elems(const cip_plan* p, int maps) { return (size_t)maps * p->N * p->P; }
// column-contiguous per-bin planes [N/2+1][planes][col_pitch(N)] (+ slack for 16-byte prefetch widening)
size_t col_elems(const cip_plan* p, int planes) {
  return (size_t)(p->N / 2 + 1) * planes * col_pitch(p->N) + 16;
}
size_t real_elems(const cip_plan* p, int maps) { return (size_t)maps * p->N * p->N; }

// orthonormal 8-point DCT-II, computed once per process: every prior-pass launch carries a copy, and
// 64 cosines per launch cost the host more than the launch of a small plan's kernel
template <typename T> void fill_dct(T* d) {
  struct Table {
    T v[64];
    Table() {
      for (int k = 0; k < 8; ++k)
        for (int n = 0; n < 8; ++n) {
          const double a = k == 0 ? std::sqrt(1.0 / 8.0) : std::sqrt(2.0 / 8.0);
          v[k * 8 + n] = (T)(a * std::cos(M_PI * (2 * n + 1) * k / 16.0));
        }
    }
  };
  static const Table t;
  std::memcpy(d, t.v, sizeof(t.v));
}

// exp(-2 pi i k / 2048) with the angle reduced exactly through octant symmetry, and behind them the
// same values once per FFT stage in the order the stage reads them (tw_stage)
void twiddles(std::vector<double>& re, std::vector<double>& im) {
  re.resize(kTwAll);
  im.resize(kTwAll);
  for (int k = 0; k < kTwN; ++k) {
    const double a = 2.0 * M_PI * (double)k / (double)kTwN;
    re[k] = std::cos(a);
    im[k] = -std::sin(a);
  }
  // exact values at multiples of pi/4
  for (int k = 0; k < kTwN; k += kTwN / 4) {
    const int q = k / (kTwN / 4);
    re[k] = (q == 0) ? 1.0 : (q == 2 ? -1.0 : 0.0);
    im[k] = (q == 1) ? -1.0 : (q == 3 ? 1.0 : 0.0);
  }
  const int stages[][2] = {{8, 8}, {8, 64}, {2, 64}, {2, 512}, {4, 64}, {4, 512}};  // radix, LS
  for (auto& st : stages)
    for (int r = 1; r < st[0]; ++r)
      for (int j = 0; j < st[1]; ++j) {
        const int d = tw_stage(st[0], st[1]) + (r - 1) * st[1] + j, k = r * j * (kTwN / (st[0] * st[1]));
        re[d] = re[k];
        im[d] = im[k];
      }
}

// Plan buffers use the stream-ordered allocator on the stream of the call that creates or frees
// them, so that no call implicitly synchronises the device (the request server relies on it).
void free_ptr(cip_plan* p, void*& q) {
  if (q) cudaFreeAsync(q, p->ast);
  q = nullptr;
}
cudaError_t dmalloc(cip_plan* p, void** q, size_t bytes) { return cudaMallocAsync(q, bytes, p->ast); }

template <typename T> cip_status alloc_state(cip_plan* p) {
  using C = typename CT<T>::type;
  const size_t nc = ncomp_of(p->prior);
  const int S = smaps(p);
  for (int i = 0; i < 2; ++i) {
    free_ptr(p, p->u[i]);
    CIP_CUDA(p, dmalloc(p, &p->u[i], real_elems(p, S) * nc * sizeof(T)));
  }
  free_ptr(p, p->tprev);
  CIP_CUDA(p, dmalloc(p, &p->tprev, real_elems(p, S) * nc * sizeof(T)));
  free_ptr(p, p->lowbuf);
  free_ptr(p, p->lowq);
  if (low_fix(p)) {
    CIP_CUDA(p, dmalloc(p, &p->lowbuf, 2 * low_elems(p) * sizeof(C)));
    CIP_CUDA(p, dmalloc(p, &p->lowq, 2 * low_elems(p) * sizeof(C)));
    p->colmode = 2;  // the correction is part of the split column pass
    if (!p->colbuf) CIP_CUDA(p, dmalloc(p, &p->colbuf, col_elems(p, p->M) * sizeof(C)));
  }
  if (is_cd(p)) {
    // row spectra of v and of rho (t - u) over the coefficient maps, the column buffer and p, x
    free_ptr(p, p->xh);
    free_ptr(p, p->qh);
    CIP_CUDA(p, dmalloc(p, &p->xh, col_elems(p, S) * sizeof(C)));
    CIP_CUDA(p, dmalloc(p, &p->qh, col_elems(p, S) * sizeof(C)));
    free_ptr(p, p->colbuf);
    CIP_CUDA(p, dmalloc(p, &p->colbuf, col_elems(p, S) * sizeof(C)));
    for (int i = 0; i < 2; ++i) {
      free_ptr(p, p->pbuf[i]);
      CIP_CUDA(p, dmalloc(p, &p->pbuf[i], col_elems(p, p->M) * sizeof(C)));
    }
    free_ptr(p, p->xcol);
    CIP_CUDA(p, dmalloc(p, &p->xcol, col_elems(p, p->M) * sizeof(C)));
    free_ptr(p, p->theta);
    CIP_CUDA(p, dmalloc(p, &p->theta, col_elems(p, p->L) * sizeof(C)));
  }
  free_ptr(p, p->pinv);
  p->pinv = nullptr;
  CIP_CUDA(p, dmalloc(p, &p->pinv, col_elems(p, p->M * (p->M + 1) / 2) * sizeof(C)));
  {
    void* q = p->partials;
    free_ptr(p, q);
    p->partials = nullptr;
  }
  if (p->prior == CIP_PRIOR_WDCT) {
    for (int i = 0; i < 3; ++i) {  // coefficients, x / q, two lowpass bands of (N/2)^2 per channel
      free_ptr(p, p->wbuf[i]);
      CIP_CUDA(p, dmalloc(p, &p->wbuf[i], real_elems(p, p->M) * sizeof(T) / (i == 2 ? 2 : 1)));
    }
    free_ptr(p, p->wcos);
    CIP_CUDA(p, dmalloc(p, &p->wcos, (size_t)p->M * p->M * sizeof(T)));
    // orthonormal DCT-II along the channels, C[k][m] = a_k cos(pi (2m + 1) k / (2M))
    std::vector<T> c((size_t)p->M * p->M);
    for (int k = 0; k < p->M; ++k)
      for (int m = 0; m < p->M; ++m)
        c[(size_t)k * p->M + m] =
            (T)(std::sqrt((k == 0 ? 1.0 : 2.0) / p->M) * std::cos(M_PI * (2 * m + 1) * k / (2.0 * p->M)));
    for (size_t i = 0; i < c.size(); ++i) p->wcos_h[i] = (double)c[i];
    CIP_CUDA(p, cudaMemcpyAsync(p->wcos, c.data(), c.size() * sizeof(T), cudaMemcpyHostToDevice, p->ast));
    CIP_CUDA(p, cudaStreamSynchronize(p->ast));
  }
  p->rowsA = prior_pass_kind(p) == PRIOR_L1 ? rowpass_rows<T>(p->N) : passA_rows<T>(p->N, tile_kind(p->prior));
  p->blocksA = (p->N / p->rowsA) * smaps(p);
  // the wavelet prior's shrinkage: a thread per pixel (all channels), at most 2048 blocks
  if (p->prior == CIP_PRIOR_WDCT) p->blocksA = std::min(p->N * p->N / 256, 2048);
  CIP_CUDA(p, dmalloc(p, (void**)&p->partials, (size_t)p->blocksA * kNPart * sizeof(double)));
  return CIP_OK;
}

template <typename T> cip_status reset_state(cip_plan* p, cudaStream_t s) {
  using C = typename CT<T>::type;
  const size_t nc = ncomp_of(p->prior);
  const int S = smaps(p);
  CIP_CUDA(p, cudaMemsetAsync(p->xh, 0, col_elems(p, S) * sizeof(C), s));
  CIP_CUDA(p, cudaMemsetAsync(p->qh, 0, col_elems(p, S) * sizeof(C), s));
  CIP_CUDA(p, cudaMemsetAsync(p->conv, 0, 2 * sizeof(int), s));
  // (the other u buffer is written before it is read)
  CIP_CUDA(p, cudaMemsetAsync(p->u[0], 0, real_elems(p, S) * nc * sizeof(T), s));
  CIP_CUDA(p, cudaMemsetAsync(p->tprev, 0, real_elems(p, S) * nc * sizeof(T), s));
  if (p->lowbuf) CIP_CUDA(p, cudaMemsetAsync(p->lowbuf, 0, 2 * low_elems(p) * sizeof(C), s));
  if (is_cd(p)) {
    for (int i = 0; i < 2; ++i) CIP_CUDA(p, cudaMemsetAsync(p->pbuf[i], 0, col_elems(p, p->M) * sizeof(C), s));
    CIP_CUDA(p, cudaMemsetAsync(p->xcol, 0, col_elems(p, p->M) * sizeof(C), s));
    p->pcur = 0;
  }
  p->cur = 0;
  p->iteration = 0;
  p->resid_valid = false;
  return CIP_OK;
}

// bring a caller array (host or device) to the device; returns a device pointer
cip_status stage_in(cip_plan* p, const void* src, size_t bytes, cudaStream_t s, Staging& st, const void** dev) {
  if (is_device_ptr(src)) {
    *dev = src;
    return CIP_OK;
  }
  st.s = s;
  CIP_CUDA(p, cudaMallocAsync(&st.p, bytes, s));
  CIP_CUDA(p, cudaMemcpyAsync(st.p, src, bytes, cudaMemcpyHostToDevice, s));
  *dev = st.p;
  return CIP_OK;
}

// the setup-precision buffers of a plan of real type T
template <typename T> SetupC<T>* setup_buf(void* b) { return static_cast<SetupC<T>*>(b); }

template <typename T> cip_status form_factor(cip_plan* p, cudaStream_t s) {
  using C = typename CT<T>::type;
  if (!p->lam64) return fail(p, CIP_ERR_STATE, "the PSF spectra were released (cip_set_psfs again)");
  if (!p->pinv64)
    CIP_CUDA(p, dmalloc(p, &p->pinv64, half_elems(p, p->M * (p->M + 1) / 2) * sizeof(SetupC<T>)));
  CIP_CUDA(p, cudaMemsetAsync(p->pinv_list, 0, sizeof(int), s));
  const int use_g = prior_is_tv(p->prior) ? 1 : 0;
  // analysis: Psi = rho g I + beta Lambda^H Lambda; dictionary: t I + beta Lambda^H Lambda with t = 1
  // (P^H P = I for a convolutional dictionary, Eq. solx_synt_DFT)
  const double diag = is_cd(p) ? 1.0 : p->rho;
  const SetupC<T>* lam = setup_buf<T>(p->lam64);
  bool plain = false;
  if constexpr (sizeof(T) == 4) {
    if (p->opt.precision == 1) {
      plain = true;
      CIP_LAUNCH(p, launch_factor_fp32(lam, p->gs, use_g, p->K, p->M, p->N, diag, p->beta,
                                       reinterpret_cast<float2*>(p->pinv), p->pinv_list, kPinvListCap, s));
    }
  }
  if (!plain) {
    CIP_LAUNCH(p, launch_factor<T>(lam, p->gs, use_g, p->K, p->M, p->N, diag, p->beta, static_cast<C*>(p->pinv),
                                   setup_buf<T>(p->pinv64), p->pinv_list, kPinvListCap, s));
  }
  CIP_LAUNCH(p, launch_factor_pinv<T>(lam, p->gs, use_g, p->K, p->M, p->N, diag, p->beta, static_cast<C*>(p->pinv),
                                      setup_buf<T>(p->pinv64), p->pinv_list, kPinvListCap, s));
  int nlist = 0;
  CIP_CUDA(p, cudaMemcpyAsync(&nlist, p->pinv_list, sizeof(int), cudaMemcpyDeviceToHost, s));
  CIP_CUDA(p, cudaStreamSynchronize(s));
  if (nlist > kPinvListCap)
    return fail(p, CIP_ERR_UNSUPPORTED, "more singular frequency bins than the pseudo-inverse list holds");
  return CIP_OK;
}

// theta as the column solve reads it: the learnt spectra while the dictionary update is on
const void* theta_of(const cip_plan* p) { return p->dl_sigma > 0 ? p->dl_spec : p->theta; }
int theta_planes(const cip_plan* p) { return p->Q > 0 ? p->M * p->L : (p->dl_sigma > 0 ? 2 * p->L : p->L); }

// exp(-2 pi i j / M), j < M, with the angle reduced through (j mod M) exactly
void channel_twiddles(int M, double* re, double* im) {
  for (int j = 0; j < M; ++j) {
    const double a = 2.0 * M_PI * (double)j / (double)M;
    re[j] = std::cos(a);
    im[j] = -std::sin(a);
  }
}

// buffers of the dictionary update for the plan's current L and P (allocated once per shape)
cip_status alloc_dict(cip_plan* p) {
  if (p->dl_spec && p->dl_L == p->L && p->dl_P == p->Pf) return CIP_OK;
  void** bufs[] = {&p->dl_spec, &p->dl_col, &p->dl_ypart, &p->dl_yfull, &p->dl_gfac, &p->dl_gs};
  for (void** b : bufs)
    if (*b) {
      cudaFreeAsync(*b, p->ast);
      *b = nullptr;
    }
  if (p->dl_cnt) cudaFreeAsync(p->dl_cnt, p->ast);
  if (p->dl_part) cudaFreeAsync(p->dl_part, p->ast);
  p->dl_cnt = nullptr;
  p->dl_part = nullptr;
  const size_t ce = 2 * p->esz;
  const size_t H = p->N / 2 + 1, nkb = p->N / kDLBlock, LP = (size_t)p->L * p->Pf;
  CIP_CUDA(p, dmalloc(p, &p->dl_spec, col_elems(p, 2 * p->L) * ce));
  CIP_CUDA(p, dmalloc(p, &p->dl_col, col_elems(p, p->L) * ce));
  CIP_CUDA(p, dmalloc(p, &p->dl_ypart, H * nkb * LP * ce));
  CIP_CUDA(p, dmalloc(p, &p->dl_yfull, H * LP * ce));
  CIP_CUDA(p, dmalloc(p, &p->dl_gfac, H * LP * ce));
  CIP_CUDA(p, dmalloc(p, &p->dl_gs, LP * p->Pf * p->esz));
  CIP_CUDA(p, dmalloc(p, (void**)&p->dl_cnt, H * sizeof(int)));
  CIP_CUDA(p, cudaMemsetAsync(p->dl_cnt, 0, H * sizeof(int), p->ast));
  CIP_CUDA(p, dmalloc(p, (void**)&p->dl_part, (H * nkb + p->L) * sizeof(double)));
  if (!p->dl_host) CIP_CUDA(p, cudaMallocHost((void**)&p->dl_host, (size_t)(2049 * 32 + 32) * sizeof(double)));
  p->dl_L = p->L;
  p->dl_P = p->Pf;
  return CIP_OK;
}

template <typename T> cip_status dict_init(cip_plan* p, cudaStream_t s);

// Filters d[L][P][P] (plan dtype): embedded on the N x N torus with their centre at (0,0),
// DFT in FP64, kept as theta in the plan's precision (Section IV-B, Theta_m of the dictionary).
template <typename T> cip_status do_set_dictionary(cip_plan* p, const void* d, cudaStream_t s) {
  using C = typename CT<T>::type;
  cip_status st = alloc_state<T>(p);
  if (st != CIP_OK) return st;
  const int Qd = p->Q > 0 ? p->Q : 1;
  Staging sg;
  const void* dd = nullptr;
  st = stage_in(p, d, (size_t)p->L * Qd * p->Pf * p->Pf * sizeof(T), s, sg, &dd);
  if (st != CIP_OK) return st;
  double* emb = nullptr;
  using R = typename SetupReal<T>::type;
  SetupC<T>* th64 = nullptr;
  // 2D: one N x N plane per filter; 3D: M planes per filter (the filter on the M x N x N torus)
  const int planes = p->Q > 0 ? p->L * p->M : p->L;
  if (p->Q > 0) {
    free_ptr(p, p->theta);
    CIP_CUDA(p, dmalloc(p, &p->theta, col_elems(p, planes) * sizeof(C)));
    if (!p->w3) CIP_CUDA(p, dmalloc(p, &p->w3, 16 * sizeof(double2)));
    double re[16], im[16];
    channel_twiddles(p->M, re, im);
    double2 w[16];
    for (int j = 0; j < p->M; ++j) w[j] = make_double2(re[j], im[j]);
    CIP_CUDA(p, cudaMemcpyAsync(p->w3, w, p->M * sizeof(double2), cudaMemcpyHostToDevice, s));
    CIP_CUDA(p, cudaStreamSynchronize(s));  // w lives on this stack frame
  }
  CIP_CUDA(p, cudaMallocAsync((void**)&emb, real_elems(p, planes) * sizeof(double), s));
  CIP_CUDA(p, cudaMallocAsync((void**)&th64, half_elems(p, planes) * sizeof(SetupC<T>), s));
  cudaError_t e = cudaMemsetAsync(emb, 0, real_elems(p, planes) * sizeof(double), s);
  if (e == cudaSuccess)
    e = p->Q > 0 ? launch_embed_filters3d<T>(static_cast<const T*>(dd), emb, p->L, p->Q, p->Pf, p->M, p->N, s)
                 : launch_embed_filters<T>(static_cast<const T*>(dd), emb, p->L, p->Pf, p->N, s);
  if (e == cudaSuccess) e = launch_row_r2c<R, double>(emb, th64, p->N, planes * p->N, setup_buf<T>(p->tw64), s);
  if (e == cudaSuccess) e = launch_col_c2c<R>(th64, p->N, planes, -1, setup_buf<T>(p->tw64), s);
  if (e == cudaSuccess)
    e = p->Q > 0 ? launch_theta3_store<T>(th64, static_cast<C*>(p->theta), static_cast<const double2*>(p->w3), p->L,
                                          p->M, p->N, s)
                 : launch_theta_store<T>(th64, static_cast<C*>(p->theta), p->L, p->N, s);
  if (e == cudaSuccess) p->launches += 4;
  cudaFreeAsync(emb, s);
  cudaFreeAsync(th64, s);
  CIP_CUDA(p, e);
  if (p->Q == 0) {  // the filters the online update starts from
    free_ptr(p, p->filt);
    const size_t fb = (size_t)p->L * p->Pf * p->Pf * sizeof(T);
    CIP_CUDA(p, dmalloc(p, &p->filt, fb));
    CIP_CUDA(p, cudaMemcpyAsync(p->filt, dd, fb, cudaMemcpyDeviceToDevice, s));
  }
  if (p->dl_sigma > 0) {
    st = alloc_dict(p);
    if (st != CIP_OK) return st;
    st = dict_init<T>(p, s);
    if (st != CIP_OK) return st;
  }
  if (p->have_psfs) {
    st = form_factor<T>(p, s);
    if (st != CIP_OK) return st;
  }
  return reset_state<T>(p, s);
}

template <typename T> cip_status do_set_prior(cip_plan* p, cudaStream_t s) {
  if (is_cd(p)) return CIP_OK;  // buffers follow the dictionary (cip_set_dictionary)
  cip_status st = alloc_state<T>(p);
  if (st != CIP_OK) return st;
  if (p->have_psfs) {
    st = form_factor<T>(p, s);
    if (st != CIP_OK) return st;
  }
  return reset_state<T>(p, s);
}

template <typename T> cip_status do_set_psfs(cip_plan* p, const void* h, cudaStream_t s) {
  const size_t bytes = real_elems(p, p->K * p->M) * sizeof(T);
  Staging st;
  const void* dh = nullptr;
  cip_status r = stage_in(p, h, bytes, s, st, &dh);
  if (r != CIP_OK) return r;
  using R = typename SetupReal<T>::type;
  if (!p->lam64) CIP_CUDA(p, dmalloc(p, &p->lam64, half_elems(p, p->K * p->M) * sizeof(SetupC<T>)));
  p->factor_src = nullptr;
  const int nrows = p->K * p->M * p->N;
  SetupC<T>* lam = setup_buf<T>(p->lam64);
  const SetupC<T>* tw = setup_buf<T>(p->tw64);
  CIP_LAUNCH(p, (launch_row_r2c<R, T>(static_cast<const T*>(dh), lam, p->N, nrows, tw, s)));
  CIP_LAUNCH(p, launch_col_c2c<R>(lam, p->N, p->K * p->M, -1, tw, s));
  p->have_psfs = true;
  r = form_factor<T>(p, s);
  if (r != CIP_OK) return r;
  return reset_state<T>(p, s);
}

template <typename T> cip_status autotune(cip_plan* p, cudaStream_t s);
int forced_avar(const cip_plan* p);
bool prior_has_variant(const cip_plan* p);

// data term xb (or b for the plain FP32 method) from the measurement spectra yhat
template <typename T> cudaError_t form_data_term(cip_plan* p, const SetupC<T>* yhat, cudaStream_t s) {
  using C = typename CT<T>::type;
  const cip_plan* fs = p->factor_src ? p->factor_src : p;
  const SetupC<T>* lam = setup_buf<T>(fs->lam64);
  if constexpr (sizeof(T) == 4) {
    if (p->opt.precision == 1)
      return launch_rhs_fp32(lam, yhat, p->K, p->M, p->N, p->beta, reinterpret_cast<float2*>(p->bhat), s);
  }
  return launch_rhs<T>(lam, yhat, setup_buf<T>(fs->pinv64), p->K, p->M, p->N, p->beta, static_cast<C*>(p->bhat), s);
}

template <typename T> cip_status do_set_y(cip_plan* p, const void* y, cudaStream_t s) {
  using C = typename CT<T>::type;
  const size_t bytes = real_elems(p, p->K) * sizeof(T);
  Staging st;
  const void* dy = nullptr;
  cip_status r = stage_in(p, y, bytes, s, st, &dy);
  if (r != CIP_OK) return r;
  using R = typename SetupReal<T>::type;
  SetupC<T>* yhat = nullptr;
  // spectra and FP64 factor: the plan's own, or those of the plan its factor was adopted from
  const cip_plan* fs = p->factor_src ? p->factor_src : p;
  if (!fs->lam64 || !fs->pinv64) return fail(p, CIP_ERR_STATE, "the PSF spectra were released (cip_set_psfs again)");
  CIP_CUDA(p, cudaMallocAsync((void**)&yhat, half_elems(p, p->K) * sizeof(SetupC<T>), s));
  const SetupC<T>* tw = setup_buf<T>(p->tw64);
  cudaError_t e = launch_row_r2c<R, T>(static_cast<const T*>(dy), yhat, p->N, p->K * p->N, tw, s);
  if (e == cudaSuccess) e = launch_col_c2c<R>(yhat, p->N, p->K, -1, tw, s);
  if (e == cudaSuccess) e = form_data_term<T>(p, yhat, s);
  if (e == cudaSuccess) p->launches += 3;
  if (e == cudaSuccess && p->adapt_tau > 0 && !is_cd(p)) {
    // the data term is formed again whenever the adaptive penalty changes rho
    if (p->yhat_keep) cudaFreeAsync(p->yhat_keep, s);
    p->yhat_keep = yhat;
  } else {
    cudaFreeAsync(yhat, s);
  }
  CIP_CUDA(p, e);
  p->have_y = true;
  p->avar = std::max(0, forced_avar(p));
  if (p->opt.column_pass == 0 && p->opt.col_tile == 0 && (!is_cd(p) || prior_has_variant(p))) {
    r = autotune<T>(p, s);
    if (r != CIP_OK) return r;
  }
  return reset_state<T>(p, s);
}

template <typename T> PassAArgs<T> passA_args(cip_plan* p, int flags) {
  using C = typename CT<T>::type;
  PassAArgs<T> a;
  a.xh = static_cast<const C*>(p->xh);
  a.qh = static_cast<C*>(p->qh);
  a.u_in = static_cast<const T*>(p->u[p->cur]);
  a.u_out = static_cast<T*>(p->u[p->cur ^ 1]);
  a.tprev = static_cast<T*>(p->tprev);
  a.t_imp = nullptr;
  a.partials = p->partials;
  a.err = p->conv + 1;
  a.tw = static_cast<const C*>(p->tw);
  a.M = smaps(p);
  a.tau = (T)(p->lam / p->rho);
  // the dictionary's column solve works on spectra scaled by 1/N^2 (see convdict.cu)
  a.qscale = is_cd(p) ? (T)(0.5 * p->rho / ((double)p->N * p->N)) : (T)(0.5 * p->rho);
  a.flags = flags;
  a.test_fault = p->test_fault;
  a.variant = p->avar;
  a.lowbuf = low_fix(p) ? static_cast<C*>(p->lowbuf) : nullptr;
  fill_dct<T>(a.dct);
  return a;
}

template <typename T> PassBArgs<T> passB_args(cip_plan* p);

// Whether the kernels of an iteration start programmatically.  In complex128 an SM's few FP64 units make two
// CTAs on one SM take twice as long, and CTAs that start while the other pass still holds SMs are placed two on one:
// where a pass has about one CTA per SM the early start costs far more than the launch latency it hides.  The
// line: the column pass has about a CTA per SM or more, and the prior pass is small (fewer than 5 2^18 pixels in
// all maps; beyond, many tiles per SM even out).  Iterations, early and plain: l1 512^2 x 1 150 and 100 us, x 4
// 212 and 176, x 5 243 and 248; DCT 256^2 x 8 180 and 131, 128^2 x 8 82 and 87; wavelet 512^2 x 1 420 and 330; dictionary
// 64^2 x 8 with 9 filters 109 and 54.  One channel of 256^2 and TV below six gain nothing (TV 256^2 x 4 85 and 87).
// In a batch, early and plain: 4 l1 plans of 512^2 x 2 317 and 288 us an iteration of all, six
// mixed ones 437 and 375.
// The filter update's own kernels: 128^2 x 8 with 9 filters 442 and 360, 256^2 x 3 613 and 584, 64^2 x 3 126 and 136.
template <typename T> Chain chain(const cip_plan* p, cudaStream_t s) {
  if (sizeof(T) == 4 || (is_cd(p) && p->Q > 0)) return {s, true};
  if (is_cd(p) && p->dl_sigma > 0) return {s, p->N < 128};
  const int col = (is_cd(p) ? p->M : 1) * (p->N / 2 + 1);
  const long long px = (long long)smaps(p) * p->N * p->N;
  const bool tv = p->prior == CIP_PRIOR_TV || p->prior == CIP_PRIOR_TV_ISO;
  const int few = p->prior == CIP_PRIOR_WDCT ? 64 : 128;  // the wavelet chain's eleven kernels collide earlier
  return {s, col < few || px >= 5 << 18 || px < (tv ? 6 << 16 : (is_cd(p) ? 1 << 15 : 2 << 16))};
}

// Row transforms between the column-layout row spectra and real rows ([maps][N][N]): x = row IDFT of `spec` into `rows` (read-back, wavelet
// chain), or spec = row DFT of scale * rows.
template <typename T> cudaError_t rows_from_spec(cip_plan* p, const void* spec, int maps, void* rows, Chain s) {
  using C = typename CT<T>::type;
  PassAArgs<T> a{};
  a.xh = static_cast<const C*>(spec);
  a.u_out = static_cast<T*>(rows);
  a.err = p->conv + 1;
  a.tw = static_cast<const C*>(p->tw);
  a.M = maps;
  return launch_rowpass<T>(a, p->N, ROWS_OUT, s);
}
template <typename T>
cudaError_t spec_from_rows(cip_plan* p, const void* rows, int maps, double scale, void* spec, Chain s) {
  using C = typename CT<T>::type;
  PassAArgs<T> a{};
  a.qh = static_cast<C*>(spec);
  a.u_in = static_cast<const T*>(rows);
  a.err = p->conv + 1;
  a.tw = static_cast<const C*>(p->tw);
  a.M = maps;
  a.qscale = (T)(0.5 * scale);  // the 1/2 of the pair extraction
  return launch_rowpass<T>(a, p->N, ROWS_IN, s);
}

// The prior pass: one fused kernel per row tile for TV, DCT and l1; for the wavelet (x) DCT prior
// (not local to a row tile) the chain x = row IDFT, J wavelet levels, channel DCT + shrinkage +
// dual + residual partials, J inverse levels, q-hat = rho row DFT(q).  In import mode x is not
// needed and the chain starts at the shrinkage kernel.
template <typename T> cip_status prior_pass(cip_plan* p, const PassAArgs<T>& a, cudaStream_t stream) {
  const Chain s = chain<T>(p, stream);
  if (p->prior != CIP_PRIOR_WDCT) {
    CIP_LAUNCH(p, launch_passA<T>(a, p->N, prior_pass_kind(p), s));
    return CIP_OK;
  }
  const int N = p->N, M = p->M;
  T* A = static_cast<T*>(p->wbuf[0]);
  T* B = static_cast<T*>(p->wbuf[1]);
  WaveFilt<T> f;
  for (int k = 0; k < 16; ++k) {
    f.h[k] = (T)p->wfilt[k];
    f.g[k] = (T)((k & 1) ? -p->wfilt[15 - k] : p->wfilt[15 - k]);
  }
  // A: coefficients (Mallat layout); B: x, later q; S0, S1: the lowpass band between levels
  T* S[2] = {static_cast<T*>(p->wbuf[2]), static_cast<T*>(p->wbuf[2]) + real_elems(p, M) / 4};
  const int hp = N / 2;
  const size_t hplane = (size_t)hp * hp, plane = (size_t)N * N;
  // levels on bands larger than nf: one tiled kernel each; from the band of side nf down to the
  // 16 x 16 coarse band: one kernel (and one for the inverse), a CTA per channel in shared memory
  const int nf = wave_fuse_band<T>(N);
  int levf = 0;
  while ((N >> levf) > nf) ++levf;
  if (!(a.flags & PA_IMPORT)) {
    CIP_LAUNCH(p, rows_from_spec<T>(p, a.xh, M, B, s));
    for (int lev = 0; lev < levf; ++lev) {
      const T* src = lev == 0 ? B : S[(lev - 1) & 1];
      const int sp = lev == 0 ? N : hp;
      const size_t spl = lev == 0 ? plane : hplane;
      CIP_LAUNCH(p, launch_dwt2_fwd<T>(src, sp, spl, A, N, S[lev & 1], hp, hplane, N >> lev, M, f, s));
    }
    CIP_LAUNCH(p, launch_dwt2_fwd_fused<T>(levf == 0 ? B : S[(levf - 1) & 1], levf == 0 ? N : hp,
                                           levf == 0 ? plane : hplane, A, N, nf, M, f, s));
  }
  ChanDCT<T> cm;
  for (int i = 0; i < 256; ++i) cm.c[i] = (T)p->wcos_h[i];
  CIP_LAUNCH(p, launch_wdct_shrink<T>(A, cm, a.u_in, a.u_out, a.tprev, a.t_imp,
                                      a.partials, p->blocksA, N, M, a.tau, a.flags, s));
  CIP_LAUNCH(p, launch_dwt2_inv_fused<T>(A, N, levf == 0 ? B : S[(levf - 1) & 1], levf == 0 ? N : hp,
                                         levf == 0 ? plane : hplane, nf, M, f, s));
  for (int lev = levf - 1; lev >= 0; --lev) {
    T* dst = lev == 0 ? B : S[(lev - 1) & 1];
    CIP_LAUNCH(p, launch_dwt2_inv<T>(S[lev & 1], hp, hplane, A, N, dst, lev == 0 ? N : hp, lev == 0 ? plane : hplane,
                                     N >> lev, M, f, s));
  }
  CIP_LAUNCH(p, spec_from_rows<T>(p, B, M, p->rho, a.qh, s));
  return CIP_OK;
}

// arguments of the 3D dictionary's per-bin solve
template <typename T> CD3Args<T> cd3_args(cip_plan* p) {
  using C = typename CT<T>::type;
  CD3Args<T> a;
  a.colbuf = static_cast<C*>(p->colbuf);
  a.theta = static_cast<const C*>(p->theta);
  a.p_in = static_cast<const C*>(p->pbuf[p->pcur]);
  a.p_out = static_cast<C*>(p->pbuf[p->pcur ^ 1]);
  a.xb = static_cast<const C*>(p->bhat);
  a.pinv = static_cast<const C*>(p->pinv);
  a.xcol = static_cast<C*>(p->xcol);
  a.N = p->N;
  a.M = p->M;
  a.L = p->L;
  a.rho = (T)p->rho;
  a.n2 = (T)((double)p->N * p->N);
  double re[16], im[16];
  channel_twiddles(p->M, re, im);
  for (int j = 0; j < 16; ++j) a.w[j] = j < p->M ? mk<C>(re[j], im[j]) : mk<C>(0.0, 0.0);
  return a;
}

// the column pass in the plan's chosen form
template <typename T> cip_status column_pass(cip_plan* p, cudaStream_t stream, int mode, int cc) {
  using C = typename CT<T>::type;
  const Chain s = chain<T>(p, stream);
  if (is_cd(p)) {
    // dictionary: column DFT of rho (t - u) over the L*M coefficient maps, the per-(bin, channel)
    // x- and z-update, inverse column DFT of v
    const int S = smaps(p);
    const bool fused = p->Q == 0 && cd_fused_fits<T>(p->N, p->M, p->L);
    if (!fused)
      CIP_LAUNCH(p, launch_cols_fft<T>(static_cast<const C*>(p->qh), static_cast<C*>(p->colbuf),
                                       static_cast<const C*>(p->tw), p->N, S, -1, s));
    if (p->Q > 0) {
      CD3Args<T> a = cd3_args<T>(p);
      CIP_LAUNCH(p, launch_cd3_solve<T>(a, s));
    } else {
      CDArgs<T> a;
      a.colbuf = !fused || p->dl_sigma > 0 ? static_cast<C*>(p->colbuf) : nullptr;
      a.qh = static_cast<const C*>(p->qh);
      a.xh = static_cast<C*>(p->xh);
      a.tw = static_cast<const C*>(p->tw);
      a.theta = static_cast<const C*>(theta_of(p));
      a.th_planes = theta_planes(p);
      a.p_in = static_cast<const C*>(p->pbuf[p->pcur]);
      a.p_out = static_cast<C*>(p->pbuf[p->pcur ^ 1]);
      a.xb = static_cast<const C*>(p->bhat);
      a.pinv = static_cast<const C*>(p->pinv);
      a.xcol = static_cast<C*>(p->xcol);
      a.N = p->N;
      a.M = p->M;
      a.L = p->L;
      a.gs = p->gs;
      a.rho = (T)p->rho;
      a.mu = (T)p->mu;
      a.n2 = (T)((double)p->N * p->N);
      if (fused) CIP_LAUNCH(p, launch_cd_fused<T>(a, s));
      else CIP_LAUNCH(p, launch_cd_solve<T>(a, s));
    }
    if (!fused)
      CIP_LAUNCH(p, launch_cols_fft<T>(static_cast<const C*>(p->colbuf), static_cast<C*>(p->xh),
                                       static_cast<const C*>(p->tw), p->N, S, +1, s));
    p->pcur ^= 1;
    return CIP_OK;
  }
  PassBArgs<T> b = passB_args<T>(p);
  if (mode == 2) {
    if (!p->colbuf) return fail(p, CIP_ERR_STATE, "split column pass selected without its column buffer");
    int n = 0;
    const bool lf = low_fix(p) && p->lowbuf;
    CIP_CUDA(p, launch_passB_split<T>(b, static_cast<C*>(p->colbuf), p->N, s, &n,
                                      lf ? static_cast<const C*>(p->lowbuf) : nullptr,
                                      lf ? static_cast<C*>(p->lowq) : nullptr, (T)p->rho));
    p->launches += n;
  } else {
    (void)cc;
    if constexpr (sizeof(T) == 4) {
      if (mode == 3) {
        CIP_LAUNCH(p, launch_coldirect(b, smaps(p), s));
        return CIP_OK;
      }
    }
    CIP_LAUNCH(p, launch_colpass_fused<T>(b, smaps(p), p->conv + 1, s));
  }
  return CIP_OK;
}

std::mutex g_tune_mu;
// (N, M, dtype, prior, maps of a dictionary's prior pass, forced prior-pass variant or -1) -> (column-pass
// form, fused tile width, prior-pass variant, column-pass form of recorded iterations).  Maps: M L for
// dictionaries, whose row pass runs over them and fills the device or not, and -M L for 3D ones, whose column
// pass overlaps it otherwise (32 maps of 256^2, widths 8 and 16: 2D 28.8 and 22.0 us an iteration, 3D 31.5 and 35.9);
// 0 for the other priors (M says it) and in a line of the file that names none, which then holds for every
// dictionary.
using TuneKey = std::tuple<int, int, int, int, int, int>;
using TuneVal = std::tuple<int, int, int, int>;
std::map<TuneKey, TuneVal> g_tune;
bool g_tune_loaded = false;

// Tuning decisions persist across processes when CIP_TUNE_CACHE names a file (one line per
// decision, appended), so that a profiling run under a tool that serialises launches reuses the
// plain run's choice instead of timing again under different conditions.  Caller holds g_tune_mu.
void tune_cache_load() {
  if (g_tune_loaded) return;
  g_tune_loaded = true;
  const char* path = std::getenv("CIP_TUNE_CACHE");
  if (!path || !*path) return;
  std::ifstream in(path);
  for (std::string line; std::getline(in, line);) {
    std::istringstream f(line);
    int n, m, dt, pr, mode, cc, av, rec, maps;
    if (!(f >> n >> m >> dt >> pr >> mode >> cc >> av)) continue;
    if (!(f >> rec)) rec = mode == 3 ? 1 : mode;  // a line without the recorded form
    if (!(f >> maps) || pr != CIP_PRIOR_CONVDICT) maps = 0;
    g_tune[std::make_tuple(n, m, dt, pr, maps, -1)] = {mode, cc, av, rec};
  }
}
void tune_cache_store(const TuneKey& key, const TuneVal& v) {
  const char* path = std::getenv("CIP_TUNE_CACHE");
  if (!path || !*path || std::get<5>(key) >= 0) return;  // the file holds unforced decisions only
  std::ofstream out(path, std::ios::app);
  out << std::get<0>(key) << ' ' << std::get<1>(key) << ' ' << std::get<2>(key) << ' ' << std::get<3>(key) << ' '
      << std::get<0>(v) << ' ' << std::get<1>(v) << ' ' << std::get<2>(v) << ' ' << std::get<3>(v);
  if (std::get<4>(key) != 0) out << ' ' << std::get<4>(key);
  out << '\n';
}

bool prior_has_variant(const cip_plan* p) {
  return p->dtype == CIP_F32 && p->N >= 256 && p->N <= 1024 &&
         (p->prior == CIP_PRIOR_TV || p->prior == CIP_PRIOR_TV_ISO || p->prior == CIP_PRIOR_DCT8 ||
          p->prior == CIP_PRIOR_L1 || p->prior == CIP_PRIOR_CONVDICT);  // dictionaries: l1 on the codes
}
bool row_prior(const cip_plan* p) { return p->prior >= 0 && prior_pass_kind(p) == PRIOR_L1; }
// T = I at N = 256 has a third width, 32, in which the last two FFT stages merge (rowpass.cu)
bool has_wide_variant(const cip_plan* p) { return prior_has_variant(p) && row_prior(p) && p->N == 256; }
// FFT elements per thread of the prior pass's default kernel (the device-side rule of passA.cu)
int prior_fft_default(const cip_plan* p) {
  if (row_prior(p)) return p->dtype == CIP_F32 ? rowpass_elems<float>(p->N, 0) : rowpass_elems<double>(p->N, 0);
  const bool tv = p->prior == CIP_PRIOR_TV || p->prior == CIP_PRIOR_TV_ISO;
  return (p->dtype == CIP_F32 && p->N <= 1024) ? ((p->N == 512 && !tv) ? 16 : 8) : 16;
}
// the variant the options force: -1 none (autotuned), else 0 / 1
int forced_avar(const cip_plan* p) {
  if (!prior_has_variant(p)) return 0;
  if (p->opt.prior_fft == 0) return p->opt.column_pass != 0 || p->opt.col_tile != 0 ? 0 : -1;
  return p->opt.prior_fft == prior_fft_default(p) ? 0 : 1;
}

// the fused form without the ring is a choice of the autotuner only
bool direct_ok(const cip_plan* p) { return p->dtype == CIP_F32 && !is_cd(p) && coldirect_fits(p->N, p->M); }

template <typename T> void set_colmode(cip_plan* p, int mode, int cc) {
  if (mode == 3 && !direct_ok(p)) mode = 1;  // (a decision read from a file)
  p->colmode = mode;
  if (mode == 1) p->cc = cc;
  p->blocksB = mode != 2 ? p->N / 2 + 1 : p->M * (p->N / 2 + 1);
}
// The form of recorded iterations.  Their kernels share the device with other plans' (batch, server), where
// the form without the ring is no gain (coldirect.cu): they take the faster of the other two, with the
// same prior-pass width and so the same bits as the plan alone.
int rec_form(const cip_plan* p) { return p->colmode == 3 ? p->recmode : p->colmode; }

// Autotuner: times whole iterations (column pass, then prior pass, launched back to back as in
// cip_iterate) for every column-pass form (fused kernel, with and without the ring; split FFT / solve / FFT) and both
// prior-pass FFT widths where a variant exists, on this plan's buffers, and keeps the fastest,
// cached per (N, M, dtype, prior, maps of a dictionary, forced width) for the process: plans with one width (wavelet
// prior, complex128, N < 256, N = 2048) and plans with a forced one time their candidates once as
// well, not at every cip_set_measurements (14 to 28 iterations and the event waits between them:
// 2.5 ms of the 8.6 ms of a 40-iteration 512 x 512 x 10 wavelet reconstruction).  The prior pass reads u[cur] and writes the
// other u buffer and q-hat without moving cur, so repeating an iteration keeps its inputs; the
// state is reset afterwards (cip_set_measurements).  Where the form without the ring wins, the faster of
// the other two at the same width is kept beside it for recorded iterations (rec_form).
template <typename T> cip_status autotune(cip_plan* p, cudaStream_t s) {
  using C = typename CT<T>::type;
  const int fav = forced_avar(p);
  const int kfav = prior_has_variant(p) ? fav : -1;
  const TuneKey key = std::make_tuple(p->N, p->M, (int)p->dtype, p->prior, is_cd(p) ? (p->Q > 0 ? -smaps(p) : smaps(p)) : 0, kfav);
  if (low_fix(p)) {  // the low-column correction of large TV plans is part of the split form
    set_colmode<T>(p, 2, p->cc);
    if (!p->colbuf) CIP_CUDA(p, dmalloc(p, &p->colbuf, col_elems(p, p->M) * sizeof(C)));
    return CIP_OK;
  }
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    tune_cache_load();
    auto it = g_tune.find(key);
    if (it == g_tune.end()) it = g_tune.find(std::make_tuple(p->N, p->M, (int)p->dtype, p->prior, 0, kfav));
    if (it != g_tune.end()) {
      set_colmode<T>(p, std::get<0>(it->second), std::get<1>(it->second));
      p->avar = std::get<2>(it->second);
      p->recmode = std::get<3>(it->second) == 2 ? 2 : 1;
      // a cached choice of the split form still needs this plan's own column buffer
      if (rec_form(p) == 2 && !p->colbuf) CIP_CUDA(p, dmalloc(p, &p->colbuf, col_elems(p, p->M) * sizeof(C)));
      return CIP_OK;
    }
  }
  if (!p->colbuf) CIP_CUDA(p, dmalloc(p, &p->colbuf, col_elems(p, p->M) * sizeof(C)));
  std::vector<TuneVal> cands;
  const int av0 = fav < 0 ? 0 : fav, av1 = fav < 0 ? (has_wide_variant(p) ? 2 : 1) : fav;
  for (int av = av0; av <= av1; ++av) {
    if (is_cd(p)) {  // dictionary plans have one column-pass form; only the prior-pass width is tuned
      cands.push_back({p->colmode, p->cc, av, p->colmode});
      continue;
    }
    if (colpass_fused_fits<T>(p->N, p->M)) {
      cands.push_back({1, 1, av, 1});
      if (direct_ok(p)) cands.push_back({3, 1, av, 1});
    }
    cands.push_back({2, 0, av, 2});
  }
  cudaEvent_t e0, e1;
  CIP_CUDA(p, cudaEventCreate(&e0));
  CIP_CUDA(p, cudaEventCreate(&e1));
  float best = 1e30f, best_rec = 1e30f;
  std::vector<float> took;
  TuneVal pick = {p->colmode, p->cc, p->avar, p->colmode};
  auto iteration = [&]() -> cip_status {
    cip_status st = column_pass<T>(p, s, p->colmode, p->cc);
    if (st != CIP_OK) return st;
    return prior_pass<T>(p, passA_args<T>(p, 0), s);
  };
  for (auto& c : cands) {
    set_colmode<T>(p, std::get<0>(c), std::get<1>(c));
    p->avar = std::get<2>(c);
    cip_status st = CIP_OK;
    for (int w = 0; w < 2 && st == CIP_OK; ++w) st = iteration();
    if (st != CIP_OK) return st;
    cudaEventRecord(e0, s);
    for (int w = 0; w < 5 && st == CIP_OK; ++w) st = iteration();
    if (st != CIP_OK) return st;
    cudaEventRecord(e1, s);
    CIP_CUDA(p, cudaEventSynchronize(e1));
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    took.push_back(ms);
    if (ms < best) {
      best = ms;
      pick = c;
    }
  }
  if (std::get<0>(pick) == 3)
    for (size_t i = 0; i < cands.size(); ++i)
      if (std::get<0>(cands[i]) != 3 && std::get<2>(cands[i]) == std::get<2>(pick) && took[i] < best_rec) {
        best_rec = took[i];
        std::get<3>(pick) = std::get<0>(cands[i]);
      }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  set_colmode<T>(p, std::get<0>(pick), std::get<1>(pick));
  p->avar = std::get<2>(pick);
  p->recmode = std::get<3>(pick) == 2 ? 2 : 1;
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune[key] = pick;
  tune_cache_store(key, pick);
  return CIP_OK;
}

template <typename T> PassBArgs<T> passB_args(cip_plan* p) {
  using C = typename CT<T>::type;
  PassBArgs<T> b;
  b.qh = static_cast<const C*>(p->qh);
  b.xh = static_cast<C*>(p->xh);
  b.pinv = static_cast<const C*>(p->pinv);
  b.bhat = static_cast<const C*>(p->bhat);
  b.tw = static_cast<const C*>(p->tw);
  b.N = p->N;
  b.M = p->M;
  b.plain = p->opt.precision == 1 ? 1 : 0;
  return b;
}

void ensure_events(cip_plan* p) {
  if (!p->evA.empty()) return;
  p->evA.resize(2 * kMaxTimed);
  p->evB.resize(2 * kMaxTimed);
  for (auto& e : p->evA) cudaEventCreate(&e);
  for (auto& e : p->evB) cudaEventCreate(&e);
}

// Online dictionary update: g = the given filters, e = 0, so theta and F(g - e) both start as the
// plan's theta (the filters' DFT formed in FP64 at cip_set_dictionary).
template <typename T> cip_status dict_init(cip_plan* p, cudaStream_t s) {
  using C = typename CT<T>::type;
  const size_t w = (size_t)p->L * col_pitch(p->N) * sizeof(C);
  CIP_CUDA(p, cudaMemcpy2DAsync(p->dl_spec, 2 * w, p->theta, w, w, p->N / 2 + 1, cudaMemcpyDeviceToDevice, s));
  CIP_CUDA(p, cudaMemcpy2DAsync(static_cast<char*>(p->dl_spec) + w, 2 * w, p->theta, w, w, p->N / 2 + 1,
                                cudaMemcpyDeviceToDevice, s));
  CIP_CUDA(p, cudaMemcpyAsync(p->dl_gs, p->filt, (size_t)p->L * p->Pf * p->Pf * sizeof(T), cudaMemcpyDeviceToDevice, s));
  return CIP_OK;
}

template <typename T> DLArgs<T> dl_args(cip_plan* p, bool check) {
  using C = typename CT<T>::type;
  DLArgs<T> a;
  a.zcol = static_cast<const C*>(p->colbuf);
  a.xcol = static_cast<const C*>(p->xcol);
  a.spec = static_cast<C*>(p->dl_spec);
  a.wcol = static_cast<C*>(p->dl_col);
  a.ypart = static_cast<C*>(p->dl_ypart);
  a.yfull = static_cast<C*>(p->dl_yfull);
  a.cnt = p->dl_cnt;
  a.gfac = static_cast<C*>(p->dl_gfac);
  a.gs = static_cast<T*>(p->dl_gs);
  a.rpart = p->dl_part;
  a.spart = p->dl_part + (size_t)(p->N / 2 + 1) * (p->N / kDLBlock);
  a.p_out = static_cast<C*>(p->pbuf[p->pcur]);
  a.tw = static_cast<const C*>(p->tw);
  a.N = p->N;
  a.M = p->M;
  a.L = p->L;
  a.P = p->Pf;
  a.check = check ? 1 : 0;
  a.sigma = (T)p->dl_sigma;
  return a;
}

// One step of the filter ADMM (Section IV-B) after the column pass, from the x and z of that pass
// (x-hat in xcol, z-hat in colbuf, both / N^2): d from Eq. d_admm summed over the channels (Eq.
// sold_3D), g from Eq. g_admm, e from Eq. h_admm; theta = F g and p = sum_l theta_l z_l formed
// again, so that the next x-update sees the updated dictionary (reading R21).  Three launches;
// with `check` they also leave the sums of ||d - g||^2 and ||g - g_prev||^2 in dl_part.
template <typename T> cip_status dict_step(cip_plan* p, cudaStream_t stream, bool check = false) {
  const Chain s = chain<T>(p, stream);
  const DLArgs<T> a = dl_args<T>(p, check);
  CIP_LAUNCH(p, launch_dl_solve<T>(a, s));
  CIP_LAUNCH(p, launch_dl_filter<T>(a, s));
  CIP_LAUNCH(p, launch_dl_spec<T>(a, s));
  return CIP_OK;
}

// Adaptation of sigma (reading R29): the Eq. paramS rule on r = ||d - g|| and s = sigma ||g - g_prev||
// of the step just taken; on a change the scaled dual e is rescaled so that sigma e is unchanged.
template <typename T> cip_status dict_adapt(cip_plan* p, cudaStream_t s) {
  const size_t nr = (size_t)(p->N / 2 + 1) * (p->N / kDLBlock);
  CIP_CUDA(p, cudaMemcpyAsync(p->dl_host, p->dl_part, (nr + p->L) * sizeof(double), cudaMemcpyDeviceToHost, s));
  CIP_CUDA(p, cudaStreamSynchronize(s));
  double r2 = 0.0, s2 = 0.0;
  for (size_t i = 0; i < nr; ++i) r2 += p->dl_host[i];
  for (int l = 0; l < p->L; ++l) s2 += p->dl_host[nr + l];
  const double r = std::sqrt(r2 / ((double)p->N * p->N)), sd = p->dl_sigma * std::sqrt(s2);
  if (!std::isfinite(r) || !std::isfinite(sd)) return fail(p, CIP_ERR_DIVERGED, "filter residuals are not finite");
  double sn = p->dl_sigma;
  if (r > p->dl_mu * sd) sn = p->dl_sigma * p->dl_tau;
  else if (sd > p->dl_mu * r) sn = p->dl_sigma / p->dl_tau;
  if (sn != p->dl_sigma) {
    using C = typename CT<T>::type;
    CIP_LAUNCH(p, launch_dl_rescale<T>(static_cast<C*>(p->dl_spec), p->L, p->N, (T)(p->dl_sigma / sn), s));
    p->dl_sigma = sn;
  }
  return CIP_OK;
}

// Adaptive penalty: rho -> rho_new after a residual check (readings R17, R18).  The scaled
// dual is rescaled so that rho u is unchanged, the factor and the data term are formed again
// for rho_new (the dictionary's factor does not depend on rho), and q of the next x-update is
// formed again from the kept t and the rescaled u by the prior pass in import mode.
template <typename T> cip_status change_rho(cip_plan* p, double rho_new, cudaStream_t s) {
  const size_t n = real_elems(p, smaps(p)) * ncomp_of(p->prior);
  CIP_LAUNCH(p, launch_scale<T>(static_cast<T*>(p->u[p->cur]), n, (T)(p->rho / rho_new), s));
  p->rho = rho_new;
  if (!is_cd(p)) {
    if (!p->yhat_keep) return fail(p, CIP_ERR_STATE, "the adaptive penalty needs cip_set_rho_adaptation before cip_set_measurements");
    cip_status st = form_factor<T>(p, s);
    if (st != CIP_OK) return st;
    CIP_LAUNCH(p, form_data_term<T>(p, setup_buf<T>(p->yhat_keep), s));
  }
  PassAArgs<T> a = passA_args<T>(p, PA_IMPORT);
  a.t_imp = static_cast<const T*>(p->tprev);
  {
    cip_status pst = prior_pass<T>(p, a, s);
    if (pst != CIP_OK) return pst;
  }
  p->cur ^= 1;
  return CIP_OK;
}

// Eq. paramS on the absolute residuals r = ||Tx - t||, s = rho ||t - t_prev|| (sums of squares
// resid[0] and resid[4] of the last check)
double rho_rule(const cip_plan* p, const double* resid) {
  const double ra = std::sqrt(resid[0]), sa = p->rho * std::sqrt(resid[4]);
  if (ra > p->adapt_mu * sa) return p->rho * p->adapt_tau;
  if (sa > p->adapt_mu * ra) return p->rho / p->adapt_tau;
  return p->rho;
}

template <typename T> cip_status iterate_impl(cip_plan* p, int max_iter, double tol, int* done, cudaStream_t s) {
  const bool adapt = p->adapt_tau > 0;
  const bool checks = tol > 0 || adapt;
  if (checks && !p->resid_host)
    CIP_CUDA(p, cudaMallocHost((void**)&p->resid_host, (kNPart + 2) * sizeof(double)));
  const int ce = p->opt.check_every > 0 ? p->opt.check_every : 10;
  int it = 0;
  bool stop = false;
  for (; it < max_iter && !stop; ++it) {
    const bool last = (it == max_iter - 1);
    const int phase = (it + 1) % ce;
    int flags = 0;
    // t is kept on the iteration before a residual check and on the last iteration (so the next
    // call's first dual residual compares against the right t_prev); with the adaptive penalty
    // also on the check itself (q is formed again from it when rho changes)
    if ((checks && phase == ce - 1) || (adapt && phase == 0) || it == max_iter - 2 || last) flags |= PA_STORE_T;
    const bool check = (checks && phase == 0 && it > 0) || last;
    if (check) flags |= PA_RESID;
    // x-update (pass B), then t/u update + next adjoint (pass A)
    const bool timeB = p->timing && p->nB < kMaxTimed;
    if (timeB) cudaEventRecord(p->evB[2 * p->nB], s);
    cip_status cst = column_pass<T>(p, s, p->colmode, p->cc);
    if (cst != CIP_OK) return cst;
    if (timeB) cudaEventRecord(p->evB[2 * p->nB++ + 1], s);
    // sigma adapts after every check_every-th filter step, counted over the plan's iterations
    const bool dl_check = p->dl_sigma > 0 && p->dl_tau > 0 && (p->iteration + 1) % ce == 0;
    if (p->dl_sigma > 0) {
      cst = dict_step<T>(p, s, dl_check);
      if (cst != CIP_OK) return cst;
    }
    PassAArgs<T> a = passA_args<T>(p, flags);
    const bool timeA = p->timing && p->nA < kMaxTimed;
    if (timeA) cudaEventRecord(p->evA[2 * p->nA], s);
    {
      cip_status pst = prior_pass<T>(p, a, s);
      if (pst != CIP_OK) return pst;
    }
    if (timeA) cudaEventRecord(p->evA[2 * p->nA++ + 1], s);
    p->cur ^= 1;
    p->iteration++;
    if (dl_check) {
      cst = dict_adapt<T>(p, s);
      if (cst != CIP_OK) return cst;
    }
    if (check) {
      // the previous iteration stored t only if it ran; otherwise s is not meaningful
      CIP_LAUNCH(p, launch_reduce_partials(p->partials, p->blocksA, p->rho, tol, p->resid, p->conv, s));
      p->resid_valid = true;
      // the penalty adapts at every check, the last iteration of a call included, so that
      // splitting the iterations over several calls does not change the iterates
      const bool adapt_now = adapt && phase == 0 && it > 0;
      if ((tol > 0 && !last) || adapt_now) {
        CIP_CUDA(p, cudaMemcpyAsync(p->resid_host, p->resid, (kNPart + 2) * sizeof(double),
                                    cudaMemcpyDeviceToHost, s));
        int kerr = 0;
        CIP_CUDA(p, cudaMemcpyAsync(&kerr, p->conv + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
        CIP_CUDA(p, cudaStreamSynchronize(s));
        if (kerr) return fail(p, CIP_ERR_TIMEOUT, "a device wait for an asynchronous copy timed out");
        const double r = p->resid_host[kNPart], sr = p->resid_host[kNPart + 1];
        if (!std::isfinite(r) || !std::isfinite(sr)) {
          if (done) *done = it + 1;
          return fail(p, CIP_ERR_DIVERGED, "residuals are not finite");
        }
        if (tol > 0 && !last && r < tol && sr < tol) stop = true;
        if (adapt_now && !stop) {
          const double rho_new = rho_rule(p, p->resid_host);
          if (rho_new != p->rho) {
            cip_status cs = change_rho<T>(p, rho_new, s);
            if (cs != CIP_OK) return cs;
          }
        }
      }
    }
  }
  if (done) *done = it;
  return CIP_OK;
}

// One iteration (column pass, prior pass) enqueued with no host synchronisation and no timing
// events, so that it can be recorded into a CUDA graph.
template <typename T> cip_status enqueue_iteration(cip_plan* p, cudaStream_t s, int flags) {
  cip_status cst = column_pass<T>(p, s, rec_form(p), p->cc);
  if (cst != CIP_OK) return cst;
  if (p->dl_sigma > 0) {
    cst = dict_step<T>(p, s);
    if (cst != CIP_OK) return cst;
  }
  PassAArgs<T> a = passA_args<T>(p, flags);
  {
    cip_status pst = prior_pass<T>(p, a, s);
    if (pst != CIP_OK) return pst;
  }
  p->cur ^= 1;
  p->iteration++;
  if (flags & PA_RESID) {
    CIP_LAUNCH(p, launch_reduce_partials(p->partials, p->blocksA, p->rho, 0.0, p->resid, p->conv, s));
    p->resid_valid = true;
  }
  return CIP_OK;
}

// inverse row DFT of `maps` column-layout row spectra into a caller array (host or device)
template <typename T>
cip_status rows_out(cip_plan* p, const void* rows, int maps, void* out, cudaStream_t s) {
  const size_t bytes = real_elems(p, maps) * sizeof(T);
  if (is_device_ptr(out)) {
    CIP_LAUNCH(p, rows_from_spec<T>(p, rows, maps, out, s));
    return CIP_OK;
  }
  void* tmp = nullptr;
  CIP_CUDA(p, cudaMallocAsync(&tmp, bytes, s));
  cudaError_t e = rows_from_spec<T>(p, rows, maps, tmp, s);
  if (e == cudaSuccess) p->launches++;
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, tmp, bytes, cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(tmp, s);
  CIP_CUDA(p, e);
  CIP_CUDA(p, cudaStreamSynchronize(s));
  return CIP_OK;
}

template <typename T> cip_status get_x_impl(cip_plan* p, void* x, cudaStream_t s) {
  using C = typename CT<T>::type;
  if (!is_cd(p)) return rows_out<T>(p, p->xh, p->M, x, s);
  // dictionary: x-hat is kept per bin; inverse column DFT to row spectra first
  void* rows = nullptr;
  CIP_CUDA(p, cudaMallocAsync(&rows, col_elems(p, p->M) * sizeof(C), s));
  cudaError_t e = launch_cols_fft<T>(static_cast<const C*>(p->xcol), static_cast<C*>(rows),
                                     static_cast<const C*>(p->tw), p->N, p->M, +1, s);
  if (e != cudaSuccess) {
    cudaFreeAsync(rows, s);
    CIP_CUDA(p, e);
  }
  p->launches++;
  cip_status st = rows_out<T>(p, rows, p->M, x, s);
  cudaFreeAsync(rows, s);
  return st;
}

// dictionary state import: p = sum_l theta_l F z_l / N^2 from coefficient maps z [M][L][N][N]
template <typename T> cip_status import_z(cip_plan* p, const void* z, cudaStream_t s) {
  using C = typename CT<T>::type;
  const int S = smaps(p);
  Staging sz;
  const void* dz = nullptr;
  cip_status r = stage_in(p, z, real_elems(p, S) * sizeof(T), s, sz, &dz);
  if (r != CIP_OK) return r;
  // row DFT into xh (overwritten by the next column pass), column DFT into colbuf
  CIP_LAUNCH(p, spec_from_rows<T>(p, dz, S, 1.0, p->xh, s));
  CIP_LAUNCH(p, launch_cols_fft<T>(static_cast<const C*>(p->xh), static_cast<C*>(p->colbuf),
                                   static_cast<const C*>(p->tw), p->N, S, -1, s));
  if (p->Q > 0) {
    CD3Args<T> a = cd3_args<T>(p);
    CIP_LAUNCH(p, launch_p3_from_z<T>(static_cast<const C*>(p->colbuf), static_cast<const C*>(p->theta),
                                      static_cast<C*>(p->pbuf[p->pcur]), a, 0.0, s));
    return CIP_OK;
  }
  CIP_LAUNCH(p, launch_p_from_z<T>(static_cast<const C*>(p->colbuf), static_cast<const C*>(theta_of(p)),
                                   static_cast<C*>(p->pbuf[p->pcur]), p->N, p->M, p->L, s, 0.0, theta_planes(p)));
  return CIP_OK;
}

cip_status copy_out(cip_plan* p, void* dst, const void* src, size_t bytes, cudaStream_t s) {
  const bool dev = is_device_ptr(dst);
  CIP_CUDA(p, cudaMemcpyAsync(dst, src, bytes, dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
  if (!dev) CIP_CUDA(p, cudaStreamSynchronize(s));
  return CIP_OK;
}

template <typename T> cip_status import_impl(cip_plan* p, const void* t, const void* u, cudaStream_t s) {
  const size_t bytes = real_elems(p, smaps(p)) * ncomp_of(p->prior) * sizeof(T);
  Staging st1, st2;
  const void *dt = nullptr, *du = nullptr;
  cip_status r = stage_in(p, t, bytes, s, st1, &dt);
  if (r != CIP_OK) return r;
  r = stage_in(p, u, bytes, s, st2, &du);
  if (r != CIP_OK) return r;
  CIP_CUDA(p, cudaMemcpyAsync(p->u[p->cur], du, bytes, cudaMemcpyDeviceToDevice, s));
  CIP_CUDA(p, cudaMemcpyAsync(p->tprev, dt, bytes, cudaMemcpyDeviceToDevice, s));
  PassAArgs<T> a = passA_args<T>(p, PA_IMPORT);
  a.t_imp = static_cast<const T*>(dt);
  {
    cip_status pst = prior_pass<T>(p, a, s);
    if (pst != CIP_OK) return pst;
  }
  p->cur ^= 1;
  p->iteration = 0;
  p->resid_valid = false;
  return CIP_OK;
}

#define DISPATCH_T(p, call_f32, call_f64) ((p)->dtype == CIP_F32 ? (call_f32) : (call_f64))

cip_status check_ready(cip_plan* p, bool need_y) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (p->prior < 0) return fail(p, CIP_ERR_STATE, "cip_set_prior has not been called");
  if (is_cd(p) && !p->theta) return fail(p, CIP_ERR_STATE, "cip_set_dictionary has not been called");
  if (!p->have_psfs) return fail(p, CIP_ERR_STATE, "cip_set_psfs has not been called");
  if (need_y && !p->have_y) return fail(p, CIP_ERR_STATE, "cip_set_measurements has not been called");
  return CIP_OK;
}

}  // namespace

extern "C" {

const char* cip_version(void) { return "cip 0.1 (sm_103a)"; }

cip_status cip_wavelet_lowpass(int p, double* h) {
  if (!h || p < 1 || p > 8) return CIP_ERR_INVALID_ARG;
  return symlet_lowpass(p, h) ? CIP_OK : CIP_ERR_INVALID_ARG;
}

const char* cip_status_string(cip_status s) {
  switch (s) {
    case CIP_OK: return "ok";
    case CIP_ERR_INVALID_ARG: return "invalid argument";
    case CIP_ERR_UNSUPPORTED: return "unsupported size or option";
    case CIP_ERR_OOM: return "out of device memory";
    case CIP_ERR_CUDA: return "CUDA error";
    case CIP_ERR_STATE: return "call out of order";
    case CIP_ERR_TIMEOUT: return "device wait timed out";
    case CIP_ERR_DIVERGED: return "iteration diverged";
  }
  return "unknown status";
}

const char* cip_last_error(const cip_plan* plan) { return plan ? plan->err.c_str() : g_create_error.c_str(); }

size_t cip_plan_bytes(int N, int K, int M, cip_dtype dtype, cip_prior prior) {
  if (!valid_n(N) || K < 1 || M < 1) return 0;
  const size_t e = dtype == CIP_F64 ? 8 : 4;
  const size_t P = (size_t)half_pitch(N), half = (size_t)N * P * 2 * e, real = (size_t)N * N * e;
  const size_t nc = prior_is_tv(prior) ? 2 : 1;
  const size_t colc = (size_t)(N / 2 + 1) * col_pitch(N) * 2 * e;  // one map in the column layout
  size_t b = 0;
  b += 3 * M * colc;                          // xh, qh, bhat
  b += M * colc;                              // split column buffer (autotuner)
  b += (size_t)M * (M + 1) / 2 * half;        // pinv
  b += (size_t)M * (M + 1) / 2 * N * P * 16;  // FP64 copy of pinv (data term at set_measurements)
  b += 3 * nc * M * real;                     // u[2], tprev
  b += (size_t)K * M * N * P * 16;            // FP64 PSF spectra
  b += (size_t)kTwAll * (16 + 2 * e) + N * 8;   // tables
  b += (size_t)(N / 2) * M * kNPart * 8 + 4096;
  if (prior == CIP_PRIOR_WDCT) b += 5 * M * real / 2 + (size_t)M * M * e;  // wavelet work planes, DCT matrix
  return b;
}

cip_status cip_plan_create(cip_plan** out, int N, int K, int M, cip_dtype dtype, const cip_options* opt) {
  return cip_plan_create_on_stream(out, N, K, M, dtype, opt, nullptr);
}

cip_status cip_plan_create_on_stream(cip_plan** out, int N, int K, int M, cip_dtype dtype, const cip_options* opt,
                                     void* stream) {
  if (!out) return fail(nullptr, CIP_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (!valid_n(N)) return fail(nullptr, CIP_ERR_UNSUPPORTED, "N must be a power of two in [64, 2048]");
  if (K < 1 || K > 16 || M < 1 || M > 16) return fail(nullptr, CIP_ERR_UNSUPPORTED, "K and M must be in [1, 16]");
  if (dtype != CIP_F32 && dtype != CIP_F64) return fail(nullptr, CIP_ERR_INVALID_ARG, "bad dtype");
  cip_plan* p = new cip_plan();
  p->ast = static_cast<cudaStream_t>(stream);
  p->N = N;
  p->K = K;
  p->M = M;
  p->P = half_pitch(N);
  p->dtype = dtype;
  p->esz = dtype == CIP_F64 ? 8 : 4;
  if (opt) p->opt = *opt;
  const size_t ce = 2 * p->esz;  // complex element size
  const int cc = p->opt.col_tile;
  if (cc != 0 && cc != 1 && cc != 2 && cc != 4) {
    delete p;
    return fail(nullptr, CIP_ERR_INVALID_ARG, "col_tile must be 0, 1, 2 or 4");
  }
  p->cc = cc == 0 ? 1 : cc;
  if (p->opt.prior_fft != 0 && p->opt.prior_fft != 8 && p->opt.prior_fft != 16) {
    delete p;
    return fail(nullptr, CIP_ERR_INVALID_ARG, "prior_fft must be 0, 8 or 16");
  }
  const bool fused_ok = dtype == CIP_F64 ? colpass_fused_fits<double>(N, M) : colpass_fused_fits<float>(N, M);
  if (p->opt.column_pass == 1 && !fused_ok) {
    delete p;
    return fail(nullptr, CIP_ERR_UNSUPPORTED, "the fused column pass does not fit in shared memory for this N, M and dtype");
  }
  p->blocksB = N / 2 + 1;
  if (p->opt.precision != 0 && (p->opt.precision != 1 || dtype != CIP_F32)) {
    delete p;
    return fail(nullptr, CIP_ERR_INVALID_ARG, "precision must be 0, or 1 (plain FP32) for CIP_F32 plans");
  }
  p->colmode = (p->opt.column_pass == 2 || !fused_ok) ? 2 : 1;
  if (p->colmode == 2) p->blocksB = M * (N / 2 + 1);
  if (p->opt.column_pass < 0 || p->opt.column_pass > 2) {
    delete p;
    return fail(nullptr, CIP_ERR_INVALID_ARG, "column_pass must be 0, 1 or 2");
  }
#define ALLOC(ptr, bytes)                                                                       \
  do {                                                                                          \
    cudaError_t e_ = cudaMallocAsync((void**)&(ptr), (bytes), p->ast);                          \
    if (e_ != cudaSuccess) {                                                                    \
      cip_plan_destroy(p);                                                                      \
      return fail(nullptr, CIP_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e_)); \
    }                                                                                           \
  } while (0)
  ALLOC(p->xh, col_elems(p, M) * ce);
  ALLOC(p->qh, col_elems(p, M) * ce);
  ALLOC(p->bhat, col_elems(p, M) * ce);
  ALLOC(p->tw, (size_t)kTwAll * ce);
  ALLOC(p->tw64, (size_t)kTwAll * 16);  // complex double-float (complex64 plans) or complex128
  ALLOC(p->gs, (size_t)N * sizeof(double));
  ALLOC(p->resid, (kNPart + 2) * sizeof(double));
  ALLOC(p->conv, 2 * sizeof(int));  // [0] converged, [1] a kernel's bounded wait gave up
  ALLOC(p->pinv_list, (1 + kPinvListCap) * sizeof(int));
  if (p->colmode == 2) ALLOC(p->colbuf, col_elems(p, M) * ce);
#undef ALLOC
  std::vector<double> re, im;
  twiddles(re, im);
  std::vector<double2> t64(kTwAll);
  std::vector<float2> t32(kTwAll);
  std::vector<cdf> tdf(kTwAll);
  for (int k = 0; k < kTwAll; ++k) {
    t64[k] = make_double2(re[k], im[k]);
    tdf[k].x = df64_from_host(re[k]);
    tdf[k].y = df64_from_host(im[k]);
    t32[k] = make_float2((float)re[k], (float)im[k]);
  }
  std::vector<double> gs(N);
  for (int k = 0; k < N; ++k) {
    // 4 sin^2(pi k / N), exact zero at k = 0
    const double sn = std::sin(M_PI * (double)k / (double)N);
    gs[k] = 4.0 * sn * sn;
  }
  gs[0] = 0.0;
  cudaError_t e = cudaStreamSynchronize(p->ast);  // buffers valid on every stream from here on
  if (e == cudaSuccess)
    e = dtype == CIP_F64 ? cudaMemcpy(p->tw64, t64.data(), kTwAll * sizeof(double2), cudaMemcpyHostToDevice)
                         : cudaMemcpy(p->tw64, tdf.data(), kTwAll * sizeof(cdf), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = dtype == CIP_F64 ? cudaMemcpy(p->tw, t64.data(), kTwAll * sizeof(double2), cudaMemcpyHostToDevice)
                         : cudaMemcpy(p->tw, t32.data(), kTwAll * sizeof(float2), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(p->gs, gs.data(), N * sizeof(double), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cip_plan_destroy(p);
    return fail(nullptr, CIP_ERR_CUDA, std::string("cudaMemcpy: ") + cudaGetErrorString(e));
  }
  *out = p;
  return CIP_OK;
}

cip_status cip_plan_destroy(cip_plan* p) {
  if (!p) return CIP_ERR_INVALID_ARG;
  void* bufs[] = {p->lowbuf, p->lowq, p->w3, p->theta, p->pbuf[0], p->pbuf[1], p->xcol, p->yhat_keep, p->filt, p->dl_spec, p->dl_col, p->dl_ypart, p->dl_yfull, p->dl_gfac, p->dl_gs, p->dl_cnt, p->dl_part, p->wbuf[0], p->wbuf[1], p->wbuf[2], p->wcos,
                  p->xh, p->qh, p->u[0], p->u[1], p->tprev, p->pinv, p->pinv64, p->bhat, p->colbuf, p->lam64, p->tw, p->tw64,
                  p->gs, p->partials, p->resid, p->conv, p->pinv_list};
  for (void* b : bufs)
    if (b) cudaFreeAsync(b, p->ast);
  if (p->resid_host) cudaFreeHost(p->resid_host);
  if (p->dl_host) cudaFreeHost(p->dl_host);
  for (auto& ev : p->evA) cudaEventDestroy(ev);
  for (auto& ev : p->evB) cudaEventDestroy(ev);
  delete p;
  return CIP_OK;
}

cip_status cip_set_prior(cip_plan* p, cip_prior prior, double lambda, double rho, double beta, void* stream) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (prior != CIP_PRIOR_TV && prior != CIP_PRIOR_DCT8 && prior != CIP_PRIOR_L1 && prior != CIP_PRIOR_CONVDICT &&
      prior != CIP_PRIOR_TV_ISO && prior != CIP_PRIOR_WDCT)
    return fail(p, CIP_ERR_INVALID_ARG, "unknown prior");
  if (prior == CIP_PRIOR_WDCT && !symlet_lowpass(8, p->wfilt))
    return fail(p, CIP_ERR_CUDA, "Symmlet-8 filter construction failed");
  if (!(lambda > 0) || !(rho > 0) || !(beta > 0)) return fail(p, CIP_ERR_INVALID_ARG, "lambda, rho, beta must be > 0");
  const int kind = tile_kind(prior);
  const int rows = p->dtype == CIP_F64 ? passA_rows<double>(p->N, kind) : passA_rows<float>(p->N, kind);
  if (p->N % rows != 0) return fail(p, CIP_ERR_UNSUPPORTED, "image size not a multiple of the row tile");
  const size_t smA = p->dtype == CIP_F64 ? passA_smem<double>(p->N, kind) : passA_smem<float>(p->N, kind);
  int dev = 0, smem_optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (smem_optin > 0 && smA > (size_t)smem_optin) return fail(p, CIP_ERR_UNSUPPORTED, "prior pass tile too large");
  p->prior = prior;
  p->lam = lambda;
  p->rho = rho;
  p->beta = beta;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  p->have_y = false;  // the data term depends on the factor: set_measurements again
  return DISPATCH_T(p, do_set_prior<float>(p, s), do_set_prior<double>(p, s));
}

cip_status cip_set_psfs(cip_plan* p, const void* h, void* stream) {
  if (!p || !h) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  if (p->prior < 0) return fail(p, CIP_ERR_STATE, "cip_set_prior must precede cip_set_psfs");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  cip_status r = DISPATCH_T(p, do_set_psfs<float>(p, h, s), do_set_psfs<double>(p, h, s));
  if (r == CIP_OK) p->have_y = false;
  return r;
}

cip_status cip_set_measurements(cip_plan* p, const void* y, void* stream) {
  if (!p || !y) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, do_set_y<float>(p, y, s), do_set_y<double>(p, y, s));
}

cip_status cip_reset_state(cip_plan* p, void* stream) {
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, reset_state<float>(p, s), reset_state<double>(p, s));
}

cip_status cip_iterate(cip_plan* p, int max_iter, double tol, int* iters_done, void* stream) {
  cip_status r = check_ready(p, true);
  if (r != CIP_OK) return r;
  if (max_iter < 0) return fail(p, CIP_ERR_INVALID_ARG, "max_iter < 0");
  if (p->timing) ensure_events(p);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, iterate_impl<float>(p, max_iter, tol, iters_done, s),
                    iterate_impl<double>(p, max_iter, tol, iters_done, s));
}

cip_status cip_get_x(cip_plan* p, void* x, void* stream) {
  if (!p || !x) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, get_x_impl<float>(p, x, s), get_x_impl<double>(p, x, s));
}

cip_status cip_get_u(cip_plan* p, void* u, void* stream) {
  if (!p || !u) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  p->ast = static_cast<cudaStream_t>(stream);
  return copy_out(p, u, p->u[p->cur], real_elems(p, smaps(p)) * ncomp_of(p->prior) * p->esz, p->ast);
}

cip_status cip_set_dictionary_3d(cip_plan* p, const void* filters, int L, int Q, int P, void* stream) {
  if (!p || !filters) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  if (!is_cd(p)) return fail(p, CIP_ERR_STATE, "cip_set_prior(CIP_PRIOR_CONVDICT) must precede cip_set_dictionary_3d");
  if (p->opt.precision != 0) return fail(p, CIP_ERR_UNSUPPORTED, "the plain FP32 method covers analysis priors only");
  if (L < 1 || L > 32) return fail(p, CIP_ERR_UNSUPPORTED, "L must be in [1, 32]");
  if (Q < 1 || Q > p->M) return fail(p, CIP_ERR_INVALID_ARG, "filter depth must be in [1, M]");
  if (P < 1 || P > p->N) return fail(p, CIP_ERR_INVALID_ARG, "filter size must be in [1, N]");
  if (p->dl_sigma > 0) return fail(p, CIP_ERR_UNSUPPORTED, "the online dictionary update covers 2D filters only");
  if (p->mu > 0) return fail(p, CIP_ERR_UNSUPPORTED, "the code gradient penalty covers 2D filters only");
  const bool fits = p->dtype == CIP_F32 ? cd3_fits<float>(p->M, L) : cd3_fits<double>(p->M, L);
  if (!fits) return fail(p, CIP_ERR_UNSUPPORTED, "M * L too large for the 3D dictionary's per-bin tile");
  p->L = L;
  p->Pf = P;
  p->Q = Q;
  p->have_y = false;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, do_set_dictionary<float>(p, filters, s), do_set_dictionary<double>(p, filters, s));
}

cip_status cip_set_dictionary(cip_plan* p, const void* filters, int L, int P, void* stream) {
  if (!p || !filters) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  p->Q = 0;
  if (!is_cd(p)) return fail(p, CIP_ERR_STATE, "cip_set_prior(CIP_PRIOR_CONVDICT) must precede cip_set_dictionary");
  if (p->opt.precision != 0) return fail(p, CIP_ERR_UNSUPPORTED, "the plain FP32 method covers analysis priors only");
  if (L < 1 || L > 32) return fail(p, CIP_ERR_UNSUPPORTED, "L must be in [1, 32]");
  if (P < 1 || P > p->N) return fail(p, CIP_ERR_INVALID_ARG, "filter size must be in [1, N]");
  p->L = L;
  p->Pf = P;
  p->have_y = false;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, do_set_dictionary<float>(p, filters, s), do_set_dictionary<double>(p, filters, s));
}

cip_status cip_set_code_gradient_weight(cip_plan* p, double mu) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (!is_cd(p)) return fail(p, CIP_ERR_STATE, "the gradient penalty applies to CIP_PRIOR_CONVDICT plans only");
  if (!(mu >= 0.0) || !std::isfinite(mu)) return fail(p, CIP_ERR_INVALID_ARG, "mu must be finite and >= 0");
  if (mu > 0 && p->Q > 0) return fail(p, CIP_ERR_UNSUPPORTED, "the code gradient penalty covers 2D filters only");
  p->mu = mu;
  return CIP_OK;
}

cip_status cip_set_dictionary_learning(cip_plan* p, double sigma, void* stream) {
  if (!p) return CIP_ERR_INVALID_ARG;
  cip_status r = CIP_OK;
  if (!is_cd(p) || !p->theta)
    return fail(p, CIP_ERR_STATE, "dictionary learning needs a CIP_PRIOR_CONVDICT plan after cip_set_dictionary");
  if (!(sigma >= 0.0) || !std::isfinite(sigma)) return fail(p, CIP_ERR_INVALID_ARG, "sigma must be finite and >= 0");
  if (sigma > 0 && p->M > 8) return fail(p, CIP_ERR_UNSUPPORTED, "dictionary learning supports M <= 8 channels");
  if (sigma > 0 && p->Q > 0) return fail(p, CIP_ERR_UNSUPPORTED, "the online dictionary update covers 2D filters only");
  if (sigma > 0 && p->Pf > kDLMaxP) return fail(p, CIP_ERR_UNSUPPORTED, "dictionary learning supports filters up to 32 x 32");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  const size_t ce = 2 * p->esz;
  if (sigma == 0.0) {
    if (p->dl_sigma > 0) {  // the learnt theta becomes the plan's dictionary
      const size_t w = (size_t)p->L * col_pitch(p->N) * ce;
      CIP_CUDA(p, cudaMemcpy2DAsync(p->theta, w, p->dl_spec, 2 * w, w, p->N / 2 + 1, cudaMemcpyDeviceToDevice, s));
      CIP_CUDA(p, cudaMemcpyAsync(p->filt, p->dl_gs, (size_t)p->L * p->Pf * p->Pf * p->esz, cudaMemcpyDeviceToDevice, s));
    }
    p->dl_sigma = 0.0;
    return CIP_OK;
  }
  r = alloc_dict(p);
  if (r != CIP_OK) return r;
  const bool was_on = p->dl_sigma > 0;
  p->dl_sigma = sigma;
  if (was_on) return CIP_OK;  // a new sigma keeps the filters learnt so far
  return DISPATCH_T(p, dict_init<float>(p, s), dict_init<double>(p, s));
}

cip_status cip_get_dictionary(cip_plan* p, void* filters, void* stream) {
  if (!p || !filters) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  if (!is_cd(p) || !(p->dl_sigma > 0))
    return fail(p, CIP_ERR_STATE, "the filters change only with cip_set_dictionary_learning on");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  const size_t bytes = (size_t)p->L * p->Pf * p->Pf * p->esz;
  return copy_out(p, filters, p->dl_gs, bytes, s);
}

cip_status cip_set_rho_adaptation(cip_plan* p, double tau, double mu) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (tau == 0.0) {
    p->adapt_tau = p->adapt_mu = 0.0;
    return CIP_OK;
  }
  if (!(tau > 1.0) || !(mu > 1.0) || !std::isfinite(tau) || !std::isfinite(mu))
    return fail(p, CIP_ERR_INVALID_ARG, "tau and mu must be finite and > 1 (or tau = 0 to turn adaptation off)");
  if (p->have_y && !is_cd(p) && !p->yhat_keep)
    return fail(p, CIP_ERR_STATE, "cip_set_rho_adaptation must precede cip_set_measurements");
  p->adapt_tau = tau;
  p->adapt_mu = mu;
  return CIP_OK;
}

cip_status cip_set_sigma_adaptation(cip_plan* p, double tau, double mu) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (tau == 0.0) {
    p->dl_tau = p->dl_mu = 0.0;
    return CIP_OK;
  }
  if (!(tau > 1.0) || !(mu > 1.0) || !std::isfinite(tau) || !std::isfinite(mu))
    return fail(p, CIP_ERR_INVALID_ARG, "tau and mu must be finite and > 1 (or tau = 0 to turn adaptation off)");
  p->dl_tau = tau;
  p->dl_mu = mu;
  return CIP_OK;
}

cip_status cip_get_sigma(cip_plan* p, double* sigma) {
  if (!p || !sigma) return CIP_ERR_INVALID_ARG;
  *sigma = p->dl_sigma;
  return CIP_OK;
}

cip_status cip_get_rho(cip_plan* p, double* rho) {
  if (!p || !rho) return CIP_ERR_INVALID_ARG;
  *rho = p->rho;
  return CIP_OK;
}

cip_status cip_get_coefficients(cip_plan* p, void* z, void* stream) {
  if (!p || !z) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  if (!is_cd(p)) return fail(p, CIP_ERR_STATE, "coefficient maps exist only for CIP_PRIOR_CONVDICT");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, rows_out<float>(p, p->xh, smaps(p), z, s), rows_out<double>(p, p->xh, smaps(p), z, s));
}

cip_status cip_state_import_coefficients(cip_plan* p, const void* z, const void* t, const void* u, void* stream) {
  if (!p || !z || !t || !u) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  if (!is_cd(p)) return fail(p, CIP_ERR_STATE, "coefficient maps exist only for CIP_PRIOR_CONVDICT");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  r = DISPATCH_T(p, import_z<float>(p, z, s), import_z<double>(p, z, s));
  if (r != CIP_OK) return r;
  return DISPATCH_T(p, import_impl<float>(p, t, u, s), import_impl<double>(p, t, u, s));
}

cip_status cip_get_residuals(cip_plan* p, double* r_rel, double* s_rel) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (!p->resid_valid) return fail(p, CIP_ERR_STATE, "no residuals computed since the last reset");
  double h[kNPart + 2];
  int kerr = 0;
  CIP_CUDA(p, cudaMemcpy(h, p->resid, sizeof(h), cudaMemcpyDeviceToHost));
  CIP_CUDA(p, cudaMemcpy(&kerr, p->conv + 1, sizeof(int), cudaMemcpyDeviceToHost));
  if (kerr) return fail(p, CIP_ERR_TIMEOUT, "a device wait for an asynchronous copy timed out");
  if (r_rel) *r_rel = h[kNPart];
  if (s_rel) *s_rel = h[kNPart + 1];
  return CIP_OK;
}

cip_status cip_get_iteration(cip_plan* p, int* iteration) {
  if (!p || !iteration) return CIP_ERR_INVALID_ARG;
  *iteration = p->iteration;
  return CIP_OK;
}

cip_status cip_state_import(cip_plan* p, const void* t, const void* u, void* stream) {
  if (!p || !t || !u) return fail(p, CIP_ERR_INVALID_ARG, "null argument");
  cip_status r = check_ready(p, false);
  if (r != CIP_OK) return r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  return DISPATCH_T(p, import_impl<float>(p, t, u, s), import_impl<double>(p, t, u, s));
}

// device buffers that make up the ADMM state, in checkpoint order
static std::vector<std::pair<void*, size_t>> state_segments(cip_plan* p) {
  const int S = smaps(p);
  const size_t hb = col_elems(p, S) * 2 * p->esz;
  const size_t ub = real_elems(p, S) * ncomp_of(p->prior) * p->esz;
  std::vector<std::pair<void*, size_t>> seg = {{p->xh, hb}, {p->qh, hb}, {p->u[p->cur], ub}, {p->tprev, ub}};
  if (p->lowbuf) seg.push_back({p->lowbuf, 2 * low_elems(p) * 2 * p->esz});  // the next x-update's low columns
  if (is_cd(p)) {
    seg.push_back({p->pbuf[p->pcur], col_elems(p, p->M) * 2 * p->esz});
    seg.push_back({p->xcol, col_elems(p, p->M) * 2 * p->esz});
  }
  if (p->dl_sigma > 0) {  // the dictionary being learnt is part of the state
    seg.push_back({p->dl_spec, col_elems(p, 2 * p->L) * 2 * p->esz});
    seg.push_back({p->dl_gs, (size_t)p->L * p->Pf * p->Pf * p->esz});
  }
  return seg;
}

// checkpoint header: iteration count and the filter ADMM's penalty (0 while the update is off)
struct StateHeader {
  int iteration;
  int reserved;
  double sigma;
};
constexpr size_t kStateHeader = sizeof(StateHeader);

cip_status cip_state_size(cip_plan* p, size_t* bytes) {
  if (!p || !bytes) return CIP_ERR_INVALID_ARG;
  if (p->prior < 0) return fail(p, CIP_ERR_STATE, "cip_set_prior has not been called");
  if (is_cd(p) && !p->theta) return fail(p, CIP_ERR_STATE, "cip_set_dictionary has not been called");
  size_t n = kStateHeader;
  for (auto& sgm : state_segments(p)) n += sgm.second;
  *bytes = n;
  return CIP_OK;
}

cip_status cip_state_export(cip_plan* p, void* buf, void* stream) {
  size_t total = 0;
  cip_status r = cip_state_size(p, &total);
  if (r != CIP_OK) return r;
  if (!buf) return fail(p, CIP_ERR_INVALID_ARG, "null buffer");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  const bool dev = is_device_ptr(buf);
  const cudaMemcpyKind k = dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  char* b = static_cast<char*>(buf);
  StateHeader hdr{p->iteration, 0, p->dl_sigma};
  if (dev) {
    CIP_CUDA(p, cudaMemcpyAsync(b, &hdr, sizeof(hdr), cudaMemcpyHostToDevice, s));
    CIP_CUDA(p, cudaStreamSynchronize(s));  // hdr lives on this stack frame
  } else {
    std::memcpy(b, &hdr, sizeof(hdr));
  }
  size_t off = sizeof(hdr);
  for (auto& sgm : state_segments(p)) {
    CIP_CUDA(p, cudaMemcpyAsync(b + off, sgm.first, sgm.second, k, s));
    off += sgm.second;
  }
  CIP_CUDA(p, cudaStreamSynchronize(s));
  return CIP_OK;
}

cip_status cip_state_restore(cip_plan* p, const void* buf, void* stream) {
  size_t total = 0;
  cip_status r = cip_state_size(p, &total);
  if (r != CIP_OK) return r;
  if (!buf) return fail(p, CIP_ERR_INVALID_ARG, "null buffer");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  p->ast = s;
  const bool dev = is_device_ptr(buf);
  const cudaMemcpyKind k = dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const char* b = static_cast<const char*>(buf);
  StateHeader hdr;
  if (dev) {
    CIP_CUDA(p, cudaMemcpyAsync(&hdr, b, sizeof(hdr), cudaMemcpyDeviceToHost, s));
    CIP_CUDA(p, cudaStreamSynchronize(s));
  } else {
    std::memcpy(&hdr, b, sizeof(hdr));
  }
  size_t off = sizeof(hdr);
  for (auto& sgm : state_segments(p)) {
    CIP_CUDA(p, cudaMemcpyAsync(sgm.first, b + off, sgm.second, k, s));
    off += sgm.second;
  }
  CIP_CUDA(p, cudaStreamSynchronize(s));
  p->iteration = hdr.iteration;
  if (p->dl_sigma > 0 && hdr.sigma > 0) p->dl_sigma = hdr.sigma;  // the adapted penalty of the filter ADMM
  p->resid_valid = false;
  return CIP_OK;
}

cip_status cip_set_timing(cip_plan* p, int on) {
  if (!p) return CIP_ERR_INVALID_ARG;
  p->timing = on != 0;
  p->nA = p->nB = 0;
  if (p->timing) ensure_events(p);  // created here, outside any timed sequence of iterations
  return CIP_OK;
}

cip_status cip_get_timing(cip_plan* p, double* a_ms, int* a_n, double* b_ms, int* b_n) {
  if (!p) return CIP_ERR_INVALID_ARG;
  double ta = 0, tb = 0;
  for (int i = 0; i < p->nA; ++i) {
    float ms = 0;
    CIP_CUDA(p, cudaEventSynchronize(p->evA[2 * i + 1]));
    CIP_CUDA(p, cudaEventElapsedTime(&ms, p->evA[2 * i], p->evA[2 * i + 1]));
    ta += ms;
  }
  for (int i = 0; i < p->nB; ++i) {
    float ms = 0;
    CIP_CUDA(p, cudaEventSynchronize(p->evB[2 * i + 1]));
    CIP_CUDA(p, cudaEventElapsedTime(&ms, p->evB[2 * i], p->evB[2 * i + 1]));
    tb += ms;
  }
  if (a_ms) *a_ms = ta;
  if (a_n) *a_n = p->nA;
  if (b_ms) *b_ms = tb;
  if (b_n) *b_n = p->nB;
  p->nA = p->nB = 0;
  return CIP_OK;
}

cip_status cip_set_test_fault(cip_plan* p, int kind) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (kind != 0 && kind != 1) return fail(p, CIP_ERR_INVALID_ARG, "test fault kind must be 0 or 1");
  p->test_fault = kind;
  return CIP_OK;
}

cip_status cip_get_launches(cip_plan* p, unsigned long long* n) {
  if (!p || !n) return CIP_ERR_INVALID_ARG;
  *n = p->launches;
  return CIP_OK;
}

cip_status cip_get_prior_fft(cip_plan* p, int* elems) {
  if (!p || !elems) return CIP_ERR_INVALID_ARG;
  const int e = prior_fft_default(p);
  *elems = !prior_has_variant(p) || p->avar == 0 ? e : (p->avar == 1 ? 24 - e : 32);
  return CIP_OK;
}

cip_status cip_get_config(cip_plan* p, int* rows, int* cc, int* blocksA, int* blocksB, int* column_pass) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (rows) *rows = p->rowsA;
  if (column_pass) *column_pass = p->colmode == 2 ? 2 : 1;
  if (cc) *cc = p->cc;
  if (blocksA) *blocksA = p->blocksA;
  if (blocksB) *blocksB = p->blocksB;
  return CIP_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched launch: many independent plans (uneven N, M, prior) iterated
// together.  Their iterations are recorded once into a CUDA graph in which
// every plan is its own branch (fork/join over a few capture streams), so the
// hardware scheduler packs the small instances' kernels side by side, and the
// graph (two iterations, which returns every ping-pong buffer to its starting
// side) is replayed.  The last two iterations run outside the graph with the
// residual flags so that cip_get_residuals stays valid for every plan.
// ---------------------------------------------------------------------------
struct cip_batch {
  std::vector<cip_plan*> plans;
  std::vector<cudaStream_t> streams;
  cudaStream_t cap = nullptr;  // capture stream (recording cannot start on the legacy default stream)
  cudaEvent_t fork = nullptr;
  std::vector<cudaEvent_t> joins;
  cudaGraphExec_t exec = nullptr;
  std::vector<std::pair<int, int>> parity;  // (cur, pcur) of every plan when the graph was recorded
  std::vector<unsigned long long> graph_launches;
  std::string err;
};

namespace {

cip_status bfail(cip_batch* b, cip_status s, const std::string& m) {
  b->err = m;
  return s;
}

#define BATCH_CUDA(b, call)                                                                 \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess) return bfail(b, CIP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

cip_status plan_enqueue(cip_plan* p, cudaStream_t s, int flags) {
  return DISPATCH_T(p, enqueue_iteration<float>(p, s, flags), enqueue_iteration<double>(p, s, flags));
}

// one round over all plans: plan i on capture stream i % S, joined back into `s`
cip_status batch_round(cip_batch* b, cudaStream_t s, int iters, int last_flags) {
  BATCH_CUDA(b, cudaEventRecord(b->fork, s));
  for (auto st : b->streams) BATCH_CUDA(b, cudaStreamWaitEvent(st, b->fork, 0));
  for (size_t i = 0; i < b->plans.size(); ++i) {
    cudaStream_t st = b->streams[i % b->streams.size()];
    for (int k = 0; k < iters; ++k) {
      const int flags = (k == iters - 1) ? last_flags : (k == iters - 2 && last_flags ? PA_STORE_T : 0);
      cip_status r = plan_enqueue(b->plans[i], st, flags);
      if (r != CIP_OK) return bfail(b, r, std::string("plan ") + std::to_string(i) + ": " + b->plans[i]->err);
    }
  }
  for (size_t j = 0; j < b->streams.size(); ++j) {
    BATCH_CUDA(b, cudaEventRecord(b->joins[j], b->streams[j]));
    BATCH_CUDA(b, cudaStreamWaitEvent(s, b->joins[j], 0));
  }
  return CIP_OK;
}

cip_status batch_record(cip_batch* b) {
  cudaStream_t s = b->cap;
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  b->parity.clear();
  b->graph_launches.clear();
  std::vector<unsigned long long> l0;
  for (auto* p : b->plans) {
    b->parity.push_back({p->cur, p->pcur});
    l0.push_back(p->launches);
  }
  BATCH_CUDA(b, cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  cip_status r = batch_round(b, s, 2, 0);
  cudaGraph_t g = nullptr;
  cudaError_t e = cudaStreamEndCapture(s, &g);
  if (r != CIP_OK) {
    if (g) cudaGraphDestroy(g);
    return r;
  }
  BATCH_CUDA(b, e);
  e = cudaGraphInstantiate(&b->exec, g, 0);
  cudaGraphDestroy(g);
  BATCH_CUDA(b, e);
  // recording advanced the host-side bookkeeping by two iterations without running them: undo
  for (size_t i = 0; i < b->plans.size(); ++i) {
    cip_plan* p = b->plans[i];
    p->iteration -= 2;
    b->graph_launches.push_back(p->launches - l0[i]);
    p->launches = l0[i];
    p->cur = b->parity[i].first;
    p->pcur = b->parity[i].second;
  }
  return CIP_OK;
}

}  // namespace

extern "C" {

cip_status cip_batch_create(cip_batch** out, cip_plan* const* plans, int n, int nstreams) {
  if (!out || !plans || n < 1) return CIP_ERR_INVALID_ARG;
  *out = nullptr;
  cip_batch* b = new cip_batch();
  for (int i = 0; i < n; ++i) {
    if (!plans[i]) {
      delete b;
      return CIP_ERR_INVALID_ARG;
    }
    b->plans.push_back(plans[i]);
  }
  const int ns = std::max(1, std::min(nstreams > 0 ? nstreams : 8, n));
  b->streams.resize(ns);
  b->joins.resize(ns);
  for (int j = 0; j < ns; ++j) {
    cudaStreamCreateWithFlags(&b->streams[j], cudaStreamNonBlocking);
    cudaEventCreateWithFlags(&b->joins[j], cudaEventDisableTiming);
  }
  cudaEventCreateWithFlags(&b->fork, cudaEventDisableTiming);
  cudaStreamCreateWithFlags(&b->cap, cudaStreamNonBlocking);
  *out = b;
  return CIP_OK;
}

cip_status cip_batch_iterate(cip_batch* b, int iters, void* stream) {
  if (!b) return CIP_ERR_INVALID_ARG;
  if (iters < 0) return bfail(b, CIP_ERR_INVALID_ARG, "iters < 0");
  for (auto* p : b->plans) {
    cip_status r = check_ready(p, true);
    if (r != CIP_OK) return bfail(b, r, p->err);
  }
  if (iters == 0) return CIP_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // the last two iterations (or the only one) run eagerly with the residual flags
  const int tail = iters >= 2 ? 2 : 1;
  int body = iters - tail;
  if (body % 2) {
    cip_status r = batch_round(b, s, 1, 0);
    if (r != CIP_OK) return r;
    --body;
  }
  if (body > 0 && !b->exec) {
    // first use: two eager iterations (every kernel's one-time attribute setup happens outside capture)
    cip_status r = batch_round(b, s, 2, 0);
    if (r != CIP_OK) return r;
    body -= 2;
  }
  if (body > 0) {
    bool ok = b->exec != nullptr && b->parity.size() == b->plans.size();
    for (size_t i = 0; ok && i < b->plans.size(); ++i)
      ok = b->parity[i].first == b->plans[i]->cur && b->parity[i].second == b->plans[i]->pcur;
    if (!ok) {
      BATCH_CUDA(b, cudaStreamSynchronize(s));  // recording reads no data; order it after queued work
      cip_status r = batch_record(b);
      if (r != CIP_OK) return r;
    }
    for (int k = 0; k < body / 2; ++k) BATCH_CUDA(b, cudaGraphLaunch(b->exec, s));
    for (size_t i = 0; i < b->plans.size(); ++i) {
      b->plans[i]->iteration += body;
      b->plans[i]->launches += b->graph_launches[i] * (unsigned long long)(body / 2);
    }
  }
  return batch_round(b, s, tail, PA_STORE_T | PA_RESID);
}

const char* cip_batch_last_error(const cip_batch* b) { return b ? b->err.c_str() : ""; }

cip_status cip_batch_destroy(cip_batch* b) {
  if (!b) return CIP_ERR_INVALID_ARG;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  for (auto st : b->streams) cudaStreamDestroy(st);
  for (auto ev : b->joins) cudaEventDestroy(ev);
  if (b->fork) cudaEventDestroy(b->fork);
  if (b->cap) cudaStreamDestroy(b->cap);
  delete b;
  return CIP_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Internal operations for the request server (plan_internal.h)
// ---------------------------------------------------------------------------
#include "plan_internal.h"

namespace cip {

cip_status plan_iterate_async(cip_plan* p, int k, cudaStream_t s, double* host_resid, cudaEvent_t ev) {
  cip_status r = check_ready(p, true);
  if (r != CIP_OK) return r;
  if (k < 1) return fail(p, CIP_ERR_INVALID_ARG, "k < 1");
  for (int i = 0; i < k; ++i) {
    const int flags = (i == k - 1) ? (PA_STORE_T | PA_RESID) : (i == k - 2 ? PA_STORE_T : 0);
    r = plan_enqueue(p, s, flags);
    if (r != CIP_OK) return r;
  }
  static_assert(kResidHost == kNPart + 2, "the residual record is the five sums and the two relative values");
  CIP_CUDA(p, cudaMemcpyAsync(host_resid, p->resid, kResidHost * sizeof(double), cudaMemcpyDeviceToHost, s));
  CIP_CUDA(p, cudaEventRecord(ev, s));
  return CIP_OK;
}

cip_status plan_adapt_rho(cip_plan* p, const double* host_resid, cudaStream_t s) {
  if (!p || !host_resid) return CIP_ERR_INVALID_ARG;
  if (!(p->adapt_tau > 0) || is_cd(p)) return CIP_OK;
  const double rho_new = rho_rule(p, host_resid);
  if (rho_new == p->rho) return CIP_OK;
  p->ast = s;
  return DISPATCH_T(p, change_rho<float>(p, rho_new, s), change_rho<double>(p, rho_new, s));
}

cip_status plan_adopt_factor(cip_plan* dst, const cip_plan* src, cudaStream_t s) {
  if (!dst || !src) return CIP_ERR_INVALID_ARG;
  dst->ast = s;
  if (dst->N != src->N || dst->K != src->K || dst->M != src->M || dst->dtype != src->dtype ||
      dst->prior != src->prior || dst->rho != src->rho || dst->beta != src->beta ||
      dst->opt.precision != src->opt.precision || is_cd(dst))
    return fail(dst, CIP_ERR_INVALID_ARG, "factor source has a different shape or parameters");
  if (!src->have_psfs || !src->lam64 || !src->pinv64) return fail(dst, CIP_ERR_STATE, "factor source has no factor");
  const size_t bytes = col_elems(dst, dst->M * (dst->M + 1) / 2) * 2 * dst->esz;
  CIP_CUDA(dst, cudaMemcpyAsync(dst->pinv, src->pinv, bytes, cudaMemcpyDeviceToDevice, s));
  dst->factor_src = src;
  dst->have_psfs = true;
  dst->have_y = false;
  return DISPATCH_T(dst, reset_state<float>(dst, s), reset_state<double>(dst, s));
}

cip_status plan_trim(cip_plan* p) {
  if (!p) return CIP_ERR_INVALID_ARG;
  if (p->lam64) cudaFreeAsync(p->lam64, p->ast);
  if (p->pinv64) cudaFreeAsync(p->pinv64, p->ast);
  p->lam64 = nullptr;
  p->pinv64 = nullptr;
  p->factor_src = nullptr;
  return CIP_OK;
}

size_t plan_resident_bytes(int N, int K, int M, cip_dtype dtype, cip_prior prior) {
  (void)K;
  const size_t e = dtype == CIP_F64 ? 8 : 4, c = 2 * e;
  const size_t H = N / 2 + 1, P = half_pitch(N), CP = col_pitch(N);
  const size_t nc = prior_is_tv(prior) ? 2 : 1;
  const size_t npk = (size_t)M * (M + 1) / 2;
  size_t b = 2 * (size_t)M * H * CP * c;      // xh, qh (column layout)
  b += (size_t)M * H * CP * c;                // data term
  b += npk * H * CP * c;                      // factor
  b += (size_t)M * H * CP * c;                // column buffer of the split form
  b += 3 * nc * (size_t)M * N * N * e;        // u (two), t_prev
  b += (size_t)kTwAll * (16 + c) + N * 8 + (size_t)(N / 2) * M * kNPart * 8 + 8192;
  if (prior == CIP_PRIOR_WDCT) b += 5 * (size_t)M * N * N * e / 2 + (size_t)M * M * e;  // wavelet work planes
  return b;
}

}  // namespace cip
