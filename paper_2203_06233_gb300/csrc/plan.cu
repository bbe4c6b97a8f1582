// Host side of libstap: plan creation and validation, workspace layout,
// host-computed tables (window, twiddles, default steering) and the C entry
// points that launch the kernels.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "batch.cuh"
#include "snapshots.cuh"
#include "stap_internal.cuh"
#include "solve_df.cuh"

using stap::DeviceStatus;

namespace {

constexpr size_t kAlign = 256;
constexpr int kMaxSlabs = 8;     // range slabs of a pipelined single-CPI run
constexpr double kPi = 3.14159265358979323846264338327950288;

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// An NVTX range around the host-side launch of one step's kernel(s), so that
// profilers and timeline tools label every launch with its step.  With no
// tool attached the push and pop return at once.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

struct Cpi {
  stap_dims d{};
  int D = 0, NB = 0;
  // snapshot geometry: Doppler rows Cd and bins per snapshot Td (C, T for
  // adjacent bins; C*T, 1 for PRI-staggered sub-windows, of which there are TW)
  int Cd = 0, Td = 0, TW = 1;
  // offsets of this CPI's tables inside the workspace
  size_t win_off = 0, tw_off = 0, steer_off = 0, g_off = 0, a_off = 0;
  std::vector<float> win;       // [P - TW + 1]
  std::vector<float> tw;        // [K][2]
  std::vector<double> steer;    // [S][D][2]
  // steer[s] = g (x) a_s for the default table: temporal factor g [T][2] and
  // spatial factors a [S][C][2]; cleared when the caller replaces the table
  // (all of them scaled: finish_steering)
  bool separable = false;
  bool sep_sym = false;   // sep_a_ff[S-1-s] is conj(sep_a_ff[s]) bit for bit
  double g_norm = 0.0, steer_sum = 0.0;   // |g|_2, the largest sum of |re| + |im| of a v_s (rounded up)
  std::vector<double> sep_g, sep_a;
  std::vector<float> steer_ff, sep_a_ff, g_ff;   // the tables as double-floats [..][4]
  size_t steer_ff_off = 0, a_ff_off = 0, g_ff_off = 0;
  stap::Tune tune;              // launch choices (autotuner or defaults)
  size_t dop_elems() const { return (size_t)Cd * d.n_dop * d.n_range; }
  size_t cov_elems() const { return (size_t)d.n_dop * NB * D * D; }
  size_t wts_elems() const { return (size_t)d.n_dop * NB * d.n_steering * D; }
};

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

stap_status validate(const stap_dims& d) {
  if (d.n_chan < 1 || d.n_pulses < 1 || d.n_dop < 1 || d.n_range < 1 || d.tdof < 1 ||
      d.training_block < 1 || d.n_steering < 1)
    return STAP_ERR_SHAPE;
  if (d.n_dop < d.n_pulses || d.tdof > d.n_dop || d.n_range % d.training_block != 0)
    return STAP_ERR_SHAPE;
  const long long D = (long long)d.n_chan * d.tdof;
  if (!is_pow2(d.n_dop) || d.n_dop > (1 << stap::kMaxLogK) || D > stap::kMaxD)
    return STAP_ERR_UNSUPPORTED;
  // keep every tensor below 2^40 elements and every grid dimension in range
  const long long NB = d.n_range / d.training_block;
  if ((long long)d.n_chan * d.n_dop * d.n_range > (1LL << 40) ||
      (long long)d.n_dop * NB * D * D > (1LL << 40) ||
      (long long)d.n_dop * NB * d.n_steering * D > (1LL << 40) || d.n_steering > 4096 ||
      d.training_block > 4096 || d.n_chan > 65535)
    return STAP_ERR_UNSUPPORTED;
  return STAP_OK;
}

// (re, im) double pairs -> (re_hi, re_lo, im_hi, im_lo) floats
void to_ff(const std::vector<double>& src, std::vector<float>& dst) {
  dst.resize(src.size() * 2);
  for (size_t i = 0; i < src.size(); ++i) {
    const float hi = (float)src[i];
    dst[2 * i] = hi;
    dst[2 * i + 1] = (float)(src[i] - (double)hi);
  }
}

// Look angle of steering vector s of S, in radians: uniform in angle over
// (-90, 90) degrees at s + 1/2 (the default steering's reading).  The upper
// half is the negated lower half, so the spatial factors of s and S-1-s are
// conjugates bit for bit (the solve combines such pairs in one pass).
double steer_theta(int s, int S) {
  if (2 * s + 1 > S) return -steer_theta(S - 1 - s, S);
  return (-90.0 + 180.0 * (s + 0.5) / S) * kPi / 180.0;
}

// Whether the double-float spatial factors [S][C] (re hi, re lo, im hi, im lo)
// satisfy a[S-1-s][c] = conj(a[s][c]) exactly.
bool conj_symmetric(const std::vector<float>& a_ff, int S, int C) {
  for (int s = 0; s < S; ++s)
    for (int c = 0; c < C; ++c) {
      const float* x = &a_ff[4 * ((size_t)s * C + c)];
      const float* y = &a_ff[4 * ((size_t)(S - 1 - s) * C + c)];
      if (!(x[0] == y[0] && x[1] == y[1] && x[2] == -y[2] && x[3] == -y[3])) return false;
    }
  return true;
}

// The exponent of the largest |re|, |im| of n numbers (0 where they are all
// zero, or not all finite), and the numbers with that exponent taken out.
int top_exponent(const double* x, size_t n) {
  double m = 0.0;
  for (size_t i = 0; i < n; ++i) m = std::max(m, std::fabs(x[i]));
  return m > 0.0 && std::isfinite(m) ? std::ilogb(m) : 0;
}
void scale_down(double* x, size_t n, int e) {
  for (size_t i = 0; i < n; ++i) x[i] = std::scalbn(x[i], -e);
}

// The weights u / sqrt(v^H u) do not depend on the steering vector's scale, so
// every table is kept with the power of two of its largest entry taken out:
// exact, nothing to undo, and neither the double-floats that the solves read
// nor the products v^H u, which are FP32 products there, leave FP32's range
// whatever the magnitudes that the caller's table or front end has.
//
// An arbitrary table: each vector by itself.
void finish_steering(Cpi& c) {
  const size_t n = 2 * (size_t)c.D;
  for (int s = 0; s < c.d.n_steering; ++s) {
    double* v = c.steer.data() + s * n;
    scale_down(v, n, top_exponent(v, n));
  }
  to_ff(c.steer, c.steer_ff);
  c.separable = false;
}

// v_s = g (x) a_s from the temporal and spatial factors, each scaled.
void finish_separable(Cpi& c) {
  const int C = c.d.n_chan, S = c.d.n_steering, T = c.d.tdof, D = c.D;
  scale_down(c.sep_g.data(), 2 * (size_t)T, top_exponent(c.sep_g.data(), 2 * (size_t)T));
  for (int s = 0; s < S; ++s) {
    double* a = &c.sep_a[2 * (size_t)s * C];
    scale_down(a, 2 * (size_t)C, top_exponent(a, 2 * (size_t)C));
    for (int t = 0; t < T; ++t)
      for (int ch = 0; ch < C; ++ch) {
        const double gr = c.sep_g[2 * t], gi = c.sep_g[2 * t + 1], ar = a[2 * ch], ai = a[2 * ch + 1];
        double* v = &c.steer[2 * ((size_t)s * D + t * C + ch)];
        v[0] = gr * ar - gi * ai;
        v[1] = gr * ai + gi * ar;
      }
  }
  c.g_norm = c.steer_sum = 0.0;
  for (double x : c.sep_g) c.g_norm += x * x;
  c.g_norm = 1.0001 * std::sqrt(c.g_norm);
  for (int s = 0; s < S; ++s) {
    double sum = 0.0;
    for (int i = 0; i < 2 * D; ++i) sum += std::fabs(c.steer[2 * (size_t)s * D + i]);
    c.steer_sum = std::max(c.steer_sum, 1.0001 * sum);
  }
  to_ff(c.steer, c.steer_ff);
  to_ff(c.sep_a, c.sep_a_ff);
  to_ff(c.sep_g, c.g_ff);
  c.separable = true;
  c.sep_sym = conj_symmetric(c.sep_a_ff, S, C);
}

void make_tables(Cpi& c) {
  const stap_dims& d = c.d;
  const int K = d.n_dop, T = d.tdof, C = d.n_chan, S = d.n_steering;
  const int P = d.n_pulses - c.TW + 1;   // window length (the sub-window's)
  std::vector<double> h(P);
  for (int p = 0; p < P; ++p)
    h[p] = (P == 1) ? 1.0 : 0.5 - 0.5 * std::cos(2.0 * kPi * p / (double)(P - 1));
  c.win.resize(P);
  for (int p = 0; p < P; ++p) c.win[p] = (float)h[p];
  c.tw.resize(2 * (size_t)K);
  for (int m = 0; m < K; ++m) {
    const double a = -2.0 * kPi * m / (double)K;
    c.tw[2 * m] = (float)std::cos(a);
    c.tw[2 * m + 1] = (float)std::sin(a);
  }
  // temporal part: the window's response at the T bin offsets around the bin;
  // staggered sub-windows all answer a bin-centre target with sum h' (offset 0)
  std::vector<double> gr(T), gi(T);
  for (int t = 0; t < T; ++t) {
    const long long m = c.TW > 1 ? 0 : t - T / 2;
    double sr = 0, si = 0;
    for (int p = 0; p < P; ++p) {
      long long n = (m * p) % K;
      if (n < 0) n += K;
      const double a = -2.0 * kPi * (double)n / (double)K;
      sr += h[p] * std::cos(a);
      si += h[p] * std::sin(a);
    }
    gr[t] = sr;
    gi[t] = si;
  }
  c.steer.assign(2 * (size_t)S * c.D, 0.0);
  c.sep_g.assign(2 * (size_t)T, 0.0);
  c.sep_a.assign(2 * (size_t)S * C, 0.0);
  for (int t = 0; t < T; ++t) {
    c.sep_g[2 * t] = gr[t];
    c.sep_g[2 * t + 1] = gi[t];
  }
  for (int s = 0; s < S; ++s) {
    const double th = steer_theta(s, S);
    const double fs = 0.5 * std::sin(th);
    for (int ch = 0; ch < C; ++ch) {
      const double a = 2.0 * kPi * fs * ch;
      c.sep_a[2 * ((size_t)s * C + ch)] = std::cos(a);
      c.sep_a[2 * ((size_t)s * C + ch) + 1] = std::sin(a);
    }
  }
  finish_separable(c);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// One step of a captured persistent batch: a persistent launch over a group
// of recorded launches, or a recorded launch issued as it is.
struct BatchStep {
  const void* batched = nullptr;
  int block = 0;
  size_t smem = 0;
  long long total = 0;
  int n = 0;
  size_t params_off = 0, prefix_off = 0, counter_off = 0;
  int record = -1;   // replay of records[record]
};


}  // namespace

struct stap_plan_s {
  std::vector<Cpi> cpis;
  stap_options opt{};
  cudaStream_t stream = nullptr;
  char* ws = nullptr;
  size_t ws_bytes = 0;
  size_t step_bytes = 0, run_bytes = 0, batch_bytes = 0;
  // streamed runs (stap_run_stream): two device cubes and two device outputs
  // beyond run_bytes
  size_t stream_bytes = 0, cube_bytes = 0, out_bytes = 0;
  cudaStream_t h2d = nullptr, d2h = nullptr;
  cudaEvent_t ev_start = nullptr, ev_in[2] = {}, ev_done[2] = {}, ev_out[2] = {}, ev_red[2] = {};
  // reduced-DOF front end (stap_plan_set_front_end): N element channels, the
  // matrix W [C][N] (c64, at fe_w_off) and the element chunk of one copy /
  // reduction; streamed runs then take element cubes
  int fe_N = 0, fe_chunk = 0;
  size_t fe_w_off = 0;
  std::vector<float> fe_w;
  size_t dop_off = 0, cov_off = 0, wts_off = 0;   // run intermediates (sized for the largest CPI)
  size_t ctr_off = 0;                             // training matrices (neighbour blocks or window)
  bool tables_ready = false;
  // polls before a pipeline wait of the tensor-core kernels gives up
  // (stap_plan_set_wait_limit)
  int wait_polls = stap::kDefaultWaitPolls;
  // batch schedule (stap_plan_set_batch_schedule) and the workspace region
  // that holds the persistent launches' parameter blocks, prefix sums and
  // counters (batch plans only)
  int batch_schedule = STAP_BATCH_PERSISTENT;
  size_t ctl_off = 0, ctl_bytes = 0;
  std::vector<BatchStep> batch_steps;                                    // the captured schedule
  std::vector<std::function<cudaError_t(cudaStream_t)>> batch_replays;  // its one-CPI launches

  // batched runs (n_cpi > 1): forked streams and the captured launch graph
  static constexpr int kSideStreams = 8;
  cudaStream_t side[kSideStreams] = {};
  cudaStream_t cap = nullptr;     // capture origin (the caller's stream may be the legacy one)
  cudaEvent_t fork_ev = nullptr, join_ev[kSideStreams] = {};
  cudaGraphExec_t graph_exec = nullptr;
  // pipelined single-CPI runs: one stream per range slab, earlier slabs at
  // higher priority
  cudaStream_t slab[kMaxSlabs] = {};
  cudaEvent_t slab_fork = nullptr, slab_join[kMaxSlabs] = {};
  std::vector<const void*> graph_cubes;   // buffers the graph was captured with
  std::vector<float*> graph_outs;
  char* graph_ws = nullptr;
  size_t graph_ws_bytes = 0;
  cudaStream_t graph_stream = nullptr;
  int graph_waves = 0;

  DeviceStatus* status() const { return reinterpret_cast<DeviceStatus*>(ws); }
  template <typename Tp>
  Tp* at(size_t off) const { return reinterpret_cast<Tp*>(ws + off); }
};

namespace {

stap_status upload_tables(stap_plan p, int only_cpi = -1) {
  for (size_t i = 0; i < p->cpis.size(); ++i) {
    if (only_cpi >= 0 && (int)i != only_cpi) continue;
    const Cpi& c = p->cpis[i];
    if (cudaMemcpyAsync(p->ws + c.win_off, c.win.data(), c.win.size() * sizeof(float),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.tw_off, c.tw.data(), c.tw.size() * sizeof(float),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.steer_off, c.steer.data(), c.steer.size() * sizeof(double),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.g_off, c.sep_g.data(), c.sep_g.size() * sizeof(double),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.a_off, c.sep_a.data(), c.sep_a.size() * sizeof(double),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.steer_ff_off, c.steer_ff.data(), c.steer_ff.size() * sizeof(float),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.a_ff_off, c.sep_a_ff.data(), c.sep_a_ff.size() * sizeof(float),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess ||
        cudaMemcpyAsync(p->ws + c.g_ff_off, c.g_ff.data(), c.g_ff.size() * sizeof(float),
                        cudaMemcpyHostToDevice, p->stream) != cudaSuccess)
      return STAP_ERR_CUDA;
  }
  if (p->fe_N && (only_cpi <= 0) &&
      cudaMemcpyAsync(p->ws + p->fe_w_off, p->fe_w.data(), p->fe_w.size() * sizeof(float),
                      cudaMemcpyHostToDevice, p->stream) != cudaSuccess)
    return STAP_ERR_CUDA;
  return STAP_OK;
}

stap_status check_launch(cudaError_t e) { return e == cudaSuccess ? STAP_OK : STAP_ERR_CUDA; }

stap_status ready(stap_plan p, size_t need) {
  if (!p) return STAP_ERR_INVALID_ARG;
  if (!p->ws || !p->tables_ready || p->ws_bytes < need) return STAP_ERR_NO_WORKSPACE;
  return STAP_OK;
}

// ----- the four steps on one CPI (arguments already validated) --------------

// Each step covers nr range cells (whole training blocks; nr < 0: all of
// them) starting at the given pointers; range-indexed tensors keep the CPI's
// full row stride R, and cov/wts hold the nr / B blocks of each bin.

stap_status do_doppler(stap_plan p, const Cpi& c, const void* cube, void* dop, cudaStream_t st,
                       int nr = -1) {
  NvtxRange range("stap_doppler");
  const stap_dims& d = c.d;
  return check_launch(stap::launch_doppler(
      static_cast<const float2*>(cube), static_cast<float2*>(dop), p->at<const float>(c.win_off),
      p->at<const float2>(c.tw_off), d.n_chan, c.TW, d.n_pulses, d.n_dop, nr < 0 ? d.n_range : nr,
      d.n_range, st, c.tune));
}

// Whether a mixed-precision plan's default apply is the (more accurate) FP32
// kernel: for short snapshots, which fit a thread's registers, while the
// tensor-core kernel's time is the splitting of the snapshots whatever S is (K
// 128 R 4096 B 128, FP32 / BF16X3 / TF32X3 / FP16S, us: D = 12 S = 16 30 / 60 / 71 /
// 96, D = 24 S = 32 87 / 103 / 105 / 208, D = 24 S = 64 155 / 139 / 130 / 278).  Beyond
// D = 24 the FP32 kernel would win for S <= 8 to 32 by up to a quarter, but the
// outputs would move by up to a few 1e-5 of their norm, where strong clutter
// cancels in the filter; the autotuner, which is asked to, still picks it.
// By the CPI's shape alone: range slabs, batches and single runs agree.
bool fp32_apply_default(const Cpi& c, int precision) {
  return c.D <= 24 && (c.d.n_steering <= 32 || precision == STAP_PREC_FP16_SCALED);
}

// lower: the chain's own buffer, of which the solve reads only the lower
// triangle (the kernels then skip the upper one)
stap_status do_covariance(stap_plan p, const Cpi& c, const void* dop, void* cov, cudaStream_t st,
                          int nr = -1, bool lower = false) {
  NvtxRange range("stap_covariance");
  const stap_dims& d = c.d;
  const int R = nr < 0 ? d.n_range : nr;
  // mixed-precision plans use the tensor cores unless the tuning kept the
  // (more accurate) FP32 kernel as the faster one
  if (stap::tc_precision(p->opt.precision) && c.tune.cov_kind != 1)
    return check_launch(stap::launch_covariance_tc(static_cast<const float2*>(dop),
                                                   static_cast<double2*>(cov), c.Cd, d.n_dop,
                                                   R, d.n_range, c.Td, d.training_block,
                                                   p->opt.precision, lower, p->status(), st,
                                                   p->wait_polls));
  return check_launch(stap::launch_covariance_fp32(static_cast<const float2*>(dop),
                                                   static_cast<double2*>(cov), c.Cd, d.n_dop,
                                                   R, d.n_range, c.Td, d.training_block, st,
                                                   c.tune, lower));
}

stap_status do_solve(stap_plan p, const Cpi& c, const void* cov, void* wts, cudaStream_t st,
                     int nr = -1, bool any_matrix = false) {
  NvtxRange range("stap_solve_weights");
  const stap_dims& d = c.d;
  const long long nb = nr < 0 ? c.NB : nr / d.training_block;
  return check_launch(stap::launch_solve(
      static_cast<const double2*>(cov), static_cast<float2*>(wts),
      p->at<const double2>(c.steer_off), c.separable ? p->at<const double2>(c.g_off) : nullptr,
      c.separable ? p->at<const double2>(c.a_off) : nullptr, p->at<const float4>(c.steer_ff_off),
      c.separable ? p->at<const float4>(c.a_ff_off) : nullptr,
      c.separable ? p->at<const float4>(c.g_ff_off) : nullptr, (long long)d.n_dop * nb,
      (long long)d.n_dop * c.NB, c.D, d.n_steering, d.n_chan, p->opt.load_factor, p->opt.refine_steps,
      p->opt.solver, p->status(), st, c.tune, c.separable && c.sep_sym, c.g_norm, c.steer_sum,
      any_matrix));
}

stap_status do_apply(stap_plan p, const Cpi& c, const void* dop, const void* wts, float* out,
                     cudaStream_t st, int nr = -1) {
  NvtxRange range("stap_apply");
  const stap_dims& d = c.d;
  const int R = nr < 0 ? d.n_range : nr;
  if (stap::tc_precision(p->opt.precision) &&
      stap::apply_tc_supported(d.training_block, d.n_steering) &&
      (c.tune.apply_kind == 3 || (c.tune.apply_kind == 0 && !fp32_apply_default(c, p->opt.precision))))
    return check_launch(stap::launch_apply_tc(static_cast<const float2*>(dop),
                                              static_cast<const float2*>(wts), out, c.Cd,
                                              d.n_dop, R, d.n_range, c.Td, d.training_block,
                                              d.n_steering, p->opt.precision, p->status(), st,
                                              p->wait_polls));
  return check_launch(stap::launch_apply(static_cast<const float2*>(dop),
                                         static_cast<const float2*>(wts), out, c.Cd, d.n_dop,
                                         R, d.n_range, c.Td, d.training_block, d.n_steering, st,
                                         c.tune));
}

// the training matrices inside a run: the lower triangles, all the solve reads
stap_status do_train(stap_plan p, const Cpi& c, const void* cov, void* ctr, cudaStream_t st) {
  if (p->opt.training == STAP_TRAIN_WINDOW) {
    NvtxRange range("stap_train_window");
    return check_launch(stap::launch_train_window(static_cast<const double2*>(cov),
                                                  static_cast<double2*>(ctr), c.d.n_dop, c.NB, c.D,
                                                  p->opt.train_guard, p->opt.train_half, st, true));
  }
  NvtxRange range("stap_train_neighbours");
  return check_launch(stap::launch_train_neighbours(static_cast<const double2*>(cov),
                                                    static_cast<double2*>(ctr), c.d.n_dop, c.NB,
                                                    c.D, st, true));
}

// ctr: the training matrices' buffer when the plan trains on neighbour blocks
// (then nr must cover the whole range)
stap_status do_chain(stap_plan p, const Cpi& c, const void* cube, float* out, char* dop, char* cov,
                     char* wts, char* ctr, cudaStream_t st, int nr = -1) {
  stap_status r;
  if ((r = do_doppler(p, c, cube, dop, st, nr)) != STAP_OK) return r;
  if ((r = do_covariance(p, c, dop, cov, st, nr, true)) != STAP_OK) return r;
  const char* trained = cov;
  if (p->opt.training != STAP_TRAIN_OWN_BLOCK) {
    if ((r = do_train(p, c, cov, ctr, st)) != STAP_OK) return r;
    trained = ctr;
  }
  if ((r = do_solve(p, c, trained, wts, st, nr)) != STAP_OK) return r;
  return do_apply(p, c, dop, wts, out, st, nr);
}

int slab_count(stap_plan p, const Cpi& c) {
  if (p->opt.training != STAP_TRAIN_OWN_BLOCK) return 1;   // blocks need their neighbours
  int ns = c.tune.slabs < 1 ? 1 : c.tune.slabs;
  if (ns > kMaxSlabs) ns = kMaxSlabs;
  if (ns > c.NB) ns = c.NB;
  return ns;
}

// One CPI in `slab_count` range slabs of whole training blocks.  Every slab's
// four-step chain is independent (its snapshots, covariances and weights lie
// inside the slab), so the chains run on their own streams: while the
// FP64-bound solve of one slab runs, the memory- and FP32-bound Doppler,
// covariance and apply kernels of the others fill the SMs.  Earlier slabs run
// at higher stream priority, so the chains stagger into a pipeline instead of
// advancing in lockstep.  Slab j's covariances and weights start at 256-byte
// aligned offsets of the run buffers (the plan reserves the slack).
stap_status run_single(stap_plan p, const void* cube, float* out) {
  const Cpi& c = p->cpis[0];
  char* dop = p->ws + p->dop_off;
  char* cov = p->ws + p->cov_off;
  char* wts = p->ws + p->wts_off;
  const int ns = slab_count(p, c);
  if (ns <= 1)
    return do_chain(p, c, cube, static_cast<float*>(out), dop, cov, wts, p->ws + p->ctr_off, p->stream);
  if (!p->slab_fork) {
    int least = 0, greatest = 0;
    if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess) return STAP_ERR_CUDA;
    if (cudaEventCreateWithFlags(&p->slab_fork, cudaEventDisableTiming) != cudaSuccess)
      return STAP_ERR_CUDA;
    for (int j = 0; j < kMaxSlabs; ++j) {
      int prio = greatest + j;            // numerically lower = higher priority
      if (prio > least) prio = least;
      if (cudaStreamCreateWithPriority(&p->slab[j], cudaStreamNonBlocking, prio) != cudaSuccess ||
          cudaEventCreateWithFlags(&p->slab_join[j], cudaEventDisableTiming) != cudaSuccess)
        return STAP_ERR_CUDA;
    }
  }
  const stap_dims& d = c.d;
  const int B = d.training_block, K = d.n_dop;
  if (cudaEventRecord(p->slab_fork, p->stream) != cudaSuccess) return STAP_ERR_CUDA;
  stap_status st = STAP_OK;
  size_t cov_at = 0, wts_at = 0;
  int j = 0;
  for (; j < ns && st == STAP_OK; ++j) {
    const int nb0 = (int)((long long)c.NB * j / ns), nb1 = (int)((long long)c.NB * (j + 1) / ns);
    const size_t rs = (size_t)nb0 * B;
    const int nr = (nb1 - nb0) * B;
    if (cudaStreamWaitEvent(p->slab[j], p->slab_fork, 0) != cudaSuccess) {
      st = STAP_ERR_CUDA;
      break;
    }
    st = do_chain(p, c, static_cast<const float2*>(cube) + rs, out + rs,
                  dop + rs * sizeof(float2), cov + cov_at, wts + wts_at, nullptr, p->slab[j], nr);
    cov_at += align_up((size_t)K * (nb1 - nb0) * c.D * c.D * 16);
    wts_at += align_up((size_t)K * (nb1 - nb0) * d.n_steering * c.D * 8);
    if (cudaEventRecord(p->slab_join[j], p->slab[j]) != cudaSuccess) st = STAP_ERR_CUDA;
  }
  // join every stream that was forked, even after a failed launch
  for (int i = 0; i < j; ++i)
    if (cudaStreamWaitEvent(p->stream, p->slab_join[i], 0) != cudaSuccess) st = STAP_ERR_CUDA;
  return st;
}

size_t inter_bytes(const stap_options& o, const Cpi& c) {
  return align_up(c.dop_elems() * 8) + align_up(c.cov_elems() * 16) + align_up(c.wts_elems() * 8) +
         (o.training != STAP_TRAIN_OWN_BLOCK ? align_up(c.cov_elems() * 16) : 0);
}

void drop_graph(stap_plan p) {
  if (p->graph_exec) cudaGraphExecDestroy(p->graph_exec);
  p->graph_exec = nullptr;
  p->graph_cubes.clear();
  p->graph_outs.clear();
}

// Batched run: CPIs packed into waves whose intermediates fit the workspace
// beyond the tables; inside a wave every CPI's four-kernel chain runs on one
// of kSideStreams forked streams, so small CPIs overlap.  The whole sequence
// is captured once into a CUDA graph and replayed while the same buffers,
// workspace and stream are passed.
stap_status run_batched_persistent(stap_plan p, const void* const* cubes, float* const* outs,
                                   cudaStream_t cs);
stap_status issue_persistent_steps(stap_plan p, cudaStream_t cs);

stap_status run_batched(stap_plan p, const void* const* cubes, float* const* outs) {
  const size_t n = p->cpis.size();
  bool same = p->graph_exec && p->graph_ws == p->ws && p->graph_ws_bytes == p->ws_bytes &&
              p->graph_stream == p->stream;
  for (size_t i = 0; same && i < n; ++i)
    same = p->graph_cubes[i] == cubes[i] && p->graph_outs[i] == outs[i];
  if (same)
    return cudaGraphLaunch(p->graph_exec, p->stream) == cudaSuccess ? STAP_OK : STAP_ERR_CUDA;

  drop_graph(p);
  if (!p->fork_ev) {
    if (cudaEventCreateWithFlags(&p->fork_ev, cudaEventDisableTiming) != cudaSuccess ||
        cudaStreamCreateWithFlags(&p->cap, cudaStreamNonBlocking) != cudaSuccess)
      return STAP_ERR_CUDA;
    for (int i = 0; i < stap_plan_s::kSideStreams; ++i)
      if (cudaStreamCreateWithFlags(&p->side[i], cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&p->join_ev[i], cudaEventDisableTiming) != cudaSuccess)
        return STAP_ERR_CUDA;
  }
  const size_t arena = p->ws_bytes - p->step_bytes;
  char* base = p->ws + p->step_bytes;
  cudaStream_t cs = p->cap;
  const bool persistent = p->batch_schedule == STAP_BATCH_PERSISTENT;
  if (persistent) {   // record, group and upload the schedule before the capture
    const stap_status ps = run_batched_persistent(p, cubes, outs, cs);
    if (ps != STAP_OK) return ps;
  }
  if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed) != cudaSuccess)
    return STAP_ERR_CUDA;
  stap_status st = STAP_OK;
  int waves = 0;
  size_t i = persistent ? n : 0;
  if (persistent) st = issue_persistent_steps(p, cs);
  while (st == STAP_OK && i < n) {
    // fork
    if (cudaEventRecord(p->fork_ev, cs) != cudaSuccess) { st = STAP_ERR_CUDA; break; }
    for (int k = 0; k < stap_plan_s::kSideStreams; ++k)
      if (cudaStreamWaitEvent(p->side[k], p->fork_ev, 0) != cudaSuccess) st = STAP_ERR_CUDA;
    size_t used = 0;
    int slot = 0;
    while (st == STAP_OK && i < n && (slot == 0 || used + inter_bytes(p->opt, p->cpis[i]) <= arena)) {
      const Cpi& c = p->cpis[i];
      char* dop = base + used;
      char* cov = dop + align_up(c.dop_elems() * 8);
      char* wts = cov + align_up(c.cov_elems() * 16);
      char* ctr = wts + align_up(c.wts_elems() * 8);
      used += inter_bytes(p->opt, c);
      st = do_chain(p, c, cubes[i], outs[i], dop, cov, wts, ctr,
                    p->side[slot % stap_plan_s::kSideStreams]);
      ++slot;
      ++i;
    }
    // join
    for (int k = 0; k < stap_plan_s::kSideStreams && st == STAP_OK; ++k)
      if (cudaEventRecord(p->join_ev[k], p->side[k]) != cudaSuccess ||
          cudaStreamWaitEvent(cs, p->join_ev[k], 0) != cudaSuccess)
        st = STAP_ERR_CUDA;
    ++waves;
  }
  cudaGraph_t graph = nullptr;
  const cudaError_t end = cudaStreamEndCapture(cs, &graph);
  if (st != STAP_OK || end != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return st != STAP_OK ? st : STAP_ERR_CUDA;
  }
  const cudaError_t inst = cudaGraphInstantiate(&p->graph_exec, graph, 0);
  cudaGraphDestroy(graph);
  if (inst != cudaSuccess) {
    p->graph_exec = nullptr;
    return STAP_ERR_CUDA;
  }
  p->graph_cubes.assign(cubes, cubes + n);
  p->graph_outs.assign(outs, outs + n);
  p->graph_ws = p->ws;
  p->graph_ws_bytes = p->ws_bytes;
  p->graph_stream = p->stream;
  p->graph_waves = waves;
  return cudaGraphLaunch(p->graph_exec, p->stream) == cudaSuccess ? STAP_OK : STAP_ERR_CUDA;
}

// Persistent schedule: the CPIs of each wave phase by phase; the launches a
// phase records for the wave's CPIs are grouped by persistent kernel and CTA
// size (one persistent launch per group, its per-CPI parameter blocks and
// prefix sums in the workspace's control region, uploaded before the
// capture); launches without a persistent form are issued as recorded.
stap_status run_batched_persistent(stap_plan p, const void* const* cubes, float* const* outs,
                                   cudaStream_t cs) {
  const size_t n = p->cpis.size();
  const size_t arena = p->ws_bytes - p->step_bytes;
  char* base = p->ws + p->step_bytes;
  stap::LaunchRecorder rec;
  std::vector<BatchStep> steps;
  p->batch_steps.clear();
  p->batch_replays.clear();
  std::vector<unsigned char> ctl(p->ctl_bytes, 0);
  size_t ctl_used = 0;
  auto take = [&](size_t bytes) -> size_t {
    const size_t at = ctl_used;
    ctl_used = align_up(ctl_used + bytes);
    return at;
  };
  stap_status st = STAP_OK;
  size_t i = 0;
  while (st == STAP_OK && i < n) {
    // the wave: CPIs whose intermediates fit the arena together
    struct Slot { size_t cpi; char *dop, *cov, *wts, *ctr; };
    std::vector<Slot> wave;
    size_t used = 0;
    while (i < n && (wave.empty() || used + inter_bytes(p->opt, p->cpis[i]) <= arena)) {
      const Cpi& c = p->cpis[i];
      Slot sl;
      sl.cpi = i;
      sl.dop = base + used;
      sl.cov = sl.dop + align_up(c.dop_elems() * 8);
      sl.wts = sl.cov + align_up(c.cov_elems() * 16);
      sl.ctr = sl.wts + align_up(c.wts_elems() * 8);
      used += inter_bytes(p->opt, c);
      wave.push_back(sl);
      ++i;
    }
    const int nphase = p->opt.training != STAP_TRAIN_OWN_BLOCK ? 5 : 4;
    for (int ph = 0; ph < nphase && st == STAP_OK; ++ph) {
      rec.records.clear();
      stap::current_recorder() = &rec;
      for (const Slot& sl : wave) {
        const Cpi& c = p->cpis[sl.cpi];
        const bool trained = p->opt.training != STAP_TRAIN_OWN_BLOCK;
        const char* solve_in = trained ? sl.ctr : sl.cov;
        stap_status r = STAP_OK;
        switch (trained ? ph : (ph < 2 ? ph : ph + 1)) {
          case 0: r = do_doppler(p, c, cubes[sl.cpi], sl.dop, cs); break;
          case 1: r = do_covariance(p, c, sl.dop, sl.cov, cs, -1, true); break;
          case 2: r = do_train(p, c, sl.cov, sl.ctr, cs); break;
          case 3: r = do_solve(p, c, solve_in, sl.wts, cs); break;
          default: r = do_apply(p, c, sl.dop, sl.wts, outs[sl.cpi], cs); break;
        }
        if (r != STAP_OK) st = r;
      }
      stap::current_recorder() = nullptr;
      if (st != STAP_OK) break;
      // group the phase's records: same persistent kernel and CTA size
      std::vector<char> done(rec.records.size(), 0);
      for (size_t a = 0; a < rec.records.size(); ++a) {
        if (done[a]) continue;
        const stap::LaunchRecord& ra = rec.records[a];
        if (!ra.batched) {   // issued as recorded, below
          done[a] = 1;
          continue;
        }
        std::vector<size_t> members;
        for (size_t b = a; b < rec.records.size(); ++b)
          if (!done[b] && rec.records[b].batched == ra.batched && rec.records[b].block == ra.block) {
            members.push_back(b);
            done[b] = 1;
          }
        BatchStep bs;
        bs.batched = ra.batched;
        bs.block = ra.block;
        bs.n = (int)members.size();
        bs.params_off = take(members.size() * stap::kMaxParamBytes);
        bs.prefix_off = take((members.size() + 1) * sizeof(long long));
        bs.counter_off = take(sizeof(unsigned long long));
        if (ctl_used > p->ctl_bytes) return STAP_ERR_NO_WORKSPACE;
        long long acc = 0;
        for (size_t m = 0; m < members.size(); ++m) {
          const stap::LaunchRecord& r = rec.records[members[m]];
          std::memcpy(&ctl[bs.params_off + m * stap::kMaxParamBytes], r.params, (size_t)r.psize);
          std::memcpy(&ctl[bs.prefix_off + m * sizeof(long long)], &acc, sizeof(long long));
          acc += r.vblocks;
          if (r.smem > bs.smem) bs.smem = r.smem;
        }
        std::memcpy(&ctl[bs.prefix_off + members.size() * sizeof(long long)], &acc, sizeof(long long));
        bs.total = acc;
        steps.push_back(bs);
      }
      // launches without a persistent form, in the order recorded
      for (size_t a = 0; a < rec.records.size(); ++a)
        if (!rec.records[a].batched) {
          BatchStep bs;
          bs.record = (int)p->batch_replays.size();
          p->batch_replays.push_back(std::move(rec.records[a].replay));
          steps.push_back(bs);
        }
    }
    // the next wave reuses the arena: its steps follow in the same stream
  }
  if (st != STAP_OK) return st;
  // parameter blocks, prefix sums and zeroed counters to the device, before the capture
  if (ctl_used && cudaMemcpy(p->ws + p->ctl_off, ctl.data(), ctl_used, cudaMemcpyHostToDevice) != cudaSuccess)
    return STAP_ERR_CUDA;
  p->batch_steps = steps;
  return STAP_OK;
}

// Issue the persistent schedule's steps on `cs` (inside the capture).
stap_status issue_persistent_steps(stap_plan p, cudaStream_t cs) {
  for (const BatchStep& bs : p->batch_steps) {
    if (bs.record >= 0) {
      if (p->batch_replays[bs.record](cs) != cudaSuccess) return STAP_ERR_CUDA;
      continue;
    }
    if (bs.total == 0) continue;
    unsigned long long* counter = p->at<unsigned long long>(p->ctl_off + bs.counter_off);
    if (cudaMemsetAsync(counter, 0, sizeof(unsigned long long), cs) != cudaSuccess) return STAP_ERR_CUDA;
    const int per_sm = stap::resident_ctas(bs.batched, bs.block, bs.smem);
    int sms = 152;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess)
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long grid = (long long)sms * per_sm;
    if (grid > bs.total) grid = bs.total;
    stap::BatchCtl ctl{p->at<const unsigned char>(p->ctl_off + bs.params_off),
                       p->at<const long long>(p->ctl_off + bs.prefix_off), counter, bs.n,
                       stap::kMaxParamBytes};
    void* args[] = {&ctl};
    if (cudaLaunchKernel(bs.batched, dim3((unsigned)grid), dim3(bs.block), args, bs.smem, cs) != cudaSuccess)
      return STAP_ERR_CUDA;
  }
  return STAP_OK;
}

// The front end over a whole element cube on the device: one pass over all N
// elements, so the reduced cube is written once (the streamed runs add chunk
// after chunk into it instead; with one chunk of all N elements they give the
// same bits).
stap_status reduce_all(stap_plan p, const float2* elem, float2* y, cudaStream_t st) {
  NvtxRange range("stap_reduce_channels");
  const stap_dims& d = p->cpis[0].d;
  return check_launch(stap::launch_reduce_channels(elem, p->at<const float2>(p->fe_w_off), y,
                                                   p->fe_N, 0, p->fe_N, d.n_chan, d.n_pulses,
                                                   d.n_range, false, st));
}

// Streamed runs with the front end: every element cube goes in chunks of
// fe_chunk elements through two device chunk buffers (copy on h2d, reduction
// into the reduced cube y on the plan's stream), then the chain runs on y and
// the output leaves on d2h.  Chunk buffer b is refilled only after the
// reduction that read it (ev_red); y is rewritten by the next cube's first
// reduction, which the plan's stream orders after this cube's chain.
stap_status run_stream_elements(stap_plan p, int64_t n, const void* const* host_cubes,
                                float* const* host_outs) {
  const stap_dims& d = p->cpis[0].d;
  const size_t PR8 = (size_t)d.n_pulses * d.n_range * 8;
  size_t off = p->run_bytes;
  float2* y = reinterpret_cast<float2*>(p->ws + off);
  off += align_up(p->cube_bytes);
  char* chunk_buf[2];
  for (int j = 0; j < 2; ++j) {
    chunk_buf[j] = p->ws + off;
    off += align_up((size_t)p->fe_chunk * PR8);
  }
  float* out_buf[2];
  for (int j = 0; j < 2; ++j) {
    out_buf[j] = reinterpret_cast<float*>(p->ws + off);
    off += align_up(p->out_bytes);
  }
  if (cudaEventRecord(p->ev_start, p->stream) != cudaSuccess ||
      cudaStreamWaitEvent(p->h2d, p->ev_start, 0) != cudaSuccess ||
      cudaStreamWaitEvent(p->d2h, p->ev_start, 0) != cudaSuccess)
    return STAP_ERR_CUDA;
  stap_status st = STAP_OK;
  long long g = 0;   // chunks queued so far
  for (int64_t i = 0; i < n && st == STAP_OK; ++i) {
    const char* src = static_cast<const char*>(host_cubes[i]);
    for (int n0 = 0; n0 < p->fe_N && st == STAP_OK; n0 += p->fe_chunk, ++g) {
      const int nc = std::min(p->fe_chunk, p->fe_N - n0);
      const int b = (int)(g & 1);
      if ((g >= 2 && cudaStreamWaitEvent(p->h2d, p->ev_red[b], 0) != cudaSuccess) ||
          cudaMemcpyAsync(chunk_buf[b], src + (size_t)n0 * PR8, (size_t)nc * PR8,
                          cudaMemcpyHostToDevice, p->h2d) != cudaSuccess ||
          cudaEventRecord(p->ev_in[b], p->h2d) != cudaSuccess ||
          cudaStreamWaitEvent(p->stream, p->ev_in[b], 0) != cudaSuccess) {
        st = STAP_ERR_CUDA;
        break;
      }
      st = check_launch(stap::launch_reduce_channels(
          reinterpret_cast<const float2*>(chunk_buf[b]), p->at<const float2>(p->fe_w_off), y,
          p->fe_N, n0, nc, d.n_chan, d.n_pulses, d.n_range, n0 > 0, p->stream));
      if (st == STAP_OK && cudaEventRecord(p->ev_red[b], p->stream) != cudaSuccess) st = STAP_ERR_CUDA;
    }
    if (st != STAP_OK) break;
    const int j = (int)(i & 1);
    if (i >= 2 && cudaStreamWaitEvent(p->stream, p->ev_out[j], 0) != cudaSuccess) {
      st = STAP_ERR_CUDA;
      break;
    }
    st = run_single(p, y, out_buf[j]);
    if (st != STAP_OK) break;
    if (cudaEventRecord(p->ev_done[j], p->stream) != cudaSuccess ||
        cudaStreamWaitEvent(p->d2h, p->ev_done[j], 0) != cudaSuccess ||
        cudaMemcpyAsync(host_outs[i], out_buf[j], p->out_bytes, cudaMemcpyDeviceToHost, p->d2h) !=
            cudaSuccess ||
        cudaEventRecord(p->ev_out[j], p->d2h) != cudaSuccess)
      st = STAP_ERR_CUDA;
  }
  if (cudaEventRecord(p->ev_start, p->h2d) != cudaSuccess ||
      cudaStreamWaitEvent(p->stream, p->ev_start, 0) != cudaSuccess ||
      cudaEventRecord(p->ev_start, p->d2h) != cudaSuccess ||
      cudaStreamWaitEvent(p->stream, p->ev_start, 0) != cudaSuccess)
    st = STAP_ERR_CUDA;
  return st;
}

stap_status single_cpi(stap_plan p) {
  if (!p) return STAP_ERR_INVALID_ARG;
  return p->cpis.size() == 1 ? STAP_OK : STAP_ERR_INVALID_ARG;
}

}  // namespace

extern "C" {

void stap_options_default(stap_options* opt) {
  if (!opt) return;
  opt->load_factor = 1e-3;
  opt->refine_steps = 1;
  opt->precision = STAP_PREC_FP32;
  opt->solver = STAP_SOLVE_FP64;
  opt->training = STAP_TRAIN_OWN_BLOCK;
  opt->train_guard = 0;
  opt->train_half = 1;
  opt->snapshots = STAP_SNAP_ADJACENT_BINS;
}

int32_t stap_abi_version(void) { return STAP_ABI_VERSION; }

stap_status stap_test_pivot_reciprocal(const double* in, double* out, int64_t n, void* cuda_stream) {
  if (n < 0 || (n > 0 && (!in || !out))) return STAP_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (stap::launch_pivot_reciprocal(static_cast<const double*>(in), out, (long long)n, s) != cudaSuccess)
    return STAP_ERR_CUDA;
  return cudaStreamSynchronize(s) == cudaSuccess ? STAP_OK : STAP_ERR_CUDA;
}

int32_t stap_checked_build(void) {
#ifdef STAP_CHECKED
  return 1;
#else
  return 0;
#endif
}

stap_status stap_check_report(int64_t* count, int32_t* site, int64_t* index, int64_t* extent) {
  if (!count) return STAP_ERR_INVALID_ARG;
  *count = 0;
  if (site) *site = 0;
  if (index) *index = 0;
  if (extent) *extent = 0;
#ifndef STAP_CHECKED
  return STAP_ERR_UNSUPPORTED;
#else
  if (cudaDeviceSynchronize() != cudaSuccess) return STAP_ERR_CUDA;
  cudaError_t (*readers[])(stap::CheckRecord*) = {
      stap::check_record_doppler, stap::check_record_covariance, stap::check_record_solve,
      stap::check_record_solve_df_small, stap::check_record_solve_df_big,
      stap::check_record_solve_df_small_any, stap::check_record_solve_df_big_any,
      stap::check_record_solve_df_small_ir, stap::check_record_solve_df_big_ir,
      stap::check_record_apply,   stap::check_record_mixed,      stap::check_record_train};
  bool first = true;
  for (auto rd : readers) {
    stap::CheckRecord r{};
    if (rd(&r) != cudaSuccess) return STAP_ERR_CUDA;
    *count += (int64_t)r.count;
    if (r.count && first) {
      first = false;
      if (site) *site = r.site;
      if (index) *index = r.index;
      if (extent) *extent = r.extent;
    }
  }
  return STAP_OK;
#endif
}

const char* stap_status_string(stap_status s) {
  switch (s) {
    case STAP_OK: return "ok";
    case STAP_ERR_INVALID_ARG: return "invalid argument";
    case STAP_ERR_SHAPE: return "invalid STAP shape";
    case STAP_ERR_UNSUPPORTED: return "shape or option not supported by the kernels";
    case STAP_ERR_CUDA: return "CUDA error";
    case STAP_ERR_NOT_POSDEF: return "loaded covariance not positive definite";
    case STAP_ERR_TIMEOUT: return "device-side wait timed out";
    case STAP_ERR_NO_WORKSPACE: return "workspace missing or too small";
    case STAP_ERR_MISALIGNED: return "buffer not 16-byte aligned";
  }
  return "unknown status";
}

stap_status stap_plan_create(const stap_dims* dims, int32_t n_cpi, const stap_options* opt,
                             void* cuda_stream, stap_plan* out, size_t* workspace_bytes) {
  if (!dims || !out || n_cpi < 1) return STAP_ERR_INVALID_ARG;
  *out = nullptr;
  stap_options o;
  stap_options_default(&o);
  if (opt) o = *opt;
  if (!(o.load_factor >= 0.0) || !std::isfinite(o.load_factor) || o.refine_steps < 0 ||
      o.refine_steps > 4)
    return STAP_ERR_INVALID_ARG;
  if (o.precision != STAP_PREC_FP32 && !stap::tc_precision(o.precision)) return STAP_ERR_UNSUPPORTED;
  if (o.solver != STAP_SOLVE_FP64 && o.solver != STAP_SOLVE_MIXED_IR) return STAP_ERR_UNSUPPORTED;
  if (o.training != STAP_TRAIN_OWN_BLOCK && o.training != STAP_TRAIN_NEIGHBOURS &&
      o.training != STAP_TRAIN_WINDOW)
    return STAP_ERR_INVALID_ARG;
  if (o.training == STAP_TRAIN_WINDOW && (o.train_guard < 0 || o.train_half < 1 ||
                                          o.train_guard > (1 << 20) || o.train_half > (1 << 20)))
    return STAP_ERR_INVALID_ARG;
  if (o.snapshots != STAP_SNAP_ADJACENT_BINS && o.snapshots != STAP_SNAP_PRI_STAGGERED)
    return STAP_ERR_INVALID_ARG;
  const bool stag = o.snapshots == STAP_SNAP_PRI_STAGGERED;
  for (int i = 0; i < n_cpi; ++i) {
    stap_status st = validate(dims[i]);
    if (st != STAP_OK) return st;
    if (o.solver == STAP_SOLVE_MIXED_IR && !stap::mir_supported(dims[i].n_chan * dims[i].tdof))
      return STAP_ERR_UNSUPPORTED;
    if (o.training == STAP_TRAIN_NEIGHBOURS && dims[i].n_range / dims[i].training_block < 2)
      return STAP_ERR_SHAPE;
    if (o.training == STAP_TRAIN_WINDOW &&
        (long long)dims[i].n_range / dims[i].training_block < 2LL * o.train_guard + 2)
      return STAP_ERR_SHAPE;
    if (stag && dims[i].tdof > dims[i].n_pulses) return STAP_ERR_SHAPE;   // sub-windows of >= 1 pulse
  }
  stap_plan p = new (std::nothrow) stap_plan_s;
  if (!p) return STAP_ERR_INVALID_ARG;
  p->opt = o;
  p->stream = static_cast<cudaStream_t>(cuda_stream);
  p->cpis.resize(n_cpi);
  size_t off = align_up(sizeof(DeviceStatus));
  size_t max_dop = 0, max_cov = 0, max_wts = 0;
  for (int i = 0; i < n_cpi; ++i) {
    Cpi& c = p->cpis[i];
    c.d = dims[i];
    c.D = c.d.n_chan * c.d.tdof;
    c.TW = stag ? c.d.tdof : 1;
    c.Cd = stag ? c.D : c.d.n_chan;
    c.Td = stag ? 1 : c.d.tdof;
    c.NB = c.d.n_range / c.d.training_block;
    make_tables(c);
    c.win_off = off;
    off = align_up(off + c.win.size() * sizeof(float));
    c.tw_off = off;
    off = align_up(off + c.tw.size() * sizeof(float));
    c.steer_off = off;
    off = align_up(off + c.steer.size() * sizeof(double));
    c.g_off = off;
    off = align_up(off + c.sep_g.size() * sizeof(double));
    c.a_off = off;
    off = align_up(off + c.sep_a.size() * sizeof(double));
    c.steer_ff_off = off;
    off = align_up(off + c.steer_ff.size() * sizeof(float));
    c.a_ff_off = off;
    off = align_up(off + c.sep_a_ff.size() * sizeof(float));
    c.g_ff_off = off;
    off = align_up(off + c.g_ff.size() * sizeof(float));
    if (c.dop_elems() > max_dop) max_dop = c.dop_elems();
    if (c.cov_elems() > max_cov) max_cov = c.cov_elems();
    if (c.wts_elems() > max_wts) max_wts = c.wts_elems();
  }
  if (n_cpi > 1) {   // persistent batch schedules: at most 5 launches per CPI and wave
    const size_t recs = 5 * (size_t)n_cpi;
    p->ctl_off = off;
    p->ctl_bytes = align_up(recs * (stap::kMaxParamBytes + 2 * sizeof(long long)) + recs * 3 * kAlign);
    off += p->ctl_bytes;
  }
  p->step_bytes = off;
  p->dop_off = off;
  off = align_up(off + max_dop * 8);
  p->cov_off = off;
  off = align_up(off + max_cov * 16);
  p->wts_off = off;
  off = align_up(off + max_wts * 8);
  if (n_cpi == 1) off += 2 * kMaxSlabs * kAlign;   // per-slab alignment of cov and wts
  p->ctr_off = off;
  if (o.training != STAP_TRAIN_OWN_BLOCK) off = align_up(off + max_cov * 16);
  p->run_bytes = off;
  size_t all = p->step_bytes;
  for (const Cpi& c : p->cpis) all += inter_bytes(o, c);
  p->batch_bytes = all > p->run_bytes ? all : p->run_bytes;
  if (n_cpi == 1) {
    const stap_dims& d = dims[0];
    p->cube_bytes = (size_t)d.n_chan * d.n_pulses * d.n_range * 8;
    p->out_bytes = (size_t)d.n_steering * d.n_dop * d.n_range * 4;
    p->stream_bytes = p->run_bytes + 2 * align_up(p->cube_bytes) + 2 * align_up(p->out_bytes);
  }
  *out = p;
  if (workspace_bytes) *workspace_bytes = p->run_bytes;
  return STAP_OK;
}

stap_status stap_plan_workspace_sizes(stap_plan p, size_t* step_bytes, size_t* run_bytes) {
  if (!p) return STAP_ERR_INVALID_ARG;
  if (step_bytes) *step_bytes = p->step_bytes;
  if (run_bytes) *run_bytes = p->run_bytes;
  return STAP_OK;
}

stap_status stap_plan_set_workspace(stap_plan p, void* dev_ptr, size_t bytes) {
  if (!p || !dev_ptr) return STAP_ERR_INVALID_ARG;
  if (!aligned16(dev_ptr)) return STAP_ERR_MISALIGNED;
  if (bytes < p->step_bytes) return STAP_ERR_NO_WORKSPACE;
  p->ws = static_cast<char*>(dev_ptr);
  p->ws_bytes = bytes;
  p->tables_ready = false;
  drop_graph(p);
  if (cudaMemsetAsync(p->ws, 0, sizeof(DeviceStatus), p->stream) != cudaSuccess) return STAP_ERR_CUDA;
  stap_status st = upload_tables(p);
  if (st != STAP_OK) return st;
  p->tables_ready = true;
  return STAP_OK;
}

stap_status stap_plan_set_wait_limit(stap_plan p, int32_t max_polls) {
  if (!p || max_polls < 0) return STAP_ERR_INVALID_ARG;
  p->wait_polls = max_polls;
  drop_graph(p);   // captured launches carry the limit
  return STAP_OK;
}

stap_status stap_plan_set_stream(stap_plan p, void* cuda_stream) {
  if (!p) return STAP_ERR_INVALID_ARG;
  p->stream = static_cast<cudaStream_t>(cuda_stream);
  return STAP_OK;
}

stap_status stap_plan_set_steering(stap_plan p, int32_t cpi, const double* host_c128) {
  if (!p || !host_c128 || cpi < 0 || cpi >= (int32_t)p->cpis.size()) return STAP_ERR_INVALID_ARG;
  if (!p->ws || !p->tables_ready) return STAP_ERR_NO_WORKSPACE;
  Cpi& c = p->cpis[cpi];
  for (size_t i = 0; i < c.steer.size(); ++i)
    if (!std::isfinite(host_c128[i])) return STAP_ERR_INVALID_ARG;
  std::memcpy(c.steer.data(), host_c128, c.steer.size() * sizeof(double));
  finish_steering(c);   // an arbitrary table: solve for every steering vector
  drop_graph(p);        // the captured launches chose the solve variant
  return upload_tables(p, cpi);
}

stap_status stap_plan_destroy(stap_plan p) {
  if (!p) return STAP_ERR_INVALID_ARG;
  drop_graph(p);
  if (p->ev_start) {
    for (cudaStream_t s : {p->h2d, p->d2h})
      if (s) {
        cudaStreamSynchronize(s);
        cudaStreamDestroy(s);
      }
    for (int j = 0; j < 2; ++j)
      for (cudaEvent_t e : {p->ev_in[j], p->ev_done[j], p->ev_out[j], p->ev_red[j]})
        if (e) cudaEventDestroy(e);
    cudaEventDestroy(p->ev_start);
  }
  if (p->fork_ev) {
    for (int i = 0; i < stap_plan_s::kSideStreams; ++i) {
      if (p->side[i]) {
        cudaStreamSynchronize(p->side[i]);
        cudaStreamDestroy(p->side[i]);
      }
      if (p->join_ev[i]) cudaEventDestroy(p->join_ev[i]);
    }
    cudaEventDestroy(p->fork_ev);
    if (p->cap) cudaStreamDestroy(p->cap);
  }
  if (p->slab_fork) {
    for (int i = 0; i < kMaxSlabs; ++i) {
      if (p->slab[i]) {
        cudaStreamSynchronize(p->slab[i]);
        cudaStreamDestroy(p->slab[i]);
      }
      if (p->slab_join[i]) cudaEventDestroy(p->slab_join[i]);
    }
    cudaEventDestroy(p->slab_fork);
  }
  // pageable-memory uploads were staged synchronously, so nothing on the
  // device still reads the host tables
  delete p;
  return STAP_OK;
}

stap_status stap_doppler(stap_plan p, const void* cube, void* dop) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!cube || !dop) return STAP_ERR_INVALID_ARG;
  if (!aligned16(cube) || !aligned16(dop)) return STAP_ERR_MISALIGNED;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  return do_doppler(p, p->cpis[0], cube, dop, p->stream);
}

stap_status stap_covariance(stap_plan p, const void* dop, void* cov) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!dop || !cov) return STAP_ERR_INVALID_ARG;
  if (!aligned16(dop) || !aligned16(cov)) return STAP_ERR_MISALIGNED;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  return do_covariance(p, p->cpis[0], dop, cov, p->stream);
}

stap_status stap_train_neighbours(stap_plan p, const void* cov, void* ctr) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!cov || !ctr || cov == ctr) return STAP_ERR_INVALID_ARG;
  if (!aligned16(cov) || !aligned16(ctr)) return STAP_ERR_MISALIGNED;
  if (p->cpis[0].NB < 2) return STAP_ERR_SHAPE;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  NvtxRange range("stap_train_neighbours");
  const Cpi& c = p->cpis[0];
  return check_launch(stap::launch_train_neighbours(static_cast<const double2*>(cov),
                                                    static_cast<double2*>(ctr), c.d.n_dop, c.NB,
                                                    c.D, p->stream));
}

stap_status stap_train_window(stap_plan p, const void* cov, void* ctr) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!cov || !ctr || cov == ctr) return STAP_ERR_INVALID_ARG;
  if (!aligned16(cov) || !aligned16(ctr)) return STAP_ERR_MISALIGNED;
  const int guard = p->opt.training == STAP_TRAIN_WINDOW ? p->opt.train_guard : 0;
  const int half = p->opt.training == STAP_TRAIN_WINDOW ? p->opt.train_half : 1;
  if ((long long)p->cpis[0].NB < 2LL * guard + 2) return STAP_ERR_SHAPE;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  NvtxRange range("stap_train_window");
  const Cpi& c = p->cpis[0];
  return check_launch(stap::launch_train_window(static_cast<const double2*>(cov),
                                                static_cast<double2*>(ctr), c.d.n_dop, c.NB, c.D,
                                                guard, half, p->stream));
}

stap_status stap_solve_weights(stap_plan p, const void* cov, void* wts) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!cov || !wts) return STAP_ERR_INVALID_ARG;
  if (!aligned16(cov) || !aligned16(wts)) return STAP_ERR_MISALIGNED;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  return do_solve(p, p->cpis[0], cov, wts, p->stream, -1, true);
}

stap_status stap_apply(stap_plan p, const void* dop, const void* wts, float* out) {
  stap_status st = single_cpi(p);
  if (st != STAP_OK) return st;
  if (!dop || !wts || !out) return STAP_ERR_INVALID_ARG;
  if (!aligned16(dop) || !aligned16(wts) || !aligned16(out)) return STAP_ERR_MISALIGNED;
  if ((st = ready(p, p->step_bytes)) != STAP_OK) return st;
  return do_apply(p, p->cpis[0], dop, wts, out, p->stream);
}

stap_status stap_run_cpi(stap_plan p, const void* const* cubes, float* const* outs) {
  NvtxRange range("stap_run_cpi");
  if (!p || !cubes || !outs) return STAP_ERR_INVALID_ARG;
  for (size_t i = 0; i < p->cpis.size(); ++i) {
    if (!cubes[i] || !outs[i]) return STAP_ERR_INVALID_ARG;
    if (!aligned16(cubes[i]) || !aligned16(outs[i])) return STAP_ERR_MISALIGNED;
  }
  stap_status st = ready(p, p->run_bytes);
  if (st != STAP_OK) return st;
  if (p->cpis.size() > 1) return run_batched(p, cubes, outs);
  return run_single(p, cubes[0], outs[0]);
}

stap_status stap_plan_set_batch_schedule(stap_plan p, int32_t schedule) {
  if (!p || (schedule != STAP_BATCH_PERSISTENT && schedule != STAP_BATCH_STREAMS))
    return STAP_ERR_INVALID_ARG;
  if (p->batch_schedule != schedule) drop_graph(p);
  p->batch_schedule = schedule;
  return STAP_OK;
}

stap_status stap_plan_get_batch_schedule(stap_plan p, int32_t* schedule) {
  if (!p || !schedule) return STAP_ERR_INVALID_ARG;
  *schedule = p->batch_schedule;
  return STAP_OK;
}

stap_status stap_plan_batch_bytes(stap_plan p, size_t* all_concurrent_bytes) {
  if (!p || !all_concurrent_bytes) return STAP_ERR_INVALID_ARG;
  *all_concurrent_bytes = p->batch_bytes;
  return STAP_OK;
}

stap_status stap_plan_stream_bytes(stap_plan p, size_t* bytes) {
  if (!p || !bytes) return STAP_ERR_INVALID_ARG;
  if (p->cpis.size() != 1) return STAP_ERR_INVALID_ARG;
  *bytes = p->stream_bytes;
  return STAP_OK;
}

stap_status stap_plan_set_front_end(stap_plan p, int32_t n_elem, const double* W,
                                    int32_t chunk_elems) {
  if (!p || !W || n_elem < 1 || p->cpis.size() != 1) return STAP_ERR_INVALID_ARG;
  if (p->ws || p->fe_N) return STAP_ERR_INVALID_ARG;   // once, before the workspace
  Cpi& c = p->cpis[0];
  const stap_dims& d = c.d;
  const int C = d.n_chan, N = n_elem, S = d.n_steering;
  const size_t PR8 = (size_t)d.n_pulses * d.n_range * 8;
  if ((size_t)N * PR8 > ((size_t)1 << 44)) return STAP_ERR_UNSUPPORTED;
  for (size_t i = 0; i < 2 * (size_t)C * N; ++i)
    if (!std::isfinite(W[i])) return STAP_ERR_INVALID_ARG;
  int chunk = chunk_elems;
  if (chunk < 1) {   // about 512 MB of element rows per copy and reduction
    const size_t want = ((size_t)512 << 20) / PR8;
    chunk = (int)std::min<size_t>(std::max<size_t>(want, 1), (size_t)N);
  }
  if (chunk > N) chunk = N;
  // spatial gains b_s[c] = sum_n conj(W[c][n]) exp(j 2 pi f_s n): the separable
  // steering's spatial factors, and v_s = g (x) b_s
  for (int s = 0; s < S; ++s) {
    const double th = steer_theta(s, S);
    const double fs = 0.5 * std::sin(th);
    for (int ch = 0; ch < C; ++ch) {
      double br = 0, bi = 0;
      for (int e = 0; e < N; ++e) {
        const double a = 2.0 * kPi * fs * e;
        const double er = std::cos(a), ei = std::sin(a);
        const double wr = W[2 * ((size_t)ch * N + e)], wi = W[2 * ((size_t)ch * N + e) + 1];
        br += wr * er + wi * ei;   // conj(w) e
        bi += wr * ei - wi * er;
      }
      c.sep_a[2 * ((size_t)s * C + ch)] = br;
      c.sep_a[2 * ((size_t)s * C + ch) + 1] = bi;
    }
  }
  finish_separable(c);
  p->fe_w.resize(2 * (size_t)C * N);
  for (size_t i = 0; i < p->fe_w.size(); ++i) p->fe_w[i] = (float)W[i];
  p->fe_N = N;
  p->fe_chunk = chunk;
  p->fe_w_off = p->run_bytes;
  p->run_bytes = align_up(p->run_bytes + p->fe_w.size() * sizeof(float));
  p->stream_bytes = p->run_bytes + align_up(p->cube_bytes) + 2 * align_up((size_t)chunk * PR8) +
                    2 * align_up(p->out_bytes);
  if (p->batch_bytes < p->run_bytes) p->batch_bytes = p->run_bytes;
  return STAP_OK;
}

stap_status stap_reduce_channels(stap_plan p, const void* elem_cube_c64, void* cube_c64) {
  if (!p || !elem_cube_c64 || !cube_c64) return STAP_ERR_INVALID_ARG;
  if (!aligned16(elem_cube_c64) || !aligned16(cube_c64)) return STAP_ERR_MISALIGNED;
  if (!p->fe_N) return STAP_ERR_INVALID_ARG;
  stap_status st = ready(p, p->run_bytes);
  if (st != STAP_OK) return st;
  return reduce_all(p, static_cast<const float2*>(elem_cube_c64), static_cast<float2*>(cube_c64),
                    p->stream);
}

// CPI i: copy-in on h2d into device cube j = i % 2, the chain on the plan's
// stream into device output j, copy-out on d2h.  Buffer j is rewritten by CPI
// i + 2 only after CPI i's chain has read it (ev_done) and its output has been
// copied out (ev_out); a wait takes the event's latest record at enqueue time,
// which is CPI i's.
stap_status stap_run_stream(stap_plan p, int64_t n, const void* const* host_cubes,
                            float* const* host_outs) {
  if (!p || n < 0 || (n > 0 && (!host_cubes || !host_outs))) return STAP_ERR_INVALID_ARG;
  if (p->cpis.size() != 1) return STAP_ERR_INVALID_ARG;
  for (int64_t i = 0; i < n; ++i)
    if (!host_cubes[i] || !host_outs[i]) return STAP_ERR_INVALID_ARG;
  stap_status st = ready(p, p->stream_bytes);
  if (st != STAP_OK || n == 0) return st;
  if (!p->ev_start) {
    if (cudaStreamCreateWithFlags(&p->h2d, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&p->d2h, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&p->ev_start, cudaEventDisableTiming) != cudaSuccess)
      return STAP_ERR_CUDA;
    for (int j = 0; j < 2; ++j)
      if (cudaEventCreateWithFlags(&p->ev_in[j], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&p->ev_done[j], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&p->ev_out[j], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&p->ev_red[j], cudaEventDisableTiming) != cudaSuccess)
        return STAP_ERR_CUDA;
  }
  if (p->fe_N) return run_stream_elements(p, n, host_cubes, host_outs);
  char* cube_buf[2];
  float* out_buf[2];
  size_t off = p->run_bytes;
  for (int j = 0; j < 2; ++j) {
    cube_buf[j] = p->ws + off;
    off += align_up(p->cube_bytes);
  }
  for (int j = 0; j < 2; ++j) {
    out_buf[j] = reinterpret_cast<float*>(p->ws + off);
    off += align_up(p->out_bytes);
  }
  // both copy streams start after the work already queued on the plan's stream
  if (cudaEventRecord(p->ev_start, p->stream) != cudaSuccess ||
      cudaStreamWaitEvent(p->h2d, p->ev_start, 0) != cudaSuccess ||
      cudaStreamWaitEvent(p->d2h, p->ev_start, 0) != cudaSuccess)
    return STAP_ERR_CUDA;
  int64_t i = 0;
  for (; i < n && st == STAP_OK; ++i) {
    const int j = (int)(i & 1);
    if (i >= 2 && cudaStreamWaitEvent(p->h2d, p->ev_done[j], 0) != cudaSuccess) { st = STAP_ERR_CUDA; break; }
    if (cudaMemcpyAsync(cube_buf[j], host_cubes[i], p->cube_bytes, cudaMemcpyHostToDevice, p->h2d) !=
            cudaSuccess ||
        cudaEventRecord(p->ev_in[j], p->h2d) != cudaSuccess ||
        cudaStreamWaitEvent(p->stream, p->ev_in[j], 0) != cudaSuccess ||
        (i >= 2 && cudaStreamWaitEvent(p->stream, p->ev_out[j], 0) != cudaSuccess)) {
      st = STAP_ERR_CUDA;
      break;
    }
    st = run_single(p, cube_buf[j], out_buf[j]);
    if (st != STAP_OK) break;
    if (cudaEventRecord(p->ev_done[j], p->stream) != cudaSuccess ||
        cudaStreamWaitEvent(p->d2h, p->ev_done[j], 0) != cudaSuccess ||
        cudaMemcpyAsync(host_outs[i], out_buf[j], p->out_bytes, cudaMemcpyDeviceToHost, p->d2h) !=
            cudaSuccess ||
        cudaEventRecord(p->ev_out[j], p->d2h) != cudaSuccess)
      st = STAP_ERR_CUDA;
  }
  // the plan's stream passes the call only after every copy it queued
  if (cudaEventRecord(p->ev_start, p->h2d) != cudaSuccess ||
      cudaStreamWaitEvent(p->stream, p->ev_start, 0) != cudaSuccess ||
      cudaEventRecord(p->ev_start, p->d2h) != cudaSuccess ||
      cudaStreamWaitEvent(p->stream, p->ev_start, 0) != cudaSuccess)
    st = STAP_ERR_CUDA;
  return st;
}

stap_status stap_plan_autotune(stap_plan p, const void* const* cubes, float* const* outs,
                               int32_t reps) {
  if (!p || !cubes || !outs) return STAP_ERR_INVALID_ARG;
  for (size_t i = 0; i < p->cpis.size(); ++i) {
    if (!cubes[i] || !outs[i]) return STAP_ERR_INVALID_ARG;
    if (!aligned16(cubes[i]) || !aligned16(outs[i])) return STAP_ERR_MISALIGNED;
  }
  stap_status st = ready(p, p->run_bytes);
  if (st != STAP_OK) return st;
  if (reps < 1) reps = 3;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return STAP_ERR_CUDA;
  const float kNever = 3.0e38f;
  // time `launch` (one untimed run first); kNever if it fails
  // time n runs of `launch` (one untimed run first); kNever if it fails
  auto timeit_n = [&](int n, auto&& launch) -> float {
    if (launch() != STAP_OK) return kNever;
    cudaEventRecord(e0, p->stream);
    for (int r = 0; r < n; ++r)
      if (launch() != STAP_OK) return kNever;
    cudaEventRecord(e1, p->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return kNever;
    float ms = kNever;
    cudaEventElapsedTime(&ms, e0, e1);
    return ms;
  };
  auto timeit = [&](auto&& launch) -> float { return timeit_n(reps, launch); };
  auto same_key = [](const stap_dims& a, const stap_dims& b) {
    return a.n_chan == b.n_chan && a.n_pulses == b.n_pulses && a.n_dop == b.n_dop &&
           a.tdof == b.tdof && a.training_block == b.training_block && a.n_steering == b.n_steering;
  };
  std::vector<char> tuned(p->cpis.size(), 0);
  char* dop = p->ws + p->dop_off;
  char* cov = p->ws + p->cov_off;
  char* wts = p->ws + p->wts_off;
  for (size_t i = 0; i < p->cpis.size() && st == STAP_OK; ++i) {
    if (tuned[i]) continue;
    Cpi& c = p->cpis[i];
    const stap_dims& d = c.d;
    const void* cube = cubes[i];
    float* out = outs[i];
    stap::Tune best = c.tune;
    auto pick = [&](auto&& set, const std::vector<int>& values, auto&& run) {
      float bt = kNever;
      int bv = 0;
      for (int v : values) {
        set(c.tune, v);
        const float ms = timeit(run);
        if (ms < bt) {
          bt = ms;
          bv = v;
        }
      }
      set(c.tune, bv);
    };
    c.tune = best;
    pick([](stap::Tune& t, int v) { t.dop_tr = v; }, {8, 16, 32},
         [&] { return do_doppler(p, c, cube, dop, p->stream); });
    {
      const bool mixed = stap::tc_precision(p->opt.precision);
      if (mixed) c.tune.cov_kind = 1;   // tune the FP32 kernel first
      std::vector<int> kts;
      for (int kt = 1; kt <= 32 && kt <= d.n_dop; kt *= 2) kts.push_back(kt);
      // as the run writes them: lower triangles
      pick([](stap::Tune& t, int v) { t.cov_kt = v; }, kts,
           [&] { return do_covariance(p, c, dop, cov, p->stream, -1, true); });
      if (mixed)   // then keep the tensor cores only where they are faster
        pick([](stap::Tune& t, int v) { t.cov_kind = v; }, {2, 1},
             [&] { return do_covariance(p, c, dop, cov, p->stream, -1, true); });
    }
    if ((st = do_covariance(p, c, dop, cov, p->stream)) != STAP_OK) break;
    // FP64 solves have launch choices; the double-float ones (faster wherever
    // they may stand in) have none
    if (stap::solve_df_eligible(p->opt.solver, p->opt.load_factor, c.D, p->opt.refine_steps)) {
      c.tune.solve_kind = c.tune.solve_ts = c.tune.solve_nw = c.tune.solve_lr = 0;
    } else if (c.D <= stap::kSmallMaxD) {
      const int nrhs = c.separable ? d.n_chan : d.n_steering;
      int base = 1;
      while (base < nrhs && base < 32) base <<= 1;
      const bool has_reg = c.D == 8 || c.D == 12 || c.D == 16;
      float bt = kNever;
      int bts = 0, bnw = 0, bkind = 0;
      for (int kind = has_reg ? 1 : 0; kind <= (has_reg ? 2 : 0); ++kind)
        for (int ts = base; ts <= 32; ts <<= 1)
          for (int nw = 1; nw <= 4; ++nw) {
            c.tune.solve_kind = kind;
            c.tune.solve_ts = ts;
            c.tune.solve_nw = nw;
            const float ms = timeit([&] { return do_solve(p, c, cov, wts, p->stream); });
            if (ms < bt) {
              bt = ms;
              bts = ts;
              bnw = nw;
              bkind = kind;
            }
          }
      c.tune.solve_kind = 3;   // one system per CTA instead of teams
      if (timeit([&] { return do_solve(p, c, cov, wts, p->stream); }) < bt) bkind = 3;
      c.tune.solve_kind = bkind;
      c.tune.solve_ts = bts;
      c.tune.solve_nw = bnw;
    } else {
      std::vector<int> lrs = {16, 32};
      if (c.D <= 64) lrs.insert(lrs.begin(), 8);
      pick([](stap::Tune& t, int v) { t.solve_lr = v; }, lrs,
           [&] { return do_solve(p, c, cov, wts, p->stream); });
      if (c.D > 64 && c.tune.solve_lr == 32)   // 8 or 16 warps
        pick([](stap::Tune& t, int v) { t.solve_nw = v; }, {0, 16},
             [&] { return do_solve(p, c, cov, wts, p->stream); });
    }
    if ((st = do_solve(p, c, cov, wts, p->stream)) != STAP_OK) break;
    if (stap::tc_precision(p->opt.precision) && stap::apply_tc_supported(d.training_block, d.n_steering))
      pick([](stap::Tune& t, int v) { t.apply_kind = v; }, {3, 1, 2},
           [&] { return do_apply(p, c, dop, wts, out, p->stream); });
    else
      pick([](stap::Tune& t, int v) { t.apply_kind = v; }, {1, 2},
           [&] { return do_apply(p, c, dop, wts, out, p->stream); });
    if (p->cpis.size() == 1) {  // the whole run, pipelined over range slabs or not
      // The candidates differ by a few percent and by how well the steps of
      // different slabs overlap, which depends on the cube being read cold
      // (as a new CPI is): before each timed run, writes to the output and
      // to every intermediate region (more than the L2 holds for the
      // standard CPI) evict it.  Seven rounds taken round-robin, reps runs
      // each; the candidate with the lowest median round wins (the minimum
      // rewarded rounds that happened to find part of the cube in L2).
      const size_t out_bytes = (size_t)d.n_steering * d.n_dop * d.n_range * sizeof(float);
      // dop, cov, wts (and training) regions; the front end's W table, kept
      // after them, must survive
      const size_t mid_bytes = (p->fe_N ? p->fe_w_off : p->run_bytes) - p->dop_off;
      auto cold_run = [&]() -> float {
        if (cudaMemsetAsync(out, 0, out_bytes, p->stream) != cudaSuccess ||
            cudaMemsetAsync(p->ws + p->dop_off, 0, mid_bytes, p->stream) != cudaSuccess)
          return kNever;
        cudaEventRecord(e0, p->stream);
        if (run_single(p, cube, out) != STAP_OK) return kNever;
        cudaEventRecord(e1, p->stream);
        if (cudaEventSynchronize(e1) != cudaSuccess) return kNever;
        float ms = kNever;
        cudaEventElapsedTime(&ms, e0, e1);
        return ms;
      };
      constexpr int kRounds = 7;
      constexpr int kCands = 4;
      const int cands[kCands] = {1, 2, 4, 8};
      float per_round[kCands][kRounds];
      // a CPI of tens of milliseconds gains nothing from overlapping its
      // short steps: one cold run decides whether to look at all
      c.tune.slabs = 1;
      const int rounds = cold_run() > 20.f ? 0 : kRounds;
      for (int round = 0; round < rounds; ++round)
        for (int k = 0; k < kCands; ++k) {
          c.tune.slabs = cands[k];
          float ms = run_single(p, cube, out) == STAP_OK ? 0.f : kNever;   // streams, untimed run
          for (int r = 0; r < reps && ms < kNever; ++r) {
            const float t = cold_run();
            ms = t >= kNever ? kNever : ms + t;
          }
          per_round[k][round] = ms;
        }
      float med[kCands];
      for (int k = 0; k < kCands; ++k) {
        med[k] = kNever;
        if (!rounds) continue;
        float v[kRounds];
        for (int r = 0; r < kRounds; ++r) v[r] = per_round[k][r];
        std::sort(v, v + kRounds);
        med[k] = v[kRounds / 2];
      }
      int bk = 0;
      for (int k = 1; k < kCands; ++k)
        if (med[k] < med[bk]) bk = k;
      c.tune.slabs = rounds ? cands[bk] : 1;
    }
    for (size_t j = i; j < p->cpis.size(); ++j)
      if (!tuned[j] && same_key(p->cpis[j].d, d)) {
        p->cpis[j].tune = c.tune;
        tuned[j] = 1;
      }
  }
  // a batch: the persistent or the multi-stream schedule, whichever replays faster
  if (st == STAP_OK && p->cpis.size() > 1) {
    float best = kNever;
    int bsched = p->batch_schedule;
    for (int sched : {(int)STAP_BATCH_PERSISTENT, (int)STAP_BATCH_STREAMS}) {
      p->batch_schedule = sched;
      drop_graph(p);
      if (run_batched(p, cubes, outs) != STAP_OK) continue;   // capture and first launch
      cudaEventRecord(e0, p->stream);
      bool ok = true;
      for (int r = 0; r < reps && ok; ++r) ok = run_batched(p, cubes, outs) == STAP_OK;
      cudaEventRecord(e1, p->stream);
      float ms = kNever;
      if (ok && cudaEventSynchronize(e1) == cudaSuccess) cudaEventElapsedTime(&ms, e0, e1);
      if (ms < best) {
        best = ms;
        bsched = sched;
      }
    }
    p->batch_schedule = bsched;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  drop_graph(p);
  // the timing runs may have counted failures: start clean
  if (cudaMemsetAsync(p->ws, 0, sizeof(DeviceStatus), p->stream) != cudaSuccess) return STAP_ERR_CUDA;
  return st;
}

stap_status stap_plan_get_tuning(stap_plan p, int32_t cpi, int32_t* choices) {
  if (!p || !choices || cpi < 0 || cpi >= (int32_t)p->cpis.size()) return STAP_ERR_INVALID_ARG;
  const stap::Tune& t = p->cpis[cpi].tune;
  const int32_t v[STAP_TUNING_LEN] = {t.dop_tr,   t.cov_kt,     t.solve_ts,   t.solve_nw, t.solve_lr,
                                      t.apply_kind, t.slabs,    t.solve_kind, t.cov_kind};
  for (int i = 0; i < STAP_TUNING_LEN; ++i) choices[i] = v[i];
  return STAP_OK;
}

stap_status stap_plan_set_tuning(stap_plan p, int32_t cpi, const int32_t* choices) {
  if (!p || !choices || cpi < 0 || cpi >= (int32_t)p->cpis.size()) return STAP_ERR_INVALID_ARG;
  for (int i = 0; i < STAP_TUNING_LEN; ++i)
    if (choices[i] < 0 || choices[i] > 64) return STAP_ERR_INVALID_ARG;
  stap::Tune& t = p->cpis[cpi].tune;
  t.dop_tr = choices[0];
  t.cov_kt = choices[1];
  t.solve_ts = choices[2];
  t.solve_nw = choices[3];
  t.solve_lr = choices[4];
  t.apply_kind = choices[5];
  t.slabs = choices[6];
  t.solve_kind = choices[7];
  t.cov_kind = choices[8];
  drop_graph(p);
  return STAP_OK;
}

stap_status stap_get_status(stap_plan p, int64_t* n_failed) {
  if (!p) return STAP_ERR_INVALID_ARG;
  if (!p->ws) return STAP_ERR_NO_WORKSPACE;
  DeviceStatus h{};
  if (cudaStreamSynchronize(p->stream) != cudaSuccess) return STAP_ERR_CUDA;
  if (cudaMemcpyAsync(&h, p->ws, sizeof(h), cudaMemcpyDeviceToHost, p->stream) != cudaSuccess ||
      cudaMemsetAsync(p->ws, 0, sizeof(DeviceStatus), p->stream) != cudaSuccess ||
      cudaStreamSynchronize(p->stream) != cudaSuccess)
    return STAP_ERR_CUDA;
  if (n_failed) *n_failed = (int64_t)h.n_failed;
  if (h.timeout) return STAP_ERR_TIMEOUT;
  return h.n_failed ? STAP_ERR_NOT_POSDEF : STAP_OK;
}

}  // extern "C"

namespace stap {
LaunchRecorder*& current_recorder() {
  thread_local LaunchRecorder* r = nullptr;
  return r;
}
}  // namespace stap
