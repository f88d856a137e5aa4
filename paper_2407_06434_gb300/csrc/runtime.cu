// Host runtime behind the C ABI of include/omp_gb300.h: handle and workspace management,
// dictionary preparation, the per-iteration launch sequence, CUDA-graph capture and replay.
//
// One solve is: set_args, init, compaction 0, then for k = 0..S-1 {correlate(k), update(k),
// compaction(k+1)}, then finalize. On the FP32 path correlate is a BF16 correlation, a selection
// and an overflow pass (filter.cu); where L2 does not hold the dictionary update is three launches
// (gather.cu); few signals take a form of their own between init and finalize (small.cu). Every
// kernel reads the live count of its iteration from device memory and returns at once past it, so
// the whole sequence is launch-invariant: it is captured once per (B, S, eps) into a CUDA graph and
// replayed with one cudaGraphLaunch, the per-call pointers travelling through a small device-side
// argument block.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"

using namespace ompk;

struct GraphEntry {
  int B, S;
  float eps;
  int prof;   // 1 if captured with profiling event nodes
  int stats;  // 1 if captured with the per-step margins recorded
  cudaGraphExec_t exec;
};

struct omp_handle_s {
  omp_desc d{};
  int dev = 0;
  int sm_count = 0;
  Ws ws{};
  TcPlan* tc = nullptr;
  const float* prepared_A = nullptr;
  CallArgs* args_dev = nullptr;
  cudaStream_t cap_stream = nullptr;
  cudaStream_t body_stream = nullptr;  // captures the body of the graph's while loop
  std::vector<GraphEntry> graphs;
  std::vector<void*> allocs;
  float* y_stage = nullptr;
  float* x_stage = nullptr;
  int* s_stage = nullptr;
  float* margin_buf = nullptr;                // Bmax x Smax per-step margins (when requested)
  unsigned long long* cand2_buf = nullptr;    // FP32 path: runner-up keys (when requested)
  // profiling: events[(kind * Smax + k) * 2 + {0: start, 1: end}], kind 0 = correlate, 1 = update
  bool prof_on = false;
  int prof_last_S = 0;
  bool prof_last_valid = false;
  std::vector<cudaEvent_t> prof_ev;
};

namespace {

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

bool fault_alloc_due() {
  // test hook: OMP_FAULT_ALLOC_AT=n makes the n-th workspace allocation of a handle fail
  static int counter = 0;
  const char* v = std::getenv("OMP_FAULT_ALLOC_AT");
  if (!v) return false;
  const int at = std::atoi(v);
  return at > 0 && ++counter == at;
}

bool device_alloc(omp_handle_s* h, void** p, size_t bytes) {
  *p = nullptr;
  // test hook: OMP_FAULT_ALLOC_BYTES=n makes allocations of more than n bytes fail
  const char* v = std::getenv("OMP_FAULT_ALLOC_BYTES");
  if (v && bytes > std::strtoull(v, nullptr, 10)) return false;
  if (cudaMalloc(p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  h->allocs.push_back(*p);
  return true;
}

// A handle's workspaces come from one allocation: each is asked for, then all pointers are set. (One
// cudaMalloc and cudaFree per workspace, about forty, made up most of creating and destroying a
// handle: 470 and 300 us, which a caller with one batch per dictionary pays every time.)
struct Arena {
  struct Want {
    void** p;
    size_t at;
  };
  std::vector<Want> wants;
  size_t bytes = 0;

  template <class T>
  bool ask(T** p, size_t count) {
    *p = nullptr;
    if (count == 0) return true;
    if (fault_alloc_due()) return false;
    wants.push_back({reinterpret_cast<void**>(p), bytes});
    bytes += (count * sizeof(T) + 511) / 512 * 512;
    return true;
  }
  bool allocate(omp_handle_s* h) {
    void* base = nullptr;
    if (!device_alloc(h, &base, bytes)) return false;
    for (const Want& w : wants) *w.p = static_cast<char*>(base) + w.at;
    return true;
  }
};

void release(omp_handle_s* h) {
  for (auto& g : h->graphs) cudaGraphExecDestroy(g.exec);
  h->graphs.clear();
  for (cudaEvent_t e : h->prof_ev) cudaEventDestroy(e);
  h->prof_ev.clear();
  if (h->tc) tc_destroy(h->tc);
  h->tc = nullptr;
  for (void* p : h->allocs) cudaFree(p);
  h->allocs.clear();
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  h->cap_stream = nullptr;
  if (h->body_stream) cudaStreamDestroy(h->body_stream);
  h->body_stream = nullptr;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

omp_status check_launch() {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

void enqueue_correlate(omp_handle_s* h, const Ws& ws, int k, int B, cudaStream_t s) {
  if (ws.prec == OMP_PREC_FP32 && !ws.filt) {
    launch_corr_simt(ws, k, B, s);
    return;
  }
  launch_corr_tc(ws, h->tc, k, B, s);
  if (ws.filt) {
    launch_filter_select(ws, k, B, s);
    launch_corr_overflow(ws, k, B, s);
  }
}

// The FP32 path's filter pays from about 3e8 products a step on, and for rows of 256 elements and
// more always: the tile kernel then takes a chain of that many products at least. Measured, us a
// step with and without: 64 x 256, 2000 signals 29 / 23; 128 x 512, 2000 29 / 27; 128 x 1024, 4000
// 33 / 48; 100 x 8000, 500 31 / 43; 256 x 512, 100 22 / 22; 256 x 1024, 1000 28 / 32; 512 x 2048,
// 16 27 / 42; 256 x 1024, 5000 44 / 81.
bool large_step(const Ws& w, int B) { return static_cast<double>(w.N) * w.Mp * B >= 3e8; }
bool filter_pays(const Ws& w, int B) { return w.Mp >= 256 || large_step(w, B); }

// FP32 path: every atom scored in FP32
void no_filter(Ws& w) {
  w.filt = 0;
  w.tcprec = w.prec;
}

// The workspace view a solve runs with: the handle's own, or -- when the caller asks for each
// step's top-two margin -- one whose kernels record it: the FP32 correlation also merges the
// runner-up's key, and the quantised paths run without the score bound (every candidate
// rescored in FP32, no pruning), which picks the same atoms (the exactness tests compare the two).
Ws solve_ws(const omp_handle_s* h, int B, bool stats) {
  Ws w = h->ws;
  if (w.filt && (stats || !filter_pays(w, B))) no_filter(w);
  if (stats) {
    w.margin = h->margin_buf;
    w.cand2 = w.prec == OMP_PREC_FP32 ? h->cand2_buf : nullptr;
    w.rescore_eps = 0.f;
    w.tau = nullptr;
    w.tau_pos = nullptr;
    w.win_pos = nullptr;
    w.ea = nullptr;
  }
  return w;
}

void prof_mark(omp_handle_s* h, bool prof, int kind, int k, int end, cudaStream_t s) {
  if (!prof) return;
  cudaEventRecordWithFlags(h->prof_ev[(static_cast<size_t>(kind) * h->ws.Smax + k) * 2 + end], s,
                           cudaEventRecordExternal);
}

// A solve of few signals (small.cu), where the sizes and options take one of those forms.
bool enqueue_small(omp_handle_s* h, const Ws& ws, int B, int S, float eps, cudaStream_t s) {
  const int form = small_form(ws, B, eps);
  if (form == 0) return false;
  launch_init(ws, h->args_dev, B, s);
  if (form == 1)
    launch_solo(ws, B, S, eps, h->d.eps_relative, s);
  else
    for (int k = 0; k < S; ++k) launch_wide(ws, h->sm_count, B, S, eps, h->d.eps_relative, s);
  launch_finalize(ws, h->args_dev, B, S, s);
  return true;
}

void enqueue_solve(omp_handle_s* h, const Ws& ws, int B, int S, float eps, bool prof, cudaStream_t s) {
  launch_init(ws, h->args_dev, B, s);
  launch_compact(ws, 0, B, S, false, s);
  for (int k = 0; k < S; ++k) {
    prof_mark(h, prof, 0, k, 0, s);
    enqueue_correlate(h, ws, k, B, s);
    prof_mark(h, prof, 0, k, 1, s);
    prof_mark(h, prof, 1, k, 0, s);
    launch_update(ws, k, B, S, eps, h->d.eps_relative, s);
    prof_mark(h, prof, 1, k, 1, s);
    if (k + 1 < S) launch_compact(ws, k + 1, B, S, true, s);
  }
  launch_finalize(ws, h->args_dev, B, S, s);
}

// The same solve as one graph whose iterations are a device-side while loop (a conditional
// node): the body (correlate, update, compact, advance) reads the iteration from the counter
// that the init kernel zeroes, and the advance kernel ends the loop after S iterations or as
// soon as no signal is live, so a batch that converges early launches no further kernels.
bool capture_while_solve(omp_handle_s* h, const Ws& ws, int B, int S, float eps, cudaGraph_t* out) {
  cudaStream_t s = h->cap_stream;
  *out = nullptr;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return false;
  launch_init(ws, h->args_dev, B, s);
  launch_compact(ws, 0, B, S, false, s);
  cudaStreamCaptureStatus st;
  cudaGraph_t g = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t nd = 0;
  bool ok = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, &deps, nullptr, &nd) == cudaSuccess &&
            st == cudaStreamCaptureStatusActive;
  cudaGraphConditionalHandle cond{};
  cudaGraphNode_t node = nullptr;
  cudaGraph_t body = nullptr;
  if (ok) ok = cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault) == cudaSuccess;
  if (ok) {
    cudaGraphNodeParams np{};
    np.type = cudaGraphNodeTypeConditional;
    np.conditional.handle = cond;
    np.conditional.type = cudaGraphCondTypeWhile;
    np.conditional.size = 1;
    ok = cudaGraphAddNode(&node, g, deps, nullptr, nd, &np) == cudaSuccess;
    if (ok) body = np.conditional.phGraph_out[0];
  }
  if (ok)
    ok = cudaStreamBeginCaptureToGraph(h->body_stream, body, nullptr, nullptr, 0,
                                       cudaStreamCaptureModeThreadLocal) == cudaSuccess;
  if (ok) {
    enqueue_correlate(h, ws, -1, B, h->body_stream);
    launch_update(ws, -1, B, S, eps, h->d.eps_relative, h->body_stream);
    launch_compact(ws, -1, B, S, true, h->body_stream);
    launch_advance(ws, S, cond, h->body_stream);
    cudaGraph_t tmp = nullptr;
    ok = cudaStreamEndCapture(h->body_stream, &tmp) == cudaSuccess;
  }
  if (ok) ok = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies) == cudaSuccess;
  if (ok) launch_finalize(ws, h->args_dev, B, S, s);
  cudaGraph_t graph = nullptr;
  const bool ended = cudaStreamEndCapture(s, &graph) == cudaSuccess && graph != nullptr;
  if (!ok || !ended) {
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    return false;
  }
  *out = graph;
  return true;
}

void enqueue_topk(omp_handle_s* h, const float* R, int B, int topk, cudaStream_t s) {
  Ws ws = h->ws;
  if (ws.filt) no_filter(ws);  // the score is an output
  // the lists are the output: no threshold, and no window, which is sized by the residual norms and
  // quantisation errors of a solve's signals
  ws.tau = nullptr;
  ws.tau_pos = nullptr;
  ws.win_pos = nullptr;
  ws.ea = nullptr;
  launch_load_rows(ws, R, B, s);
  launch_compact(ws, 0, B, 1, false, s);
  enqueue_correlate(h, ws, 0, B, s);
  launch_topk_out(ws, h->args_dev, B, topk, s);
}

omp_status prepare(omp_handle_s* h, const float* A, cudaStream_t s) {
  if (h->ws.ea && cudaMemsetAsync(h->ws.ea, 0, sizeof(float), s) != cudaSuccess) return OMP_ERR_CUDA;
  launch_prep(h->ws, A, s);
  launch_gram_simt(h->ws, s);
  const omp_status st = check_launch();
  if (st == OMP_OK) h->prepared_A = A;
  return st;
}

omp_status run_solve(omp_handle_s* h, int B, int S, float eps, bool stats, cudaStream_t stream) {
  const bool prof = h->prof_on;
  h->prof_last_S = S;
  h->prof_last_valid = prof;
  const Ws ws = solve_ws(h, B, stats);
  if (!h->d.use_graph) {
    if (prof || !enqueue_small(h, ws, B, S, eps, stream)) enqueue_solve(h, ws, B, S, eps, prof, stream);
    return check_launch();
  }
  for (auto& g : h->graphs)
    if (g.prof == static_cast<int>(prof) && g.stats == static_cast<int>(stats) && g.B == B &&
        g.S == S && g.eps == eps)
      return cudaGraphLaunch(g.exec, stream) == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
  // capture on the handle's own stream (capture only records; the replay below runs in the
  // caller's stream order)
  // The unrolled form is the default: on GB300 each pass of a conditional while node costs about
  // 5.5 us more than an unrolled iteration, which is about what three launches that return at
  // once cost, so the loop saves nothing even when a batch converges early. The profiled form
  // is always unrolled, with an event pair around each kernel.
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  bool ok = false;
  if (prof) {
    ok = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      enqueue_solve(h, ws, B, S, eps, prof, h->cap_stream);
      ok = cudaStreamEndCapture(h->cap_stream, &graph) == cudaSuccess && graph != nullptr;
    }
  } else if (h->d.use_graph == 2) {
    ok = capture_while_solve(h, ws, B, S, eps, &graph);
  } else {
    ok = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      if (!enqueue_small(h, ws, B, S, eps, h->cap_stream)) enqueue_solve(h, ws, B, S, eps, false, h->cap_stream);
      ok = cudaStreamEndCapture(h->cap_stream, &graph) == cudaSuccess && graph != nullptr;
    }
  }
  if (ok) ok = cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess;
  if (graph) cudaGraphDestroy(graph);
  if (!ok) {
    cudaGetLastError();
    return OMP_ERR_CUDA;
  }
  h->graphs.push_back(GraphEntry{B, S, eps, static_cast<int>(prof), static_cast<int>(stats), exec});
  return cudaGraphLaunch(exec, stream) == cudaSuccess ? OMP_OK : OMP_ERR_CUDA;
}

omp_status validate_solve(omp_handle_s* h, const float* A, const float* Y, int64_t B, int32_t S,
                          float eps, const void* X, const void* sup) {
  if (!h || !A || !Y || !X || !sup) return OMP_ERR_INVALID_ARGUMENT;
  if (B < 1 || B > h->d.max_batch) return OMP_ERR_INVALID_ARGUMENT;
  if (S < 1 || S > h->d.max_iters) return OMP_ERR_INVALID_ARGUMENT;
  if (!(eps >= 0.f) || !std::isfinite(eps)) return OMP_ERR_INVALID_ARGUMENT;
  if (!aligned16(A) || !aligned16(Y) || !aligned16(X) || !aligned16(sup))
    return OMP_ERR_INVALID_ARGUMENT;
  return OMP_OK;
}

}  // namespace

extern "C" {

void omp_desc_default(omp_desc* d, int64_t M, int64_t N) {
  if (!d) return;
  std::memset(d, 0, sizeof(*d));
  d->M = M;
  d->N = N;
  d->max_batch = 4096;
  int64_t s = M < N ? M : N;
  d->max_iters = static_cast<int32_t>(s < 64 ? s : 64);
  d->precision = OMP_PREC_BF16;
  d->rescore_topk = 8;
  d->eps_relative = 1;
  d->use_graph = 1;
  d->device = 0;
}

const char* omp_status_string(omp_status s) {
  switch (s) {
    case OMP_OK: return "OMP_OK";
    case OMP_ERR_INVALID_ARGUMENT: return "OMP_ERR_INVALID_ARGUMENT";
    case OMP_ERR_UNSUPPORTED_DEVICE: return "OMP_ERR_UNSUPPORTED_DEVICE";
    case OMP_ERR_OUT_OF_MEMORY: return "OMP_ERR_OUT_OF_MEMORY";
    case OMP_ERR_CUDA: return "OMP_ERR_CUDA";
    case OMP_ERR_DEVICE_TIMEOUT: return "OMP_ERR_DEVICE_TIMEOUT";
    case OMP_ERR_NUMERICAL: return "OMP_ERR_NUMERICAL";
  }
  return "OMP_ERR_UNKNOWN";
}

// |quantised score - FP32 score| <= bound ||a|| ||r|| (the FP8 score taken in the units of the
// residual's scale). BF16 rounding of a and r (unit roundoff u = 2^-8) gives 2u + u^2 of
// sum |a_m r_m| <= ||a|| ||r||. E4M3 with a per-row scale s = amax / 448 rounds each element to
// within u |x| + beta s, u = 2^-4 in the normal range and beta = 2^-10 (half the subnormal
// spacing) below it; with s <= ||x|| / 448 and sum |x_m| <= sqrt(Mp) ||x|| that is
// 2u + u^2 + 2 sqrt(Mp) b (1 + u) + Mp b^2 with b = 2^-10 / 448. The tensor-core accumulation is
// allowed 2^-22 and the FP32 rescoring 2^-24 per addition over Mp terms; 1% covers the rounding
// of inv_norm, of the scales and of the stored ||r||.
float omp_score_error_bound(int32_t precision, int64_t Mp) {
  if (Mp < 1) return 0.f;
  const double m = static_cast<double>(Mp);
  const double g_tc = m * std::ldexp(1.0, -22) / (1.0 - m * std::ldexp(1.0, -22));
  const double g_32 = m * std::ldexp(1.0, -24) / (1.0 - m * std::ldexp(1.0, -24));
  if (precision == OMP_PREC_BF16) {
    const double u = std::ldexp(1.0, -8);
    return static_cast<float>(1.01 * (2 * u + u * u + (1 + u) * (1 + u) * g_tc + g_32));
  }
  if (precision == OMP_PREC_FP8_E4M3) {
    const double u = std::ldexp(1.0, -4), b = std::ldexp(1.0, -10) / 448.0, sb = std::sqrt(m) * b;
    return static_cast<float>(
        1.01 * (2 * u + u * u + 2 * sb * (1 + u) + m * b * b + (1 + u + sb) * (1 + u + sb) * g_tc + g_32));
  }
  return 0.f;
}

omp_status omp_create(const omp_desc* desc, omp_handle* out) {
  if (!desc || !out) return OMP_ERR_INVALID_ARGUMENT;
  *out = nullptr;
  const omp_desc d = *desc;
  if (d.M < 1 || d.M > 8192 || d.N < 2 || d.N > 65536 || d.max_batch < 1 ||
      d.max_batch > (1 << 24) || d.max_iters < 1 || d.max_iters > 256 || d.max_iters > d.M ||
      d.max_iters > d.N || d.precision < 0 || d.precision > 2 || d.rescore_topk < 0 ||
      d.rescore_topk > kMaxTopk || d.use_graph < 0 || d.use_graph > 2 || d.gather24 < 0 ||
      d.gather24 > 1)
    return OMP_ERR_INVALID_ARGUMENT;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || d.device < 0 || d.device >= ndev) {
    cudaGetLastError();
    return OMP_ERR_UNSUPPORTED_DEVICE;
  }
  int major = 0, minor = 0, sms = 0;  // (the attributes alone: the whole property record takes long to fill)
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, d.device) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, d.device) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d.device) != cudaSuccess)
    return OMP_ERR_CUDA;
  if (major != 10 || minor != 3) return OMP_ERR_UNSUPPORTED_DEVICE;
  DeviceGuard guard(d.device);

  omp_handle_s* h = new (std::nothrow) omp_handle_s();
  if (!h) return OMP_ERR_OUT_OF_MEMORY;
  h->d = d;
  if (h->d.rescore_topk == 0) h->d.rescore_topk = kMaxTopk;
  h->dev = d.device;
  h->sm_count = sms;
  Ws& ws = h->ws;
  ws.sms = sms;
  ws.M = static_cast<int>(d.M);
  // one tensor-core K stage is 128 bytes: 64 BF16 or 128 E4M3 elements
  const int64_t malign = d.precision == OMP_PREC_FP8_E4M3 ? 2 * kMpAlign : kMpAlign;
  ws.Mp = static_cast<int>((d.M + malign - 1) / malign * malign);
  ws.N = static_cast<int>(d.N);
  ws.ldg = (ws.N + 3) / 4 * 4;
  ws.Smax = d.max_iters;
  ws.Bmax = static_cast<int>(d.max_batch);
  ws.Bpad = (ws.Bmax + kSigTile - 1) / kSigTile * kSigTile;
  ws.prec = d.precision;
  ws.topk = d.precision == OMP_PREC_FP32 ? 1 : h->d.rescore_topk;
  // (test hook: OMP_RESCORE_ALWAYS=1 turns the score bound, and all that uses it, off)
  const char* always = std::getenv("OMP_RESCORE_ALWAYS");
  ws.rescore_eps = always && std::atoi(always) == 1 ? 0.f : omp_score_error_bound(ws.prec, ws.Mp);
  {
    const double m = static_cast<double>(ws.Mp);
    ws.gam_tc = static_cast<float>(m * std::ldexp(1.0, -22) / (1.0 - m * std::ldexp(1.0, -22)));
    ws.gam_32 = static_cast<float>(m * std::ldexp(1.0, -24) / (1.0 - m * std::ldexp(1.0, -24)));
  }
  // padded to 4 entries so each signal's FP32 factor starts on a 16-byte boundary
  ws.Fstride = (static_cast<int64_t>(ws.Smax) * (ws.Smax + 1) / 2 + 3) / 4 * 4;
  ws.upd_w = update_default_warps(ws.Mp);
  const bool hook = always && std::atoi(always) == 1;
  ws.tc_cl = 1;
  const size_t N = ws.N, Mp = ws.Mp, Bm = ws.Bmax, Bp = ws.Bpad, Sm = ws.Smax;
  const size_t Npad = (N + 255) / 256 * 256;
  // Every workspace, or (lean) all but those that only make solves faster: the FP32 path's filter, the
  // longer candidate lists and the rows of a gather in a launch of its own.
  auto ask_all = [&](Arena& ar, bool lean) {
    // The FP32 path filters its atoms with a BF16 correlation, if a batch of this handle can gain by it.
    // (The test hook that turns the score bound off turns this off too.)
    ws.filt = d.precision == OMP_PREC_FP32 && !hook && !lean && filter_pays(ws, ws.Bmax) ? 1 : 0;
    ws.tcprec = ws.filt ? OMP_PREC_BF16 : ws.prec;
    const bool tc = ws.tcprec != OMP_PREC_FP32;
    if (tc) tc_fill_sched(ws, h->sm_count, lean ? kLeanPieces : kPieces);
    const size_t qbytes = ws.tcprec == OMP_PREC_BF16 ? 2 : 1;
    bool ok = true;
    ok = ok && ar.ask(&ws.A32, N * Mp);
    if (d.gather24) ok = ok && ar.ask(&ws.A24h, N * Mp) && ar.ask(&ws.A24l, N * Mp);
    if (ws.tcprec == OMP_PREC_BF16) ok = ok && ar.ask(&ws.A16, N * Mp);
    if (d.precision == OMP_PREC_FP8_E4M3) ok = ok && ar.ask(&ws.A8, N * Mp) && ar.ask(&ws.sa, N);
    if (tc) ok = ok && ar.ask(&ws.escale, Npad);
    ok = ok && ar.ask(&ws.inv_norm, N) && ar.ask(&ws.norm2, N) && ar.ask(&ws.gram, N * ws.ldg);
    ok = ok && ar.ask(&ws.R32, Bm * Mp);
    if (tc) {
      ok = ok && ar.ask(reinterpret_cast<uint8_t**>(&ws.Rq[0]), Bp * Mp * qbytes) &&
           ar.ask(reinterpret_cast<uint8_t**>(&ws.Rq[1]), Bp * Mp * qbytes);
      ok = ok && ar.ask(&ws.sr[0], Bp) && ar.ask(&ws.sr[1], Bp);
      ok = ok && ar.ask(&ws.cand_s, Bp * ws.pieces * kMaxTopk) &&
           ar.ask(&ws.cand_i, Bp * ws.pieces * kMaxTopk);
    }
    // The pruning thresholds (and the data-driven bound they carry): on BF16 always; on E4M3,
    // whose worst-case bound is too loose to prune, only where the one-warp update quantises the
    // next row itself and so can measure its rounding error (padded lengths up to 1024).
    const bool want_tau = ws.prec == OMP_PREC_BF16 ||
                          (ws.prec == OMP_PREC_FP8_E4M3 && update_default_warps(ws.Mp) == 1);
    if (want_tau && ws.rescore_eps > 0.f && ws.Smax <= kTauSmax)
      ok = ok && ar.ask(&ws.tau, Bm) && ar.ask(&ws.tau_pos, Bp) && ar.ask(&ws.win_pos, Bp) &&
           (ws.prec != OMP_PREC_FP8_E4M3 || ar.ask(&ws.ea, 1));
    if (ws.filt)
      ok = ok && ar.ask(&ws.win_pos, Bp) && ar.ask(&ws.ea, 1) && ar.ask(&ws.ovf, Bm) &&
           ar.ask(&ws.ovf_cnt, Sm + 1);
    ok = ok && ar.ask(&ws.live[0], Bm) && ar.ask(&ws.live[1], Bm);
    ok = ok && ar.ask(&ws.livek[0], Bm) && ar.ask(&ws.livek[1], Bm);
    ok = ok && ar.ask(&ws.cnt, Sm + 2) && ar.ask(&ws.kdev, 1) && ar.ask(&ws.flag, Bm) && ar.ask(&ws.cand1, Bm);
    ok = ok && ar.ask(&ws.upd_ctr, Sm + 1);
    if (!lean && gather_apart_shape(ws.N, ws.Mp, ws.Bmax)) ok = ok && ar.ask(&ws.sel, Bm) && ar.ask(&ws.Q, Bm * Mp);
    ok = ok && ar.ask(&ws.score, small_score_floats(ws.N, ws.Bmax));
    ok = ok && ar.ask(&ws.F, Bm * static_cast<size_t>(ws.Fstride)) &&
         ar.ask(&ws.F32, Bm * static_cast<size_t>(ws.Fstride)) && ar.ask(&ws.bv, Bm * Sm) &&
         ar.ask(&ws.sup, Bm * Sm);
    ok = ok && ar.ask(&ws.drop, Bm * Sm) && ar.ask(&ws.fb, Bm);
    ok = ok && ar.ask(&ws.ynorm, Bm) && ar.ask(&ws.rnorm, Bm) && ar.ask(&ws.niter, Bm) &&
         ar.ask(&ws.stop, Bm) && ar.ask(&ws.err, 1) && ar.ask(&h->args_dev, 1);
    ok = ok && ar.ask(&h->y_stage, Bm * static_cast<size_t>(ws.M)) &&
         ar.ask(&h->x_stage, Bm * Sm) && ar.ask(&h->s_stage, Bm * Sm) &&
         ar.ask(&h->margin_buf, Bm * Sm);
    if (d.precision == OMP_PREC_FP32) ok = ok && ar.ask(&h->cand2_buf, Bm);
    return ok;
  };
  Arena full, lean;
  const bool ok = ask_all(full, false) && (full.allocate(h) || (ask_all(lean, true) && lean.allocate(h)));
  if (!ok) {
    release(h);
    delete h;
    return OMP_ERR_OUT_OF_MEMORY;
  }
  const bool tc = ws.tcprec != OMP_PREC_FP32;
  bool cuda_ok = cudaMemset(ws.err, 0, sizeof(unsigned)) == cudaSuccess &&
                 (!ws.escale || cudaMemset(ws.escale, 0, Npad * sizeof(float)) == cudaSuccess) &&
                 cudaMemset(ws.cand1, 0, Bm * sizeof(unsigned long long)) == cudaSuccess &&
                 (!h->cand2_buf || cudaMemset(h->cand2_buf, 0, Bm * sizeof(unsigned long long)) == cudaSuccess) &&
                 (!ws.tau || cudaMemset(ws.tau, 0xff, Bm * sizeof(TauRec)) == cudaSuccess) &&
                 (!ws.tau_pos || cudaMemset(ws.tau_pos, 0, Bp * sizeof(float)) == cudaSuccess) &&
                 (!ws.win_pos || cudaMemset(ws.win_pos, 0, Bp * sizeof(float)) == cudaSuccess) &&
                 cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking) == cudaSuccess &&
                 (d.use_graph != 2 ||
                  cudaStreamCreateWithFlags(&h->body_stream, cudaStreamNonBlocking) == cudaSuccess) &&
                 configure_update_kernels(ws) == cudaSuccess && configure_corr_simt(ws) == cudaSuccess &&
                 configure_small(ws) == cudaSuccess;
  if (cuda_ok && tc) cuda_ok = tc_setup(ws, h->sm_count, &h->tc) == cudaSuccess;
  if (cuda_ok) cuda_ok = cudaDeviceSynchronize() == cudaSuccess;
  if (!cuda_ok) {
    cudaGetLastError();
    release(h);
    delete h;
    return OMP_ERR_CUDA;
  }
  *out = h;
  return OMP_OK;
}

omp_status omp_destroy(omp_handle h) {
  if (!h) return OMP_OK;
  {
    DeviceGuard guard(h->dev);
    cudaDeviceSynchronize();
    release(h);
  }
  delete h;
  return OMP_OK;
}

omp_status omp_prepare_dictionary(omp_handle h, const float* A, void* stream) {
  if (!h || !A || !aligned16(A)) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  return prepare(h, A, static_cast<cudaStream_t>(stream));
}

omp_status omp_solve_batch_ex(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S,
                              float eps, float* X_out, int32_t* support_out, int32_t* n_iter_out,
                              float* resid_norm_out, float* margin_out, int32_t* stop_out,
                              void* stream) {
  omp_status st = validate_solve(h, A, Y, B, S, eps, X_out, support_out);
  if (st != OMP_OK) return st;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A != h->prepared_A) {
    st = prepare(h, A, s);
    if (st != OMP_OK) return st;
  }
  CallArgs a{};
  a.Y = Y;
  a.X = X_out;
  a.support = support_out;
  a.n_iter = n_iter_out;
  a.resid = resid_norm_out;
  a.stop = stop_out;
  a.margin = margin_out;
  launch_set_args(h->args_dev, a, s);
  st = check_launch();
  if (st != OMP_OK) return st;
  return run_solve(h, static_cast<int>(B), S, eps, margin_out != nullptr, s);
}

omp_status omp_solve_batch_trace(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S,
                                 float eps, float* X_out, int32_t* support_out, float* drop_out,
                                 void* stream) {
  omp_status st = validate_solve(h, A, Y, B, S, eps, X_out, support_out);
  if (st != OMP_OK || !drop_out) return st != OMP_OK ? st : OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A != h->prepared_A) {
    st = prepare(h, A, s);
    if (st != OMP_OK) return st;
  }
  CallArgs a{};
  a.Y = Y;
  a.X = X_out;
  a.support = support_out;
  a.drop = drop_out;
  launch_set_args(h->args_dev, a, s);
  st = check_launch();
  if (st != OMP_OK) return st;
  return run_solve(h, static_cast<int>(B), S, eps, false, s);
}

omp_status omp_solve_batch_gram(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S,
                                float eps, float* X_out, int32_t* support_out, int32_t* n_iter_out,
                                float* resid_norm_out, int32_t* stop_out, void* stream) {
  omp_status st = validate_solve(h, A, Y, B, S, eps, X_out, support_out);
  if (st != OMP_OK) return st;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (!h->ws.c0) {  // first use: the first-correlation workspace and the kernel's shared memory
    if (configure_gram_solve(h->ws) != cudaSuccess) {
      cudaGetLastError();
      return OMP_ERR_INVALID_ARGUMENT;
    }
    if (configure_c0_simt() != cudaSuccess) return OMP_ERR_CUDA;
    if (fault_alloc_due() || !device_alloc(h, reinterpret_cast<void**>(&h->ws.c0),
                                           static_cast<size_t>(h->ws.Bmax) * h->ws.ldg * sizeof(float)))
      return OMP_ERR_OUT_OF_MEMORY;
  }
  if (A != h->prepared_A) {
    st = prepare(h, A, s);
    if (st != OMP_OK) return st;
  }
  CallArgs a{};
  a.Y = Y;
  a.X = X_out;
  a.support = support_out;
  a.n_iter = n_iter_out;
  a.resid = resid_norm_out;
  a.stop = stop_out;
  launch_set_args(h->args_dev, a, s);
  const Ws& ws = h->ws;
  launch_init(ws, h->args_dev, static_cast<int>(B), s);
  launch_c0_simt(ws, static_cast<int>(B), s);
  launch_gram_solve(ws, h->args_dev, static_cast<int>(B), S, eps, h->d.eps_relative, s);
  launch_finalize(ws, h->args_dev, static_cast<int>(B), S, s);
  return check_launch();
}

namespace {
omp_status solve_candidates(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S, float eps,
                            omp_proposal p, const int32_t* cand, int32_t K, const float* tau, float* X_out,
                            int32_t* support_out, int32_t* n_iter_out, float* resid_norm_out,
                            int32_t* fallback_out, cudaStream_t s);
}

omp_status omp_solve_batch_candidates(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S,
                                      float eps, const int32_t* cand, int32_t K, const float* tau,
                                      float* X_out, int32_t* support_out, int32_t* n_iter_out,
                                      float* resid_norm_out, int32_t* fallback_out, void* stream) {
  omp_status st = validate_solve(h, A, Y, B, S, eps, X_out, support_out);
  if (st != OMP_OK) return st;
  if (!cand || !tau || K < 1 || K > 256 || K > h->d.N) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  return solve_candidates(h, A, Y, B, S, eps, nullptr, cand, K, tau, X_out, support_out, n_iter_out,
                          resid_norm_out, fallback_out, static_cast<cudaStream_t>(stream));
}

omp_status omp_solve_batch_learned(omp_handle h, omp_proposal p, const float* A, const float* Y,
                                   int64_t B, int32_t S, float eps, float* X_out,
                                   int32_t* support_out, int32_t* n_iter_out,
                                   float* resid_norm_out, int32_t* fallback_out, void* stream) {
  omp_status st = validate_solve(h, A, Y, B, S, eps, X_out, support_out);
  if (st != OMP_OK) return st;
  if (!p || S > proposal_tau_len(p)) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  return solve_candidates(h, A, Y, B, S, eps, p, proposal_candidates(p), proposal_topk(p), proposal_tau(p),
                          X_out, support_out, n_iter_out, resid_norm_out, fallback_out,
                          static_cast<cudaStream_t>(stream));
}

}  // extern "C"

namespace {
// Candidate-restricted OMP followed by the dense loop for the signals that fell back. With a
// proposal `p`, its inference (features, MLP, top-K) fills `cand` first.
omp_status solve_candidates(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S, float eps,
                            omp_proposal p, const int32_t* cand, int32_t K, const float* tau, float* X_out,
                            int32_t* support_out, int32_t* n_iter_out, float* resid_norm_out,
                            int32_t* fallback_out, cudaStream_t s) {
  omp_status st;
  if (A != h->prepared_A) {
    st = prepare(h, A, s);
    if (st != OMP_OK) return st;
  }
  CallArgs a{};
  a.Y = Y;
  a.X = X_out;
  a.support = support_out;
  a.n_iter = n_iter_out;
  a.resid = resid_norm_out;
  a.fallback = fallback_out;
  launch_set_args(h->args_dev, a, s);
  const int b = static_cast<int>(B);
  Ws ws = solve_ws(h, b, false);
  // the dense loop has few signals left, often none, so that the filter's two launches a step count
  // (one signal, 16 steps, 256 x 1024: 390 us a solve with them, 272 without)
  if (ws.filt && !large_step(ws, b)) no_filter(ws);
  launch_init(ws, h->args_dev, b, s);
  if (p && !proposal_run_inference(p, A, Y, b, s)) return OMP_ERR_CUDA;
  if (!launch_restricted(ws, h->args_dev, cand, K, tau, b, S, eps, h->d.eps_relative, ws.fb, s))
    return OMP_ERR_CUDA;
  // signals that failed the residual-drop check continue in the dense loop
  launch_compact(ws, 0, b, S, false, s);
  for (int k = 0; k < S; ++k) {
    enqueue_correlate(h, ws, k, b, s);
    launch_update(ws, k, b, S, eps, h->d.eps_relative, s);
    if (k + 1 < S) launch_compact(ws, k + 1, b, S, true, s);
  }
  launch_finalize(ws, h->args_dev, b, S, s);
  return check_launch();
}
}  // namespace

extern "C" {

omp_status omp_autotune(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S, float eps,
                        int32_t repeats, int32_t* choice_out, void* stream) {
  if (!h || !A || !Y || B < 1 || B > h->d.max_batch || S < 1 || S > h->d.max_iters || repeats < 1)
    return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const char* cache = std::getenv("OMP_AUTOTUNE_CACHE");
  char key[256];
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, h->dev) != cudaSuccess) return OMP_ERR_CUDA;
  std::snprintf(key, sizeof(key), "%.64s M=%d N=%d prec=%d B=%lld S=%d", prop.name, h->ws.M, h->ws.N,
                h->ws.prec, static_cast<long long>(B), S);
  const bool tc = h->ws.prec != OMP_PREC_FP32;
  // a launch shape: update warps per signal, correlation stages, persistent CTAs (asked for;
  // a pair launch takes the largest even number whose pairs fit at once), update persistent
  // form, correlation CTAs per cluster (1, or 2 for the 2-SM MMA pair)
  struct Shape {
    int w, stages, grid, persist, cl;
  };
  auto fitted = [&](const Shape& c) {
    return tc ? tc_fit_grid(h->ws.prec, c.stages, c.cl, c.grid) : c.grid;
  };
  auto valid = [&](const Shape& c) {
    return update_slots(h->ws.Mp, c.w) != 0 && (c.persist == 0 || c.persist == 1) &&
           (!tc || (c.stages >= 2 && c.stages <= 6 && c.grid >= 1 && c.grid <= h->sm_count &&
                    (c.cl == 1 || c.cl == 2) && fitted(c) >= c.cl));
  };
  const Shape saved{h->ws.upd_w, h->ws.tc_stages, h->ws.tc_grid, h->ws.upd_persist, h->ws.tc_cl};
  Shape best{0, saved.stages, saved.grid, saved.persist, saved.cl};
  if (cache) {  // a previous run's choice: "key|w", "key|w,stages,grid", "key|w,stages,grid,persist"
                // or "key|w,stages,grid,persist,cluster"
    if (FILE* f = std::fopen(cache, "r")) {
      char line[512];
      while (std::fgets(line, sizeof(line), f)) {
        char* bar = std::strrchr(line, '|');
        Shape c = saved;
        const int n = bar ? std::sscanf(bar + 1, "%d,%d,%d,%d,%d", &c.w, &c.stages, &c.grid, &c.persist,
                                        &c.cl)
                          : 0;
        if (std::strncmp(line, key, std::strlen(key)) == 0 && line[std::strlen(key)] == '|' &&
            (n == 1 || n == 3 || n == 4 || n == 5) && valid(c))
          best = c;
      }
      std::fclose(f);
    }
  }
  // a solve that takes a few-signals form launches none of the kernels tuned here
  if (!best.w && h->d.use_graph != 2 && small_form(solve_ws(h, static_cast<int>(B), false), static_cast<int>(B), eps) != 0)
    best.w = saved.w;
  if (!best.w) {
    omp_status st = OMP_OK;
    if (A != h->prepared_A) st = prepare(h, A, s);
    if (st != OMP_OK) return st;
    CallArgs a{};
    a.Y = Y;
    a.X = h->x_stage;
    a.support = h->s_stage;
    launch_set_args(h->args_dev, a, s);
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return OMP_ERR_CUDA;
    bool failed = false;
    const int b = static_cast<int>(B);
    auto apply = [&](const Shape& c) {
      h->ws.upd_w = c.w;
      h->ws.tc_stages = c.stages;
      h->ws.tc_grid = fitted(c);
      h->ws.upd_persist = c.persist;
      h->ws.tc_cl = c.cl;
    };
    // One shape's solve as a solve runs it: a graph replay when the handle uses graphs (its
    // kernels' arguments are fixed at capture), else direct launches.
    struct Run {
      Shape c;
      cudaGraphExec_t exec;
    };
    auto make_run = [&](const Shape& c, Run* r) {
      apply(c);
      r->c = c;
      r->exec = nullptr;
      if (!h->d.use_graph) return true;
      cudaGraph_t g = nullptr;
      bool ok = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
      if (ok) {
        enqueue_solve(h, solve_ws(h, b, false), b, S, eps, false, h->cap_stream);
        ok = cudaStreamEndCapture(h->cap_stream, &g) == cudaSuccess && g != nullptr;
      }
      if (ok) ok = cudaGraphInstantiate(&r->exec, g, 0) == cudaSuccess;
      if (g) cudaGraphDestroy(g);
      if (!ok) cudaGetLastError();
      return ok;
    };
    auto launch_run = [&](const Run& r) {
      if (r.exec) {
        if (cudaGraphLaunch(r.exec, s) != cudaSuccess) failed = true;
      } else {
        apply(r.c);
        enqueue_solve(h, solve_ws(h, b, false), b, S, eps, false, s);
      }
    };
    auto time_run = [&](const Run& r) {
      cudaEventRecord(e0, s);
      launch_run(r);
      cudaEventRecord(e1, s);
      float ms = 0.f;
      if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess)
        failed = true;
      return ms;
    };
    Run inc{};
    auto drop = [](Run& r) {
      if (r.exec) cudaGraphExecDestroy(r.exec);
      r.exec = nullptr;
    };
    // The first valid shape (the default) is the incumbent. A challenger is timed alternately
    // with it, `repeats` solves each after one warm-up of each, so that clock ramp and drift fall
    // on both alike, and replaces it only when clearly faster (3% less time), so that noise does
    // not move a solve off a good shape.
    auto trial = [&](const Shape& c) {
      if (failed || !valid(c)) return;
      if (!best.w) {
        if (!make_run(c, &inc)) {
          failed = true;
          return;
        }
        best = c;
        for (int r = 0; r < 2 && !failed; ++r) time_run(inc);  // warm-up of the GPU and the shape
        return;
      }
      Run ch{};
      if (!make_run(c, &ch)) {
        failed = true;
        return;
      }
      time_run(ch);  // warm-up
      float t_inc = 0.f, t_ch = 0.f;
      for (int r = 0; r < repeats && !failed; ++r) {
        t_inc += time_run(inc);
        t_ch += time_run(ch);
      }
      if (!failed && t_ch < 0.97f * t_inc) {
        drop(inc);
        inc = ch;
        best = c;
      } else {
        drop(ch);
      }
    };
    // the update's warps per signal first (with the default correlation), then the correlation's
    // CTAs per tile (one, or a pair), pipeline depth and grid with the best of those, then the
    // update's persistent form
    for (int w = 1; w <= 8; w <<= 1) trial(Shape{w, saved.stages, saved.grid, 0, saved.cl});
    if (tc && !failed) {
      const Shape b0 = best;
      for (int cl = 1; cl <= 2; ++cl)
        if (cl != b0.cl) trial(Shape{b0.w, b0.stages, b0.grid, 0, cl});
      const Shape b1 = best;
      for (int st : {4, 3, 2, 6})
        if (st != b1.stages) trial(Shape{b1.w, st, b1.grid, 0, b1.cl});
      const Shape b2 = best;
      trial(Shape{b2.w, b2.stages, h->sm_count - h->sm_count / 8, 0, b2.cl});
    }
    if (!failed) {
      const Shape b3 = best;
      trial(Shape{b3.w, b3.stages, b3.grid, 1, b3.cl});
    }
    drop(inc);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (failed) {
      h->ws.upd_w = saved.w;
      h->ws.tc_stages = saved.stages;
      h->ws.tc_grid = saved.grid;
      h->ws.upd_persist = saved.persist;
      h->ws.tc_cl = saved.cl;
      return OMP_ERR_CUDA;
    }
    if (cache) {
      if (FILE* f = std::fopen(cache, "a")) {
        std::fprintf(f, "%s|%d,%d,%d,%d,%d\n", key, best.w, best.stages, best.grid, best.persist, best.cl);
        std::fclose(f);
      }
    }
  }
  const int best_grid = fitted(best);
  if (best.w != saved.w || best.stages != saved.stages || best_grid != saved.grid ||
      best.persist != saved.persist || best.cl != saved.cl || best.w != h->ws.upd_w ||
      best.stages != h->ws.tc_stages || best_grid != h->ws.tc_grid ||
      best.persist != h->ws.upd_persist || best.cl != h->ws.tc_cl) {
    // captured graphs hold the old launch shapes
    for (auto& g : h->graphs) cudaGraphExecDestroy(g.exec);
    h->graphs.clear();
  }
  h->ws.upd_w = best.w;
  h->ws.upd_persist = best.persist;
  if (tc) {
    h->ws.tc_stages = best.stages;
    h->ws.tc_grid = best_grid;
    h->ws.tc_cl = best.cl;
  }
  if (choice_out) *choice_out = best.w;
  return check_launch();
}

omp_status omp_tuning(omp_handle h, int32_t* update_warps, int32_t* update_persistent,
                      int32_t* corr_stages, int32_t* corr_ctas, int32_t* corr_cluster) {
  if (!h) return OMP_ERR_INVALID_ARGUMENT;
  const bool tc = h->ws.prec != OMP_PREC_FP32;
  if (update_warps) *update_warps = h->ws.upd_w;
  if (update_persistent) *update_persistent = h->ws.upd_persist;
  if (corr_stages) *corr_stages = tc ? h->ws.tc_stages : 0;
  if (corr_ctas) *corr_ctas = tc ? h->ws.tc_grid : 0;
  if (corr_cluster) *corr_cluster = tc ? h->ws.tc_cl : 0;
  return OMP_OK;
}

omp_status omp_handle_info(omp_handle h, omp_desc* desc_out, int32_t* sm_count_out) {
  if (!h) return OMP_ERR_INVALID_ARGUMENT;
  if (desc_out) *desc_out = h->d;
  if (sm_count_out) *sm_count_out = h->sm_count;
  return OMP_OK;
}

omp_status omp_loop_passes(omp_handle h, int32_t* passes_out, void* stream) {
  if (!h || !passes_out) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int v = 0;
  if (cudaMemcpyAsync(&v, h->ws.kdev, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return OMP_ERR_CUDA;
  *passes_out = v;
  return OMP_OK;
}

omp_status omp_solve_batch(omp_handle h, const float* A, const float* Y, int64_t B, int32_t S,
                           float eps, float* X_out, int32_t* support_out, void* stream) {
  return omp_solve_batch_ex(h, A, Y, B, S, eps, X_out, support_out, nullptr, nullptr, nullptr,
                            nullptr, stream);
}

omp_status omp_solve_batch_host(omp_handle h, const float* A, const float* Y_host, int64_t B,
                                int32_t S, float eps, float* X_host, int32_t* support_host,
                                void* stream) {
  if (!h || !Y_host || !X_host || !support_host) return OMP_ERR_INVALID_ARGUMENT;
  if (B < 1 || B > h->d.max_batch || S < 1 || S > h->d.max_iters) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const size_t ybytes = static_cast<size_t>(B) * h->ws.M * sizeof(float);
  if (cudaMemcpyAsync(h->y_stage, Y_host, ybytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return OMP_ERR_CUDA;
  omp_status st = omp_solve_batch_ex(h, A, h->y_stage, B, S, eps, h->x_stage, h->s_stage, nullptr,
                                     nullptr, nullptr, nullptr, stream);
  if (st != OMP_OK) return st;
  const size_t obytes = static_cast<size_t>(B) * S * sizeof(float);
  if (cudaMemcpyAsync(X_host, h->x_stage, obytes, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(support_host, h->s_stage, obytes, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return OMP_ERR_CUDA;
  return OMP_OK;
}

omp_status omp_correlate_topk(omp_handle h, const float* A, const float* R, int64_t B,
                              int32_t topk, int32_t* idx_out, float* score_out, void* stream) {
  if (!h || !A || !R || !idx_out || !score_out) return OMP_ERR_INVALID_ARGUMENT;
  if (B < 1 || B > h->d.max_batch) return OMP_ERR_INVALID_ARGUMENT;
  const int want = h->ws.prec == OMP_PREC_FP32 ? 1 : h->ws.topk;
  if (topk != want) return OMP_ERR_INVALID_ARGUMENT;
  if (!aligned16(A) || !aligned16(R)) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (A != h->prepared_A) {
    const omp_status st = prepare(h, A, s);
    if (st != OMP_OK) return st;
  }
  CallArgs a{};
  a.topk_idx = idx_out;
  a.topk_score = score_out;
  launch_set_args(h->args_dev, a, s);
  enqueue_topk(h, R, static_cast<int>(B), topk, s);
  return check_launch();
}

omp_status omp_profile_enable(omp_handle h, int32_t enable) {
  if (!h) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  if (enable && h->prof_ev.empty()) {
    const size_t n = static_cast<size_t>(h->ws.Smax) * 4;
    h->prof_ev.resize(n, nullptr);
    for (size_t i = 0; i < n; ++i)
      if (cudaEventCreate(&h->prof_ev[i]) != cudaSuccess) return OMP_ERR_CUDA;
  }
  h->prof_on = enable != 0;
  return OMP_OK;
}

omp_status omp_profile_read(omp_handle h, int32_t S, float* corr_ms_host, float* update_ms_host,
                            int32_t* live_host, void* stream) {
  if (!h || !corr_ms_host || !update_ms_host) return OMP_ERR_INVALID_ARGUMENT;
  if (!h->prof_last_valid || S != h->prof_last_S) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaStreamSynchronize(s) != cudaSuccess) return OMP_ERR_CUDA;
  for (int kind = 0; kind < 2; ++kind)
    for (int k = 0; k < S; ++k) {
      const size_t i = (static_cast<size_t>(kind) * h->ws.Smax + k) * 2;
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, h->prof_ev[i], h->prof_ev[i + 1]) != cudaSuccess) return OMP_ERR_CUDA;
      (kind == 0 ? corr_ms_host : update_ms_host)[k] = ms;
    }
  if (live_host) {
    if (cudaMemcpy(live_host, h->ws.cnt + 1, sizeof(int) * S, cudaMemcpyDeviceToHost) != cudaSuccess)
      return OMP_ERR_CUDA;
  }
  return OMP_OK;
}

omp_status omp_get_error(omp_handle h, int32_t* flags, void* stream) {
  if (!h) return OMP_ERR_INVALID_ARGUMENT;
  DeviceGuard guard(h->dev);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  unsigned v = 0;
  if (cudaMemcpyAsync(&v, h->ws.err, sizeof(v), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemsetAsync(h->ws.err, 0, sizeof(unsigned), s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return OMP_ERR_CUDA;
  if (flags) *flags = static_cast<int32_t>(v);
  if (v & OMP_DEVERR_WAIT_TIMEOUT) return OMP_ERR_DEVICE_TIMEOUT;
  if (v & OMP_DEVERR_NONFINITE) return OMP_ERR_NUMERICAL;
  return OMP_OK;
}

}  // extern "C"
