// api.cu -- the C ABI of include/bpmf.h.
//
// Argument checking, device allocation, host<->device copies and the order of
// launches of one Gibbs iteration (Algorithm 1).  No arithmetic of the
// sampler happens here; every step runs in the kernels of structure.cu,
// hyper.cu, rows.cu, binned.cu and predict.cu.
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "bpmf_impl.cuh"
#include "rows.cuh"

namespace gb {

static thread_local char g_err[512] = "";

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

namespace {

template <typename T>
int dalloc(T** p, int64_t n) {
  *p = nullptr;
  if (n <= 0) n = 1;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), sizeof(T) * (size_t)n);
  if (e != cudaSuccess) {
    cudaGetLastError();
    set_error("cudaMalloc of %lld bytes: %s", (long long)(sizeof(T) * n), cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? BPMF_ENOMEM : BPMF_ECUDA;
  }
  return BPMF_OK;
}

void dfree(void* p) {
  if (p) cudaFree(p);
}

void free_handle(Handle* h) {
  if (!h) return;
  drop_graph(h);
  release_timers(h);
  if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
  if (h->aux) cudaStreamDestroy(h->aux);
  if (h->ev_fork) cudaEventDestroy(h->ev_fork);
  if (h->ev_join) cudaEventDestroy(h->ev_join);
  if (h->aux2) cudaStreamDestroy(h->aux2);
  if (h->ev_fork2) cudaEventDestroy(h->ev_fork2);
  if (h->ev_join2) cudaEventDestroy(h->ev_join2);
  for (int s = 0; s < 2; ++s) {
    SideDev& sd = h->side[s];
    dfree(sd.tiny_pre);
    if (sd.piece_own) dfree(sd.piece_mem);
  }
  dfree(h->block); dfree(h->tblock); dfree(h->hub_part);
  delete h;
}

// n elements on the device: where they live already, or a copy in space taken
// from c (which only adds up bytes as long as it has no block).
template <typename T>
int to_device(const T* src, int64_t n, bool devptr, T** dst, Carve& c, cudaStream_t st) {
  *dst = const_cast<T*>(src);
  if (devptr || n == 0) return BPMF_OK;
  *dst = c.take<T>(n);
  if (*dst) BPMF_CUDA_CHECK(cudaMemcpyAsync(*dst, src, sizeof(T) * n, cudaMemcpyHostToDevice, st));
  return BPMF_OK;
}

constexpr int64_t kPieceBlock = 8192;  // bytes of a side's pieces in the sampler's block

// The sampler's arrays of fixed size; the words that start at zero are
// consecutive, from status to d_navg.
void carve_handle(Handle* h, Carve& c) {
  const int64_t K = h->K, KK = K * K, KP = (K + 31) & ~31;
  for (SideDev& sd : h->side) {
    sd.ptr = c.take<int64_t>(sd.R + 1);
    sd.idx = c.take<int32_t>(h->nnz);
    sd.val = c.take<float>(h->nnz);
    sd.perm = c.take<int32_t>(sd.R);
    sd.work = c.take<int4>(sd.R);
    sd.X = c.take<float>(sd.R * K);
    sd.lam = c.take<double>(KK);
    sd.mu = c.take<double>(K);
    sd.lamaug = c.take<float>((K + 1) * (K + 1));
    sd.lchol = c.take<float>(KK);
    sd.linvT = c.take<float>(KP * (KP + 4));
    if (h->cfg.path == BPMF_PATH_MIXED) {
      sd.KS = (int)((K + 7) & ~7);
      sd.Xhi = c.take<__nv_bfloat16>(sd.R * sd.KS);
      sd.Xlo = c.take<__nv_bfloat16>(sd.R * sd.KS);
    }
    sd.xbar = c.take<double>(K);
    sd.S = c.take<double>(KK);
    sd.piece_mem = c.take<char>(kPieceBlock);
    sd.piece_bytes = kPieceBlock;
  }
  h->red = c.take<double>(h->red_len);
  h->wscr = c.take<double>(6 * KK + 8 * K);
  h->red2 = c.take<double>(h->red_len);
  h->wscr2 = c.take<double>(6 * KK + 8 * K);
  h->mu0 = c.take<double>(K);
  h->W0inv = c.take<double>(KK);
  h->flag_rows = c.take<int32_t>(std::max(h->M, h->N));
  h->terr = c.take<double>(2);
  h->status = c.take<int>(1);
  h->flag_count = c.take<int32_t>(1);
  h->redo_count = c.take<int32_t>(1);
  h->redo_ticket = c.take<int>(1);
  h->test_ticket = c.take<int>(1);
  h->ws_counter = c.take<int>(1);
  h->d_iter = c.take<uint32_t>(1);
  h->d_navg = c.take<int64_t>(1);
}

// Doubles of the reduction partials.
int64_t red_length(int K, int num_sms) {
  return std::max<int64_t>({2LL * num_sms * K * K, 2LL * num_sms * K, 16LL * num_sms + 1024, 4096});
}

// The test set's arrays.
void carve_test(Handle* h, int64_t n, Carve& k) {
  h->trow = k.take<int32_t>(n);
  h->tcol = k.take<int32_t>(n);
  h->tval = k.take<float>(n);
  h->tsum = k.take<float2>(n);
}

// Scratch of bpmf_init beside the ratings from the host: what the structure
// takes or, after it, the factors of the autotuner's sweeps.
size_t init_work_bytes(int64_t M, int64_t N, int64_t nnz, const bpmf_config& cfg) {
  return std::max(structure_bytes(nnz, M, N),
                  cfg.autotune ? sizeof(float) * (size_t)(std::max(M, N) * cfg.K) : 0);
}

}  // namespace

int64_t sampler_bytes(int64_t M, int64_t N, int64_t nnz, int64_t n_test, const bpmf_config& cfg, int num_sms) {
  Handle h;
  h.M = M;
  h.N = N;
  h.nnz = nnz;
  h.K = cfg.K;
  h.cfg = cfg;
  h.side[BPMF_USERS].R = M;
  h.side[BPMF_MOVIES].R = N;
  h.red_len = red_length(cfg.K, num_sms);
  Carve held, init, test;
  carve_handle(&h, held);
  if (n_test > 0) carve_test(&h, n_test, held);
  // pieces of both sides and the partials of one: at most a piece per plen
  // ratings and one more per hub
  const int64_t hub = cfg.hub_min >= 0 ? std::max(1, cfg.hub_min) : cfg.autotune ? kTuneHubMin : 2 * kPiece;
  const int64_t pieces = nnz / piece_length(hub) + nnz / hub + 1;
  for (int s = 0; s < 2; ++s) {
    held.take<int64_t>(2 * pieces);
    held.take<int32_t>(2 * pieces);
  }
  held.take<float>(nnz >= hub ? pieces * partial_floats_per_piece(cfg.K) : 0);
  // L^-1 of the other side's rows, where a row with ratings can be in the tiny bin
  if (cfg.path != BPMF_PATH_PLAIN && (cfg.tiny_max > 0 || (cfg.tiny_max < 0 && cfg.autotune)))
    for (const int64_t n : {M, N}) held.take<float>(rank1_pre_floats(cfg.K, n, M + N - n, nnz));
  // scratch, released before the call returns
  for (int i = 0; i < 3; ++i) {
    init.take<int32_t>(nnz);
    test.take<int32_t>(n_test);
  }
  init.take<char>((int64_t)init_work_bytes(M, N, nnz, cfg));
  test.take<char>((int64_t)test_sort_bytes(n_test));
  return (int64_t)(held.bytes + std::max(init.bytes, test.bytes));
}

// Reads and clears the device status word; maps bits to a status code.
int check_status(Handle* h, const char* where) {
  int st = 0;
  BPMF_CUDA_CHECK(cudaMemcpyAsync(&st, h->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  if (st) BPMF_CUDA_CHECK(cudaMemsetAsync(h->status, 0, sizeof(int), h->stream));
  if (st & kStatusNotPD) {
    set_error("%s: a precision matrix is not positive definite in FP64", where);
    return BPMF_ENOTPD;
  }
  if (st & kStatusRng) {
    set_error("%s: Gamma sampler exceeded its rejection cap", where);
    return BPMF_ERNG;
  }
  if (st & kStatusIndex) {
    set_error("%s: index out of range", where);
    return BPMF_EINVAL;
  }
  if (st & kStatusTimeout) {
    set_error("%s: a tensor-core pipeline wait timed out", where);
    return BPMF_ECUDA;
  }
  if (st & kStatusValue) {
    set_error("%s: an input value is not finite", where);
    return BPMF_EINVAL;
  }
  return BPMF_OK;
}

namespace {

int valid_side(int side) { return side == BPMF_USERS || side == BPMF_MOVIES; }

// Records which entry point rejected its arguments and returns BPMF_EINVAL.
int einval(const char* what) {
  set_error("%s: invalid argument (null handle, side, pointer or size)", what);
  return BPMF_EINVAL;
}

int sweep_one(Handle* h, int s) {
  BPMF_TRY(launch_sweep(h, s));
  return BPMF_OK;
}

int read_fp64_rows(Handle* h, int s) {
  int32_t n = 0;
  BPMF_CUDA_CHECK(cudaMemcpyAsync(&n, h->redo_count, sizeof(int32_t), cudaMemcpyDeviceToHost,
                                  h->stream));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  h->side[s].fp64_rows = n;
  return BPMF_OK;
}

// One Gibbs iteration (Algorithm 1): per side in the configured order the
// hyperparameter draw then the row draws, then the test predictions, then
// the iteration word advances.  The second side's hyperparameter draw reads
// only that side's factors, which the first side's draw and sweep leave
// alone, so it runs on aux2 beside them (with its own scratch) and joins
// before the second sweep: the FP64 draws of the two sides, a cluster of 4 to
// 16 CTAs each, overlap, and the second side's reductions fill SMs the first side
// leaves idle.
// Everything that changes from one iteration to the next lives in device
// memory, so the same launches serve every iteration.
int step_body(Handle* h) {
  const int first = h->cfg.order == 0 ? BPMF_USERS : BPMF_MOVIES, second = 1 - first;
  const bool fork = h->aux2 != nullptr;
  int rc = BPMF_OK;
  if (fork) {
    BPMF_CUDA_CHECK(cudaEventRecord(h->ev_fork2, h->stream));
    BPMF_CUDA_CHECK(cudaStreamWaitEvent(h->aux2, h->ev_fork2, 0));
    rc = launch_hyper(h, second, h->aux2, true);
    // the join is recorded and waited for whatever happened, so that a
    // capture never ends with the branch unjoined
    if (cudaEventRecord(h->ev_join2, h->aux2) != cudaSuccess && rc == BPMF_OK) rc = BPMF_ECUDA;
  }
  if (rc == BPMF_OK) rc = launch_hyper(h, first);
  if (rc == BPMF_OK) rc = sweep_one(h, first);
  if (fork) {
    if (cudaStreamWaitEvent(h->stream, h->ev_join2, 0) != cudaSuccess && rc == BPMF_OK) rc = BPMF_ECUDA;
  } else if (rc == BPMF_OK) {
    rc = launch_hyper(h, second);
  }
  if (rc != BPMF_OK) return rc;
  BPMF_TRY(sweep_one(h, second));
  return h->n_test > 0 ? launch_test_step(h) : launch_advance_iter(h);
}

// Records step_body into an executable graph.  The capture runs on a private
// stream (the legacy default stream cannot be captured); replays go to the
// handle's stream.  Phase timers become event-record nodes whose pairs are
// read after every replay.
int capture_step(Handle* h) {
  if (!h->cap_stream)
    BPMF_CUDA_CHECK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  const int64_t k0 = h->kernels;
  const size_t p0 = h->pending.size();
  cudaStream_t user = h->stream;
  h->stream = h->cap_stream;
  BPMF_CUDA_CHECK(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeRelaxed));
  h->capturing = true;
  int rc = step_body(h);
  cudaGraph_t g = nullptr;
  const cudaError_t ec = cudaStreamEndCapture(h->stream, &g);
  h->capturing = false;
  h->stream = user;
  const int64_t per = h->kernels - k0;
  h->kernels = k0;
  std::vector<Handle::Pending> timers(h->pending.begin() + (std::ptrdiff_t)p0, h->pending.end());
  h->pending.resize(p0);
  if (rc == BPMF_OK && ec != cudaSuccess) {
    set_error("bpmf_step: graph capture: %s", cudaGetErrorString(ec));
    rc = BPMF_ECUDA;
  }
  cudaGraphExec_t ex = nullptr;
  if (rc == BPMF_OK) {
    const cudaError_t ei = cudaGraphInstantiate(&ex, g, 0);
    if (ei != cudaSuccess) {
      set_error("bpmf_step: graph instantiate: %s", cudaGetErrorString(ei));
      rc = BPMF_ECUDA;
    }
  }
  if (g) cudaGraphDestroy(g);
  if (rc != BPMF_OK) {
    cudaGetLastError();
    for (auto& p : timers) {
      h->event_pool.push_back(p.a);
      h->event_pool.push_back(p.b);
    }
    return rc;
  }
  h->graph = ex;
  h->graph_timing = h->timing;
  h->graph_kernels = per;
  h->graph_timers = timers;
  return BPMF_OK;
}

}  // namespace

// Queues one Gibbs iteration on the handle's stream without waiting for it.
int step_async(Handle* h) {
  if (h->use_graph) {
    if (h->graph && h->graph_timing != h->timing) drop_graph(h);
    if (!h->graph) BPMF_TRY(capture_step(h));
    BPMF_CUDA_CHECK(cudaGraphLaunch(h->graph, h->stream));
    h->kernels += h->graph_kernels;
  } else {
    BPMF_TRY(step_body(h));
  }
  if (h->n_test > 0) {
    if (h->iter >= h->cfg.burnin) h->n_avg += 1;
    h->have_rmse = true;
  }
  h->iter += 1;
  return BPMF_OK;
}

namespace {

// Adds the phase times of the last replay (the stream is idle).
int resolve_graph_timers(Handle* h) {
  for (auto& p : h->graph_timers) {
    float ms = 0.f;
    BPMF_CUDA_CHECK(cudaEventElapsedTime(&ms, p.a, p.b));
    h->t_ms[p.id] += ms;
    h->t_cnt[p.id] += 1;
  }
  return BPMF_OK;
}

}  // namespace
}  // namespace gb

using namespace gb;

extern "C" {

void bpmf_config_default(bpmf_config* c, int32_t K) {
  if (!c) return;
  memset(c, 0, sizeof(*c));
  c->K = K;
  c->path = BPMF_PATH_MIXED;
  c->alpha = 2.0;
  c->beta0 = 2.0;
  c->nu0 = (double)K;
  c->mu0 = nullptr;
  c->W0 = nullptr;
  c->seed = 0;
  c->order = 0;
  c->burnin = 0;
  c->light_max = -1;
  c->hub_min = -1;
  c->tiny_max = -1;
  c->heavy_kernel = 0;
  c->autotune = 0;
  c->pivot_rel = 5e-2;
}

const char* bpmf_strerror(int code) {
  switch (code) {
    case BPMF_OK: return "ok";
    case BPMF_EINVAL: return "invalid argument";
    case BPMF_ENOMEM: return "out of memory";
    case BPMF_ECUDA: return "CUDA error";
    case BPMF_ENOTPD: return "matrix not positive definite";
    case BPMF_ERNG: return "random sampler rejection cap reached";
    case BPMF_ESTATE: return "call out of order";
    case BPMF_EBUSY: return "not finished yet";
    default: return "unknown status";
  }
}

const char* bpmf_last_error(void) { return g_err; }

int bpmf_init(bpmf_t** out, int64_t M, int64_t N, int64_t nnz, const int32_t* row,
              const int32_t* col, const float* val, const bpmf_config* cfg, void* stream,
              uint32_t flags) {
  g_err[0] = 0;
  if (!out || !cfg) {
    set_error("bpmf_init: null output or config");
    return BPMF_EINVAL;
  }
  *out = nullptr;
  const int K = cfg->K;
  if (K < 1 || K > kMaxK || M < 1 || N < 1 || M >= (1LL << 31) || N >= (1LL << 31) || nnz < 0 ||
      nnz >= (1LL << 31) || (nnz > 0 && (!row || !col || !val)) || !(cfg->alpha > 0.0) ||
      !isfinite(cfg->alpha) || !(cfg->beta0 > 0.0) || !isfinite(cfg->beta0) ||
      !(cfg->nu0 > (double)K - 1.0) || !isfinite(cfg->nu0) || !(cfg->pivot_rel >= 0.0) ||
      !(cfg->pivot_rel < 1.0) || cfg->path < BPMF_PATH_PLAIN ||
      cfg->path > BPMF_PATH_MIXED || (cfg->order != 0 && cfg->order != 1) || cfg->burnin < 0 ||
      cfg->heavy_kernel < 0 || cfg->heavy_kernel > 2 || cfg->tiny_max > kTinyDegreeMax) {
    set_error("bpmf_init: invalid shape or configuration (K=%d M=%lld N=%lld nnz=%lld)", K,
              (long long)M, (long long)N, (long long)nnz);
    return BPMF_EINVAL;
  }
  const bool dev = (flags & BPMF_DEVPTR) != 0;
  Handle* h = new Handle();
  h->M = M;
  h->N = N;
  h->nnz = nnz;
  h->K = K;
  h->cfg = *cfg;
  h->cfg.mu0 = nullptr;
  h->cfg.W0 = nullptr;
  h->stream = (cudaStream_t)stream;
  int rc = BPMF_OK;
  int32_t *d_row = nullptr, *d_col = nullptr;
  float* d_val = nullptr;
  char* scratch = nullptr;
  do {
    if (cudaGetDevice(&h->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device) !=
            cudaSuccess) {
      set_error("bpmf_init: no CUDA device");
      rc = BPMF_ECUDA;
      break;
    }
    if (cudaStreamCreateWithFlags(&h->aux, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming) != cudaSuccess ||
        cudaStreamCreateWithFlags(&h->aux2, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_fork2, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&h->ev_join2, cudaEventDisableTiming) != cudaSuccess) {
      set_error("bpmf_init: stream or event creation failed");
      rc = BPMF_ECUDA;
      break;
    }
    h->side[BPMF_USERS].R = M;
    h->side[BPMF_MOVIES].R = N;
    const int64_t KK = (int64_t)K * K;
    h->red_len = red_length(K, h->num_sms);
    {
      Carve size, c;
      carve_handle(h, size);
      if ((rc = dalloc(&h->block, (int64_t)size.bytes))) break;
      c.base = h->block;
      carve_handle(h, c);
    }
    if (cudaMemsetAsync(h->status, 0, reinterpret_cast<char*>(h->d_navg + 1) - reinterpret_cast<char*>(h->status),
                        h->stream) != cudaSuccess) {
      rc = BPMF_ECUDA;
      break;
    }
    // prior
    std::vector<double> mu0(K, 0.0), W0(KK, 0.0);
    for (int k = 0; k < K; ++k) {
      if (cfg->mu0) mu0[k] = cfg->mu0[k];
      W0[(int64_t)k * K + k] = 1.0;
    }
    if (cfg->W0) std::copy(cfg->W0, cfg->W0 + KK, W0.begin());
    for (int64_t e = 0; e < KK; ++e)
      if (!isfinite(W0[e])) rc = BPMF_EINVAL;
    for (int k = 0; k < K; ++k)
      if (!isfinite(mu0[k])) rc = BPMF_EINVAL;
    if (rc) {
      set_error("bpmf_init: non-finite prior");
      break;
    }
    double* d_W0 = h->wscr + 4 * KK;  // temporary slot inside the scratch
    if (cudaMemcpyAsync(h->mu0, mu0.data(), sizeof(double) * K, cudaMemcpyHostToDevice,
                        h->stream) != cudaSuccess ||
        cudaMemcpyAsync(d_W0, W0.data(), sizeof(double) * KK, cudaMemcpyHostToDevice,
                        h->stream) != cudaSuccess) {
      set_error("bpmf_init: prior copy failed");
      rc = BPMF_ECUDA;
      break;
    }
    if ((rc = wish_cluster(K, &h->wish_ctas))) break;
    if ((rc = launch_spd_inverse_f64(d_W0, h->W0inv, K, h->wish_ctas, h->wscr, h->status, h->stream))) break;
    if ((rc = check_status(h, "bpmf_init (W0)"))) {
      set_error("bpmf_init: W0 is not symmetric positive definite");
      rc = BPMF_EINVAL;
      break;
    }
    // ratings
    const size_t work = init_work_bytes(M, N, nnz, *cfg);
    char* ws = nullptr;
    for (int pass = 0; pass < 2 && rc == BPMF_OK; ++pass) {
      Carve c;
      c.base = scratch;
      if ((rc = to_device(row, nnz, dev, &d_row, c, h->stream))) break;
      if ((rc = to_device(col, nnz, dev, &d_col, c, h->stream))) break;
      if ((rc = to_device(val, nnz, dev, &d_val, c, h->stream))) break;
      ws = c.take<char>((int64_t)work);
      if (pass == 0) rc = dalloc(&scratch, (int64_t)c.bytes);
    }
    if (rc) break;
    if ((rc = build_structure(h, d_row, d_col, d_val, ws))) break;  // waits for its work
    if (!cfg->autotune) {  // before the bins' own memory is taken
      dfree(scratch);
      scratch = nullptr;
    }
    if ((rc = setup_bins(h, BPMF_USERS))) break;
    if ((rc = setup_bins(h, BPMF_MOVIES))) break;
    if ((rc = launch_init_factors(h, BPMF_USERS))) break;
    if ((rc = launch_init_factors(h, BPMF_MOVIES))) break;
    if ((rc = launch_refresh_shadow(h, BPMF_USERS))) break;
    if ((rc = launch_refresh_shadow(h, BPMF_MOVIES))) break;
    if (cfg->autotune) {
      rc = autotune_bins(h, BPMF_USERS, reinterpret_cast<float*>(ws));
      if (rc == BPMF_OK) rc = autotune_bins(h, BPMF_MOVIES, reinterpret_cast<float*>(ws));
      if (rc == BPMF_OK) rc = check_status(h, "bpmf_init (autotune)");
      if (rc) break;
    }
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) {
      set_error("bpmf_init: %s", cudaGetErrorString(cudaGetLastError()));
      rc = BPMF_ECUDA;
      break;
    }
  } while (0);
  if (scratch) {
    cudaStreamSynchronize(h->stream);
    dfree(scratch);
  }
  if (rc != BPMF_OK) {
    free_handle(h);
    return rc;
  }
  *out = reinterpret_cast<bpmf_t*>(h);
  return BPMF_OK;
}

int bpmf_set_test(bpmf_t* hh, int64_t n, const int32_t* row, const int32_t* col, const float* val,
                  uint32_t flags) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || n < 0 || n >= (1LL << 31) || (n > 0 && (!row || !col || !val))) {
    set_error("bpmf_set_test: invalid arguments");
    return BPMF_EINVAL;
  }
  const bool dev = (flags & BPMF_DEVPTR) != 0;
  cudaStream_t st = h->stream;
  drop_graph(h);  // the captured iteration holds the old test arrays
  BPMF_CUDA_CHECK(cudaMemsetAsync(h->d_navg, 0, sizeof(int64_t), st));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(st));
  dfree(h->tblock);
  h->tblock = nullptr;
  h->trow = h->tcol = nullptr;
  h->tval = nullptr;
  h->tsum = nullptr;
  h->n_test = 0;
  h->n_avg = 0;
  h->have_rmse = false;
  if (n == 0) return BPMF_OK;
  int32_t *d_row = nullptr, *d_col = nullptr;
  float* d_val = nullptr;
  char *scratch = nullptr, *ws = nullptr;
  int rc = BPMF_OK;
  do {
    for (int pass = 0; pass < 2 && rc == BPMF_OK; ++pass) {
      Carve c;  // scratch
      c.base = scratch;
      if ((rc = to_device(row, n, dev, &d_row, c, st))) break;
      if ((rc = to_device(col, n, dev, &d_col, c, st))) break;
      if ((rc = to_device(val, n, dev, &d_val, c, st))) break;
      ws = c.take<char>((int64_t)test_sort_bytes(n));
      Carve k;  // kept
      k.base = h->tblock;
      carve_test(h, n, k);
      if (pass == 0 && (rc = dalloc(&scratch, (int64_t)c.bytes)) == BPMF_OK)
        rc = dalloc(&h->tblock, (int64_t)k.bytes);
    }
    if (rc) break;
    // validate, then sort by user (stable) for gather locality
    rc = sort_test_set(h, d_row, d_col, d_val, n, ws);
    if (rc) break;
    if (cudaMemsetAsync(h->tsum, 0, sizeof(float2) * n, st) != cudaSuccess) {
      rc = BPMF_ECUDA;
      break;
    }
    h->n_test = n;
    rc = check_status(h, "bpmf_set_test");
  } while (0);
  if (scratch) {
    cudaStreamSynchronize(st);
    dfree(scratch);
  }
  if (rc != BPMF_OK) h->n_test = 0;
  return rc;
}

int bpmf_sample_hyper(bpmf_t* hh, int side) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side)) return einval("bpmf_sample_hyper");
  BPMF_TRY(launch_hyper(h, side));
  return check_status(h, "bpmf_sample_hyper");
}

int bpmf_sweep(bpmf_t* hh, int side) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side)) return einval("bpmf_sweep");
  if (!h->side[side].have_hyper) {
    set_error("bpmf_sweep: no hyperparameters drawn or set for this side");
    return BPMF_ESTATE;
  }
  BPMF_TRY(sweep_one(h, side));
  BPMF_TRY(read_fp64_rows(h, side));
  return check_status(h, "bpmf_sweep");
}

int bpmf_step(bpmf_t* hh) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_step");
  BPMF_TRY(step_async(h));
  const int rc = check_status(h, "bpmf_step");
  if (rc == BPMF_OK && h->use_graph && h->timing) BPMF_TRY(resolve_graph_timers(h));
  return rc;
}

int bpmf_set_limits(bpmf_t* hh, int32_t gamma_cap, int64_t wait_ns) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || gamma_cap > kGammaCap) return einval("bpmf_set_limits");
  drop_graph(h);  // the captured iteration holds the old limits
  h->gamma_cap = gamma_cap < 0 ? kGammaCap : gamma_cap;
  h->wait_ns = wait_ns > 0 ? (uint64_t)wait_ns : kWaitNsDefault;
  return BPMF_OK;
}

int bpmf_set_test_hold(bpmf_t* hh, int32_t hold) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || (hold != 0 && hold != 1)) return einval("bpmf_set_test_hold");
  drop_graph(h);
  h->hold_arrive = hold;
  return BPMF_OK;
}

int bpmf_set_graph(bpmf_t* hh, int enable) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_set_graph");
  drop_graph(h);
  h->use_graph = enable != 0;
  return BPMF_OK;
}

int bpmf_predict(bpmf_t* hh, int64_t n, const int32_t* row, const int32_t* col, float* out,
                 uint32_t flags) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || n < 0 || (n > 0 && (!row || !col || !out))) return einval("bpmf_predict");
  if (n == 0) return BPMF_OK;
  const bool dev = (flags & BPMF_DEVPTR) != 0;
  int32_t *d_row = nullptr, *d_col = nullptr;
  float* d_out = dev ? out : nullptr;
  char* scratch = nullptr;
  int rc = BPMF_OK;
  do {
    for (int pass = 0; pass < 2 && rc == BPMF_OK; ++pass) {
      Carve c;
      c.base = scratch;
      if ((rc = to_device(row, n, dev, &d_row, c, h->stream))) break;
      if ((rc = to_device(col, n, dev, &d_col, c, h->stream))) break;
      if (dev) break;
      d_out = c.take<float>(n);
      if (pass == 0) rc = dalloc(&scratch, (int64_t)c.bytes);
    }
    if (rc) break;
    if ((rc = launch_predict(h, n, d_row, d_col, d_out))) break;
    if (!dev && cudaMemcpyAsync(out, d_out, sizeof(float) * n, cudaMemcpyDeviceToHost,
                                h->stream) != cudaSuccess) {
      rc = BPMF_ECUDA;
      break;
    }
    rc = check_status(h, "bpmf_predict");
  } while (0);
  if (scratch) {
    cudaStreamSynchronize(h->stream);
    dfree(scratch);
  }
  return rc;
}

int bpmf_test_rmse(bpmf_t* hh, double* rmse_sample, double* rmse_mean) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_test_rmse");
  if (!h->have_rmse) {
    set_error("bpmf_test_rmse: no test set or no iteration yet");
    return BPMF_ESTATE;
  }
  double e[2];
  BPMF_CUDA_CHECK(cudaMemcpyAsync(e, h->terr, sizeof(e), cudaMemcpyDeviceToHost, h->stream));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  if (rmse_sample) *rmse_sample = e[0];
  if (rmse_mean) *rmse_mean = h->n_avg > 0 ? e[1] : NAN;
  return BPMF_OK;
}

int bpmf_get_state(bpmf_t* hh, float* U, float* V, double* hyper, int64_t* iter, uint32_t flags) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_get_state");
  const cudaMemcpyKind kind = (flags & BPMF_DEVPTR) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  const int K = h->K;
  const int64_t KK = (int64_t)K * K;
  if (U) BPMF_CUDA_CHECK(cudaMemcpyAsync(U, h->side[0].X, sizeof(float) * h->M * K, kind, h->stream));
  if (V) BPMF_CUDA_CHECK(cudaMemcpyAsync(V, h->side[1].X, sizeof(float) * h->N * K, kind, h->stream));
  if (hyper) {
    for (int s = 0; s < 2; ++s) {
      double* base = hyper + s * (KK + K);
      BPMF_CUDA_CHECK(cudaMemcpyAsync(base, h->side[s].lam, sizeof(double) * KK,
                                      cudaMemcpyDeviceToHost, h->stream));
      BPMF_CUDA_CHECK(cudaMemcpyAsync(base + KK, h->side[s].mu, sizeof(double) * K,
                                      cudaMemcpyDeviceToHost, h->stream));
    }
  }
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  if (iter) *iter = h->iter;
  return BPMF_OK;
}

int bpmf_set_state(bpmf_t* hh, const float* U, const float* V, const double* hyper, int64_t iter,
                   uint32_t flags) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || iter < 0) return einval("bpmf_set_state");
  const cudaMemcpyKind kind = (flags & BPMF_DEVPTR) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  const int K = h->K;
  const int64_t KK = (int64_t)K * K;
  if (U) BPMF_CUDA_CHECK(cudaMemcpyAsync(h->side[0].X, U, sizeof(float) * h->M * K, kind, h->stream));
  if (V) BPMF_CUDA_CHECK(cudaMemcpyAsync(h->side[1].X, V, sizeof(float) * h->N * K, kind, h->stream));
  if (U) BPMF_TRY(launch_refresh_shadow(h, 0));
  if (V) BPMF_TRY(launch_refresh_shadow(h, 1));
  if (hyper) {
    for (int s = 0; s < 2; ++s) {
      const double* base = hyper + s * (KK + K);
      for (int64_t e = 0; e < KK + K; ++e)
        if (!isfinite(base[e])) {
          set_error("bpmf_set_state: non-finite hyperparameter");
          return BPMF_EINVAL;
        }
      BPMF_CUDA_CHECK(cudaMemcpyAsync(h->side[s].lam, base, sizeof(double) * KK,
                                      cudaMemcpyHostToDevice, h->stream));
      BPMF_CUDA_CHECK(cudaMemcpyAsync(h->side[s].mu, base + KK, sizeof(double) * K,
                                      cudaMemcpyHostToDevice, h->stream));
      BPMF_TRY(launch_check_spd_f64(h->side[s].lam, K, h->status, h->side[s].lchol, h->stream));
      BPMF_TRY(launch_hyper_to_f32(h, s));
    }
    const int rc = check_status(h, "bpmf_set_state");
    if (rc == BPMF_ENOTPD) {
      set_error("bpmf_set_state: a Lambda is not positive definite");
      return BPMF_EINVAL;
    }
    if (rc) return rc;
    h->side[0].have_hyper = h->side[1].have_hyper = true;
  }
  h->iter = iter;
  const uint32_t t32 = (uint32_t)iter;
  BPMF_CUDA_CHECK(cudaMemcpyAsync(h->d_iter, &t32, sizeof(uint32_t), cudaMemcpyHostToDevice,
                                  h->stream));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  return BPMF_OK;
}

int bpmf_get_structure(bpmf_t* hh, int side, int64_t* ptr, int32_t* idx, float* val, int32_t* perm,
                       double* mean) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side)) return einval("bpmf_get_structure");
  SideDev& sd = h->side[side];
  cudaStream_t st = h->stream;
  if (ptr) BPMF_CUDA_CHECK(cudaMemcpyAsync(ptr, sd.ptr, sizeof(int64_t) * (sd.R + 1), cudaMemcpyDeviceToHost, st));
  if (idx && h->nnz) BPMF_CUDA_CHECK(cudaMemcpyAsync(idx, sd.idx, sizeof(int32_t) * h->nnz, cudaMemcpyDeviceToHost, st));
  if (val && h->nnz) BPMF_CUDA_CHECK(cudaMemcpyAsync(val, sd.val, sizeof(float) * h->nnz, cudaMemcpyDeviceToHost, st));
  if (perm) BPMF_CUDA_CHECK(cudaMemcpyAsync(perm, sd.perm, sizeof(int32_t) * sd.R, cudaMemcpyDeviceToHost, st));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(st));
  if (mean) *mean = h->mean;
  return BPMF_OK;
}

int bpmf_get_hyper_stats(bpmf_t* hh, int side, double* xbar, double* S) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side)) return einval("bpmf_get_hyper_stats");
  SideDev& sd = h->side[side];
  if (!sd.have_stats) return BPMF_ESTATE;
  const int K = h->K;
  if (xbar) BPMF_CUDA_CHECK(cudaMemcpyAsync(xbar, sd.xbar, sizeof(double) * K, cudaMemcpyDeviceToHost, h->stream));
  if (S) BPMF_CUDA_CHECK(cudaMemcpyAsync(S, sd.S, sizeof(double) * K * K, cudaMemcpyDeviceToHost, h->stream));
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  return BPMF_OK;
}

int bpmf_get_thresholds(bpmf_t* hh, int side, int64_t thresholds[5]) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side) || !thresholds) return einval("bpmf_get_thresholds");
  const SideDev& sd = h->side[side];
  thresholds[0] = sd.tiny_max;
  thresholds[1] = sd.light_max;
  thresholds[2] = sd.hub_min;
  const bool mixed = h->cfg.path == BPMF_PATH_MIXED;
  thresholds[3] = !mixed ? 0 : (sd.Xhi && ws_supported(h->K) && !sd.heavy_tc) ? 1
                             : (tc_supported(h->K) ? 2 : 0);
  thresholds[4] = thresholds[3] == 1 ? sd.ws_cons : 0;
  return BPMF_OK;
}

int bpmf_set_thresholds(bpmf_t* hh, int side, const int64_t thresholds[5]) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side) || !thresholds) return einval("bpmf_set_thresholds");
  if (h->cfg.path == BPMF_PATH_PLAIN) {
    // one kernel for every row: only the values in effect are accepted
    int64_t cur[5];
    bpmf_get_thresholds(hh, side, cur);
    for (int i = 0; i < 5; ++i)
      if (thresholds[i] != cur[i]) {
        set_error("bpmf_set_thresholds: the plain path keeps its single schedule");
        return BPMF_EINVAL;
      }
    return BPMF_OK;
  }
  return set_thresholds(h, side, thresholds);
}

int bpmf_get_sweep_info(bpmf_t* hh, int side, int64_t bins[4], int64_t* fp64_rows) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h || !valid_side(side)) return einval("bpmf_get_sweep_info");
  SideDev& sd = h->side[side];
  if (bins)
    for (int b = 0; b < 4; ++b) bins[b] = sd.bin_count[b];
  if (fp64_rows) *fp64_rows = sd.fp64_rows;
  return BPMF_OK;
}

void bpmf_destroy(bpmf_t* hh) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream);
  else cudaDeviceSynchronize();
  free_handle(h);
}

}  // extern "C"

namespace gb {

static cudaEvent_t take_event(Handle* h) {
  if (!h->event_pool.empty()) {
    cudaEvent_t e = h->event_pool.back();
    h->event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  if (cudaEventCreate(&e) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return e;
}

PhaseTimer::PhaseTimer(Handle* h_, int id_, cudaStream_t st_)
    : h(h_), id(id_), st(st_ ? st_ : h_->stream) {
  if (!h->timing) return;
  a = take_event(h);
  if (!a) return;
  if (h->capturing) cudaEventRecordWithFlags(a, st, cudaEventRecordExternal);
  else cudaEventRecord(a, st);
}

PhaseTimer::~PhaseTimer() {
  if (!h->timing || !a) return;
  cudaEvent_t b = take_event(h);
  if (!b) {
    h->event_pool.push_back(a);
    return;
  }
  if (h->capturing) cudaEventRecordWithFlags(b, st, cudaEventRecordExternal);
  else cudaEventRecord(b, st);
  h->pending.push_back({a, b, id});
}

int resolve_timers(Handle* h) {
  if (h->pending.empty()) return BPMF_OK;
  BPMF_CUDA_CHECK(cudaStreamSynchronize(h->stream));
  for (auto& p : h->pending) {
    float ms = 0.f;
    BPMF_CUDA_CHECK(cudaEventElapsedTime(&ms, p.a, p.b));
    h->t_ms[p.id] += ms;
    h->t_cnt[p.id] += 1;
    h->event_pool.push_back(p.a);
    h->event_pool.push_back(p.b);
  }
  h->pending.clear();
  return BPMF_OK;
}

void drop_graph(Handle* h) {
  if (h->graph) {
    if (h->stream) cudaStreamSynchronize(h->stream);
    else cudaDeviceSynchronize();
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  for (auto& p : h->graph_timers) {
    h->event_pool.push_back(p.a);
    h->event_pool.push_back(p.b);
  }
  h->graph_timers.clear();
  h->graph_kernels = 0;
}

void release_timers(Handle* h) {
  for (auto& p : h->pending) {
    cudaEventDestroy(p.a);
    cudaEventDestroy(p.b);
  }
  h->pending.clear();
  for (auto e : h->event_pool) cudaEventDestroy(e);
  h->event_pool.clear();
}

}  // namespace gb

extern "C" {

int bpmf_set_timing(bpmf_t* hh, int enable) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_set_timing");
  BPMF_TRY(resolve_timers(h));
  for (int i = 0; i < BPMF_NUM_TIMERS; ++i) {
    h->t_ms[i] = 0.0;
    h->t_cnt[i] = 0;
  }
  h->kernels = 0;
  h->timing = enable != 0;
  return BPMF_OK;
}

int bpmf_get_timing(bpmf_t* hh, double* ms, int64_t* phase_count, int64_t* kernels) {
  Handle* h = reinterpret_cast<Handle*>(hh);
  if (!h) return einval("bpmf_get_timing");
  if (!h->timing) return BPMF_ESTATE;
  BPMF_TRY(resolve_timers(h));
  for (int i = 0; i < BPMF_NUM_TIMERS; ++i) {
    if (ms) ms[i] = h->t_ms[i];
    if (phase_count) phase_count[i] = h->t_cnt[i];
  }
  if (kernels) *kernels = h->kernels;
  return BPMF_OK;
}

}  // extern "C"
