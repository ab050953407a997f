// C ABI of libtpcg (include/tpcg.h): plan setup and the PCG driver.
//
// tpcg_solve runs Algorithm 1 with every scalar (alpha, beta, rho, the stop
// test) on the device.  The host only enqueues kernels in chunks of
// iterations and reads the device state between chunks; kernels of an
// iteration that starts after convergence return immediately.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <chrono>
#include <new>
#include <thread>

#include "tpcg_dev.cuh"

namespace tpcg {

void launch_apply_laplacian(const tpcg_plan* p, const Geom& g, const double* x, double* w);
void launch_init_residual(const tpcg_plan* p, const Geom& g, const double* eta, const double* U, bool zero_guess);
void launch_eta_sum(const tpcg_plan* p, const Geom& g, const double* eta, const double* U0);
void launch_direction(const tpcg_plan* p, const Geom& g);
void launch_update(const tpcg_plan* p, const Geom& g, double* U, bool zero_guess_first);
void launch_true_residual(const tpcg_plan* p, const Geom& g, const double* eta, const double* U, bool force);
void launch_form_u(const tpcg_plan* p, const Geom& g, double* U, bool force);
void launch_center_u(const tpcg_plan* p, const Geom& g, double* U, bool force);
void launch_zero(const tpcg_plan* p, long long N, double* U);
void launch_to_lp(const tpcg_plan* p, const Geom& g, const double* r);
void launch_norm_shift(const tpcg_plan* p, const Geom& g, const double* r);
void launch_f32_to_f64(const tpcg_plan* p, long long N, const float* a, double* b);
void launch_fixed_to_f64(const tpcg_plan* p, long long N, const int* a, int kp, double* b);
void launch_rhs_add_bc(const tpcg_plan* p, const Geom& g, double* eta, const double* bv);
void launch_efield(const tpcg_plan* p, const Geom& g, const double* U, const double* bval, double* ex, double* ey,
                   double* ez);
int setup_fx_grids(tpcg_plan* p);
void run_precond_f64(const tpcg_plan* pl, const double* R, double* Z, SolveState* st);
void run_precond_cmp(const tpcg_plan* p, const Geom& g, const double* R, double* Z, SolveState* st);
int run_precond_tc(const tpcg_plan* pl, float* Z, SolveState* st);
int tc_plan_setup(tpcg_plan* pl);
int oz_plan_setup(tpcg_plan* pl);
bool oz_axis_ok(int l);
void tc_plan_release(tpcg_plan* pl);
int tc_launches_per_apply(const tpcg_plan* pl);
void tc_apply_grain(tpcg_plan* pl);

const char* kernel_kind_name(int kind) {
  static const char* names[kKindCount] = {"eta_sum", "init_residual", "direction", "update", "true_residual",
                                          "center", "laplacian", "modeprod_f64", "modeprod_tc", "convert",
                                          "form_u"};
  return (kind >= 0 && kind < kKindCount) ? names[kind] : "unknown";
}

namespace {

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) == cudaSuccess && prev != dev) cudaSetDevice(dev);
    else prev = -1;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

int pad_to(int v, int m) { return ((v + m - 1) / m) * m; }

Geom make_geom(const tpcg_plan* p) {
  Geom g{};
  g.nx = p->nx;
  g.ny = p->ny;
  g.nz = p->nz;
  for (int m = 0; m < 3; ++m) {
    g.bc[m] = p->bc[m];
    g.ih2[m] = 1.0 / (p->h[m] * p->h[m]);
  }
  if (p->nz == 1) g.ih2[2] = 0.0;
  for (int m = 0; m < 3; ++m) {
    g.ih2f[m] = (float)g.ih2[m];
    g.nih2[m] = -g.ih2[m];
  }
  g.uniform = (g.ih2[0] == g.ih2[1]) && (p->nz == 1 || g.ih2[2] == g.ih2[0]);
  g.N = p->N;
  return g;
}

// The six (3D) or four (2D) mode-product passes of Algorithm 7.  Each pass
// contracts the contiguous index of its input; its output strides make the
// next contraction index contiguous.  padv = row-pitch granularity (elements).
void build_stages(tpcg_plan* p, int padv, int first_pitch) {
  const int n = p->nx, q = p->ny, t = p->nz;
  const int np = pad_to(n, padv), qp = pad_to(q, padv), tp = pad_to(t, padv);
  std::vector<StageParams> S;
  auto mk = [](int A, int B, int C, int pitch, int axis, int dir, long long oa, long long ob, long long oc) {
    StageParams s{};
    s.A = A; s.B = B; s.C = C; s.Cout = C; s.in_pitch = pitch; s.axis = axis; s.dir = dir;
    s.oa = oa; s.ob = ob; s.oc = oc;
    s.lamA = s.lamB = s.lamC = 0;
    return s;
  };
  if (t > 1) {
    StageParams s1 = mk(t, q, n, first_pitch, 0, 0, qp, 1, (long long)t * qp);         // -> [n][t][q]
    s1.out_rows = n * t; s1.out_C = q; s1.out_pitch_elems = qp;
    StageParams s2 = mk(n, t, q, qp, 1, 0, (long long)q * tp, 1, tp);                  // -> [n][q][t]
    s2.out_rows = n * q; s2.out_C = t; s2.out_pitch_elems = tp;
    StageParams s3 = mk(n, q, t, tp, 2, 0, (long long)q * tp, tp, 1);                  // -> [n][q][t], x G
    s3.scale = 1; s3.lamA = 0; s3.lamB = 1; s3.lamC = 2;
    s3.out_rows = n * q; s3.out_C = t; s3.out_pitch_elems = tp;
    StageParams s4 = mk(n, q, t, tp, 2, 1, qp, 1, (long long)n * qp);                  // -> [t][n][q]
    s4.out_rows = t * n; s4.out_C = q; s4.out_pitch_elems = qp;
    StageParams s5 = mk(t, n, q, qp, 1, 1, (long long)q * np, 1, np);                  // -> [t][q][n]
    s5.out_rows = t * q; s5.out_C = n; s5.out_pitch_elems = np;
    StageParams s6 = mk(t, q, n, np, 0, 1, (long long)q * n, n, 1);                    // -> Z [t][q][n]
    s6.final_stage = 1;
    s6.out_rows = t * q; s6.out_C = n; s6.out_pitch_elems = n;
    S = {s1, s2, s3, s4, s5, s6};
  } else {
    StageParams s1 = mk(1, q, n, first_pitch, 0, 0, qp, 1, qp);                        // -> [n][q]
    s1.out_rows = n; s1.out_C = q; s1.out_pitch_elems = qp;
    StageParams s2 = mk(n, 1, q, qp, 1, 0, qp, 0, 1);                                   // -> [n][q], x G
    s2.scale = 1; s2.lamA = 0; s2.lamB = 2; s2.lamC = 1;
    s2.out_rows = n; s2.out_C = q; s2.out_pitch_elems = qp;
    StageParams s5 = mk(1, n, q, qp, 1, 1, np, 1, np);                                  // -> [q][n]
    s5.out_rows = q; s5.out_C = n; s5.out_pitch_elems = np;
    StageParams s6 = mk(1, q, n, np, 0, 1, (long long)q * n, n, 1);                    // -> Z [q][n]
    s6.final_stage = 1;
    s6.out_rows = q; s6.out_C = n; s6.out_pitch_elems = n;
    S = {s1, s2, s5, s6};
  }
  p->stages = S;
  size_t mx = 0;
  for (const auto& s : S)
    if (!s.final_stage) mx = std::max(mx, (size_t)s.out_rows * (size_t)s.out_pitch_elems);
  p->t_elems = mx;
}

template <class T>
int dalloc(tpcg_plan* p, T** ptr, size_t count) {
  *ptr = nullptr;
  if (count == 0) count = 1;
  if (cudaMalloc((void**)ptr, count * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return TPCG_ERR_OOM;
  }
  p->device_bytes += count * sizeof(T);
  return TPCG_OK;
}

void free_plan(tpcg_plan* p) {
  if (!p) return;
  if (p->stream) cudaStreamSynchronize(p->stream);
  else cudaDeviceSynchronize();
  graph_reset(p);
  tc_plan_release(p);
  for (int a = 0; a < 3; ++a) {
    for (int d = 0; d < 2; ++d) {
      cudaFree(p->d_W64[a][d]);
      cudaFree(p->d_Wt16[a][d]);
      cudaFree(p->d_oz[a][d]);
    }
    cudaFree(p->d_lam64[a]);
    cudaFree(p->d_lam32[a]);
  }
  cudaFree(p->d_G);
  cudaFree(p->d_R);
  cudaFree(p->d_P[0]);
  if (p->prec == TPCG_FP64) cudaFree(p->d_P[1]);  // mixed forms: one allocation for the ring
  cudaFree(p->d_W);
  cudaFree(p->d_Z);
  cudaFree(p->d_Rlp);
  cudaFree(p->d_T[0]);
  cudaFree(p->d_T[1]);
  cudaFree(p->d_eta_h);
  cudaFree(p->d_ups_h);
  cudaFree(p->d_eta_h2);
  cudaFree(p->d_ups_h2);
  for (int i = 0; i < 2; ++i) {
    if (p->ev_in[i]) cudaEventDestroy(p->ev_in[i]);
    if (p->ev_solved[i]) cudaEventDestroy(p->ev_solved[i]);
    if (p->ev_out[i]) cudaEventDestroy(p->ev_out[i]);
  }
  if (p->s_in) cudaStreamDestroy(p->s_in);
  if (p->s_out) cudaStreamDestroy(p->s_out);
  cudaFree(p->d_state);
  cudaFree(p->d_partials);
  if (p->h_state) cudaFreeHost(p->h_state);
  if (p->ev_state) cudaEventDestroy(p->ev_state);
  for (cudaEvent_t e : p->prof.pool) cudaEventDestroy(e);
  delete p;
}

uint16_t host_bf16(double x) {
  // FP64 -> BF16, one round-to-nearest-even step on the FP64 bit pattern
  // (eigenbasis entries are finite and far inside the BF16 normal range).
  uint64_t u;
  std::memcpy(&u, &x, 8);
  const uint32_t sign = (uint32_t)(u >> 48) & 0x8000u;
  const int e = (int)((u >> 52) & 0x7ff);
  const int eb = e - 1023 + 127;
  if (e == 0 || eb <= 0) return (uint16_t)sign;
  const uint64_t mant = u & 0xfffffffffffffull;
  const uint32_t top = (uint32_t)(mant >> 45);
  const uint64_t rest = mant & ((1ull << 45) - 1);
  uint32_t bits = ((uint32_t)eb << 7) | top;
  if (rest > (1ull << 44) || (rest == (1ull << 44) && (top & 1u))) bits += 1;
  return (uint16_t)(sign | bits);
}

// The value of a BF16 bit pattern (exact in FP64).
double host_bf16_value(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return (double)f;
}

// FP64 -> TF32 in an FP32 container: one round-to-nearest-even step at the 10-bit mantissa, on the FP64 bit
// pattern (eigenbasis entries are finite, |x| <= 1, far inside the normal range).
float host_tf32(double x) {
  uint64_t u;
  std::memcpy(&u, &x, 8);
  const uint64_t sign = u >> 63;
  const int e = (int)((u >> 52) & 0x7ff);
  if (e == 0 || e - 1023 + 127 <= 0) return sign ? -0.0f : 0.0f;
  const uint64_t mant = u & 0xfffffffffffffull;
  uint64_t top = mant >> 42;                 // 10 kept bits
  const uint64_t rest = mant & ((1ull << 42) - 1), half = 1ull << 41;
  uint32_t bits = ((uint32_t)(e - 1023 + 127) << 23) | (uint32_t)(top << 13);
  if (rest > half || (rest == half && (top & 1u))) bits += 1u << 13;  // carry may bump the exponent: correct
  bits |= (uint32_t)sign << 31;
  float f;
  std::memcpy(&f, &bits, 4);
  return f;
}

uint16_t host_f16(double x) {
  // FP64 -> FP16 (binary16), one round-to-nearest-even step, subnormals kept
  uint64_t u;
  std::memcpy(&u, &x, 8);
  const uint32_t sign = (uint32_t)(u >> 48) & 0x8000u;
  const int e = (int)((u >> 52) & 0x7ff);
  if (e == 0) return (uint16_t)sign;
  const int E = e - 1023;
  if (E > 15) return (uint16_t)(sign | 0x7bffu);
  const uint64_t m = (u & 0xfffffffffffffull) | (1ull << 52);
  int sh = 42;
  uint32_t ef = 0;
  if (E >= -14) ef = (uint32_t)(E + 15);
  else {
    sh = 28 - E;
    if (sh > 62) return (uint16_t)sign;
  }
  const uint64_t qv = m >> sh, rem = m & ((1ull << sh) - 1), half = 1ull << (sh - 1);
  uint32_t bits = ef ? ((ef << 10) | ((uint32_t)qv & 0x3ffu)) : (uint32_t)qv;
  if (rem > half || (rem == half && (qv & 1ull))) bits += 1;
  if (bits >= 0x7c00u) bits = 0x7bffu;
  return (uint16_t)(sign | bits);
}

int run_precond(const tpcg_plan* p, const double* R, void* Z, SolveState* st) {
  if (p->prec == TPCG_FP64) {
    if (p->pc_kind == TPCG_PRECOND_PINV) run_precond_f64(p, R, (double*)Z, st);
    else run_precond_cmp(p, make_geom(p), R, (double*)Z, st);
    return TPCG_OK;
  }
  return run_precond_tc(p, (float*)Z, st);
}

// Whether a wait of an earlier application outside a solve gave up, once.
bool take_give_up(tpcg_plan* p) {
  volatile int* word = p->h_err;
  if (!*word) return false;
  *word = 0;
  return true;
}

int last_cuda_error() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    fprintf(stderr, "libtpcg: CUDA error %s\n", cudaGetErrorString(e));
    return TPCG_ERR_CUDA;
  }
  return TPCG_OK;
}

int enqueue_state_readback(tpcg_plan* p) {
  if (cudaMemcpyAsync(p->h_state, p->d_state, sizeof(SolveState), cudaMemcpyDeviceToHost, p->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  if (cudaEventRecord(p->ev_state, p->stream) != cudaSuccess) return TPCG_ERR_CUDA;
  return last_cuda_error();
}

// The launches of `count` iterations starting at j.issued.  A chunk ends with one check of the true residual: the
// iterations after the one whose recurrence met the tolerance return at once (paused()), so the check sees the
// iterate it would have seen directly behind that iteration, and neither the checks of the other iterations nor the
// application of the preconditioner behind a last one are launched (a launch that returns at once still takes 2.3 us:
// at 64 x 64 x 32 they were 8 of a solve's 35).  An application is due before every iteration but the first, whose
// Z the set-up formed.  The comparators' kernels run unconditionally: check and application behind every iteration.
int launch_iterations(SolveJob& j, int count) {
  tpcg_plan* p = j.p;
  const Geom g = make_geom(p);
  const bool cmp = p->pc_kind != TPCG_PRECOND_PINV;
  for (int c = 0; c < count; ++c) {
    const int k = j.issued + c;
    if (!cmp && k > 0) {
      const int rc = run_precond(p, p->d_R, p->d_Z, p->d_state);  // Z = M R, rho, beta
      if (rc) return rc;
    }
    launch_direction(p, g);                             // direction P, W = L P, alpha
    launch_update(p, g, j.ups, k == 0 && (j.flags & TPCG_ZERO_GUESS));  // U and R updates
    if (p->defer_u) launch_form_u(p, g, j.ups, false);  // deferred U updates, when a check is due or the ring is full
    if (cmp) {
      launch_true_residual(p, g, j.eta, j.ups, false);  // stop test
      const int rc = run_precond(p, p->d_R, p->d_Z, p->d_state);
      if (rc) return rc;
    }
  }
  if (!cmp) launch_true_residual(p, g, j.eta, j.ups, false);  // stop test
  // singular operators: centre U on the device if the stop test succeeded inside this chunk
  if (p->singular) launch_center_u(p, g, j.ups, false);
  return TPCG_OK;
}

// Graphs kept per plan; the least recently used is dropped beyond this.
constexpr size_t kGraphCap = 48;

// Runs the launch sequence `launch` on the plan's stream, as a CUDA graph when the plan allows it: the
// sequence of `key` is captured the first time it is needed (stream capture of the same launches) and
// replayed afterwards.  The kernels read the solve's buffers from the device state, so a captured sequence
// serves every solve of the plan.  Profiling (per-launch events) and the legacy default stream launch
// directly; a sequence that fails to capture turns graphs off for the plan.
template <class F>
int run_graphed(tpcg_plan* p, const GraphKey& key, F&& launch) {
  if (!p->use_graphs || !p->stream || p->prof.on) return launch();
  auto it = p->graphs.find(key);
  if (it == p->graphs.end()) {
    cudaGraph_t graph = nullptr;
    if (cudaStreamBeginCapture(p->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      p->use_graphs = 0;
      return launch();
    }
    const unsigned long long lc0 = p->launch_count;
    const int rc = launch();
    const cudaError_t ec = cudaStreamEndCapture(p->stream, &graph);
    const unsigned long long kernels = p->launch_count - lc0;
    p->launch_count = lc0;
    cudaGraphExec_t exec = nullptr;
    if (rc != TPCG_OK || ec != cudaSuccess || !graph || cudaGraphInstantiate(&exec, graph, 0ull) != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      if (rc != TPCG_OK) return rc;
      p->use_graphs = 0;
      return launch();
    }
    cudaGraphDestroy(graph);
    if (p->graphs.size() >= kGraphCap) {
      auto old = p->graphs.begin();
      for (auto q = p->graphs.begin(); q != p->graphs.end(); ++q)
        if (q->second.used < old->second.used) old = q;
      cudaGraphExecDestroy(old->second.exec);
      p->graphs.erase(old);
    }
    it = p->graphs.emplace(key, GraphEntry{exec, kernels, 0}).first;
  }
  it->second.used = ++p->graph_clock;
  p->launch_count += it->second.kernels;
  return cudaGraphLaunch(it->second.exec, p->stream) == cudaSuccess ? TPCG_OK : TPCG_ERR_CUDA;
}

unsigned graph_flags(const SolveJob& j) {
  return ((j.flags & TPCG_ZERO_GUESS) ? 1u : 0u) | ((((uintptr_t)j.eta & 15) == 0) ? 2u : 0u) |
         ((((uintptr_t)j.ups & 15) == 0) ? 4u : 0u);
}

// `count` iterations of the PCG loop of Algorithm 1; kernels of iterations after
// convergence return at once
int enqueue_iterations(SolveJob& j, int count) {
  tpcg_plan* p = j.p;
  const int rc = run_graphed(p, GraphKey{1, j.issued > 0 ? 1 : 0, count, graph_flags(j), p->graph_gen},
                             [&]() { return launch_iterations(j, count); });
  if (rc) return rc;
  j.base = j.issued;
  j.issued += count;
  return TPCG_OK;
}

}  // namespace

// Drop the plan's captured launch sequences (an option or a buffer they hold has changed).
void graph_reset(tpcg_plan* p) {
  for (auto& kv : p->graphs) cudaGraphExecDestroy(kv.second.exec);
  p->graphs.clear();
  p->graph_gen += 1;
}

int job_start(SolveJob& j) {
  tpcg_plan* p = j.p;
  if (!p || !j.eta || !j.ups) return TPCG_ERR_INVALID_ARG;
  if (!(j.tol > 0.0) || !(j.tol < 1.0) || j.maxit < 1) return TPCG_ERR_INVALID_ARG;
  const Geom g = make_geom(p);
  const bool zero_guess = (j.flags & TPCG_ZERO_GUESS) != 0;
  SolveState* hs = p->h_state;
  std::memset(hs, 0, sizeof(SolveState));
  hs->maxit = j.maxit;
  hs->tol2 = j.tol * j.tol;
  hs->first = 1;
  hs->zero_guess = zero_guess ? 1 : 0;
  hs->u_valid = zero_guess ? 0 : 1;  // mixed forms: U holds the initial guess
  hs->singular = p->singular ? 1 : 0;
  hs->status = TPCG_OK;
  hs->eta = j.eta;
  hs->ups = j.ups;
  if (cudaMemcpyAsync(p->d_state, hs, sizeof(SolveState), cudaMemcpyHostToDevice, p->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  // Algorithm 1 set-up: initial residual, Z_0, rho_0 (eq. centering first when singular)
  int rc = run_graphed(p, GraphKey{0, 0, 0, graph_flags(j), p->graph_gen}, [&]() {
    launch_eta_sum(p, g, j.eta, zero_guess ? nullptr : j.ups);  // mean, first low-precision exponent, max|U_0|
    launch_init_residual(p, g, j.eta, j.ups, zero_guess);
    if (p->lp_kind == 2 && !zero_guess) launch_to_lp(p, g, p->d_R);  // re-scale FP16 copy to the actual R_0
    return run_precond(p, p->d_R, p->d_Z, p->d_state);
  });
  if (rc) return rc;
  j.issued = 0;
  // first chunk: the iteration count of the plan's previous converged solve (similar problems repeat
  // on a plan), so that one read-back usually finds the solve finished; later chunks are short
  const int deflt = (p->prec == TPCG_FP64) ? 2 : 4;
  j.chunk = p->last_iters > 0 ? std::min(std::min(p->last_iters, 12), j.maxit + 1) : deflt;
  if ((rc = enqueue_iterations(j, j.chunk))) return rc;
  j.chunk = (p->prec == TPCG_FP64) ? 1 : 2;
  j.phase = 1;
  return enqueue_state_readback(p);
}

bool job_ready(const SolveJob& j) { return cudaEventQuery(j.p->ev_state) != cudaErrorNotReady; }

int job_step(SolveJob& j) {
  tpcg_plan* p = j.p;
  SolveState* hs = p->h_state;
  if (cudaEventSynchronize(p->ev_state) != cudaSuccess) return last_cuda_error() ? TPCG_ERR_CUDA : TPCG_ERR_CUDA;
  if (j.phase == 1) {
    j.issued = hs->iter;  // iterations that paused behind a check count for nothing
    // A chunk completes at least one iteration or ends the solve; a wait that gave up ends it too (the limit of
    // every wait of the iterations left would pass before the same error).
    if (!hs->done && !hs->timeout && j.issued > j.base && j.issued <= j.maxit + 1) {
      int rc = enqueue_iterations(j, j.chunk);
      if (rc) return rc;
      return enqueue_state_readback(p);
    }
    const Geom g = make_geom(p);
    j.status_host = hs->status;
    j.done_host = hs->done;
    j.phase = 2;
    // converged: U was centred on the device behind the chunk (singular operators), the state just
    // read back is final
    const bool finished = hs->done == 1 && hs->status == TPCG_OK;
    if (!finished) {
      if (p->defer_u) launch_form_u(p, g, j.ups, true);  // apply any deferred U updates
      if (hs->done == 2) {
        launch_zero(p, g.N, j.ups);  // eta_hat = 0: minimum-norm solution is 0
      } else {
        if (!hs->done || hs->status == TPCG_ERR_BREAKDOWN) {
          launch_true_residual(p, g, j.eta, j.ups, true);  // report the true residual of the returned iterate
          if (!hs->done) j.status_host = TPCG_ERR_NOT_CONVERGED;
        }
        if (p->singular) launch_center_u(p, g, j.ups, true);
      }
      return enqueue_state_readback(p);
    }
  }
  if (j.phase == 2) {
    int status = hs->status;
    if (!j.done_host) status = j.status_host;
    if (hs->timeout) status = TPCG_ERR_TIMEOUT;
    tpcg_info& info = j.info;
    info.status = status;
    info.iters = hs->iter;
    info.precond_applies = hs->precond_applies;
    info.prec = p->prec;
    const double en = sqrt(hs->eta_norm2);
    info.eta_norm = en;
    info.rel_res_true = (j.done_host == 2 || en == 0.0) ? 0.0 : sqrt(hs->true_rr) / en;
    info.rel_res_recur = (en == 0.0) ? 0.0 : sqrt(hs->rr) / en;
    info.removed_mean = p->singular ? hs->mean_eta : 0.0;
    info.null_component = (p->singular && j.done_host != 2) ? hs->sumU / (double)p->N : 0.0;
    info.checks = hs->checks;
    j.status = status;
    j.phase = 3;
    if (status == TPCG_OK) p->last_iters = hs->iter;
  }
  return TPCG_OK;
}

namespace {

int solve_impl(tpcg_plan* p, const double* eta, double* ups, double tol, int maxit, unsigned flags, tpcg_info* info) {
  SolveJob j;
  j.p = p;
  j.eta = eta;
  j.ups = ups;
  j.tol = tol;
  j.maxit = maxit;
  j.flags = flags;
  int rc = job_start(j);
  while (!rc && j.phase != 3) rc = job_step(j);
  if (rc) return rc;
  if (info) *info = j.info;
  return j.status;
}

}  // namespace
}  // namespace tpcg

using namespace tpcg;

extern "C" {

int tpcg_plan_create(int nx, int ny, int nz, const int bc[3], const double h[3], int prec, void* stream,
                     tpcg_plan** out) {
  if (!out) return TPCG_ERR_INVALID_ARG;
  *out = nullptr;
  if (!bc || !h) return TPCG_ERR_INVALID_ARG;
  if (nx < 3 || ny < 3 || !(nz == 1 || nz >= 3)) return TPCG_ERR_INVALID_ARG;
  const int naxes = (nz == 1) ? 2 : 3;
  for (int m = 0; m < naxes; ++m) {
    if (bc[m] < 0 || bc[m] > 4) return TPCG_ERR_INVALID_ARG;
    if (!(h[m] > 0.0) || !std::isfinite(h[m])) return TPCG_ERR_INVALID_ARG;
  }
  if (prec != TPCG_FP64 && prec != TPCG_MIXED_BF16 && prec != TPCG_MIXED_TF32 && prec != TPCG_MIXED_FP16 &&
      prec != TPCG_MIXED_BF16X3)
    return TPCG_ERR_INVALID_ARG;
  if (prec != TPCG_FP64 && (nx > 256 || ny > 256 || nz > 256)) return TPCG_ERR_UNSUPPORTED;
  const long long N = (long long)nx * ny * nz;
  if (N > (1LL << 31)) return TPCG_ERR_UNSUPPORTED;

  tpcg_plan* p = new (std::nothrow) tpcg_plan();
  if (!p) return TPCG_ERR_OOM;
  p->nx = nx; p->ny = ny; p->nz = nz;
  for (int m = 0; m < 3; ++m) {
    p->bc[m] = (m < naxes) ? bc[m] : kBcN;
    p->h[m] = (m < naxes) ? h[m] : 1.0;
  }
  p->prec = prec;
  p->lp_kind = (prec == TPCG_MIXED_BF16)   ? 1
               : (prec == TPCG_MIXED_FP16) ? 2
               : (prec == TPCG_MIXED_TF32) ? 3
               : (prec == TPCG_MIXED_BF16X3) ? 4
                                             : 0;
  p->stream = (cudaStream_t)stream;
  p->is2d = (nz == 1);
  p->N = N;
  p->singular = true;
  for (int m = 0; m < naxes; ++m)
    if (!(p->bc[m] == kBcP || p->bc[m] == kBcN)) p->singular = false;
  if (cudaGetDevice(&p->device) != cudaSuccess) { delete p; return TPCG_ERR_CUDA; }
  cudaDeviceGetAttribute(&p->num_sms, cudaDevAttrMultiProcessorCount, p->device);
  if (p->num_sms <= 0) p->num_sms = 1;
  int sm_shared = 0;
  cudaDeviceGetAttribute(&sm_shared, cudaDevAttrMaxSharedMemoryPerMultiprocessor, p->device);
  if ((size_t)sm_shared > kSmSharedBytes) { delete p; return TPCG_ERR_UNSUPPORTED; }  // sole_smem

  // Algorithm 5: eigenpairs per axis (closed forms, checked)
  const int lens[3] = {nx, ny, nz};
  for (int m = 0; m < 3; ++m) {
    if (build_axis(lens[m], p->bc[m], p->h[m], p->ax[m]) != 0) { delete p; return TPCG_ERR_EIGENBASIS; }
  }

  int rc = TPCG_OK;
  const int padv = (prec == TPCG_FP64) ? 1 : 8;
  for (int m = 0; m < 3; ++m) p->pitch16[m] = pad_to(lens[m], 8);
  build_stages(p, padv, (prec == TPCG_FP64) ? nx : p->pitch16[0]);

  // eigenbases on the device
  for (int m = 0; m < 3 && !rc; ++m) {
    const int l = lens[m];
    const AxisBasis& A = p->ax[m];
    std::vector<float> lam32(A.lam.begin(), A.lam.end());
    lam32.resize((size_t)pad_to(l, 16) + 16, 0.0f);  // 16-wide epilogue reads stay in bounds
    // FP64 matrices of the axes whose FP64 products run on the FP64 pipe; the others keep digit images
    const bool f64 = prec == TPCG_FP64 && !oz_axis_ok(l);
    if (f64 && (rc = dalloc(p, &p->d_W64[m][0], (size_t)l * l))) break;
    if (f64 && (rc = dalloc(p, &p->d_W64[m][1], (size_t)l * l))) break;
    if ((rc = dalloc(p, &p->d_lam64[m], (size_t)l))) break;
    if ((rc = dalloc(p, &p->d_lam32[m], lam32.size()))) break;
    if (f64) {
      std::vector<double> VT((size_t)l * l);
      for (int i = 0; i < l; ++i)
        for (int j = 0; j < l; ++j) VT[(size_t)j * l + i] = A.V[(size_t)i * l + j];
      cudaMemcpy(p->d_W64[m][0], A.V.data(), sizeof(double) * l * l, cudaMemcpyHostToDevice);   // W = V
      cudaMemcpy(p->d_W64[m][1], VT.data(), sizeof(double) * l * l, cudaMemcpyHostToDevice);    // W = V^T
    }
    cudaMemcpy(p->d_lam64[m], A.lam.data(), sizeof(double) * l, cudaMemcpyHostToDevice);
    cudaMemcpy(p->d_lam32[m], lam32.data(), sizeof(float) * lam32.size(), cudaMemcpyHostToDevice);
    if (prec == TPCG_MIXED_TF32) {
      // K-major W^T in TF32 (FP32 containers rounded to nearest even at the TF32 mantissa), as below
      const int lp = p->pitch16[m];
      std::vector<float> f0((size_t)l * lp, 0.0f), f1((size_t)l * lp, 0.0f);
      for (int r = 0; r < l; ++r)
        for (int c = 0; c < l; ++c) {
          f0[(size_t)r * lp + c] = host_tf32(A.V[(size_t)c * l + r]);
          f1[(size_t)r * lp + c] = host_tf32(A.V[(size_t)r * l + c]);
        }
      float *d0 = nullptr, *d1 = nullptr;
      if ((rc = dalloc(p, &d0, f0.size()))) break;
      p->d_Wt16[m][0] = d0;
      if ((rc = dalloc(p, &d1, f1.size()))) break;
      p->d_Wt16[m][1] = d1;
      cudaMemcpy(d0, f0.data(), f0.size() * 4, cudaMemcpyHostToDevice);
      cudaMemcpy(d1, f1.data(), f1.size() * 4, cudaMemcpyHostToDevice);
    } else if (prec != TPCG_FP64) {
      // K-major W^T in BF16 / FP16: dir 0 (W = V) -> element [c'][c] = V[c][c']; dir 1 (W = V^T) -> V[c'][c].
      // The split form stores a second plane after the first: lo = bf16(v - hi), hi = bf16(v).
      const int lp = p->pitch16[m];
      const size_t plane = (size_t)l * lp;
      const bool split = (prec == TPCG_MIXED_BF16X3);
      std::vector<uint16_t> b0(plane * (split ? 2 : 1), 0), b1(plane * (split ? 2 : 1), 0);
      for (int r = 0; r < l; ++r)
        for (int c = 0; c < l; ++c) {
          const double v0 = A.V[(size_t)c * l + r], v1 = A.V[(size_t)r * l + c];
          const size_t o = (size_t)r * lp + c;
          b0[o] = (prec == TPCG_MIXED_FP16) ? host_f16(v0) : host_bf16(v0);
          b1[o] = (prec == TPCG_MIXED_FP16) ? host_f16(v1) : host_bf16(v1);
          if (split) {
            b0[plane + o] = host_bf16(v0 - host_bf16_value(b0[o]));
            b1[plane + o] = host_bf16(v1 - host_bf16_value(b1[o]));
          }
        }
      uint16_t *d0 = nullptr, *d1 = nullptr;
      if ((rc = dalloc(p, &d0, b0.size()))) break;
      p->d_Wt16[m][0] = d0;
      if ((rc = dalloc(p, &d1, b1.size()))) break;
      p->d_Wt16[m][1] = d1;
      cudaMemcpy(d0, b0.data(), b0.size() * 2, cudaMemcpyHostToDevice);
      cudaMemcpy(d1, b1.data(), b1.size() * 2, cudaMemcpyHostToDevice);
    }
  }
  // PCG workspaces
  if (!rc) rc = dalloc(p, &p->d_R, (size_t)N);
  if (p->prec == TPCG_FP64) {
    for (int b = 0; b < 2 && !rc; ++b) {
      double* d = nullptr;
      rc = dalloc(p, &d, (size_t)N);
      p->d_P[b] = d;
    }
  } else if (!rc) {  // int32 directions: two slots; the ring of kPRing is allocated with TPCG_OPT_DEFER_U
    int* d = nullptr;
    rc = dalloc(p, &d, (size_t)N * 2);
    for (int b = 0; b < 2 && !rc; ++b) p->d_P[b] = d + (size_t)N * b;
    p->p_slots = 2;
  }
  if (!rc && p->prec == TPCG_FP64) rc = dalloc(p, &p->d_W, (size_t)N);
  if (!rc) {
    if (prec == TPCG_FP64) {
      double* z = nullptr;
      rc = dalloc(p, &z, (size_t)N);
      p->d_Z = z;
    } else {
      float* z = nullptr;
      rc = dalloc(p, &z, (size_t)N);
      p->d_Z = z;
    }
  }
  // 16-bit words per tensor-core operand: TF32 in FP32 containers; the split form in two planes of
  // BF16 words (hi, then lo), each plane a multiple of 64 words so the lo plane starts 128-byte aligned
  const size_t lp_elem = (prec == TPCG_MIXED_TF32 || prec == TPCG_MIXED_BF16X3) ? 2 : 1;
  if (prec == TPCG_MIXED_BF16X3) {
    p->lp_plane = (size_t)pad_to(nz * ny * p->pitch16[0], 64);
    p->t_plane = (size_t)pad_to((int)p->t_elems, 64);
  }
  if (!rc && prec != TPCG_FP64) {
    uint16_t* r = nullptr;
    rc = dalloc(p, &r, p->lp_plane ? 2 * p->lp_plane : (size_t)nz * ny * p->pitch16[0] * lp_elem);
    p->d_Rlp = r;
  }
  for (int i = 0; i < 2 && !rc && prec != TPCG_FP64; ++i) {  // (FP64 form: its intermediates use W and Z)
    uint16_t* t = nullptr;
    const size_t words = p->t_plane ? 2 * p->t_plane : p->t_elems * lp_elem;
    rc = dalloc(p, &t, words);
    p->d_T[i] = t;
    if (!rc) cudaMemset(t, 0, words * 2);
  }
  if (!rc) rc = dalloc(p, &p->d_state, 1);
  {
    // one slot of 4 doubles per block of the largest reducing launch
    const int bx = (nx + 31) / 32, by = (ny + 7) / 8;
    long long most = (long long)bx * by * nz + (long long)p->num_sms * 8;
    const StageParams& fs = p->stages.back();
    most = std::max(most, (((long long)fs.A * fs.B + 63) / 64) * ((fs.Cout + 63) / 64));
    p->partial_slots = (size_t)std::max(16384LL, most) * 4;
  }
  if (!rc) rc = dalloc(p, &p->d_partials, p->partial_slots);
  if (!rc && cudaMallocHost((void**)&p->h_state, sizeof(SolveState) + sizeof(int)) != cudaSuccess) rc = TPCG_ERR_OOM;
  if (!rc && cudaEventCreateWithFlags(&p->ev_state, cudaEventDisableTiming) != cudaSuccess) rc = TPCG_ERR_CUDA;
  if (!rc) {
    cudaMemset(p->d_state, 0, sizeof(SolveState));
    p->h_err = reinterpret_cast<int*>(p->h_state + 1);
    *p->h_err = 0;
  }
  // launch configuration, fixed per plan (reproducible reductions)
  if (!rc) {
    p->st_block = dim3(32, 8, 1);
    if (!rc && setup_fx_grids(p)) rc = TPCG_ERR_CUDA;
    for (int i = 0; i < kFxCount && !rc; ++i)
      if ((size_t)p->fx_blocks[i] * 4 > p->partial_slots) rc = TPCG_ERR_UNSUPPORTED;
  }
  if (!rc) rc = (prec != TPCG_FP64) ? tc_plan_setup(p) : oz_plan_setup(p);
  // the set-up copies ran on the legacy stream; wait for them only (not for other streams' work)
  if (!rc && cudaStreamSynchronize(0) != cudaSuccess) rc = TPCG_ERR_CUDA;
  if (rc) {
    cudaGetLastError();
    free_plan(p);
    return rc;
  }
  *out = p;
  return TPCG_OK;
}

int tpcg_plan_destroy(tpcg_plan* plan) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  free_plan(plan);
  return TPCG_OK;
}

int tpcg_plan_set_stream(tpcg_plan* plan, void* stream) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  plan->stream = (cudaStream_t)stream;
  return TPCG_OK;
}

int tpcg_plan_device_bytes(const tpcg_plan* plan, size_t* bytes) {
  if (!plan || !bytes) return TPCG_ERR_INVALID_ARG;
  *bytes = plan->device_bytes;
  return TPCG_OK;
}

int tpcg_solve(tpcg_plan* plan, const double* eta, double* ups, double tol, int maxit, unsigned flags,
               tpcg_info* info) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  const int rc = solve_impl(plan, eta, ups, tol, maxit, flags, info);
  if (info && rc != info->status) info->status = rc;
  return rc;
}

int tpcg_solve_batched(tpcg_plan* const* plans, int nsolves, const int* nrhs, const double* const* eta,
                       double* const* ups, const double* tol, int maxit, unsigned flags, tpcg_info* infos) {
  if (nsolves < 0 || (nsolves > 0 && (!plans || !eta || !ups))) return TPCG_ERR_INVALID_ARG;
  if (nsolves == 0) return TPCG_OK;
  for (int s = 0; s < nsolves; ++s) {
    if (!plans[s] || !eta[s] || !ups[s]) return TPCG_ERR_INVALID_ARG;
    if (nrhs && nrhs[s] < 0) return TPCG_ERR_INVALID_ARG;
    if (tol && !(tol[s] > 0.0 && tol[s] < 1.0)) return TPCG_ERR_INVALID_ARG;
  }
  if (maxit < 1) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plans[0]->device);
  // one queue per distinct plan (a plan's workspace serves one solve at a time);
  // queues of different plans advance concurrently on the plans' streams
  struct Item {
    const double* eta;
    double* ups;
    double tol;
    int info_index;
  };
  std::vector<tpcg_plan*> qplan;
  std::vector<std::vector<Item>> queue;
  int index = 0;
  for (int s = 0; s < nsolves; ++s) {
    size_t q = 0;
    while (q < qplan.size() && qplan[q] != plans[s]) ++q;
    if (q == qplan.size()) {
      qplan.push_back(plans[s]);
      queue.emplace_back();
    }
    const int nr = nrhs ? nrhs[s] : 1;
    for (int r = 0; r < nr; ++r) {
      const size_t off = (size_t)r * (size_t)plans[s]->N;
      queue[q].push_back(Item{eta[s] + off, ups[s] + off, tol ? tol[s] : 1e-10, index++});
    }
  }
  std::vector<SolveJob> job(qplan.size());
  std::vector<size_t> next(qplan.size(), 0);
  int first_bad = TPCG_OK;
  auto start_next = [&](size_t q) -> int {
    while (next[q] < queue[q].size()) {
      const Item& it = queue[q][next[q]];
      SolveJob j;
      j.p = qplan[q];
      j.eta = it.eta;
      j.ups = it.ups;
      j.tol = it.tol;
      j.maxit = maxit;
      j.flags = flags;
      job[q] = j;
      const int rc = job_start(job[q]);
      if (!rc) return TPCG_OK;
      if (rc == TPCG_ERR_CUDA) return rc;
      if (infos) {
        std::memset(&infos[it.info_index], 0, sizeof(tpcg_info));
        infos[it.info_index].status = rc;
      }
      if (first_bad == TPCG_OK) first_bad = rc;
      ++next[q];
    }
    job[q].phase = -1;  // queue exhausted
    return TPCG_OK;
  };
  int rc = TPCG_OK;
  for (size_t q = 0; q < qplan.size() && !rc; ++q) rc = start_next(q);
  size_t active = qplan.size();
  while (!rc && active > 0) {
    active = 0;
    bool progressed = false;
    for (size_t q = 0; q < qplan.size() && !rc; ++q) {
      if (job[q].phase == -1) continue;
      ++active;
      if (!job_ready(job[q])) continue;
      progressed = true;
      if ((rc = job_step(job[q]))) break;
      if (job[q].phase == 3) {
        const Item& it = queue[q][next[q]];
        if (infos) infos[it.info_index] = job[q].info;
        if (job[q].status != TPCG_OK && first_bad == TPCG_OK) first_bad = job[q].status;
        ++next[q];
        rc = start_next(q);
      }
    }
    if (!progressed && active > 0) std::this_thread::sleep_for(std::chrono::microseconds(20));
  }
  if (rc) return rc;
  return first_bad;
}

int tpcg_solve_host(tpcg_plan* plan, const double* eta_host, double* ups_host, double tol, int maxit, unsigned flags,
                    tpcg_info* info) {
  if (!plan || !eta_host || !ups_host) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  const size_t bytes = sizeof(double) * (size_t)plan->N;
  if (!plan->d_eta_h) {
    if (dalloc(plan, &plan->d_eta_h, (size_t)plan->N) || dalloc(plan, &plan->d_ups_h, (size_t)plan->N))
      return TPCG_ERR_OOM;
  }
  if (cudaMemcpyAsync(plan->d_eta_h, eta_host, bytes, cudaMemcpyHostToDevice, plan->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  if (!(flags & TPCG_ZERO_GUESS) &&
      cudaMemcpyAsync(plan->d_ups_h, ups_host, bytes, cudaMemcpyHostToDevice, plan->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  const int rc = solve_impl(plan, plan->d_eta_h, plan->d_ups_h, tol, maxit, flags, info);
  if (rc == TPCG_ERR_CUDA || rc == TPCG_ERR_INVALID_ARG) return rc;
  if (cudaMemcpyAsync(ups_host, plan->d_ups_h, bytes, cudaMemcpyDeviceToHost, plan->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  if (cudaStreamSynchronize(plan->stream) != cudaSuccess) return TPCG_ERR_CUDA;
  return rc;
}

// Two slots: solve i uses slot i % 2.  The copy in of solve i+1 (stream s_in) waits until the copy out
// of solve i-1, which used the same slot, has finished; the solve waits for its copy in; the copy out of
// solve i (stream s_out) waits for the solve.  Copies in and out thereby overlap the neighbouring solves.
int tpcg_solve_host_stream(tpcg_plan* plan, int nrhs, const double* const* eta_host, double* const* ups_host,
                           double tol, int maxit, unsigned flags, tpcg_info* infos) {
  if (!plan || nrhs < 0 || (nrhs > 0 && (!eta_host || !ups_host))) return TPCG_ERR_INVALID_ARG;
  if (!(tol > 0.0) || !(tol < 1.0) || maxit < 1) return TPCG_ERR_INVALID_ARG;
  for (int i = 0; i < nrhs; ++i)
    if (!eta_host[i] || !ups_host[i]) return TPCG_ERR_INVALID_ARG;
  if (nrhs == 0) return TPCG_OK;
  DeviceGuard dg(plan->device);
  if (!plan->d_eta_h && (dalloc(plan, &plan->d_eta_h, (size_t)plan->N) || dalloc(plan, &plan->d_ups_h, (size_t)plan->N)))
    return TPCG_ERR_OOM;
  if (!plan->d_eta_h2 &&
      (dalloc(plan, &plan->d_eta_h2, (size_t)plan->N) || dalloc(plan, &plan->d_ups_h2, (size_t)plan->N)))
    return TPCG_ERR_OOM;
  if (!plan->s_in) {
    if (cudaStreamCreateWithFlags(&plan->s_in, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&plan->s_out, cudaStreamNonBlocking) != cudaSuccess)
      return TPCG_ERR_CUDA;
    for (int i = 0; i < 2; ++i)
      if (cudaEventCreateWithFlags(&plan->ev_in[i], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&plan->ev_solved[i], cudaEventDisableTiming) != cudaSuccess ||
          cudaEventCreateWithFlags(&plan->ev_out[i], cudaEventDisableTiming) != cudaSuccess)
        return TPCG_ERR_CUDA;
  }
  double* const de[2] = {plan->d_eta_h, plan->d_eta_h2};
  double* const du[2] = {plan->d_ups_h, plan->d_ups_h2};
  const size_t bytes = sizeof(double) * (size_t)plan->N;
  const bool warm = !(flags & TPCG_ZERO_GUESS);
  // earlier work on the plan's stream (a previous call's solve) precedes this call's copies
  if (cudaEventRecord(plan->ev_solved[0], plan->stream) != cudaSuccess ||
      cudaStreamWaitEvent(plan->s_in, plan->ev_solved[0], 0) != cudaSuccess)
    return TPCG_ERR_CUDA;
  auto copy_in = [&](int i) -> bool {
    const int s = i & 1;
    if (i >= 2 && cudaStreamWaitEvent(plan->s_in, plan->ev_out[s], 0) != cudaSuccess) return false;
    if (cudaMemcpyAsync(de[s], eta_host[i], bytes, cudaMemcpyHostToDevice, plan->s_in) != cudaSuccess) return false;
    if (warm && cudaMemcpyAsync(du[s], ups_host[i], bytes, cudaMemcpyHostToDevice, plan->s_in) != cudaSuccess)
      return false;
    return cudaEventRecord(plan->ev_in[s], plan->s_in) == cudaSuccess;
  };
  int result = TPCG_OK, rc = TPCG_OK;
  if (!copy_in(0)) rc = TPCG_ERR_CUDA;
  for (int i = 0; i < nrhs && !rc; ++i) {
    const int s = i & 1;
    if (i + 1 < nrhs && !copy_in(i + 1)) {
      rc = TPCG_ERR_CUDA;
      break;
    }
    if (cudaStreamWaitEvent(plan->stream, plan->ev_in[s], 0) != cudaSuccess) {
      rc = TPCG_ERR_CUDA;
      break;
    }
    const int st = solve_impl(plan, de[s], du[s], tol, maxit, flags, infos ? &infos[i] : nullptr);
    if (st == TPCG_ERR_CUDA || st == TPCG_ERR_INVALID_ARG) {
      rc = st;
      break;
    }
    if (st != TPCG_OK && result == TPCG_OK) result = st;
    if (cudaEventRecord(plan->ev_solved[s], plan->stream) != cudaSuccess ||
        cudaStreamWaitEvent(plan->s_out, plan->ev_solved[s], 0) != cudaSuccess ||
        cudaMemcpyAsync(ups_host[i], du[s], bytes, cudaMemcpyDeviceToHost, plan->s_out) != cudaSuccess ||
        cudaEventRecord(plan->ev_out[s], plan->s_out) != cudaSuccess)
      rc = TPCG_ERR_CUDA;
  }
  const bool synced = cudaStreamSynchronize(plan->s_in) == cudaSuccess && cudaStreamSynchronize(plan->s_out) == cudaSuccess;
  if (rc) return rc;
  return synced ? result : TPCG_ERR_CUDA;
}

int tpcg_plan_set_option(tpcg_plan* plan, int option, int value) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  if (option == TPCG_OPT_SWEEP_GRAIN) {
    if (value < 1 || value > 64) return TPCG_ERR_INVALID_ARG;
    DeviceGuard dg(plan->device);
    const int old = plan->sweep_grain;
    plan->sweep_grain = value;
    if (setup_fx_grids(plan)) {
      plan->sweep_grain = old;
      setup_fx_grids(plan);
      return TPCG_ERR_CUDA;
    }
    tc_apply_grain(plan);
    graph_reset(plan);
    return TPCG_OK;
  }
  if (value != 0 && value != 1) return TPCG_ERR_INVALID_ARG;
  if (option == TPCG_OPT_DEFER_U) {
    if (plan->prec == TPCG_FP64) return TPCG_OK;  // the FP64 form always updates U in place
    if (value && plan->p_slots < kPRing) {  // the recorded directions need the whole ring
      DeviceGuard dg(plan->device);
      // work already enqueued on the plan's stream may still read or write the two-slot block: let it
      // finish before the block is replaced (a solve's first direction does not read the previous slot)
      if (cudaStreamSynchronize(plan->stream) != cudaSuccess) return last_cuda_error() ? TPCG_ERR_CUDA : TPCG_ERR_CUDA;
      const size_t N = (size_t)plan->nx * plan->ny * plan->nz;
      int* d = nullptr;
      if (dalloc(plan, &d, N * kPRing) != TPCG_OK) return TPCG_ERR_OOM;
      cudaFree(plan->d_P[0]);
      plan->device_bytes -= N * (size_t)plan->p_slots * sizeof(int);
      for (int b = 0; b < kPRing; ++b) plan->d_P[b] = d + N * b;
      plan->p_slots = kPRing;
    }
    plan->defer_u = value;
    graph_reset(plan);
    return TPCG_OK;
  }
  if (option == TPCG_OPT_FUSE_G) {
    plan->tc_fuse = value;
    graph_reset(plan);
    return TPCG_OK;
  }
  if (option == TPCG_OPT_SLICES) {
    plan->tc_slab = value;
    graph_reset(plan);
    return TPCG_OK;
  }
  if (option == TPCG_OPT_GRAPHS) {
    plan->use_graphs = value;
    graph_reset(plan);
    return TPCG_OK;
  }
  return TPCG_ERR_INVALID_ARG;
}

int tpcg_precond_apply(tpcg_plan* plan, const double* r, double* z) {
  if (!plan || !r || !z || r == z) return TPCG_ERR_INVALID_ARG;
  if (take_give_up(plan)) return TPCG_ERR_TIMEOUT;  // an earlier application's
  DeviceGuard dg(plan->device);
  int rc;
  if (plan->prec == TPCG_FP64) {
    if (plan->pc_kind == TPCG_PRECOND_PINV) run_precond_f64(plan, r, z, nullptr);
    else run_precond_cmp(plan, make_geom(plan), r, z, nullptr);
    return last_cuda_error();
  }
  const Geom g = make_geom(plan);
  launch_norm_shift(plan, g, r);
  launch_to_lp(plan, g, r);
  if ((rc = run_precond_tc(plan, (float*)plan->d_Z, nullptr))) return rc;
  launch_f32_to_f64(plan, plan->N, (const float*)plan->d_Z, z);
  return last_cuda_error();
}

int tpcg_apply_laplacian(tpcg_plan* plan, const double* x, double* w) {
  if (!plan || !x || !w || x == w) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  launch_apply_laplacian(plan, make_geom(plan), x, w);
  return last_cuda_error();
}

int tpcg_rhs_add_bc(tpcg_plan* plan, double* eta, const double bval[6]) {
  if (!plan || !eta || !bval) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  launch_rhs_add_bc(plan, make_geom(plan), eta, bval);
  return last_cuda_error();
}

int tpcg_plan_set_precond(tpcg_plan* plan, int kind, int p, double omega) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  if (kind != TPCG_PRECOND_PINV && kind != TPCG_PRECOND_NONE && kind != TPCG_PRECOND_JACOBI)
    return TPCG_ERR_INVALID_ARG;
  if (kind == TPCG_PRECOND_JACOBI && (p < 1 || p > 64 || !(omega >= 1.0) || !(omega < 1e300)))
    return TPCG_ERR_INVALID_ARG;
  if (kind != TPCG_PRECOND_PINV && plan->prec != TPCG_FP64) return TPCG_ERR_UNSUPPORTED;
  plan->pc_kind = kind;
  if (kind == TPCG_PRECOND_JACOBI) {
    plan->jac_p = p;
    plan->jac_omega = omega;
    // diagonal of L per axis and boundary class: the corner entries (alpha, beta) of eq. (lap1d)
    double dg[3][3];
    const int len[3] = {plan->nx, plan->ny, plan->nz};
    for (int m = 0; m < 3; ++m) {
      const double ih2 = 1.0 / (plan->h[m] * plan->h[m]);
      if (len[m] == 1) {
        dg[m][0] = dg[m][1] = dg[m][2] = 0.0;  // absent z axis: L_t = [0]
        continue;
      }
      double alpha = 2.0, beta = 2.0;
      switch (plan->bc[m]) {
        case TPCG_BC_N: alpha = 1.0; beta = 1.0; break;
        case TPCG_BC_DN: beta = 1.0; break;
        case TPCG_BC_ND: alpha = 1.0; break;
        default: break;
      }
      dg[m][0] = alpha * ih2;
      dg[m][1] = 2.0 * ih2;
      dg[m][2] = beta * ih2;
    }
    for (int cz = 0; cz < 3; ++cz)
      for (int cy = 0; cy < 3; ++cy)
        for (int cx = 0; cx < 3; ++cx)
          plan->jac_invd[cx + 3 * cy + 9 * cz] = 1.0 / (omega * (dg[0][cx] + dg[1][cy] + dg[2][cz]));
  }
  graph_reset(plan);
  return TPCG_OK;
}

int tpcg_efield(tpcg_plan* plan, const double* ups, const double bval[6], double* ex, double* ey, double* ez) {
  if (!plan || !ups || !ex || !ey || (plan->nz > 1 && !ez)) return TPCG_ERR_INVALID_ARG;
  if (ex == ups || ey == ups || (ez && ez == ups)) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  launch_efield(plan, make_geom(plan), ups, bval, ex, ey, plan->nz > 1 ? ez : nullptr);
  return last_cuda_error();
}

int tpcg_plan_autotune(tpcg_plan* plan, const char* cache_path, int applies, tpcg_tune_result* out) {
  if (!plan || !out || applies < 1 || applies > 1000) return TPCG_ERR_INVALID_ARG;
  std::memset(out, 0, sizeof(*out));
  out->slices = plan->tc_slab;
  out->fuse_g = plan->tc_fuse;
  if (plan->prec == TPCG_FP64) return TPCG_OK;  // one launch sequence only
  DeviceGuard dg(plan->device);
  char key[96];
  std::snprintf(key, sizeof(key), "%d %d %d %d", plan->nx, plan->ny, plan->nz, plan->prec);
  // a cached choice for this (grid, precision): "nx ny nz prec slices fuse_g us_per_apply" per line
  if (cache_path) {
    if (FILE* f = std::fopen(cache_path, "r")) {
      char line[256];
      while (std::fgets(line, sizeof(line), f)) {
        int a[6];
        double us = 0.0;
        if (std::sscanf(line, "%d %d %d %d %d %d %lf", &a[0], &a[1], &a[2], &a[3], &a[4], &a[5], &us) == 7 &&
            a[0] == plan->nx && a[1] == plan->ny && a[2] == plan->nz && a[3] == plan->prec && (a[4] == 0 || a[4] == 1) &&
            (a[5] == 0 || a[5] == 1)) {
          plan->tc_slab = a[4];
          plan->tc_fuse = a[5];
          graph_reset(plan);
          out->slices = a[4];
          out->fuse_g = a[5];
          out->us_per_apply = us;
          out->from_cache = 1;
        }
      }
      std::fclose(f);
      if (out->from_cache) return TPCG_OK;
    }
  }
  // time every distinct launch sequence: the preconditioner alone, on a constant 16-bit input in the
  // plan's own buffers (R~ in, Z out; nothing is allocated), events on the plan's stream
  const int slab0 = plan->tc_slab, fuse0 = plan->tc_fuse;
  const size_t lp_bytes = plan->lp_plane ? 4 * plan->lp_plane
                                         : (size_t)plan->nz * plan->ny * plan->pitch16[0] * (plan->lp_kind == 3 ? 4 : 2);
  if (cudaMemsetAsync(plan->d_Rlp, 0x3c, lp_bytes, plan->stream) != cudaSuccess) return TPCG_ERR_CUDA;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return TPCG_ERR_CUDA;
  }
  double best = -1.0;
  int best_s = slab0, best_f = fuse0, rc = TPCG_OK;
  std::vector<int> seen;  // launch counts per sequence, to skip options that change nothing
  for (int sl = 1; sl >= 0 && !rc; --sl)
    for (int fu = 1; fu >= 0 && !rc; --fu) {
      plan->tc_slab = sl;
      plan->tc_fuse = fu;
      if (sl && !plan->slab_state) continue;
      const int id = (sl && plan->slab_state ? 100 : 0) + tc_launches_per_apply(plan);
      bool dup = false;
      for (int v : seen) dup = dup || v == id;
      if (dup) continue;
      seen.push_back(id);
      for (int w = 0; w < 2 && !rc; ++w) rc = run_precond_tc(plan, (float*)plan->d_Z, nullptr);
      if (rc) break;
      cudaEventRecord(e0, plan->stream);
      for (int k = 0; k < applies && !rc; ++k) rc = run_precond_tc(plan, (float*)plan->d_Z, nullptr);
      cudaEventRecord(e1, plan->stream);
      float ms = 0.0f;
      if (rc || cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
        rc = rc ? rc : TPCG_ERR_CUDA;
        break;
      }
      const double us = 1e3 * (double)ms / applies;
      ++out->candidates;
      if (best < 0.0 || us < best) {
        best = us;
        best_s = sl;
        best_f = fu;
      }
    }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (!rc && take_give_up(plan)) rc = TPCG_ERR_TIMEOUT;
  plan->tc_slab = rc ? slab0 : best_s;
  plan->tc_fuse = rc ? fuse0 : best_f;
  graph_reset(plan);
  if (rc) {
    last_cuda_error();
    return rc;
  }
  if (last_cuda_error()) return TPCG_ERR_CUDA;
  out->slices = best_s;
  out->fuse_g = best_f;
  out->us_per_apply = best;
  if (cache_path) {
    if (FILE* f = std::fopen(cache_path, "a")) {
      std::fprintf(f, "%s %d %d %.3f\n", key, best_s, best_f, best);
      std::fclose(f);
    }
  }
  return TPCG_OK;
}

int tpcg_plan_cg_scalars(tpcg_plan* plan, tpcg_cg_scalars* out) {
  if (!plan || !out) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  SolveState* hs = plan->h_state;
  if (cudaMemcpyAsync(hs, plan->d_state, sizeof(SolveState), cudaMemcpyDeviceToHost, plan->stream) != cudaSuccess ||
      cudaStreamSynchronize(plan->stream) != cudaSuccess)
    return last_cuda_error() ? TPCG_ERR_CUDA : TPCG_ERR_CUDA;
  std::memset(out, 0, sizeof(*out));
  out->iter = hs->iter;
  out->alpha = hs->alpha;
  out->beta = hs->beta;
  out->rho = hs->rho;
  out->wp = hs->pWp;
  out->rr = hs->rr;
  out->sum_r = hs->sumR;
  out->mean_z = hs->mZ;
  out->lp_shift = (plan->lp_kind == 2 || plan->lp_kind == 4) ? hs->lp_shift_applied : 0;
  out->direction_exponent = (plan->prec == TPCG_FP64) ? 0 : hs->kp;
  return TPCG_OK;
}

int tpcg_plan_cg_vectors(tpcg_plan* plan, double* R, double* Z, double* P) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  const long long N = plan->N;
  SolveState* hs = plan->h_state;
  if (cudaMemcpyAsync(hs, plan->d_state, sizeof(SolveState), cudaMemcpyDeviceToHost, plan->stream) != cudaSuccess ||
      cudaStreamSynchronize(plan->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  const int k = hs->iter > 0 ? hs->iter - 1 : 0;  // index of the last direction formed
  const size_t bytes = sizeof(double) * (size_t)N;
  if (R && cudaMemcpyAsync(R, plan->d_R, bytes, cudaMemcpyDeviceToDevice, plan->stream) != cudaSuccess)
    return TPCG_ERR_CUDA;
  if (plan->prec == TPCG_FP64) {
    if (Z && cudaMemcpyAsync(Z, plan->d_Z, bytes, cudaMemcpyDeviceToDevice, plan->stream) != cudaSuccess)
      return TPCG_ERR_CUDA;
    if (P && cudaMemcpyAsync(P, plan->d_P[k & 1], bytes, cudaMemcpyDeviceToDevice, plan->stream) != cudaSuccess)
      return TPCG_ERR_CUDA;
  } else {
    if (Z) launch_f32_to_f64(plan, N, (const float*)plan->d_Z, Z);
    if (P) launch_fixed_to_f64(plan, N, (const int*)plan->d_P[k % plan->p_slots], hs->kp, P);
  }
  if (cudaStreamSynchronize(plan->stream) != cudaSuccess) return TPCG_ERR_CUDA;
  return last_cuda_error();
}

int tpcg_plan_eigenpairs(const tpcg_plan* plan, int axis, double* lam, double* V) {
  if (!plan || axis < 0 || axis > 2 || !lam || !V) return TPCG_ERR_INVALID_ARG;
  const AxisBasis& A = plan->ax[axis];
  std::memcpy(lam, A.lam.data(), sizeof(double) * A.len);
  std::memcpy(V, A.V.data(), sizeof(double) * (size_t)A.len * A.len);
  return TPCG_OK;
}

int tpcg_plan_launch_count(const tpcg_plan* plan, unsigned long long* launches) {
  if (!plan || !launches) return TPCG_ERR_INVALID_ARG;
  *launches = plan->launch_count;
  return TPCG_OK;
}

int tpcg_plan_precond_launches(const tpcg_plan* plan, int* launches) {
  if (!plan || !launches) return TPCG_ERR_INVALID_ARG;
  *launches = (plan->prec == TPCG_FP64) ? 0 : tc_launches_per_apply(plan);
  return TPCG_OK;
}

int tpcg_profile_begin(tpcg_plan* plan) {
  if (!plan) return TPCG_ERR_INVALID_ARG;
  Profiler& pr = plan->prof;
  pr.recs.clear();
  pr.used = 0;
  for (int k = 0; k < kKindCount; ++k) {
    pr.ms[k] = 0.0;
    pr.timed[k] = 0;
  }
  pr.on = true;
  return TPCG_OK;
}

int tpcg_profile_end(tpcg_plan* plan, tpcg_kernel_stat* stats, int max_stats, int* n_stats) {
  if (!plan || (max_stats > 0 && !stats) || !n_stats) return TPCG_ERR_INVALID_ARG;
  DeviceGuard dg(plan->device);
  Profiler& pr = plan->prof;
  pr.on = false;
  if (cudaStreamSynchronize(plan->stream) != cudaSuccess) return last_cuda_error();
  for (auto& r : pr.recs) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, r.second.first, r.second.second) == cudaSuccess) {
      pr.ms[r.first] += ms;
      pr.timed[r.first] += 1;
    }
  }
  cudaGetLastError();
  pr.recs.clear();
  pr.used = 0;
  int n = 0;
  for (int k = 0; k < kKindCount; ++k) {
    if (!pr.timed[k]) continue;
    if (n < max_stats) {
      std::memset(stats[n].name, 0, sizeof(stats[n].name));
      std::strncpy(stats[n].name, kernel_kind_name(k), sizeof(stats[n].name) - 1);
      stats[n].launches = pr.timed[k];
      stats[n].total_ms = pr.ms[k];
    }
    ++n;
  }
  *n_stats = n < max_stats ? n : max_stats;
  return TPCG_OK;
}

const char* tpcg_strerror(int status) {
  switch (status) {
    case TPCG_OK: return "ok";
    case TPCG_ERR_INVALID_ARG: return "invalid argument";
    case TPCG_ERR_OOM: return "out of memory";
    case TPCG_ERR_CUDA: return "CUDA error";
    case TPCG_ERR_NOT_CONVERGED: return "not converged within maxit";
    case TPCG_ERR_BREAKDOWN: return "breakdown (non-positive or non-finite CG scalar)";
    case TPCG_ERR_TIMEOUT: return "bounded device wait timed out";
    case TPCG_ERR_UNSUPPORTED: return "unsupported configuration";
    case TPCG_ERR_EIGENBASIS: return "eigenbasis accuracy check failed";
    case TPCG_ERR_ADMISSION: return "request exceeds the server's device-memory budget";
    case TPCG_PENDING: return "pending";
    case TPCG_ERR_UNKNOWN_TICKET: return "unknown ticket";
    case TPCG_ERR_CANCELLED: return "cancelled";
    default: return "unknown status";
  }
}

}  // extern "C"
