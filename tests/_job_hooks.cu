// Test hooks: ends of a solve and of an application that only a held-up GPU reaches, presented to the host code.
#include <cstddef>

#include "tpcg_dev.cuh"

namespace tpcg {
int job_start(SolveJob& j);
int job_step(SolveJob& j);
}  // namespace tpcg

// The plan's application word as a wait that gave up leaves it.
extern "C" void hook_give_up(tpcg_plan* p) { *p->h_err = 1; }

// A solve whose first chunk reads back without a completed iteration (timeout = 0), or with the word of a wait that gave
// up (timeout = 1).  *steps: job_step calls until the solve ended (at most 20); returns its status, or -1 for a failed
// call.
extern "C" int hook_stalled_chunk(tpcg_plan* p, const double* eta, double* ups, int timeout, int* steps) {
  tpcg::SolveJob j;
  j.p = p;
  j.eta = eta;
  j.ups = ups;
  j.tol = 1e-10;
  j.maxit = 50;
  j.flags = TPCG_ZERO_GUESS;
  if (tpcg::job_start(j) || cudaStreamSynchronize(p->stream) != cudaSuccess) return -1;
  tpcg::SolveState* hs = p->h_state;
  hs->done = 0;
  hs->status = TPCG_OK;
  if (timeout) {
    hs->timeout = 1;
    char* word = reinterpret_cast<char*>(p->d_state) + offsetof(tpcg::SolveState, timeout);
    if (cudaMemcpy(word, &timeout, sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess) return -1;
  } else {
    hs->iter = 0;
  }
  for (*steps = 0; j.phase != 3 && *steps < 20; ++*steps) {
    if (tpcg::job_step(j)) return -1;
  }
  return j.phase == 3 ? j.status : -1;
}
