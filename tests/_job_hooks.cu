// Test hooks: ends of an application that only a held-up GPU reaches, presented to the host code.
#include "tpcg_dev.cuh"

// The plan's application word as a wait that gave up leaves it.
extern "C" void hook_give_up(tpcg_plan* p) { *p->h_err = 1; }
