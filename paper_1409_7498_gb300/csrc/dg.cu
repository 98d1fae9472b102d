// Device-driven runs of a single system.  A conditional node between two MD
// steps of a CUDA graph costs ~7.7 us on GB300 even when it is not taken,
// about a tenth of a 1M-bead step.  Instead, prx_run launches a device graph
// holding a few steps (the step kernel(s) of each, then k_dg_next), and
// k_dg_next decides on the device what follows: the rebuild graph when a
// particle moved more than skin/2, the reaction graph after every Theta-th
// step, then the step graph itself until the run's steps are done, each as a
// tail launch (tail launches run in the order they were made, each after the
// previous one and the launching graph completed; the host stream sees the
// whole chain as the one graph it launched).
//
// k_dg_next and the tail launch of the step graph cost ~3 us per round, so the
// graph holds up to four steps (build_device_graphs has the measurements: 1M
// beads 87.3 -> 84.5 us per step, 250,007 33.8 -> 31.5): a step after which
// something else must come first (a rebuild, a reaction step, the run's end)
// sets ctl->hold, and the graph's further step kernels return at once.
//
// This file alone is compiled with relocatable device code (device-side graph
// launches need it); the step kernel itself is not.
#include <cuda_runtime.h>

#include "prx_internal.cuh"

namespace prx {

namespace {

__global__ void k_dg_arm(Ctl* ctl, unsigned long long steps, unsigned int theta, unsigned long long rebuild,
                         unsigned long long react) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    ctl->steps_left = steps;
    ctl->until_rx = theta ? theta - (unsigned int)(ctl->step % theta) : 0u;
    ctl->dg_on = steps != 0ull;
    ctl->hold = ctl->rx_due = 0;
    ctl->dg_rebuild = rebuild;
    ctl->dg_react = react;
  }
}

// After the graph's steps (the last one's epilogue left its verdict in the
// control block): what runs next.  A failed launch sets PRX_ECUDA and ends the
// chain.
__global__ void k_dg_next(Ctl* ctl) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const int rebuild = ctl->rebin_flag, react = ctl->rx_due;  // (loads side by side)
  const unsigned long long left = ctl->steps_left, runs = ctl->dg_runs;
  ctl->dg_runs = runs + 1ull;
  ctl->hold = ctl->rx_due = 0;
  bool ok = true;
  if (rebuild) ok = cudaGraphLaunch((cudaGraphExec_t)ctl->dg_rebuild, cudaStreamGraphTailLaunch) == cudaSuccess;
  if (ok && react) ok = cudaGraphLaunch((cudaGraphExec_t)ctl->dg_react, cudaStreamGraphTailLaunch) == cudaSuccess;
  if (ok && left) ok = cudaGraphLaunch(cudaGetCurrentGraphExec(), cudaStreamGraphTailLaunch) == cudaSuccess;
  if (!ok || !left) {
    ctl->dg_on = 0;
    mark_run(ctl);
  }
  if (!ok) atomicCAS(&ctl->status, 0, PRX_ECUDA);
}

__global__ void k_dgb_arm(BatchCtl* c, unsigned long long steps, unsigned long long phase,
                          unsigned long long theta, int any_rx, unsigned long long rebuild,
                          unsigned long long react) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    c->steps_left = steps;
    c->phase = phase;
    c->theta = theta;
    c->any_rx = any_rx;
    c->dg_rebuild = rebuild;
    c->dg_react = react;
  }
}

// Persistent runs (engine.cu) of more than one launch: the graph is one launch
// and k_eng_next, so that the host queues one graph however long the run is.
// Queued one by one, the launches of two long runs filled the stream's queue
// (1,024 entries) and prx_run waited for the device.
__global__ void k_eng_arm(Ctl* ctl, unsigned long long steps) {
  if (threadIdx.x == 0 && blockIdx.x == 0) ctl->steps_left = steps;
}
__global__ void k_eng_next(Ctl* ctl, unsigned long long* bar) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const unsigned long long left = ctl->steps_left;
  const int status = ctl->status;
  bar[0] = bar[16] = 0ull;  // the launch's barrier words
  const unsigned long long rest = status == PRX_ETIMEOUT || left <= ENG_STEPS ? 0ull : left - ENG_STEPS;
  ctl->steps_left = rest;
  const bool ok = !rest || cudaGraphLaunch(cudaGetCurrentGraphExec(), cudaStreamGraphTailLaunch) == cudaSuccess;
  if (!ok) {
    ctl->steps_left = 0ull;
    atomicCAS(&ctl->status, 0, PRX_ECUDA);
  }
  if (!ok || !rest) mark_run(ctl);
}

// After a batch step (the last member's epilogue left its decision in
// rebuild_now): the rebuild of the members that need one, the reaction step
// when the batch's phase wraps, the next step.
__global__ void k_dgb_next(BatchCtl* c) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  bool ok = true;
  if (c->rebuild_now)
    ok = cudaGraphLaunch((cudaGraphExec_t)c->dg_rebuild, cudaStreamGraphTailLaunch) == cudaSuccess;
  c->phase = c->theta ? (c->phase + 1ull) % c->theta : 0ull;
  if (ok && c->any_rx && c->phase == 0ull)
    ok = cudaGraphLaunch((cudaGraphExec_t)c->dg_react, cudaStreamGraphTailLaunch) == cudaSuccess;
  if (ok && c->steps_left > 1ull) {
    c->steps_left -= 1ull;
    ok = cudaGraphLaunch(cudaGetCurrentGraphExec(), cudaStreamGraphTailLaunch) == cudaSuccess;
  } else {
    c->steps_left = 0ull;
  }
  if (!ok) c->dg_err = 1;
}

}  // namespace

void launch_dgb_arm(BatchCtl* c, cudaStream_t st, unsigned long long steps, unsigned long long phase,
                    unsigned long long theta, int any_rx, unsigned long long rebuild,
                    unsigned long long react) {
  k_dgb_arm<<<1, 32, 0, st>>>(c, steps, phase, theta, any_rx, rebuild, react);
}

void launch_dgb_next(BatchCtl* c, cudaStream_t st) { k_dgb_next<<<1, 32, 0, st>>>(c); }

void launch_dg_arm(const Sys& S, cudaStream_t st, unsigned long long steps,
                   unsigned long long rebuild, unsigned long long react) {
  k_dg_arm<<<1, 32, 0, st>>>(S.ctl, steps, S.has_rx ? S.theta : 0u, rebuild, react);
}

void launch_eng_arm(const Sys& S, cudaStream_t st, unsigned long long steps) { k_eng_arm<<<1, 32, 0, st>>>(S.ctl, steps); }

void launch_eng_next(const Sys& S, cudaStream_t st, unsigned long long* bar) { k_eng_next<<<1, 32, 0, st>>>(S.ctl, bar); }

void launch_dg_next(const Sys& S, cudaStream_t st) { k_dg_next<<<1, 32, 0, st>>>(S.ctl); }

}  // namespace prx
