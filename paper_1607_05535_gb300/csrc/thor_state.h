// Handle structs behind the C ABI, shared by the translation units.
#pragma once

#include <memory>

#include "grid.h"
#include "thor_impl.cuh"

struct thor_mlp;

struct thor_grid {
  thor::HostGrid h;
};

// One state's use of a network, known to both: the state's stream, and an
// event after the last launch there that reads the network (or, where the
// evaluation runs on the network's own stream, after its features).
struct ClosureUse {
  cudaStream_t stream = nullptr;
  cudaEvent_t read = nullptr;
  ~ClosureUse() {
    if (read) cudaEventDestroy(read);
  }
};

// learned closure attached to a state (thor_closure_attach)
struct ClosureBinding {
  thor_mlp* net = nullptr;
  std::shared_ptr<ClosureUse> use;
  const float *in_mean = nullptr, *in_std = nullptr, *out_mean = nullptr, *out_std = nullptr;
  float* y = nullptr;                 // output of every column
  void* act[2] = {nullptr, nullptr};  // bfloat16 layer inputs of every column (two of the widest layer), one allocation
  float* x = nullptr;                 // float32 features over the same memory (the thread-staged path)
  int period = 1;                     // large steps per closure window
  long long counter = 0;              // large steps since attach
};

// zonal band means accumulated over time (thor_zonal_accumulate)
struct ZonalAcc {
  int nlat = 0;                       // bands (0: nothing allocated)
  int* order = nullptr;               // [ncol] columns in the order of their bands
  void* chunk = nullptr;              // [nchunk] band, first and last + 1 of order
  int nchunk = 0;
  double* basis = nullptr;            // [6][colp] east and north unit vectors
  double* tmp = nullptr;              // [nv][nlat][9] sums of one state
  double* acc = nullptr;              // [nv][nlat][9] accumulated band means and covariances
  double* wsum = nullptr;             // [nv][colp] time sum of w at the centres of every cell
  long long samples = 0;
};

// scratch of thor_coarse_grain, kept with the coarse state: the fine columns
// of every coarse column, listed on the device from the caller's map
struct CoarseWork {
  void* buf = nullptr;
  size_t bytes = 0;
  cudaEvent_t ready = nullptr;        // the fine state's stream, where it is another than the coarse one's
};

struct thor_state {
  thor_grid* grid = nullptr;
  int precision = THOR_FP64;
  int check_finite = 0;
  ClosureBinding closure;
  ZonalAcc zonal;
  CoarseWork coarse;
  std::unique_ptr<thor::ImplBase> impl;
};

namespace thor {
int closure_large_step(thor_state* s, int n_small, double dt);   // thor_mlp.cu
void closure_release(thor_state* s);
void coarse_release(CoarseWork& w);
void zonal_release(ZonalAcc& z);                                  // thor_climate.cu
}
