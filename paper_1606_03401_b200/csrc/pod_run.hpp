// Arguments and launch of the pod kernel.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "pod.hpp"
#include "team.hpp"

namespace mebptt {
namespace pod {

struct Args {
  int L, I, H, O, B, S;
  Config c;
  size_t off_states;                   // states, by pod
  int64_t n_blocks;
  int parts;
  char* ws;
  size_t off_wf[team::kMaxLayers], off_wr;
  size_t off_dz, off_hk, off_dy, off_carry, off_dc;
  char* stages;                        // ws + off_dz
  const void* x;
  const float *bias, *b_out, *targets;
  const Task* tasks;
  int n_tasks, phases, fwd_ops, bwd_ops;
  uint32_t polls, extra_bytes;         // a wait gives up after so many polls of 20 us; bytes a phase expects and nobody sends (testing aid)
  int* status;
  int64_t* counters;
};

using Fn = void (*)(const Args);
// wide: the states of a pod pass 4 GB, or locations count parts of a block
Fn kernel(int dtype, bool gru, int nb, bool wide);

// Packs the weights in the order the kernel keeps them, lays the initial state out, clears what a step
// starts from at zero.
struct PackArgs {
  int L, I, H, O, B;
  Config c;
  const void *W, *W_out, *h0;
  const float* c0;
  char *wf[kMaxLayers], *wr, *states;  // the initial state goes to block `init` of each pod's states
  int64_t n_blocks, init;
  int parts;
  size_t w_off[kMaxLayers];
  float* zero;
  size_t n_zero;
  int64_t* counters;
};
void launch_pack(int dtype, bool gru, const PackArgs& p, cudaStream_t s);

}  // namespace pod
}  // namespace mebptt
