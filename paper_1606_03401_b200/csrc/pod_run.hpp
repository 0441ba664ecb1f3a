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
  int T;
  team::Dims d;
  int ns_f[team::kMaxLayers], ns_b[team::kMaxLayers], ns_r;
  uint64_t resident;
  int slot_floats, red_floats;
  size_t hc, csz_off, plane, gsz, rec_gates;   // bytes: layer stride of a hidden state, its c part, gate plane, a layer's planes, planes in a record
  char* ws;
  size_t off_wf[team::kMaxLayers], off_wb[team::kMaxLayers], off_wr;
  size_t off_dz, off_hk, off_hp, off_dy, off_carry, off_dc;
  const void *x, *h0;
  const float *c0, *bias, *b_out, *targets;
  const Task* tasks;
  int n_tasks, phases;
  int* status;
  int64_t* counters;
};

using Fn = void (*)(const Args);
Fn kernel(int dtype, bool gru, int nb);

}  // namespace pod
}  // namespace mebptt
