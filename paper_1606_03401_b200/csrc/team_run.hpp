// What the executor calls of the team path.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "layout.hpp"
#include "plan.hpp"
#include "tc.hpp"

namespace mebptt {
namespace team {

// Enqueues one training step; returns a status.  With dry = true nothing is enqueued and the number of
// kernel launches is returned instead.
int64_t run_step(const Layout& y, const Plan* p, const tc::StepPtrs& io, bool want_dx, cudaStream_t s, bool dry);
// The schedules that run_step keeps per (problem, plan): drops those of a plan that is being freed; makes (or
// finds) one ahead of a step and returns a status; adds to out[0..3] as tc::prepare_stats.
void forget_plan(uint64_t plan_id);
int prepare_host(const Layout& y, const Plan* p);
void prepare_stats(int64_t* out);

}  // namespace team
}  // namespace mebptt
