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
// Drops the schedules kept for a plan that is being freed.
void forget_plan(uint64_t plan_id);

}  // namespace team
}  // namespace mebptt
