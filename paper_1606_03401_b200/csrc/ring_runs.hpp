// Runs of the bfloat16 recurrence for 513 to 1024 hidden units, whose exchange goes through a ring in the L2.
#pragma once

#include "cluster_runs.hpp"

namespace mebptt {
namespace tc {

constexpr int RING_SLOTS = 4;    // steps a ring holds
constexpr int RING_CLUSTER = 4;  // CTAs that share the contraction index of a backward step

// Widths that nothing else serves.  (A device without clusters of more than eight CTAs has 257 to 512 units here as well.)
inline bool ring_runs_supported(int H, int B) { return H % 8 == 0 && H > 16 * CU && H <= 32 * CU && B <= 64; }
// CTAs of a group of batch rows: 32 units each, whole clusters (the last ones may have no unit)
inline int ring_ctas(int H) { return (H + RING_CLUSTER * CU - 1) / (RING_CLUSTER * CU) * RING_CLUSTER; }
// Units whose dz a step of a backward run waits for, likewise (fwd_waited_units).
__host__ __device__ inline int bwd_waited_units(int H) { return (H + RING_CLUSTER * CU - 1) / (RING_CLUSTER * CU) * RING_CLUSTER * CU; }
// Rows of a slot: whole groups of 8 or of 16, whichever the device gets, whether they exist or not.  A piece of eight units is
// then a line of 128 bytes that one warp writes.  (With as many rows as there are, lines of several writers: 9 rows at
// H = 608 16 % slower, 36 at H = 800 17 %.)  Up to 8 rows are one group either way, which fits with 8 if it does with 16.
inline int ring_slot_rows(int B) { return B <= 8 ? 8 : (B + 15) / 16 * 16; }
// bytes of both rings, two sets each: launches alternate between them
inline size_t ring_bytes(int H, int B) {
  const size_t rows = (size_t)ring_slot_rows(B), row = (size_t)ring_ctas(H) * CU * 2;
  return 2 * RING_SLOTS * rows * (row + 4 * row) + 256;
}
// Those of them that the workspace has a place for.  One stage of h in place of two, of h_{k-1} and of h_k, has made room for
// 4 (S - 1) bytes a unit and row, S >= 32, and budgets are to hold no fewer states than with both: a ring takes 80 bytes a
// unit and row of a slot (99 where H is no multiple of 128), more than that below four rows.  The ring of so few lies in the
// second copy of the input projections, which then are not computed ahead.
inline size_t ring_place(int H, int B) { return B > 3 ? ring_bytes(H, B) : 0; }

struct RingArgs {
  char* ring;            // slots of this launch's set: words of ones wherever nothing has been written
  char* other;           // the other set, which the launch before used and this one clears
  const char* never;     // 16 bytes of ones that nobody writes
  uint32_t fault;        // testing aid: wait for those as well
  uint32_t poll_limit;
  int first;             // the launch's first group of batch rows
};
// The sets of launch number `id` of its direction.
RingArgs ring_args(char* rings, int H, int B, bool backward, int id, bool fault, uint32_t poll_limit);

// Tensor maps: boxes of 64 columns by 128 rows, as for the cluster kernels.
// Batch rows of a group (8 or 16) and groups a launch takes, all of them where the device keeps their CTAs resident at once;
// otherwise they take turns (batch rows never mix), and where it has no room for one, rows = 0.
struct RingFit { int rows, groups; };
RingFit ring_fit(int B, int H);
int ring_smem(bool backward, int H, int rows);   // dynamic shared memory of a CTA
cudaError_t ring_forward(const CUtensorMap& tm_w, const ClusterFwdArgs& a, const RingArgs& r, RingFit fit, cudaStream_t s);
cudaError_t ring_backward(const CUtensorMap& tm_wt, const ClusterBwdArgs& a, const RingArgs& r, RingFit fit, cudaStream_t s);

}  // namespace tc
}  // namespace mebptt
