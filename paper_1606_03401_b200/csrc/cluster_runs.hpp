// Runs of the bfloat16 recurrence whose exchange stays inside a thread-block cluster: at most 512 hidden units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mebptt {
namespace tc {

struct DevOp;

constexpr int CU = 32;   // hidden units per CTA
constexpr int CB = 16;   // rows of a tile of states: the least N of an MMA with M = 128

// A cluster holds all hidden units of a layer: 32 a CTA, 16 CTAs at most.
inline bool cluster_runs_supported(int H) { return H % 8 == 0 && H >= 64 && H <= 16 * CU; }

// Units whose h a step of a forward run waits for, those past the last unit included (zeros): every warp of the gates sends
// its eight, so that nobody is a step behind what the MMAs have begun.  (A barrier can be waited for by its parity only
// while the phase after that is not over; a warp that sent nothing would be kept in step by timing alone.)
__host__ __device__ inline int fwd_waited_units(int H) { return (H + CU - 1) / CU * CU; }

struct ClusterFwdArgs {
  const DevOp* ops;      // this launch's operations (consecutive forward operations)
  int n;
  char* ws;              // workspace base
  const float* zx;       // [n][B][4H]: input projection + bias, gate columns permuted (4 u + q)
  int* status;
  int64_t* counters;
  int B, H;
  uint32_t plane16;      // distance between gate planes, in 16-byte units
  uint32_t hsz16;        // distance from h to c inside a hidden block, in 16-byte units
  uint32_t extra;        // bytes a step is told to expect too many (0; a testing aid asks for 16)
  uint32_t poll_limit;   // polls of a barrier before the wait gives up
};
struct ClusterBwdArgs {
  const DevOp* ops;        // consecutive backward operations, k descending, all in one chunk
  int n;
  char* ws;
  const float* dha;        // [S][B][H]: gradient entering h_k from the readout, row block (k-1) % S
  void* dz;                // [S][B][4H] bfloat16 staging, row block (k-1) % S, gate columns permuted
  float* dh;               // [B][H] carried dL/dh (in: from step k_hi + 1; out: for step k_lo - 1)
  float* dc;               // [B][H] carried dL/dc
  const float* loss_part;  // [S][loss_parts]
  float* loss_t;           // [t]
  int* status;
  int64_t* counters;
  int B, H, S;
  uint32_t plane16;
  const float* zleaf;      // leaf batch: [S][B][4H] pre-activations z_k (gate columns permuted); NULL otherwise
  int loss_parts;          // partial sums of the loss per step
  uint32_t extra, poll_limit;
};

// Tensor maps of the two kernels: W_hh with permuted gate rows and its transpose (boxes of 64 columns, 128 rows).
bool cluster_maps(CUtensorMap* tm_w, CUtensorMap* tm_wt, const void* wp_hh, const void* wpT_hh, int H);
// Batch rows a cluster takes (8 or 12), so that all clusters are on the device at once where that can be; 0 where
// the device cannot run clusters of this size (those of more than eight CTAs, which more than 256 units take, need not
// fit a partition of a device).  Sets the kernels' attributes as well.
int cluster_rows(int B, int H);
int cluster_smem(bool backward, int H, int rows);   // dynamic shared memory of a CTA
cudaError_t cluster_forward(const CUtensorMap& tm_w, const ClusterFwdArgs& a, int rows, cudaStream_t s);
cudaError_t cluster_backward(const CUtensorMap& tm_wt, const ClusterBwdArgs& a, int rows, cudaStream_t s);

}  // namespace tc
}  // namespace mebptt
