// The forward operations of a batch of leaves (bfloat16, one layer).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mebptt {
namespace tc {

struct DevOp;

struct LeafArgs {
  const DevOp* ops;       // the leaves, k descending
  int n;                  // consecutive steps; rows of the products are (step, batch row), ascending
  const char* ws;         // workspace base
  const float* bias;      // [4H], gate columns permuted (4 u + q), as those of z and of the weights
  float* z;               // [n][B][4H]: out, pre-activations
  __nv_bfloat16* h;       // [B][H]: out, h_k of the last step (that of the others is the next one's h_{k-1}); NULL: not wanted
  int64_t* counters;
  int* status;
  int B, I, H;
  int first;              // 64-wide blocks of h in the first part of its contraction (lstm_dev.cuh)
};
// x [n][B][I], hprev [n][B][H]: row-major operands; wp_ih [4H][I], wp_hh [4H][H].  Returns a status.
int leaf_products(const LeafArgs& a, const void* x, const void* wp_ih, const void* hprev, const void* wp_hh, cudaStream_t s);

}  // namespace tc
}  // namespace mebptt
