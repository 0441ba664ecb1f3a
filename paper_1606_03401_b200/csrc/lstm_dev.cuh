// What the kernels of the bfloat16 recurrence share: the tape as they read it and the gate functions.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace mebptt {
namespace tc {

// Tape entry as the kernels see it.  Offsets are in units of 16 bytes from the workspace base.
struct DevOp {
  int32_t k;
  uint32_t stage;          // FWD: where h_k goes besides, for the chunk that is backpropagated next, 0 = nowhere
  uint32_t h_src, c_src;   // FWD: state k-1.            BWD: h_{k-1}, c_{k-1}
  uint32_t h_dst, c_dst;   // FWD: where h_k, c_k go.    BWD: h_k, c_k of the stored internal state
  uint32_t gates;          // FWD: gate planes to write, 0 = none.   BWD: gate planes to read
  uint32_t in_copy;        // FWD: hidden block receiving the copy of state k-1, 0 = none
};
static_assert(sizeof(DevOp) == 32, "DevOp layout");

// 1 / (1 + 2^(-x log2 e)): in the forms of the two instructions that flush denormals, where they change nothing (a
// power too small is added to 1, a sum too large has 0 for its reciprocal either way) and spare the code around them.
__device__ __forceinline__ float sigmoid_fast(float x) {
  float p, y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(x * -1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(1.f + p));
  return y;
}
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float bf16_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

// The contraction with W_hh is summed in two parts from 513 units on, z = (Zx + part 0) + part 1, and the batched
// products of a leaf batch add them in that order, so that both give the same bits.  64-wide blocks in the first part:
// (Through the ring in two parts at any width: each leaves something to poll for all of the four warps that poll it, which
// below 289 units the larger of the halves first would not.)
__host__ __device__ inline int ring_first_part_blocks(int H) { return ((H + 63) / 64 + (H > 512 ? 1 : 0)) / 2; }
__host__ __device__ inline int fwd_first_part_blocks(int H) { return H > 512 ? ring_first_part_blocks(H) : (H + 63) / 64; }

}  // namespace tc
}  // namespace mebptt
