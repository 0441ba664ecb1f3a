// What the kernels that walk runs of the bfloat16 recurrence share on the device: pushes between the CTAs of a cluster,
// operands in tensor memory, the inputs of a backward step.
#pragma once

#include <cuda_bf16.h>

#include "cluster_runs.hpp"
#include "lstm_dev.cuh"
#include "sm100.cuh"

namespace mebptt {
namespace tc {
namespace {

using namespace sm100;

constexpr uint32_t W_TILE = 128 * 128;   // [128 rows][64 contraction indices]

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void push16(uint32_t addr, uint4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
               : "memory");
}
// Bounded wait for bytes that peers push, over at once where this CTA has given up.
__device__ __forceinline__ bool wait_pushed(uint64_t* bar, uint32_t parity, volatile int* failed, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait_pushed(smem_u32(bar), parity)) return true;
    if (i > 256) {
      if (*failed) return false;
      __nanosleep(64);
    }
  }
  *failed = 1;
  return false;
}
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_32x32(uint32_t taddr, const uint4 (&q)[8]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(q[0].x), "r"(q[0].y), "r"(q[0].z), "r"(q[0].w), "r"(q[1].x), "r"(q[1].y), "r"(q[1].z), "r"(q[1].w),
        "r"(q[2].x), "r"(q[2].y), "r"(q[2].z), "r"(q[2].w), "r"(q[3].x), "r"(q[3].y), "r"(q[3].z), "r"(q[3].w),
        "r"(q[4].x), "r"(q[4].y), "r"(q[4].z), "r"(q[4].w), "r"(q[5].x), "r"(q[5].y), "r"(q[5].z), "r"(q[5].w),
        "r"(q[6].x), "r"(q[6].y), "r"(q[6].z), "r"(q[6].w), "r"(q[7].x), "r"(q[7].y), "r"(q[7].z), "r"(q[7].w)
      : "memory");
}
// Four MMAs over 64 contraction indices with the A operand in tensor memory (a lane per row, two values a column) and
// the K = 16 slices of B `b_step` descriptor units (16 bytes each) apart.
template <int b_step>
__device__ __forceinline__ void mma_tmem_x4(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, t;\n\t.reg .b32 a1, a2, a3;\n\t.reg .b64 b1, b2, b3;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.eq.b32 t, 0, 0;\n\t"
      "add.s32 a1, %1, 8;\n\tadd.s64 b1, %2, %5;\n\t"
      "add.s32 a2, %1, 16;\n\tadd.s64 b2, %2, %6;\n\t"
      "add.s32 a3, %1, 24;\n\tadd.s64 b3, %2, %7;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a1], b1, %3, t;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a2], b2, %3, t;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [a3], b3, %3, t;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "n"(b_step), "n"(2 * b_step), "n"(3 * b_step)
      : "memory");
}
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// A CTA that gave up may still be pushed to; nothing of it is left in flight once every peer has given up as well
// (or has finished) and the last stores have had time to land.
__device__ __forceinline__ void settle(bool failed) {
  if (failed)
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
}

// bytes of one sender's partial sums: [RB / 4 groups of batch rows][32 columns of dh][4 rows]
__host__ __device__ constexpr uint32_t recv_slot(int RB) { return (uint32_t)(CU * RB * 4); }

// What a step reads from memory does not depend on the recurrence.  A warp of its own (the scheduler of a warp of the
// gates has nothing else to issue, so what such a warp does beside its chain is paid for in full: 600 to 1300 cycles a
// step) asks for it two steps ahead, in pieces of 16 bytes that land here.  Rows are padded so that lanes with eight
// units and four groups of rows meet no bank twice.
template <int RB>
struct GateStage {
  union {
    __nv_bfloat16 g[4][RB][CU + 8];   // stored gates [gate][row][unit]
    float4 z[RB][CU + 1];             // of a leaf, for which no internal state was stored: z_k [row][unit]
  };
  float f[3][RB][CU + 4];             // gradient from the readout, c_{k-1}, c_k (not of a leaf)
};
__device__ __forceinline__ void copy16_async(void* to, const void* from) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(to)), "l"(from) : "memory");
}
// One warp; rows, units: of the cluster's rows and the CTA's units that exist.  e0: element of the first of both.
template <int RB, class Args>
__device__ __forceinline__ void ask_for(const Args& a, const DevOp& op, size_t blk, size_t e0, int rows, int units, int lane,
                                        GateStage<RB>& st) {
  const bool leaf = a.zleaf != nullptr;
  {
    const int c = 4 * (lane & 7);
    const float* d = a.dha + blk + e0 + c;
    const float* cp = reinterpret_cast<const float*>(a.ws + (size_t)op.c_src * 16) + e0 + c;
    const float* ct = reinterpret_cast<const float*>(a.ws + (size_t)op.c_dst * 16) + e0 + c;
#pragma unroll
    for (int y = 0; y < RB / 4; ++y) {
      const int r = 4 * y + (lane >> 3);
      if (r < rows && c < units) {
        const uint32_t o = (uint32_t)(r * a.H);
        copy16_async(&st.f[0][r][c], d + o);
        copy16_async(&st.f[1][r][c], cp + o);
        if (!leaf) copy16_async(&st.f[2][r][c], ct + o);
      }
    }
  }
  if (leaf) {
    const float* z = a.zleaf + 4 * (blk + e0 + lane);
#pragma unroll
    for (int r = 0; r < RB; ++r)
      if (r < rows && lane < units) copy16_async(&st.z[r][lane], z + (size_t)r * 4 * a.H);
  } else {
    const int c = 8 * (lane & 3);
    const __nv_bfloat16* g = reinterpret_cast<const __nv_bfloat16*>(a.ws + (size_t)op.gates * 16) + e0 + c;
#pragma unroll
    for (int y = 0; y < (RB + 7) / 8; ++y) {
      const int r = 8 * y + (lane >> 2);
      if (r < rows && c < units)
#pragma unroll
        for (int q = 0; q < 4; ++q) copy16_async(&st.g[q][r][c], g + (uint32_t)(r * a.H) + (size_t)q * a.plane16 * 8);
    }
  }
}
// The values of one unit and NV rows as the derivatives want them (ct: the tanh of c_k).  A leaf's forward operation is
// redone from the pre-activations with the arithmetic of the forward kernel, gates rounded as they would have been stored.
template <int NV>
struct GateIn { float g[4][NV], ct[NV], cp[NV], d[NV]; };
template <int NV, int RB>
__device__ __forceinline__ void pick_out(bool leaf, const GateStage<RB>& st, int u, int r0, GateIn<NV>& in) {
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const int r = r0 + v;
    in.d[v] = st.f[0][r][u];
    in.cp[v] = st.f[1][r][u];
    float c;
    if (leaf) {
      const float4 z = st.z[r][u];
      const float iv = sigmoid_fast(z.x), fv = sigmoid_fast(z.y), gv = tanh_fast(z.z), ov = sigmoid_fast(z.w);
      c = fmaf(fv, in.cp[v], iv * gv);
      in.g[0][v] = round_bf16(iv); in.g[1][v] = round_bf16(fv); in.g[2][v] = round_bf16(gv); in.g[3][v] = round_bf16(ov);
    } else {
      c = st.f[2][r][u];
#pragma unroll
      for (int q = 0; q < 4; ++q) in.g[q][v] = __bfloat162float(st.g[q][r][u]);
    }
    in.ct[v] = tanh_fast(c);
  }
}

}  // namespace
}  // namespace tc
}  // namespace mebptt
