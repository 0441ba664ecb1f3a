// The forward operations of a batch of leaves: z_k = (W_ih x_k + b) + W_hh h_{k-1}, the h_{k-1} all memorised, and h_k.
//
// As products that accumulate in memory and an element-wise kernel behind them that was three to four kernels in a chain,
// 4 to 11 us each, in front of every backward run of leaves: what bounds them is not their loops but what surrounds
// them, and z passing through memory in between.  Here the parts of the contraction are accumulated side by side in
// tensor memory and added in registers, in the order and with the roundings of the products they replace (and so of the
// forward kernels: input projection with bias, then the recurrent part in the parts of fwd_first_part_blocks); a thread
// then has the four gates of eight units of a row side by side, and where the row is one of the last step, whose h_k
// nobody has yet (the others are memorised: the operand of the next step), it makes that as well.
//
// One CTA per 128 rows x BN gate columns: BN = 32 where 128 would leave most SMs without a tile.  A thread requests tiles of
// 64 contraction indices of both operands, one issues the MMAs, all four warps write: as in tc_gemm.cu.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "launch.hpp"
#include "leaf_products.hpp"
#include "lstm_dev.cuh"
#include "mebptt.h"
#include "sm100.cuh"
#include "tmap.hpp"

namespace mebptt {
namespace tc {

namespace {

using namespace sm100;

constexpr int BM = 128, BK = 64, STAGES = 4;
constexpr int A_BYTES = BM * BK * 2;

template <int BN>
__global__ void __launch_bounds__(128, 2) leaf_products_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_wih,
                                                               const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_whh,
                                                               const LeafArgs a, int parts, uint32_t cols) {
  constexpr int B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[STAGES], empty[STAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;

  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int M = a.n * a.B, G = 4 * a.H;
  // tiles of the contraction: the input's, then those of h, the first nk1 of them in part 1
  const int nk0 = (a.I + BK - 1) / BK, KB = (a.H + BK - 1) / BK, nk1 = a.first, nk = nk0 + KB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(&done, 1);
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_x);
    tma_prefetch_desc(&tm_wih);
    tma_prefetch_desc(&tm_h);
    tma_prefetch_desc(&tm_whh);
  }
  if (warp == 1) tmem_alloc(&tmem_slot, cols);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();
  grid_dep_launch();

  if (warp == 0 && lane == 0) {
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % STAGES;
      if (kb >= STAGES && !mbar_wait(&empty[s], ((kb / STAGES) - 1) & 1)) { failed = 1; break; }
      uint8_t* sA = ring + s * STAGE_BYTES;
      const bool in = kb < nk0;
      const int x = (in ? kb : kb - nk0) * BK;
      mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
      tma_load_2d(sA, in ? &tm_x : &tm_h, x, m0, &full[s]);
      tma_load_2d(sA + A_BYTES, in ? &tm_wih : &tm_whh, x, n0, &full[s]);
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = make_idesc(1, BM, BN, false, false);
    const uint64_t a_desc = make_desc_sw128(smem_u32(ring), 16, 1024), b_desc = make_desc_sw128(smem_u32(ring) + A_BYTES, 16, 1024);
    bool ok = true;
    for (int kb = 0; kb < nk && ok; ++kb) {
      const int s = kb % STAGES;
      if (!mbar_wait(&full[s], (kb / STAGES) & 1)) { failed = 1; ok = false; break; }
      tc_fence_after_sync();
      const int q = kb < nk0 ? 0 : kb - nk0 < nk1 ? 1 : 2;
      const bool first = kb == 0 || kb == nk0 || kb == nk0 + nk1;
      if (elect_one()) {
        mma_f16_x4(tmem + (uint32_t)(q * BN), a_desc + (uint64_t)(s * (STAGE_BYTES >> 4)), b_desc + (uint64_t)(s * (STAGE_BYTES >> 4)), idesc,
                   first ? 0u : 1u);
        mma_commit(&empty[s]);
      }
      __syncwarp();
    }
    if (elect_one()) mma_commit(&done);
    __syncwarp();
  }

  __syncwarp();
  const bool ok = mbar_wait(&done, 0) && !*(volatile int*)&failed;
  tc_fence_after_sync();
  const int row = m0 + 32 * warp + lane;             // step row / B of the batch (ascending), batch row row % B
  const bool live = ok && row < M;
  const int step = live ? row / a.B : 0, b = live ? row - step * a.B : 0;
  const bool makes_h = live && a.h && step == a.n - 1;
  const float* cprev = reinterpret_cast<const float*>(a.ws + (size_t)a.ops[0].c_src * 16) + (size_t)b * a.H;
  const uint32_t lanes = tmem + ((uint32_t)(32 * warp) << 16);
#pragma unroll 1
  for (int c = 0; c < BN; c += 32) {
    if (n0 + c >= G) break;                          // (G is a multiple of 32)
    float z[32];
    {
      uint32_t r0[32], r1[32];
      tmem_ld_32x32(lanes + (uint32_t)c, r0);
      tmem_ld_32x32(lanes + (uint32_t)(BN + c), r1);
      tmem_ld_wait();
      const float4* bias = reinterpret_cast<const float4*>(a.bias + n0 + c);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 v = bias[j];
        z[4 * j] = (__uint_as_float(r0[4 * j]) + v.x) + __uint_as_float(r1[4 * j]);
        z[4 * j + 1] = (__uint_as_float(r0[4 * j + 1]) + v.y) + __uint_as_float(r1[4 * j + 1]);
        z[4 * j + 2] = (__uint_as_float(r0[4 * j + 2]) + v.z) + __uint_as_float(r1[4 * j + 2]);
        z[4 * j + 3] = (__uint_as_float(r0[4 * j + 3]) + v.w) + __uint_as_float(r1[4 * j + 3]);
      }
      if (parts > 2) {
        tmem_ld_32x32(lanes + (uint32_t)(2 * BN + c), r0);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) z[j] += __uint_as_float(r0[j]);
      }
    }
    if (!live) continue;
    float4* zp = reinterpret_cast<float4*>(a.z + (size_t)row * G + n0 + c);
#pragma unroll
    for (int j = 0; j < 8; ++j) zp[j] = make_float4(z[4 * j], z[4 * j + 1], z[4 * j + 2], z[4 * j + 3]);
    if (!makes_h) continue;
    // the eight units of these columns, with the arithmetic of the forward kernels
    const int u0 = (n0 + c) / 4;
    const float4 c0 = *reinterpret_cast<const float4*>(cprev + u0), c1 = *reinterpret_cast<const float4*>(cprev + u0 + 4);
    const float cp[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
    float h[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float iv = sigmoid_fast(z[4 * j]), fv = sigmoid_fast(z[4 * j + 1]), gv = tanh_fast(z[4 * j + 2]), ov = sigmoid_fast(z[4 * j + 3]);
      h[j] = ov * tanh_fast(fmaf(fv, cp[j], iv * gv));
    }
    *reinterpret_cast<uint4*>(a.h + (size_t)b * a.H + u0) =
        make_uint4(pack_bf16x2(h[0], h[1]), pack_bf16x2(h[2], h[3]), pack_bf16x2(h[4], h[5]), pack_bf16x2(h[6], h[7]));
  }
  if (!ok && threadIdx.x == 0) *a.status = MEBPTT_ERR_TIMEOUT;
  if (failed && warp == 0 && lane == 0)
    for (int s = 0; s < STAGES; ++s) (void)mbar_wait(&full[s], 0);   // loads may still be in flight
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, cols);
  if (ok && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) a.counters[0] += a.n;
}

}  // namespace

int leaf_products(const LeafArgs& a, const void* x, const void* wp_ih, const void* hprev, const void* wp_hh, cudaStream_t s) {
  const int M = a.n * a.B, G = 4 * a.H, parts = a.first < (a.H + BK - 1) / BK ? 3 : 2;
  const int wide_tiles = (G + 127) / 128 * ((M + BM - 1) / BM);
  const bool narrow = wide_tiles <= 74;   // tiles of 128 columns would occupy half the SMs at most
  const int BN = narrow ? 32 : 128;
  CUtensorMap tx, twi, th, twh;
  if (!make_tmap_2d(&tx, x, 2, (uint64_t)a.I, (uint64_t)M, (uint64_t)a.I * 2, 64, BM) ||
      !make_tmap_2d(&twi, wp_ih, 2, (uint64_t)a.I, (uint64_t)G, (uint64_t)a.I * 2, 64, (uint32_t)BN) ||
      !make_tmap_2d(&th, hprev, 2, (uint64_t)a.H, (uint64_t)M, (uint64_t)a.H * 2, 64, BM) ||
      !make_tmap_2d(&twh, wp_hh, 2, (uint64_t)a.H, (uint64_t)G, (uint64_t)a.H * 2, 64, (uint32_t)BN))
    return MEBPTT_ERR_UNSUPPORTED;
  const int smem = STAGES * (A_BYTES + BN * BK * 2) + 1024;
  auto* fn = narrow ? leaf_products_kernel<32> : leaf_products_kernel<128>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  const uint32_t used = (uint32_t)(parts * BN), cols = used <= 64 ? 64u : used <= 128 ? 128u : used <= 256 ? 256u : 512u;
  if (e == cudaSuccess)
    e = launch_pdl(fn, dim3((unsigned)((G + BN - 1) / BN), (unsigned)((M + BM - 1) / BM)), dim3(128), (size_t)smem, s, tx, twi, th, twh, a, parts, cols);
  if (e != cudaSuccess) { cudaGetLastError(); return MEBPTT_ERR_CUDA; }
  return MEBPTT_OK;
}

}  // namespace tc
}  // namespace mebptt
