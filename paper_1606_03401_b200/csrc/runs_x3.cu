// The LSTM recurrence on the tensor cores for float32 storage (MEBPTT_TF32), one layer: persistent
// kernels that walk a run of consecutive operations, as tc_lstm.cu has them for bfloat16.
//
// Operation by operation (stepwise_x3.cu) a forward operation is a contraction over [x ; h] and a cell
// kernel, a backward one a gate kernel and a contraction, each a launch that must wait for the one
// before: 15 to 20 us an operation at H = 1024, B = 32, of which the arithmetic is a tenth.  Here a
// run of n operations is one launch with the halves of W_hh resident in shared memory.
//
// The product of two float32 values is hi hi + hi mid + mid hi of their bfloat16 halves, as in
// stepwise_x3.cu.  Both operands carry their halves as rows: the M side of the MMA is 32 rows of hi
// and 32 rows of mid of the weights, the N side 32 batch rows of hi and 32 of mid of the vector, so that
// one 64 x 64 MMA yields all products of a K = 16 slice (and mid mid, which nobody reads).
//
//   fwd_run_x3   CTA c of a group (32 batch rows) owns hidden units 8 c .. 8 c + 7: 32 gate rows.
//                h_{k-1} comes from an exchange buffer [2][groups][hi, mid][32][H] that the owners
//                fill, in slabs of 128 columns through a ring (at H = 1024 weights and vector are
//                128 KB each, more than a CTA has); x W_ih + b is batched over the run beforehand.
//   bwd_run_x3   clusters of four CTAs share 32 columns of dh: CTA r contracts the derivatives of gate
//                r (again [hi, mid][32][H] of an exchange buffer) against the matching block of W_hh^T,
//                and the partial tiles are added by the owners of 8 columns each, in the order of r.
//
// Every CTA needs the whole vector each step: 128 KB a CTA, 16.8 MB in all at H = 1024, so a step is
// bound by the L2 (about 2.5 us of it) and by the signalling round, as on the bfloat16 path.
#include "kernels.hpp"
#include "launch.hpp"
#include "sm100.cuh"
#include "tc.hpp"
#include "tmap.hpp"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace mebptt {
namespace stepwise3 {

namespace {

using namespace sm100;
using tc::GemmOut;
using tc::gemm_bf16;
typedef __nv_bfloat16 bf16;

constexpr int RU = 8;                    // hidden units a CTA owns
constexpr int RB = 32;                   // batch rows of a group
constexpr int CS = 4;                    // CTAs of a cluster of the backward kernel: one per gate
constexpr int SLAB = 2;                  // K tiles (64 columns) per copy
constexpr int RING = 4;                  // slabs in flight
constexpr uint32_t TILE = 64 * 128;      // [64 rows][64 columns] of either operand
constexpr int PART_LD = 4 * RU + 4;      // row stride of the handed-over accumulators (floats)
constexpr int RECV_LD = RB + 4;          // row stride of a partial column of dh (floats)
constexpr int SYNC_STRIDE = 32;          // words between the step counters of two groups
constexpr int TMEM_COLS = 64;

inline __host__ __device__ int whole_boxes(int KB) { return (KB + 3) / 4 * 4; }   // weights come in boxes of four tiles
inline int fwd_smem(int KB) { return lone_smem((whole_boxes(KB) + RING * SLAB) * (int)TILE + 2 * RB * PART_LD * 4 + 1024); }
inline int bwd_smem(int KB) { return lone_smem((whole_boxes(KB) + RING * SLAB) * (int)TILE + 2 * CS * 2 * RU * RECV_LD * 4 + 1024); }

__device__ __forceinline__ float sigmoidf_(float a) { return 1.0f / (1.0f + expf(-a)); }
__device__ __forceinline__ void split2(float v, bf16& hi, bf16& mid) {
  hi = __float2bfloat16_rn(v);
  mid = __float2bfloat16_rn(v - __bfloat162float(hi));
}
// halves of two neighbouring values: hi.x | hi.y and mid.x | mid.y
__device__ __forceinline__ void split_pair(float2 v, __nv_bfloat162& hi, __nv_bfloat162& mid) {
  split2(v.x, hi.x, mid.x);
  split2(v.y, hi.y, mid.y);
}
// (what a caller hands in is aligned to its elements only)
__device__ __forceinline__ float2 ld2(const float* p) { return make_float2(p[0], p[1]); }

struct FwdX3Args {
  stepwise::FwdRunStep op[32];
  const float* zx;        // [n][B][4H]: input projection and bias
  bf16* exch;             // [2][groups][64][HP]
  uint32_t* sync;
  int* status;
  int64_t* counters;
  size_t plane;           // elements between gate planes
  int n, B, H, HP, ncg, groups;
  uint32_t expect, poll_limit;
};
struct BwdX3Args {
  stepwise::BwdRunStep op[32];   // in the order of execution, time descending
  const float* dha;       // [n][B][H], row block n - 1 - i for operation i
  float *dh, *dc;         // carried gradients
  bf16* exch;             // [2][groups][4][64][HP]
  bf16* st_dz3;           // stage rows of the run's first step in time: [hi | hi | mid] of width 3 * 4H
  bf16* st_hp2;           // [hi | mid] of h_{k-1}
  bf16* st_in2;           // likewise of x_k
  uint32_t* sync;
  int* status;
  int64_t* counters;
  size_t plane;
  const float* loss_part; // [n][loss_parts] in ascending time, and where the loss terms go
  float* loss_t;
  int loss_parts;
  int n, B, H, HP, I, ncg, groups;
  uint32_t expect, poll_limit;
};

// What both kernels' producer and MMA warps do: each step the rows `row(i)` .. + 63 of the exchange
// buffer come in slabs of SLAB tiles through a ring of RING and are multiplied with the resident tiles.
struct Pipe {
  uint64_t wfull, full[RING], empty[RING], acc;
};
__device__ __forceinline__ void pipe_init(Pipe& p) {
  mbar_init(&p.wfull, 1);
  for (int s = 0; s < RING; ++s) { mbar_init(&p.full[s], 1); mbar_init(&p.empty[s], 1); }
  mbar_init(&p.acc, 1);
}
// One lane.  `steps` operations; step i waits for the counter to reach (i + 1) expect.
template <class Row>
__device__ __forceinline__ void produce(Pipe& p, uint8_t* sW, uint8_t* ring, const CUtensorMap* tm_w, int w_row,
                                        const CUtensorMap* tm_v, Row row, int KB, int n, const uint32_t* sync, uint32_t expect,
                                        uint32_t limit, volatile int* failed) {
  const int slabs = (KB + SLAB - 1) / SLAB;
  uint32_t it = 0;
  const bool any = !*failed;
  if (any) {
    const int boxes = whole_boxes(KB) / 4;   // (a box counts in full, also where it is filled with zeros)
    mbar_arrive_expect_tx(&p.wfull, (uint32_t)boxes * 4 * TILE);
    for (int q = 0; q < boxes; ++q) tma_load_3d(sW + q * 4 * TILE, tm_w, 0, w_row, 4 * q, &p.wfull);
  }
  for (int i = 0; i < n; ++i) {
    if (*failed || !wait_counter(sync, (uint32_t)(i + 1) * expect, failed, limit)) break;
    fence_proxy_async_global();
    for (int s = 0; s < slabs; ++s, ++it) {
      const uint32_t slot = it % RING, use = it / RING;
      if (use > 0 && !wait_or_fail(&p.empty[slot], (use - 1) & 1, failed)) break;
      mbar_arrive_expect_tx(&p.full[slot], SLAB * TILE);
      tma_load_3d(ring + slot * SLAB * TILE, tm_v, 0, row(i), s * SLAB, &p.full[slot]);
    }
    if (i == n - 1) grid_dep_launch();
  }
  if (*failed && any) {
    // copies that were requested may still be landing: give them a bounded chance
    (void)mbar_wait(&p.wfull, 0);
    for (uint32_t u = it > (uint32_t)RING ? it - RING : 0; u < it; ++u) (void)mbar_wait(&p.full[u % RING], (u / RING) & 1);
  }
}
// The whole warp.
__device__ __forceinline__ void multiply(Pipe& p, const uint8_t* sW, const uint8_t* ring, uint32_t tmem, int KB, int n,
                                         volatile int* failed) {
  constexpr uint32_t idesc = make_idesc(1, 64, 64, false, false);
  const int slabs = (KB + SLAB - 1) / SLAB;
  const uint64_t w0 = make_desc_sw128(smem_u32(sW), 16, 1024), v0 = make_desc_sw128(smem_u32(ring), 16, 1024);
  bool ok = !*failed && wait_or_fail(&p.wfull, 0, failed);
  uint32_t it = 0;
  for (int i = 0; i < n; ++i) {
    for (int s = 0; s < slabs && ok; ++s, ++it) {
      const uint32_t slot = it % RING;
      ok = wait_or_fail(&p.full[slot], (it / RING) & 1, failed);
      if (!ok) break;
      tc_fence_after_sync();
      const int tiles = min(SLAB, KB - s * SLAB);
      if (elect_one()) {
        for (int j = 0; j < tiles; ++j)
          mma_f16_x4(tmem, w0 + (uint64_t)((s * SLAB + j) * (TILE >> 4)), v0 + (uint64_t)((slot * SLAB + j) * (TILE >> 4)), idesc,
                     (s | j) ? 1u : 0u);
        mma_commit(&p.empty[slot]);
      }
      __syncwarp();
    }
    if (elect_one()) mma_commit(&p.acc);   // always: the epilogue counts on one arrival per step
    __syncwarp();
  }
}

__global__ void __launch_bounds__(192, 1) fwd_run_x3(const __grid_constant__ CUtensorMap tm_h, const __grid_constant__ CUtensorMap tm_w,
                                                     const __grid_constant__ FwdX3Args a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Pipe pipe;
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int KB = a.HP / 64;
  uint8_t* ring = sm + whole_boxes(KB) * TILE;
  float* part = reinterpret_cast<float*>(ring + RING * SLAB * TILE);   // [2][RB][PART_LD]: weights' hi rows, mid rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x / a.ncg, cta = blockIdx.x % a.ncg;
  uint32_t* const sync = a.sync + grp * SYNC_STRIDE;
  if (tid == 0) {
    pipe_init(pipe);
    mbar_fence_init();
    tma_prefetch_desc(&tm_h);
    tma_prefetch_desc(&tm_w);
  }
  if (warp == 4) tmem_alloc(&tmem_slot, TMEM_COLS);
  grid_dep_wait();
  if (tid == 0) failed = *a.status != 0;   // after a failure every later launch only walks through
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;

  if (warp == 4) {
    if (lane == 0)
      produce(pipe, sm, ring, &tm_w, cta * 64, &tm_h, [&](int i) { return ((i & 1) * a.groups + grp) * 64; }, KB, a.n, sync,
              a.expect, a.poll_limit, &failed);
    __syncwarp();
  } else if (warp == 5) {
    multiply(pipe, sm, ring, tmem, KB, a.n, &failed);
  } else {
    // as a reader of TMEM: warp w, lanes 0 .. 15 hold rows 16 w .. 16 w + 15 (two warps hi, two mid);
    // as an owner of state: batch row tid / 4 of the group, hidden units 2 (tid % 4), + 1 of the CTA
    const int bl = tid >> 2, u0 = 2 * (tid & 3);
    const int b = grp * RB + bl, j0 = cta * RU + u0;
    const size_t e0 = (size_t)b * a.H + j0;
    auto give = [&](int par, float2 h) {
      bf16* x = a.exch + ((size_t)(par * a.groups + grp) * 64 + bl) * a.HP + j0;
      __nv_bfloat162 hi, mid;
      split_pair(h, hi, mid);
      *reinterpret_cast<__nv_bfloat162*>(x) = hi;
      *reinterpret_cast<__nv_bfloat162*>(x + (size_t)RB * a.HP) = mid;
    };
    float2 h = ld2((const float*)a.op[0].h_prev + e0), c = ld2(a.op[0].c_prev + e0);
    float2 zx[4];
    auto fetch = [&](int i) {
      const float* z = a.zx + ((size_t)i * a.B + b) * 4 * a.H + j0;
#pragma unroll
      for (int q = 0; q < 4; ++q) zx[q] = *reinterpret_cast<const float2*>(z + (size_t)q * a.H);
    };
    give(0, h);
    named_barrier(1, 128);
    if (tid == 0) red_release_add(sync, 1u);
    fetch(0);
    for (int i = 0; i < a.n; ++i) {
      const stepwise::FwdRunStep op = a.op[i];
      const bool got = wait_or_fail(&pipe.acc, (uint32_t)i & 1, &failed);
      tc_fence_after_sync();
      uint32_t r0[32], r1[32];
      tmem_ld_32x32(tmem + ((uint32_t)(32 * warp) << 16), r0);
      tmem_ld_32x32(tmem + ((uint32_t)(32 * warp) << 16) + 32, r1);
      tmem_ld_wait();
      if (lane < 16) {
        float* dst = part + (size_t)(warp >> 1) * RB * PART_LD + 16 * (warp & 1) + lane;
#pragma unroll
        for (int v = 0; v < RB; ++v)
          dst[v * PART_LD] = warp < 2 ? __uint_as_float(r0[v]) + __uint_as_float(r1[v]) : __uint_as_float(r0[v]);
      }
      tc_fence_before_sync();
      named_barrier(1, 128);
      float g[2][4], hv[2], cv[2];   // gates i, f, g, o of the two units
      const float cp[2] = {c.x, c.y};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4 p0 = *reinterpret_cast<const float4*>(part + (size_t)bl * PART_LD + 4 * (u0 + u));
        const float4 p1 = *reinterpret_cast<const float4*>(part + (size_t)(RB + bl) * PART_LD + 4 * (u0 + u));
        g[u][0] = sigmoidf_((u ? zx[0].y : zx[0].x) + (p0.x + p1.x));
        g[u][1] = sigmoidf_((u ? zx[1].y : zx[1].x) + (p0.y + p1.y));
        g[u][2] = tanhf((u ? zx[2].y : zx[2].x) + (p0.z + p1.z));
        g[u][3] = sigmoidf_((u ? zx[3].y : zx[3].x) + (p0.w + p1.w));
        cv[u] = fmaf(g[u][1], cp[u], g[u][0] * g[u][2]);
        hv[u] = g[u][3] * tanhf(cv[u]);
      }
      const float2 hn = make_float2(hv[0], hv[1]);
      if (i + 1 < a.n) give((i + 1) & 1, hn);
      named_barrier(1, 128);   // this CTA's stores precede the release; the parts are free again
      if (tid == 0 && i + 1 < a.n) red_release_add(sync, 1u);
      if (i + 1 < a.n) fetch(i + 1);
      if (got) {
        *reinterpret_cast<float2*>((float*)op.h_out + e0) = hn;
        *reinterpret_cast<float2*>(op.c_out + e0) = make_float2(cv[0], cv[1]);
        if (op.gates) {
          float* gp = (float*)op.gates + e0;
#pragma unroll
          for (int q = 0; q < 4; ++q) *reinterpret_cast<float2*>(gp + q * a.plane) = make_float2(g[0][q], g[1][q]);
        }
        if (op.h_in_copy) {
          *reinterpret_cast<float2*>((float*)op.h_in_copy + e0) = h;
          *reinterpret_cast<float2*>(op.c_in_copy + e0) = c;
        }
      }
      h = hn;
      c = make_float2(cv[0], cv[1]);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (blockIdx.x == 0) a.counters[0] += a.n;
  }
  if (warp == 4) tmem_dealloc(tmem, TMEM_COLS);
}

__global__ void __launch_bounds__(192, 1) bwd_run_x3(const __grid_constant__ CUtensorMap tm_dz, const __grid_constant__ CUtensorMap tm_wt,
                                                     const __grid_constant__ BwdX3Args a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ Pipe pipe;
  __shared__ uint64_t pready[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int KB = a.HP / 64;
  uint8_t* ring = sm + whole_boxes(KB) * TILE;
  // partial sums received from the cluster: [2 buffers][CS senders][hi rows, mid rows][RU columns][RECV_LD]
  float* recv = reinterpret_cast<float*>(ring + RING * SLAB * TILE);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x / a.ncg, cta = blockIdx.x % a.ncg, cl = cta / CS;
  const uint32_t rank = cluster_ctarank();   // = cta % CS: the gate whose derivatives this CTA contracts
  uint32_t* const sync = a.sync + grp * SYNC_STRIDE;
  if (tid == 0) {
    pipe_init(pipe);
    mbar_init(&pready[0], CS);
    mbar_init(&pready[1], CS);
    mbar_fence_init();
    tma_prefetch_desc(&tm_dz);
    tma_prefetch_desc(&tm_wt);
  }
  if (warp == 4) tmem_alloc(&tmem_slot, TMEM_COLS);
  grid_dep_wait();
  if (tid == 0) failed = *a.status != 0;
  tc_fence_before_sync();
  cluster_sync();                            // peers arrive on each other's barriers: all must be initialised
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;

  if (warp == 4) {
    if (lane == 0)
      produce(pipe, sm, ring, &tm_wt, (cl * CS + (int)rank) * 64, &tm_dz,
              [&](int i) { return (((i & 1) * a.groups + grp) * CS + (int)rank) * 64; }, KB, a.n, sync, a.expect, a.poll_limit, &failed);
    __syncwarp();
  } else if (warp == 5) {
    multiply(pipe, sm, ring, tmem, KB, a.n, &failed);
  } else {
    const int bl = tid >> 2, u0 = 2 * (tid & 3);
    const int b = grp * RB + bl, j0 = cl * CS * RU + (int)rank * RU + u0;
    const bool owner = j0 < a.H;             // (H is a multiple of 8: all units of a CTA or none)
    const size_t e0 = (size_t)b * a.H + j0, G = 4 * (size_t)a.H;
    float dh[2] = {0.f, 0.f}, dc[2] = {0.f, 0.f};
    if (owner) {
      const float2 v = *reinterpret_cast<const float2*>(a.dh + e0), w = *reinterpret_cast<const float2*>(a.dc + e0);
      dh[0] = v.x; dh[1] = v.y; dc[0] = w.x; dc[1] = w.y;
    }
    struct { float2 g[4], ct, cp, hp, da; } in = {};
    auto fetch = [&](int i) {
      const stepwise::BwdRunStep& op = a.op[i];
      const float* gp = (const float*)op.gates + e0;
#pragma unroll
      for (int q = 0; q < 4; ++q) in.g[q] = *reinterpret_cast<const float2*>(gp + q * a.plane);
      in.ct = *reinterpret_cast<const float2*>(op.c_t + e0);
      in.cp = ld2(op.c_prev + e0);
      in.hp = ld2((const float*)op.h_prev + e0);
      in.da = *reinterpret_cast<const float2*>(a.dha + (size_t)(a.n - 1 - i) * a.B * a.H + e0);
    };
    // Product `it` into this thread's dh: each row of the accumulators goes to the CTA that owns its
    // column, which adds what the four senders sent in the order of their ranks.
    auto reduce = [&](int it) {
      float* buf = recv + (size_t)(it & 1) * CS * 2 * RU * RECV_LD;
      const bool got = wait_or_fail(&pipe.acc, (uint32_t)it & 1, &failed);
      tc_fence_after_sync();
      uint32_t r0[32], r1[32];
      tmem_ld_32x32(tmem + ((uint32_t)(32 * warp) << 16), r0);
      tmem_ld_32x32(tmem + ((uint32_t)(32 * warp) << 16) + 32, r1);
      tmem_ld_wait();
      if (lane < 16) {
        const int col = 16 * (warp & 1) + lane;      // of the cluster's 32
        float* dst = buf + (((size_t)rank * 2 + (warp >> 1)) * RU + (col % RU)) * RECV_LD;
        float v[RB];
#pragma unroll
        for (int i = 0; i < RB; ++i)
          v[i] = warp < 2 ? __uint_as_float(r0[i]) + __uint_as_float(r1[i]) : __uint_as_float(r0[i]);
#pragma unroll
        for (int i = 0; i < RB / 4; ++i)
          st_peer_f4(dst + 4 * i, (uint32_t)(col / RU), make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
      }
      tc_fence_before_sync();
      named_barrier(1, 128);
      if (tid < CS) mbar_arrive_peer(&pready[it & 1], (uint32_t)tid);   // release: the stores above are visible
      bool all = false;
      for (uint32_t spin = 0; spin < kSpinLimit; ++spin) {
        if (mbar_try_wait_cluster(&pready[it & 1], (uint32_t)(it >> 1) & 1)) { all = true; break; }
        if (spin > 256) {
          if (*(volatile int*)&failed) break;
          __nanosleep(64);
        }
      }
      if (!all) failed = 1;
      if (got && all) {
        float sum[2] = {0.f, 0.f};
#pragma unroll
        for (int p = 0; p < CS; ++p) {
          const float* src = buf + ((size_t)p * 2 * RU + u0) * RECV_LD + bl;
#pragma unroll
          for (int u = 0; u < 2; ++u) sum[u] += src[u * RECV_LD] + src[(RU + u) * RECV_LD];
        }
        dh[0] = sum[0]; dh[1] = sum[1];
      }
    };
    if (owner) fetch(0);
    for (int i = 0; i < a.n; ++i) {
      if (i > 0) reduce(i - 1);
      __nv_bfloat162 hi[4], mid[4];
      float2 hp = in.hp;
      if (owner) {
        float v[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float gi = u ? in.g[0].y : in.g[0].x, gf = u ? in.g[1].y : in.g[1].x;
          const float gg = u ? in.g[2].y : in.g[2].x, go = u ? in.g[3].y : in.g[3].x;
          const float d = (u ? in.da.y : in.da.x) + dh[u];
          const float th = tanhf(u ? in.ct.y : in.ct.x);
          const float dcv = fmaf(d * go, 1.f - th * th, dc[u]);
          v[u][0] = dcv * gg * gi * (1.f - gi);
          v[u][1] = dcv * (u ? in.cp.y : in.cp.x) * gf * (1.f - gf);
          v[u][2] = dcv * gi * (1.f - gg * gg);
          v[u][3] = d * th * go * (1.f - go);
          dc[u] = dcv * gf;
        }
        bf16* x = a.exch + ((size_t)(((i & 1) * a.groups + grp) * CS) * 64 + bl) * a.HP + j0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          split_pair(make_float2(v[0][q], v[1][q]), hi[q], mid[q]);
          *reinterpret_cast<__nv_bfloat162*>(x + (size_t)q * 64 * a.HP) = hi[q];
          *reinterpret_cast<__nv_bfloat162*>(x + (size_t)(q * 64 + RB) * a.HP) = mid[q];
        }
      }
      named_barrier(1, 128);   // this CTA's derivatives precede the release
      if (tid == 0) red_release_add(sync, 1u);
      if (i == 0 && blockIdx.x == 0 && tid < a.n) {   // loss terms, their parts in a fixed order
        float sum = 0.f;
        for (int p = 0; p < a.loss_parts; ++p) sum += a.loss_part[tid * a.loss_parts + p];
        a.loss_t[tid] = sum;
      }
      // off the recurrence: the next operation's inputs, the stages of the weight gradients
      const int blk = a.n - 1 - i;   // row block of the stages, from the run's first step in time
      if (owner) {
        if (i + 1 < a.n) fetch(i + 1);
        if (!*(volatile int*)&failed) {
          bf16* z = a.st_dz3 + ((size_t)blk * a.B + b) * 3 * G + j0;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            *reinterpret_cast<__nv_bfloat162*>(z + (size_t)q * a.H) = hi[q];
            *reinterpret_cast<__nv_bfloat162*>(z + G + (size_t)q * a.H) = hi[q];
            *reinterpret_cast<__nv_bfloat162*>(z + 2 * G + (size_t)q * a.H) = mid[q];
          }
          __nv_bfloat162 h0, h1;
          split_pair(hp, h0, h1);
          bf16* o = a.st_hp2 + ((size_t)blk * a.B + b) * 2 * a.H + j0;
          *reinterpret_cast<__nv_bfloat162*>(o) = h0;
          *reinterpret_cast<__nv_bfloat162*>(o + a.H) = h1;
        }
      }
      const float* x = (const float*)a.op[i].in;
      for (int e = blockIdx.x * 128 + tid; e < a.B * a.I; e += gridDim.x * 128) {
        const int r = e / a.I, c = e % a.I;
        bf16 x0, x1;
        split2(x[e], x0, x1);
        bf16* o = a.st_in2 + ((size_t)blk * a.B + r) * 2 * a.I + c;
        o[0] = x0; o[a.I] = x1;
      }
    }
    reduce(a.n - 1);
    if (owner && !*(volatile int*)&failed) {
      *reinterpret_cast<float2*>(a.dh + e0) = make_float2(dh[0], dh[1]);
      *reinterpret_cast<float2*>(a.dc + e0) = make_float2(dc[0], dc[1]);
    }
  }
  tc_fence_before_sync();
  cluster_sync();   // no CTA leaves while a peer may still send to it or signal it
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (blockIdx.x == 0) a.counters[1] += a.n;
  }
  if (warp == 4) tmem_dealloc(tmem, TMEM_COLS);
}

// ---- the resident operands, once per training step -------------------------------------------------
// W_hh as the forward kernel holds it: row 64 cta + 32 p + 4 u + q is half p of gate q of unit 8 cta + u,
// padded with zeros to HP columns.
__global__ void pack_runs_fwd(const float* W, int K, int I, int H, int HP, bf16* out) {
  grid_dep_wait();
  grid_dep_launch();
  const size_t n = (size_t)4 * H * HP;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % HP), r = (int)(e / HP), u = r >> 2, q = r & 3;
    bf16 hi, mid;
    split2(c < H ? W[((size_t)q * H + u) * K + I + c] : 0.f, hi, mid);
    bf16* o = out + ((size_t)(u / RU) * 64 + 4 * (u % RU) + q) * HP + c;
    o[0] = hi;
    o[(size_t)32 * HP] = mid;
  }
}
// W_hh^T as the backward kernel holds it: row (4 cl + q) 64 + 32 p + c is half p of column 32 cl + c of
// gate q's block.  A block of 32 x 8 threads transposes 32 x 32 elements (x: columns / 32, y: units / 32, z: q).
__global__ void pack_runs_bwd(const float* W, int K, int I, int H, int HP, bf16* out) {
  __shared__ float t[32][33];
  grid_dep_wait();
  grid_dep_launch();
  const int cl = blockIdx.x, jb = blockIdx.y * 32, q = blockIdx.z;
  for (int y = threadIdx.y; y < 32; y += 8) {
    const int c = cl * 32 + threadIdx.x, j = jb + y;
    t[y][threadIdx.x] = c < H && j < H ? W[((size_t)q * H + j) * K + I + c] : 0.f;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8) {
    bf16 hi, mid;
    split2(t[threadIdx.x][y], hi, mid);
    bf16* o = out + ((size_t)(cl * CS + q) * 64 + y) * HP + jb + threadIdx.x;
    o[0] = hi;
    o[(size_t)32 * HP] = mid;
  }
}

// The cells of a batch of leaves from the products of their h_{k-1}: z1 = h_hi W_f, z2 = h_mid W_f over the rows
// of w_f, summed as the forward kernel sums them.
struct LeafPtrs { const float* c_prev[X3_LEAVES]; };
__global__ void leaf_cells(const LeafPtrs src, const float* zx, const float* z1, const float* z2, float* out, size_t plane, int B, int H,
                           int64_t* counters) {
  grid_dep_wait();
  grid_dep_launch();
  const int leaf = blockIdx.y;
  const float* cpv = src.c_prev[leaf];
  float* o = out + (size_t)leaf * 6 * plane;
  const size_t n = (size_t)B * H;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / H), j = (int)(e % H);
    const size_t row = (size_t)leaf * B + b;
    const size_t at = row * 8 * H + (size_t)(j / RU) * 64 + 4 * (j % RU);
    const float4 hh = *reinterpret_cast<const float4*>(z1 + at), mh = *reinterpret_cast<const float4*>(z1 + at + 32);
    const float4 hm = *reinterpret_cast<const float4*>(z2 + at);
    const float* zr = zx + row * 4 * H + j;
    const float gi = sigmoidf_(zr[0] + ((hh.x + hm.x) + mh.x));
    const float gf = sigmoidf_(zr[H] + ((hh.y + hm.y) + mh.y));
    const float gg = tanhf(zr[2 * (size_t)H] + ((hh.z + hm.z) + mh.z));
    const float go = sigmoidf_(zr[3 * (size_t)H] + ((hh.w + hm.w) + mh.w));
    const float c = fmaf(gf, cpv[e], gi * gg);
    o[e] = gi; o[plane + e] = gf; o[2 * plane + e] = gg; o[3 * plane + e] = go;
    o[4 * plane + e] = c;
    o[5 * plane + e] = go * tanhf(c);
  }
  if (blockIdx.x == 0 && leaf == 0 && threadIdx.x == 0) counters[0] += gridDim.y;
}

inline int round64(int v) { return (v + 63) / 64 * 64; }

}  // namespace

bool runs_begin(RunsX3& r, int I, int H, int B, const float* W, cudaStream_t s) {
  const int HP = round64(H), K = I + H, ncl = (H + CS * RU - 1) / (CS * RU);
  r.I = I; r.H = H; r.B = B; r.HP = HP; r.groups = B / RB;
  launch_pdl(pack_runs_fwd, dim3(1184), dim3(256), 0, s, W, K, I, H, HP, r.w_f);
  launch_pdl(pack_runs_bwd, dim3(ncl, HP / 32, 4), dim3(32, 8), 0, s, W, K, I, H, HP, r.w_b);
  // (the columns that pad a row to HP are read, and multiplied by zeros)
  cudaMemsetAsync(r.exch_f, 0, (size_t)2 * r.groups * 64 * HP * 2, s);
  cudaMemsetAsync(r.exch_b, 0, (size_t)2 * r.groups * CS * 64 * HP * 2, s);
  cudaMemsetAsync(r.sync, 0, r.n_sync * 4, s);
  r.launches = 0;
  const int KB = HP / 64;
  cudaFuncSetAttribute(fwd_run_x3, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd_smem(KB));
  cudaFuncSetAttribute(bwd_run_x3, cudaFuncAttributeMaxDynamicSharedMemorySize, bwd_smem(KB));
  return make_tmap_blocks64(&r.tm_h, r.exch_f, HP, (uint64_t)2 * r.groups * 64, (uint64_t)HP * 2, 64, SLAB) &&
         make_tmap_blocks64(&r.tm_w, r.w_f, HP, (uint64_t)H / RU * 64, (uint64_t)HP * 2, 64, 4) &&
         make_tmap_blocks64(&r.tm_dz, r.exch_b, HP, (uint64_t)2 * r.groups * CS * 64, (uint64_t)HP * 2, 64, SLAB) &&
         make_tmap_blocks64(&r.tm_wt, r.w_b, HP, (uint64_t)ncl * CS * 64, (uint64_t)HP * 2, 64, 4);
}

int runs_smem(bool backward, int H) { return backward ? bwd_smem(round64(H) / 64) : fwd_smem(round64(H) / 64); }

int forward_run(RunsX3& r, const stepwise::FwdRunStep* st, int n, const float* zx, size_t plane_elems, int64_t* counters,
                int* status, cudaStream_t s) {
  FwdX3Args a{};
  for (int i = 0; i < n; ++i) a.op[i] = st[i];
  const int fault = tc::wait_fault_mask();
  a.zx = zx; a.exch = r.exch_f; a.sync = r.sync + (size_t)r.launches++ * 2 * SYNC_STRIDE;
  a.status = status; a.counters = counters; a.plane = plane_elems;
  a.n = n; a.B = r.B; a.H = r.H; a.HP = r.HP; a.ncg = r.H / RU; a.groups = r.groups;
  a.expect = (uint32_t)a.ncg + ((fault & 1) ? 1u : 0u);
  a.poll_limit = (fault & 1) ? tc::fault_poll_limit : (kSpinLimit >> 1);
  void* args[] = {(void*)&r.tm_h, (void*)&r.tm_w, (void*)&a};
  return launch_coop((const void*)fwd_run_x3, r.groups * a.ncg, 192, fwd_smem(r.HP / 64), s, args, 1) == cudaSuccess
             ? MEBPTT_OK : MEBPTT_ERR_CUDA;
}

int backward_run(RunsX3& r, const stepwise::BwdRunStep* st, int n, const float* dha, float* dh, float* dc, __nv_bfloat16* st_dz3,
                 __nv_bfloat16* st_hp2, __nv_bfloat16* st_in2, size_t plane_elems, const float* loss_part, int loss_parts, float* loss_t,
                 int64_t* counters, int* status, cudaStream_t s) {
  BwdX3Args a{};
  a.loss_part = loss_part; a.loss_parts = loss_parts; a.loss_t = loss_t;
  for (int i = 0; i < n; ++i) a.op[i] = st[i];
  const int fault = tc::wait_fault_mask();
  a.dha = dha; a.dh = dh; a.dc = dc; a.exch = r.exch_b; a.st_dz3 = st_dz3; a.st_hp2 = st_hp2; a.st_in2 = st_in2;
  a.sync = r.sync + (size_t)r.launches++ * 2 * SYNC_STRIDE;
  a.status = status; a.counters = counters; a.plane = plane_elems;
  a.n = n; a.B = r.B; a.H = r.H; a.HP = r.HP; a.I = r.I; a.groups = r.groups;
  a.ncg = (r.H + CS * RU - 1) / (CS * RU) * CS;
  a.expect = (uint32_t)a.ncg + ((fault & 2) ? 1u : 0u);
  a.poll_limit = (fault & 2) ? tc::fault_poll_limit : (kSpinLimit >> 1);
  void* args[] = {(void*)&r.tm_dz, (void*)&r.tm_wt, (void*)&a};
  return launch_coop((const void*)bwd_run_x3, r.groups * a.ncg, 192, bwd_smem(r.HP / 64), s, args, CS, false) == cudaSuccess
             ? MEBPTT_OK : MEBPTT_ERR_CUDA;
}

// A leaf on its own is a launch of a persistent kernel each way, a readout and a projection (H = 1000, B = 32:
// some 80 us); batched, the forward operations are two products and a cell kernel, and the readout and the
// backward operations of up to X3_LEAVES leaves are one run (150 steps at full memory: 12.2 -> 4.4 ms).
int forward_leaves(RunsX3& r, const __nv_bfloat16* hp2, const float* const* c_prev, int n, const float* zx, float* z, float* out,
                   size_t plane_elems, int64_t* counters, int* status, cudaStream_t s) {
  const int M = n * r.B, N = 8 * r.H;
  float* z2 = z + (size_t)M * N;
  for (int half = 0; half < 2; ++half) {
    const int rc = gemm_bf16(hp2 + (size_t)half * r.H, 2 * r.H, false, r.w_f, r.HP, false,
                             GemmOut{GemmOut::STORE_F32, half ? z2 : z, N, nullptr, 0}, M, N, r.H, status, s);
    if (rc != MEBPTT_OK) return rc;
  }
  LeafPtrs ptrs{};
  for (int a = 0; a < n; ++a) ptrs.c_prev[a] = c_prev[a];
  const size_t blocks = ((size_t)r.B * r.H + 255) / 256;
  launch_pdl(leaf_cells, dim3((unsigned)(blocks > 128 ? 128 : blocks), (unsigned)n), dim3(256), 0, s, ptrs, zx, (const float*)z,
             (const float*)z2, out, plane_elems, r.B, r.H, counters);
  return MEBPTT_OK;
}

}  // namespace stepwise3
}  // namespace mebptt
