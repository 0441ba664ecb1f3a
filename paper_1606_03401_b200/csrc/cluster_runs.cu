// Runs of the bfloat16 recurrence for at most 512 hidden units: a thread-block cluster holds all of W_hh and
// walks a run for 8 or 12 batch rows; what a step produces travels between shared memories, never through the L2.
//
// What bounds a step is the trip of the new state to everyone who needs it.  Through global memory (the
// kernels of tc_lstm.cu, which wider layers need) that trip is a store, a release that waits for it, a counter, a
// poll and a fetch: 2.8 us an operation at H = 256 and 3.2 at H = 512, of which the products are a fifth.
// Here the batch rows of an LSTM, which never mix, are cut into groups of 8 or 12 (cluster_rows), and each group is one
// cluster of ceil(H / 32) CTAs, a CTA with 32 hidden units: its 128 gate rows are a full MMA tile, the N is 16, the least
// that an M of 128 allows.
//
//   forward    z[128 gate rows][16] = W_hh[rows of this CTA][H] h_{k-1}, the weights in tensor memory, h_{k-1} in shared
//              memory; the gates; h_k goes to every CTA of the cluster, straight into the operand its next MMA reads (without
//              swizzle: below), by asynchronous stores that count their bytes on the receiver's barrier.
//   backward   dz of the CTA's 32 units (128 gate columns) never leaves the CTA for the recurrence: it is multiplied
//              by all H columns of W_hh it meets (K = 128), and the partial sums of dh go to the CTAs that own the
//              columns, which add them in the order of the ranks.  (Gathering dz instead would send four times h.)
//
// Two buffers of what is received: a CTA that pushes for step i + 2 has received every peer's push for step i + 1,
// made after that peer had consumed step i.  Clusters wait for no one outside, so the launch is not cooperative.
// All waits are bounded; a CTA that gives up stops pushing, and all meet at the barrier of the cluster at the end.  (The
// barrier that dz crosses, bar.sync 1, has no limit of its own: it ends because every warp comes to it once a step, at
// most one step apart, whatever has run out.)
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "cluster_runs.hpp"
#include "env.hpp"
#include "launch.hpp"
#include "lstm_dev.cuh"
#include "mebptt.h"
#include "runs_dev.cuh"
#include "sm100.cuh"
#include "tmap.hpp"

namespace mebptt {
namespace tc {

namespace {

using namespace sm100;

constexpr uint32_t H_TILE = CB * 128;    // [16 batch rows][64 contraction indices]
constexpr int ZROW = 40;                 // floats a batch row of a warp's accumulators takes: 32 gate rows; lanes that read
                                         // four rows and two units side by side then meet no bank twice
constexpr int THREADS = 160;             // of the forward kernel: warps 0-3: gates; warp 4: copies and MMAs

__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// The CTA's weights from the tiles they were copied to into tensor memory, from column 0 on, 32 columns a tile: warp w
// moves the rows 32 w .. 32 w + 31, a lane a row.  (The MMA reads a stationary operand there at 11 cycles a K = 16
// slice; out of shared memory, where 4 KB a slice pass at 128 bytes a cycle, it takes 38.)
__device__ __forceinline__ void weights_to_tmem(const uint8_t* tiles, int n, uint64_t* ready, uint32_t tmem, int warp, int lane, volatile int* failed) {
  const uint8_t* row = tiles + (32 * warp + lane) * 128;
  for (int k = 0; k < n; ++k) {
    (void)wait_or_fail(&ready[k], 0, failed);
    __syncwarp();
    uint4 q[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) q[c] = *reinterpret_cast<const uint4*>(row + k * W_TILE + ((c ^ (lane & 7)) * 16));
    tmem_st_32x32(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(32 * k), q);
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  tc_fence_before_sync();
}
// Bounded wait for MMAs that are committed in every step, whatever has run out: not over early.  What may pass before they
// are issued is two waits of the others (a step's inputs, then what peers push), each at most kSpinLimit polls.
__device__ __forceinline__ bool wait_committed(uint64_t* bar, uint32_t parity, volatile int* failed) {
  for (int turn = 0; turn < 4; ++turn)
    for (uint32_t i = 0; i < kSpinLimit; ++i) {
      if (mbar_try_wait(bar, parity)) return true;
      if (i > 256 || turn) __nanosleep(64);
    }
  *failed = 1;
  return false;
}
__host__ __device__ inline uint32_t tmem_cols(int used) { return used <= 64 ? 64u : used <= 128 ? 128u : used <= 256 ? 256u : 512u; }
// ------------------------------------------------------------------------------------------
// forward run
// ------------------------------------------------------------------------------------------
// h_{k-1} lies without swizzle, in pieces [8 hidden units][16 rows][16 bytes]: what a warp makes of a step, its own
// 8 units, is then 256 consecutive bytes of every receiver.  (A remote store of 16 bytes costs its receiver some
// 2 cycles where those of a warp are side by side and 5 where they are 128 bytes apart, as in a swizzled tile: an
// exchange of 16 CTAs 1505 and 2337 cycles.)
constexpr uint32_t PIECE = CB * 16;

struct FwdStage {                 // per warp
  float z[CB][ZROW];              // accumulators [batch row][gate row of the warp's 8 units]
  __nv_bfloat16 v[5][CB][8];      // h, i, f, g, o [batch row][unit]
};

template <int RB>
__global__ void __launch_bounds__(THREADS, 1) fwd_run_cluster(const __grid_constant__ CUtensorMap tm_w, const ClusterFwdArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t wfull[8], first, full[2], acc;
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  __shared__ __align__(16) FwdStage stage[4];

  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int KT = (a.H + 63) / 64;
  uint8_t* sW = sm;                           // KT tiles: this CTA's gate rows of W_hh
  uint8_t* sH = sm + KT * W_TILE;             // [2][8 KT] pieces: the group's rows of h_{k-1}
  const uint32_t h_buf = (uint32_t)KT * 8 * PIECE;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank(), cs = cluster_size();
  const int grp = blockIdx.x / (int)cs;

  if (tid == 0) {
    for (int k = 0; k < 8; ++k) mbar_init(&wfull[k], 1);
    mbar_init(&first, 4);
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&acc, 1);
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_w);
  }
  // pieces past the CTAs' units and rows past RB are never pushed
  for (uint32_t e = tid; e < 2 * h_buf / 16; e += THREADS) reinterpret_cast<uint4*>(sH)[e] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_shared();
  const uint32_t acc_col = 32 * (uint32_t)KT;   // the accumulators, behind the weights
  if (warp == 4) tmem_alloc(&tmem_slot, tmem_cols(32 * KT + CB));
  tc_fence_before_sync();
  cluster_sync();                             // peers push onto each other's barriers: all must be initialised
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();

  if (warp == 4) {
    constexpr uint32_t idesc = make_idesc(1, 128, CB, false, false);
    const uint32_t bytes = (uint32_t)(RB * fwd_waited_units(a.H) * 2) + a.extra;
    if (lane == 0) {
      for (int kb = 0; kb < KT; ++kb) {
        mbar_arrive_expect_tx(&wfull[kb], W_TILE);
        tma_load_2d(sW + kb * W_TILE, &tm_w, kb * 64, (int)rank * 4 * CU, &wfull[kb]);
      }
      if (a.n > 1) mbar_arrive_expect_tx(&full[1], bytes);
      if (a.n > 2) mbar_arrive_expect_tx(&full[0], bytes);
    }
    __syncwarp();
    bool ok = true;
    for (int i = 0; i < a.n; ++i) {
      const int b = i & 1;
      if (ok)
        ok = __all_sync(0xffffffffu, i == 0 ? wait_or_fail(&first, 0, &failed)
                                            : wait_pushed(&full[b], (uint32_t)((i - 1) >> 1) & 1, &failed, a.poll_limit));
      if (ok) {
        fence_proxy_async_shared();           // what the peers stored, before the MMAs read it
        tc_fence_after_sync();
        const uint64_t h_desc = make_desc_plain(smem_u32(sH + b * h_buf), PIECE, 128);
        if (elect_one()) {
          for (int kb = 0; kb < KT; ++kb)
            mma_tmem_x4<2 * PIECE / 16>(tmem + acc_col, tmem + 32 * kb, h_desc + (uint64_t)(kb * (8 * PIECE >> 4)), idesc, kb ? 1u : 0u);
        }
        __syncwarp();
      }
      if (elect_one()) {
        mma_commit(&acc);                     // always: the gates count on one arrival per step
        // (only a phase that is over: a barrier takes one arrival a phase)
        if (ok && i >= 1 && i + 2 < a.n) mbar_arrive_expect_tx(&full[b], bytes);
      }
      __syncwarp();
      if (i == a.n - 1 && lane == 0) grid_dep_launch();
    }
    if (failed && lane == 0)
      for (int kb = 0; kb < KT; ++kb) (void)mbar_wait(&wfull[kb], 0);   // loads that were requested may still be landing
  } else if (warp < 4) {
    // Lane l of warp w holds gate row 32 w + l of the accumulators (gate l % 4 of unit 8 w + l / 4); through the
    // warp's own stage it gets the four gates of that unit for the rows l % 4 + 4 v.  States leave in pieces of 16
    // bytes: eight units, the warp's own, of one row.
    const int u = lane >> 2, r0 = lane & 3;
    const int j = (int)rank * CU + 8 * warp + u;             // hidden unit
    const int jw = (int)rank * CU + 8 * warp;                // the warp's first
    const bool wvalid = jw < a.H;                            // H is a multiple of 8
    const int brow = grp * RB;
    constexpr int ROWS = RB == 8 ? 8 : 16, PEERS = 32 / ROWS;   // a warp pushes to so many peers at a time
    const int prow = lane & (ROWS - 1);                      // the row whose pieces this lane stores and pushes
    const bool pvalid = wvalid && prow < RB && brow + prow < a.B;
    const size_t ep = (size_t)(brow + prow) * a.H + jw;
    FwdStage& st = stage[warp];
    const DevOp op0 = a.ops[0];
    {
      // the state the run starts from, rows past the batch as zeros
      const __nv_bfloat16* h0 = reinterpret_cast<const __nv_bfloat16*>(a.ws + (size_t)op0.h_src * 16);
      for (int p = tid / ROWS; p < a.H / 8; p += 128 / ROWS) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (prow < RB && brow + prow < a.B) v = *reinterpret_cast<const uint4*>(h0 + (size_t)(brow + prow) * a.H + 8 * p);
        *reinterpret_cast<uint4*>(sH + p * PIECE + prow * 16) = v;
      }
      fence_proxy_async_shared();
    }
    constexpr int NV = RB / 4;                               // rows of a thread
    bool rvalid[NV];
    size_t er[NV];
    float c[NV];
    float4 zx[NV];
    uint4 hprev = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int b = brow + r0 + 4 * v;
      rvalid[v] = wvalid && b < a.B;
      er[v] = (size_t)b * a.H + j;
      c[v] = 0.f;
      zx[v] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (rvalid[v]) {
        c[v] = reinterpret_cast<const float*>(a.ws + (size_t)op0.c_src * 16)[er[v]];
        zx[v] = *reinterpret_cast<const float4*>(a.zx + 4 * er[v]);
      }
    }
    if (pvalid) hprev = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(a.ws + (size_t)op0.h_src * 16) + ep);
    weights_to_tmem(sW, KT, wfull, tmem, warp, lane, &failed);
    __syncwarp();
    if (lane == 0) mbar_arrive(&first);
    const uint32_t piece = smem_u32(sH) + (uint32_t)(jw >> 3) * PIECE + (uint32_t)prow * 16;
    const uint32_t bar0 = smem_u32(&full[0]), bar1 = smem_u32(&full[1]);

    for (int i = 0; i < a.n; ++i) {
      const DevOp op = a.ops[i];
      const bool got = wait_or_fail(&acc, (uint32_t)i & 1, &failed) && !*(volatile int*)&failed;
      tc_fence_after_sync();
      uint32_t r[ROWS];
      if constexpr (RB == 8) tmem_ld_32x8(tmem + ((uint32_t)(32 * warp) << 16) + acc_col, r);
      else tmem_ld_32x16(tmem + ((uint32_t)(32 * warp) << 16) + acc_col, r);
      tmem_ld_wait();
      tc_fence_before_sync();
#pragma unroll
      for (int n = 0; n < RB; ++n) st.z[n][lane] = __uint_as_float(r[n]);
      __syncwarp();
      float cin[NV], gate[NV][4];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float4 p = *reinterpret_cast<const float4*>(&st.z[r0 + 4 * v][4 * u]);
        const float iv = sigmoid_fast(zx[v].x + p.x), fv = sigmoid_fast(zx[v].y + p.y);
        const float gv = tanh_fast(zx[v].z + p.z), ov = sigmoid_fast(zx[v].w + p.w);
        cin[v] = c[v];
        c[v] = fmaf(fv, c[v], iv * gv);
        const float hv = ov * tanh_fast(c[v]);
        st.v[0][r0 + 4 * v][u] = __float2bfloat16_rn(hv);
        gate[v][0] = iv; gate[v][1] = fv; gate[v][2] = gv; gate[v][3] = ov;
      }
      __syncwarp();
      // (Past the last unit these are zeros: its weights and Zx are.  A row with a NaN has one there as well, beside NaNs in
      // all of its units.)
      const uint4 hnew = *reinterpret_cast<const uint4*>(&st.v[0][prow][0]);
      if (got && prow < RB && i + 1 < a.n) {
        // h_k to every CTA, the next in rank first
        const uint32_t dst = piece + (((uint32_t)i + 1) & 1) * h_buf, bar = (i & 1) ? bar0 : bar1;
        for (uint32_t p = lane / ROWS; p < cs; p += PEERS) {
          uint32_t peer = rank + 1 + p;
          peer = peer >= cs ? peer - cs : peer;
          push16(map_rank(dst, peer), hnew, map_rank(bar, peer));
        }
      }
      // the rest of the state, off the critical path
      if (got) {
        if (pvalid && lane < RB) {
          *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.h_dst * 16) + ep) = hnew;
          if (op.stage) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.stage * 16) + ep) = hnew;
        }
        if (op.gates) {
#pragma unroll
          for (int v = 0; v < NV; ++v)
#pragma unroll
            for (int q = 0; q < 4; ++q) st.v[1 + q][r0 + 4 * v][u] = __float2bfloat16_rn(gate[v][q]);
          __syncwarp();
          __nv_bfloat16* gp = reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.gates * 16) + ep;
          const size_t pl = (size_t)a.plane16 * 8;   // elements
#pragma unroll
          for (int h = 0; h < ROWS / 8; ++h) {
            const int q = PEERS * h + lane / ROWS;
            if (pvalid) *reinterpret_cast<uint4*>(gp + q * pl) = *reinterpret_cast<const uint4*>(&st.v[1 + q][prow][0]);
          }
        }
        if (op.in_copy && pvalid && lane < RB)
          *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.in_copy * 16) + ep) = hprev;
        hprev = hnew;
        float* cd = reinterpret_cast<float*>(a.ws + (size_t)op.c_dst * 16);
        float* ci = op.in_copy ? reinterpret_cast<float*>(a.ws + ((size_t)op.in_copy + a.hsz16) * 16) : nullptr;
#pragma unroll
        for (int v = 0; v < NV; ++v)
          if (rvalid[v]) {
            cd[er[v]] = c[v];
            if (ci) ci[er[v]] = cin[v];
            if (i + 1 < a.n) zx[v] = *reinterpret_cast<const float4*>(a.zx + 4 * ((size_t)(i + 1) * a.B * a.H + er[v]));
          }
      }
      __syncwarp();   // the stage is free again
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  settle(failed != 0);
  cluster_sync();     // no CTA leaves while a peer may still push to it
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (blockIdx.x == 0) a.counters[0] += a.n;
  }
  if (warp == 4) tmem_dealloc(tmem, tmem_cols(32 * KT + CB));
}

// ------------------------------------------------------------------------------------------
// backward run
// ------------------------------------------------------------------------------------------
constexpr int BWD_THREADS = 224;   // warps 0-3: gates; 4: MMAs; 5: what is read and dz, in and out; 6: loss terms

// Shared memory behind the alignment: weights, dz, partial sums received, two stages of inputs.
template <int RB>
struct BwdSmem {
  static __host__ __device__ uint32_t weights(int H) { return (uint32_t)((H + 127) / 128 * 2) * W_TILE; }
  static __host__ __device__ uint32_t dz(int H) { return weights(H); }                     // [2][2] tiles [16 batch rows][64 gate columns]
  static __host__ __device__ uint32_t recv(int H) { return dz(H) + 4 * H_TILE; }           // [2][CTAs] partial sums
  static __host__ __device__ uint32_t stages(int H) { return recv(H) + 2 * (uint32_t)((H + CU - 1) / CU) * recv_slot(RB); }
  static __host__ __device__ uint32_t total(int H) { return 1024 + stages(H) + 2 * (uint32_t)sizeof(GateStage<RB>); }
};

template <int RB>
__global__ void __launch_bounds__(BWD_THREADS, 1) bwd_run_cluster(const __grid_constant__ CUtensorMap tm_wt, const ClusterBwdArgs a) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t wfull[8], full[2], inready[2], acc;
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;
  typedef BwdSmem<RB> Smem;
  constexpr uint32_t SLOT = recv_slot(RB);

  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int MT = (a.H + 127) / 128;                // tiles of 128 columns of dh
  uint8_t* const sW = sm;                          // [MT][2] tiles: W_hh^T, rows of dh by this CTA's gate columns
  uint8_t* const sZ = sm + Smem::dz(a.H);
  uint8_t* const sR = sm + Smem::recv(a.H);
  GateStage<RB>* const sI = reinterpret_cast<GateStage<RB>*>(sm + Smem::stages(a.H));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank(), cs = cluster_size();
  const int grp = blockIdx.x / (int)cs;

  if (tid == 0) {
    for (int k = 0; k < 8; ++k) mbar_init(&wfull[k], 1);
    for (int b = 0; b < 2; ++b) { mbar_init(&full[b], 1); mbar_init(&inready[b], 32); }
    mbar_init(&acc, 1);
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_wt);
  }
  for (uint32_t e = tid; e < 4 * H_TILE / 16; e += BWD_THREADS) reinterpret_cast<uint4*>(sZ)[e] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_shared();
  const uint32_t acc_col = 64 * (uint32_t)MT;      // the accumulators, behind the weights
  if (warp == 4) tmem_alloc(&tmem_slot, tmem_cols((64 + CB) * MT));
  tc_fence_before_sync();
  cluster_sync();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();

  const int brow = grp * RB, rows = a.B - brow;                          // the cluster's batch rows (RB of them, or fewer)
  const int unit0 = (int)rank * CU, units = a.H - unit0;                 // the CTA's hidden units (likewise)
  const int s_hi = (a.ops[0].k - 1) % a.S;                               // row block of the run's first step; those after it descend

  if (warp == 4) {
    constexpr uint32_t idesc = make_idesc(1, 128, CB, false, false);
    const uint32_t bytes = cs * SLOT + a.extra;
    if (lane == 0) {
      for (int t = 0; t < 2 * MT; ++t) {
        mbar_arrive_expect_tx(&wfull[t], W_TILE);
        tma_load_2d(sW + t * W_TILE, &tm_wt, unit0 * 4 + 64 * (t & 1), 128 * (t >> 1), &wfull[t]);
      }
      mbar_arrive_expect_tx(&full[0], bytes);
      if (a.n > 1) mbar_arrive_expect_tx(&full[1], bytes);
    }
    __syncwarp();
    const uint64_t z_desc = make_desc_sw128(smem_u32(sZ), 16, 1024);
    for (int i = 0; i < a.n; ++i) {
      named_barrier(1, 192);                  // dz is there (at first the weights as well): every warp of the gates arrives
      tc_fence_after_sync();                  // once a step, whatever happens
      if (elect_one()) {
        const uint64_t zd = z_desc + (uint64_t)((i & 1) * (2 * H_TILE >> 4));
        for (int m = 0; m < MT; ++m)
          for (int kb = 0; kb < 2; ++kb)
            mma_tmem_x4<2>(tmem + acc_col + m * CB, tmem + 32 * (2 * m + kb), zd + (uint64_t)(kb * (H_TILE >> 4)), idesc, kb ? 1u : 0u);
        mma_commit(&acc);
        // the buffer of step i - 1 has been read by now, unless a wait ran out: every warp has said so with its dz
        if (i >= 1 && i + 1 < a.n && !*(volatile int*)&failed) mbar_arrive_expect_tx(&full[(i + 1) & 1], bytes);
      }
      __syncwarp();
      if (i == a.n - 1 && lane == 0) grid_dep_launch();
    }
    if (failed && lane == 0)
      for (int t = 0; t < 2 * MT; ++t) (void)mbar_wait(&wfull[t], 0);   // loads that were requested may still be landing
  } else if (warp == 5) {
    const size_t e0 = (size_t)brow * a.H + unit0, bh = (size_t)a.B * a.H;
    __nv_bfloat16* const dz = reinterpret_cast<__nv_bfloat16*>(a.dz);
    auto fill = [&](const DevOp& op, int i) {
      ask_for<RB>(a, op, (size_t)(s_hi - i) * bh, e0, rows < RB ? rows : RB, units < CU ? units : CU, lane, sI[i & 1]);
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&inready[i & 1])) : "memory");
    };
    DevOp next = a.ops[0];
    for (int i = 0; i < 2 && i < a.n; ++i) {
      const DevOp op = next;
      if (i + 1 < a.n) next = a.ops[i + 1];
      fill(op, i);
    }
    if (a.n > 2) next = a.ops[2];
    for (int i = 0; i < a.n; ++i) {
      named_barrier(1, 192);                  // dz of step i is there, its inputs have been used
      // dz to its stage: a row is 64 gate columns a tile, 16-byte piece p at p ^ (row % 8)
      const uint8_t* zs = sZ + (i & 1) * 2 * H_TILE;
      __nv_bfloat16* out = dz + 4 * ((size_t)(s_hi - i) * bh + e0);
#pragma unroll
      for (int y = 0; y < RB / 2; ++y) {
        const int r = 2 * y + (lane >> 4), p = lane & 15;                // 16 pieces a row
        if (r < rows && 2 * p < units)
          *reinterpret_cast<uint4*>(out + (size_t)r * 4 * a.H + 8 * p) =
              *reinterpret_cast<const uint4*>(zs + (p >> 3) * H_TILE + r * 128 + (((p & 7) ^ (r & 7)) * 16));
      }
      if (i + 2 < a.n) {
        const DevOp op = next;
        if (i + 3 < a.n) next = a.ops[i + 3];
        fill(op, i + 2);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == 6) {
    // loss terms of the run: the partial sums of a step in a fixed order
    if (blockIdx.x == 0)
      for (int i = lane; i < a.n; i += 32) {
        float sum = 0.f;
        for (int p = 0; p < a.loss_parts; ++p) sum += a.loss_part[(s_hi - i) * a.loss_parts + p];
        a.loss_t[a.ops[0].k - 1 - i] = sum;
      }
  } else {
    // lane l of warp w owns hidden unit 8 w + l % 8 of the CTA for NV batch rows from NV (l / 8) on
    constexpr int NV = RB == 8 ? 2 : 4;
    const int u = 8 * warp + (lane & 7), r0 = NV * (lane >> 3);
    const int rp = r0 < RB ? r0 : 0;               // (lanes with rows past RB pick their neighbours')
    const bool leaf = a.zleaf != nullptr;
    const size_t e = (size_t)(brow + r0) * a.H + unit0 + u;
    bool valid[NV];
    float dh[NV], dc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      valid[v] = u < units && r0 + v < RB && r0 + v < rows;
      dh[v] = valid[v] ? a.dh[e + (size_t)v * a.H] : 0.f;
      dc[v] = valid[v] ? a.dc[e + (size_t)v * a.H] : 0.f;
    }
    // dz of (row r, unit u): four gate columns, 8 bytes of a swizzled row
    uint8_t* const zt = sZ + (u >> 4) * H_TILE + ((uint32_t)u & 1) * 8;
    uint32_t zoff[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) zoff[v] = (uint32_t)(r0 + v) * 128 + (((((uint32_t)u & 15) >> 1) ^ ((uint32_t)(r0 + v) & 7)) * 16);
    // partial sums: lane l of warp w holds column 128 m + 32 w + l of dh, which CTA 4 m + w owns
    uint32_t to[4], tb[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const uint32_t peer = (uint32_t)(4 * m + warp) < cs ? (uint32_t)(4 * m + warp) : 0u;
      to[m] = map_rank(smem_u32(sR) + rank * SLOT + (uint32_t)lane * 16, peer);
      tb[m] = map_rank(smem_u32(&full[0]), peer);
    }
    const float* const mine = reinterpret_cast<const float*>(sR) + (rp >> 2) * 4 * CU + 4 * u + (rp & 3);   // of sender 0, buffer 0

    // dh of this thread from the partial sums of product `it`, added in the order of the ranks
    auto receive = [&](int it) {
      const bool got = wait_pushed(&full[it & 1], (uint32_t)(it >> 1) & 1, &failed, a.poll_limit);
      if (!got) return;
      const float* src = mine + (it & 1) * (cs * (SLOT / 4));
      float s[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] = 0.f;
#pragma unroll 4
      for (uint32_t p = 0; p < cs; ++p, src += SLOT / 4) {
        if constexpr (NV == 4) {
          const float4 x = *reinterpret_cast<const float4*>(src);
          s[0] += x.x; s[1] += x.y; s[2] += x.z; s[3] += x.w;
        } else {
          const float2 x = *reinterpret_cast<const float2*>(src);
          s[0] += x.x; s[1] += x.y;
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v) dh[v] = s[v];
    };

    weights_to_tmem(sW, 2 * MT, wfull, tmem, warp, lane, &failed);
    GateIn<NV> in;
    (void)wait_or_fail(&inready[0], 0, &failed);
    pick_out<NV, RB>(leaf, sI[0], u, rp, in);
    for (int i = 0; i < a.n; ++i) {
      if (i > 0) receive(i - 1);
      uint8_t* const zb = zt + (i & 1) * 2 * H_TILE;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const float gi = in.g[0][v], gf = in.g[1][v], gg = in.g[2][v], go = in.g[3][v];
        const float dht = in.d[v] + dh[v];
        const float th = in.ct[v];
        const float d_o = dht * th;
        const float dct = fmaf(dht * go, 1.f - th * th, dc[v]);
        const float zi = dct * gg * gi * (1.f - gi);
        const float zf = dct * in.cp[v] * gf * (1.f - gf);
        const float zg = dct * gi * (1.f - gg * gg);
        const float zo = d_o * go * (1.f - go);
        dc[v] = dct * gf;
        if (valid[v]) *reinterpret_cast<uint2*>(zb + zoff[v]) = make_uint2(pack_bf16x2(zi, zf), pack_bf16x2(zg, zo));
      }
      fence_proxy_async_shared();
      tc_fence_before_sync();
      asm volatile("bar.arrive 1, 192;" ::: "memory");
      // beside the products: the inputs of the next (earlier) step
      if (i + 1 < a.n) {
        (void)wait_or_fail(&inready[(i + 1) & 1], (uint32_t)((i + 1) >> 1) & 1, &failed);
        pick_out<NV, RB>(leaf, sI[(i + 1) & 1], u, rp, in);
      }
      // (not over because another wait ran out: barrier 1 has no limit and counts warps, not which, so no warp may come
      // to it for a step before all have for the one before)
      const bool got = wait_committed(&acc, (uint32_t)i & 1, &failed) && !*(volatile int*)&failed;
      tc_fence_after_sync();
      constexpr int COLS = RB == 8 ? 8 : 16;
      uint32_t r[4][COLS];
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (m < MT) {
          if constexpr (RB == 8) tmem_ld_32x8(tmem + ((uint32_t)(32 * warp) << 16) + acc_col + (uint32_t)(m * CB), r[m]);
          else tmem_ld_32x16(tmem + ((uint32_t)(32 * warp) << 16) + acc_col + (uint32_t)(m * CB), r[m]);
        }
      tmem_ld_wait();
      tc_fence_before_sync();
      const uint32_t obuf = (uint32_t)(i & 1) * cs * SLOT, bbuf = (uint32_t)(i & 1) * 8;
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (got && (uint32_t)(4 * m + warp) < cs)
#pragma unroll
          for (int v = 0; v < RB / 4; ++v)
            push16(to[m] + obuf + v * (CU * 16), make_uint4(r[m][4 * v], r[m][4 * v + 1], r[m][4 * v + 2], r[m][4 * v + 3]), tb[m] + bbuf);
    }
    receive(a.n - 1);
    if (!*(volatile int*)&failed) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (valid[v]) {
          a.dh[e + (size_t)v * a.H] = dh[v];
          a.dc[e + (size_t)v * a.H] = dc[v];
        }
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  settle(failed != 0);
  cluster_sync();
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (blockIdx.x == 0) a.counters[1] += a.n;
  }
  if (warp == 4) tmem_dealloc(tmem, tmem_cols((64 + CB) * MT));
}

int cluster_ctas(int H) { return (H + CU - 1) / CU; }
int fwd_smem(int H) { return lone_smem((H + 63) / 64 * (int)(W_TILE + 2 * 8 * PIECE) + 1024); }
int bwd_smem(int H, int RB) { return lone_smem((int)(RB == 8 ? BwdSmem<8>::total(H) : BwdSmem<12>::total(H))); }
const void* kernel(int dir, int RB) {
  if (dir) return RB == 8 ? (const void*)bwd_run_cluster<8> : (const void*)bwd_run_cluster<12>;
  return RB == 8 ? (const void*)fwd_run_cluster<8> : (const void*)fwd_run_cluster<12>;
}

cudaError_t launch_cluster(const void* fn, int threads, int groups, int cs, int smem, void** args, cudaStream_t s) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(groups * cs)); cfg.blockDim = dim3((unsigned)threads); cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = counted(s);
  cfg.attrs = at; cfg.numAttrs = pdl_enabled() ? 2u : 1u;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace

bool cluster_maps(CUtensorMap* tm_w, CUtensorMap* tm_wt, const void* wp_hh, const void* wpT_hh, int H) {
  const uint64_t h = (uint64_t)H;
  return make_tmap_2d(tm_w, wp_hh, 2, h, 4 * h, h * 2, 64, 128) && make_tmap_2d(tm_wt, wpT_hh, 2, 4 * h, h, 8 * h, 64, 128);
}

int cluster_rows(int B, int H) {
  const int cs = cluster_ctas(H);
  if (env::run_cluster() > 0 && cs > env::run_cluster()) return 0;
  int fit = run_sms() / cs;
  for (int RB : {8, 12})
    for (int dir = 0; dir < 2; ++dir) {
      const void* fn = kernel(dir, RB);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)cs); cfg.blockDim = dim3(dir ? BWD_THREADS : THREADS); cfg.dynamicSmemBytes = (size_t)(dir ? bwd_smem(H, RB) : fwd_smem(H));
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at; cfg.numAttrs = 1;
      int n = 0;
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, dir ? bwd_smem(16 * CU, RB) : fwd_smem(16 * CU)) != cudaSuccess ||
          cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
          cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
      }
      if (n < fit) fit = n;
    }
  if (fit < 1) return 0;
  // Fewer rows make a step shorter (all that is sent and most of what a thread does is in proportion to them), as long
  // as the clusters need not take turns.  Forward and backward operation, B = 64, 8, 12 and 16 rows, in us: H = 256 0.78,
  // 1.02, 1.22 and 0.90, 1.21, 1.29; H = 512, where seven clusters fit, 2.1 (in turns), 1.32, 1.57 and 2.5, 1.73, 1.91.
  // (So 16 rows are never taken: 64 are six clusters of 12.)
  return (B + 7) / 8 <= fit ? 8 : 12;
}

int cluster_smem(bool backward, int H, int rows) { return backward ? bwd_smem(H, rows) : fwd_smem(H); }

cudaError_t cluster_forward(const CUtensorMap& tm_w, const ClusterFwdArgs& a, int rows, cudaStream_t s) {
  void* args[] = {(void*)&tm_w, (void*)&a};
  return launch_cluster(kernel(0, rows), THREADS, (a.B + rows - 1) / rows, cluster_ctas(a.H), fwd_smem(a.H), args, s);
}

cudaError_t cluster_backward(const CUtensorMap& tm_wt, const ClusterBwdArgs& a, int rows, cudaStream_t s) {
  void* args[] = {(void*)&tm_wt, (void*)&a};
  return launch_cluster(kernel(1, rows), BWD_THREADS, (a.B + rows - 1) / rows, cluster_ctas(a.H), bwd_smem(a.H, rows), args, s);
}

}  // namespace tc
}  // namespace mebptt
