// Runs of the bfloat16 recurrence for 513 to 1024 hidden units.
//
// W_hh is too much for the CTAs of one cluster, so what a step makes has to reach others through the L2.  What that
// costs, one after the other, when it is done by the book -- store, release (which waits for the stores), counter, poll,
// copy of the state into shared memory -- is 3 us of the 4.2 (forward) and 4.6 (backward) an operation took.  Here a
// state is its own signal: it is stored in pieces of 16 bytes into a ring of slots that hold ones everywhere else, and
// every reader polls the very pieces it needs, into registers and from there into the operand of its MMA.  (A word of
// ones is two NaNs with every payload bit set: no conversion to bfloat16 makes one.)  An exchange between 32 CTAs, 32
// KB each, takes 2250 cycles that way.
//
// What makes that cheap enough is tensor memory: with the weights there (448 columns; two tiles of 64 contraction
// indices stay in shared memory) a CTA holds 128 gate rows of a whole W_hh, twice what shared memory does, so that 32
// CTAs serve a group of 8 or 16 batch rows: half the bytes to every CTA, half the CTAs to a group, and an MMA takes 11
// cycles a K = 16 slice instead of 38.
//
//   forward    a CTA makes h_k of its 32 units; every CTA of the group polls all of it.  The contraction is summed in
//              two parts (fwd_first_part_blocks), as the batched products of a leaf batch are.
//   backward   a CTA makes dz_k of its 32 units.  The CTAs of a cluster of four share the contraction index: CTA r
//              polls the dz_k of a quarter of the units and multiplies it by the 128 columns of dh its cluster owns;
//              the partial sums go to the columns' owners inside the cluster and are added in the order of the ranks.
//              (Clusters of eight would halve what is polled, but only 15 of the 16 that 1024 units and 64 rows take fit.)
//
// The ring: step i uses slot i mod 4.  Forward, a CTA that has all of h_i knows that everybody has consumed h_{i-1}, so
// it puts ones over its own pieces of that; backward that holds for dz_{i-2} (what a CTA receives at step i comes from
// CTAs whose step i - 1 had everybody's dz_{i-1}).  A fence of the writer between that and what it writes next, and one of
// each polling thread between two steps, see to it that a slot is seen cleared before it is polled again: the thread
// that polls a piece polls the same writer's pieces in every step.  A launch leaves its ring as it is and clears the set
// of the launch before it.
//
// The launch is cooperative (its CTAs wait for one another), and every wait is bounded.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "launch.hpp"
#include "lstm_dev.cuh"
#include "mebptt.h"
#include "ring_runs.hpp"
#include "runs_dev.cuh"
#include "sm100.cuh"

namespace mebptt {
namespace tc {

namespace {

using namespace sm100;

constexpr int TM_TILES = 14;             // tiles of weights in tensor memory (32 columns each), the others stay in shared memory
constexpr uint32_t ACC = 32 * TM_TILES;  // column of the accumulators
constexpr int STG = 4;                   // tiles on their way to tensor memory at a time: even, so that a stage is always moved by the same team of warps
constexpr uint32_t PIECE = 256;          // operand of an MMA without swizzle: [16-byte piece of K][16 rows][16 bytes]
constexpr int ZROW = 40;
constexpr int POLLERS = 8;               // warps that poll

__device__ __forceinline__ uint4 load_piece(const char* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_piece(char* p, uint4 v) {
  asm volatile("st.relaxed.gpu.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint4 ones() { return make_uint4(~0u, ~0u, ~0u, ~0u); }
__device__ __forceinline__ bool there(const uint4& v) { return v.x != ~0u && v.y != ~0u && v.z != ~0u && v.w != ~0u; }
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// N pieces a lane: piece x of this lane lies at from + x * stride and goes to smem + x * to_stride; `want` has a bit for
// each that is to come.  False, for the whole warp, if the wait of a lane ran out (or another warp's did).
template <int N>
__device__ __forceinline__ bool poll_lane(const char* from, uint32_t stride, uint8_t* to, uint32_t to_stride, uint32_t want, volatile int* failed,
                                            uint32_t limit) {
  if (!want) return true;
  // One piece first, until it is there, then all of them: eight warps that poll eight pieces a lane keep the memory pipe so
  // full that MMAs leave at a third of their pace.
  const char* const last = from + (31 - __clz(want)) * stride;
  uint32_t i = 0;
  while (!there(load_piece(last)))
    if (++i >= limit || (i > 4096 && *failed)) { *failed = 1; return false; }
  for (; want; ++i) {
    if (i >= limit || (i > 4096 && *failed)) { *failed = 1; return false; }
    uint4 v[N];
#pragma unroll
    for (int x = 0; x < N; ++x)
      if (want >> x & 1) v[x] = load_piece(from + x * stride);
#pragma unroll
    for (int x = 0; x < N; ++x)
      if ((want >> x & 1) && there(v[x])) {
        *reinterpret_cast<uint4*>(to + x * to_stride) = v[x];
        want &= ~(1u << x);
      }
  }
  return true;
}

template <int N>
__device__ __forceinline__ bool poll_pieces(const char* from, uint32_t stride, uint8_t* to, uint32_t to_stride, uint32_t want, volatile int* failed,
                                            uint32_t limit) {
  return __all_sync(0xffffffffu, poll_lane<N>(from, stride, to, to_stride, want, failed, limit));
}

// MMAs over a tile of 64 contraction indices in shared memory (128-byte swizzle) and B as above
__device__ __forceinline__ void mma_smem_x4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
#pragma unroll
  for (int k = 0; k < 4; ++k)
    mma_f16(d_tmem, a_desc + 2 * k, b_desc + (uint64_t)k * (2 * PIECE / 16), idesc, k ? 1u : accumulate);
}

// Tiles [lo, hi) of the contraction into one accumulator: first those whose weights are in tensor memory.
__device__ __forceinline__ void mma_tiles(uint32_t d, uint32_t tmem, uint64_t w_desc, uint64_t b_desc, int lo, int hi, uint32_t idesc, uint32_t add) {
  uint64_t bd = b_desc + (uint64_t)(lo * (8 * PIECE >> 4));
  const int mid = hi < TM_TILES ? hi : TM_TILES;
  uint32_t at = tmem + 32u * (uint32_t)lo;
#pragma unroll 1
  for (int t = lo; t < mid; ++t, at += 32, bd += 8 * PIECE >> 4, add = 1) mma_tmem_x4<2 * PIECE / 16>(d, at, bd, idesc, add);
#pragma unroll 1
  for (int t = mid; t < hi; ++t, w_desc += W_TILE >> 4, bd += 8 * PIECE >> 4, add = 1) mma_smem_x4(d, w_desc, bd, idesc, add);
}

// The way of the weights to tensor memory: tile t < TM_TILES through stage t mod STG, the others to where they stay.
struct Weights {
  uint64_t full[STG], empty[STG], rest;
};
__device__ __forceinline__ void weights_init(Weights& w) {
  for (int s = 0; s < STG; ++s) { mbar_init(&w.full[s], 1); mbar_init(&w.empty[s], 4); }
  mbar_init(&w.rest, 1);
}
// One lane: requests the tiles (x(t), y(t): coordinates of tile t).  Bounded; what was requested lands before the gates go on.
template <class XY>
__device__ __forceinline__ void weights_request(Weights& w, const CUtensorMap* tm, int tiles, uint8_t* stages, uint8_t* stay, XY xy, volatile int* failed) {
  if (tiles > TM_TILES) mbar_arrive_expect_tx(&w.rest, (uint32_t)(tiles - TM_TILES) * W_TILE);
  for (int t = TM_TILES; t < tiles; ++t) {
    const int2 c = xy(t);
    tma_load_2d(stay + (t - TM_TILES) * W_TILE, tm, c.x, c.y, &w.rest);
  }
  for (int t = 0; t < tiles && t < TM_TILES; ++t) {
    const int s = t % STG, it = t / STG;
    if (it > 0 && !wait_or_fail(&w.empty[s], (uint32_t)(it - 1) & 1, failed)) return;
    const int2 c = xy(t);
    mbar_arrive_expect_tx(&w.full[s], W_TILE);
    tma_load_2d(stages + s * W_TILE, tm, c.x, c.y, &w.full[s]);
  }
}
// Warps of the gates: warp w moves rows 32 (w mod 4) .. + 31 of every tile, or of every other where there are eight warps.
__device__ __forceinline__ void weights_move(Weights& w, int tiles, const uint8_t* stages, uint32_t tmem, int warp, int lane, int teams, volatile int* failed) {
  const int q = warp & 3;
  for (int t = warp >> 2; t < tiles && t < TM_TILES; t += teams) {
    const int s = t % STG;
    (void)wait_or_fail(&w.full[s], (uint32_t)(t / STG) & 1, failed);
    __syncwarp();
    const uint8_t* row = stages + s * W_TILE + (32 * q + lane) * 128;
    uint4 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = *reinterpret_cast<const uint4*>(row + ((c ^ (lane & 7)) * 16));
    tmem_st_32x32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(32 * t), v);
    // (behind what takes the values: loads still under way when the stage is given back would see the next tile)
    __syncwarp();
    if (lane == 0) mbar_arrive(&w.empty[s]);
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  tc_fence_before_sync();
}

// ------------------------------------------------------------------------------------------
// forward run
// ------------------------------------------------------------------------------------------
// Warps 0 .. 4 G - 1: gates, each for 8 units and 8 rows (G = RB / 8); then one for copies and MMAs; then those that poll.
struct RingFwdStage {              // per warp of the gates
  float z[2][8][ZROW];             // accumulators of both parts [batch row][gate row of the warp's 8 units]
  __nv_bfloat16 v[5][8][8];        // h, i, f, g, o [batch row][unit]
};
template <int RB>
struct FwdShape {
  static constexpr int G = RB / 8, GATES = 4 * G, THREADS = 32 * (GATES + 1 + POLLERS);
  static __host__ __device__ uint32_t stay(int) { return 0; }
  static __host__ __device__ uint32_t stages(int KT) { return (uint32_t)(KT > TM_TILES ? KT - TM_TILES : 0) * W_TILE; }
  static __host__ __device__ uint32_t h(int KT) { return stages(KT) + STG * W_TILE; }
  static __host__ __device__ uint32_t out(int KT) { return h(KT) + 2 * (uint32_t)KT * 8 * PIECE; }
  static __host__ __device__ uint32_t total(int KT) { return out(KT) + GATES * (uint32_t)sizeof(RingFwdStage) + 1024; }
};

template <int RB>
__global__ void __launch_bounds__(FwdShape<RB>::THREADS, 1) fwd_run_ring(const __grid_constant__ CUtensorMap tm_w, const ClusterFwdArgs a,
                                                                         const RingArgs g, int ncta, int KT0) {
  typedef FwdShape<RB> Shape;
  constexpr int GATES = Shape::GATES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Weights wt;
  __shared__ uint64_t ready, hfull[2][2], acc[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;

  uint8_t* const sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int KT = (a.H + 63) / 64;                  // tiles of 64 contraction indices, KT0 of them in the first part
  uint8_t* const sH = sm + Shape::h(KT);           // [2][8 KT] pieces of h_{k-1}
  const uint32_t h_buf = (uint32_t)KT * 8 * PIECE;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = g.first + (int)blockIdx.x / ncta, cta = (int)blockIdx.x % ncta, groups = (a.B + RB - 1) / RB;
  // (a slot: the groups one after the other, [8 units][RB rows][16 bytes] each)
  const uint32_t group_bytes = (uint32_t)ncta * CU * RB * 2, slot_bytes = group_bytes * groups;

  if (tid == 0) {
    weights_init(wt);
    mbar_init(&ready, GATES);
    for (int b = 0; b < 2; ++b)
      for (int q = 0; q < 2; ++q) mbar_init(&hfull[b][q], POLLERS / 2);
    for (int b = 0; b < 2; ++b) mbar_init(&acc[b], 1);
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_w);
  }
  for (uint32_t e = tid; e < 2 * h_buf / 16; e += Shape::THREADS) reinterpret_cast<uint4*>(sH)[e] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_shared();
  if (warp == GATES) tmem_alloc(&tmem_slot, 512);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();

  const int brow = grp * RB;
  if (warp == GATES) {
    constexpr uint32_t idesc = make_idesc(1, 128, CB, false, false);
    if (lane == 0)
      weights_request(wt, &tm_w, KT, sm + Shape::stages(KT), sm + Shape::stay(KT), [&](int t) { return make_int2(64 * t, cta * 4 * CU); }, &failed);
    __syncwarp();
    bool ok = __all_sync(0xffffffffu, wait_or_fail(&ready, 0, &failed));
    if (ok && KT > TM_TILES) ok = __all_sync(0xffffffffu, wait_or_fail(&wt.rest, 0, &failed));
    const uint64_t w_desc = make_desc_sw128(smem_u32(sm + Shape::stay(KT)), 16, 1024);
    for (int i = 0; i < a.n; ++i) {
      const int b = i & 1;
      const uint64_t h_desc = make_desc_plain(smem_u32(sH + b * h_buf), PIECE, 128);
      for (int q = 0; q < 2; ++q) {
        if (ok) ok = __all_sync(0xffffffffu, wait_or_fail(&hfull[b][q], (uint32_t)(i >> 1) & 1, &failed));
        if (!ok) break;
        tc_fence_after_sync();
        if (elect_one()) {
          // (two sets of accumulators: the part this CTA's units are not in may be here before its gates have read the set
          // of the step before)
          const uint32_t d = tmem + ACC + (uint32_t)(2 * b + q) * CB;
          mma_tiles(d, tmem, w_desc, h_desc, q ? KT0 : 0, q ? KT : KT0, idesc, 0u);
        }
        __syncwarp();
      }
      if (elect_one()) mma_commit(&acc[b]);   // always: the gates count on one arrival per step
      __syncwarp();
      if (i == a.n - 1 && lane == 0) grid_dep_launch();
    }
    if (failed && lane == 0) {
      // loads that were requested may still be landing
      if (KT > TM_TILES) (void)mbar_wait(&wt.rest, 0);
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
  } else if (warp > GATES) {
    // ---- polling: half the warps for each part of the contraction.  A lane has one row; its pieces are 8 units each -----
    constexpr int ROWS = RB, PER = 32 / ROWS;                       // pieces of 8 units a warp has in hand at a time
    constexpr int N = 64 / (PER * POLLERS / 2);                     // 64 pieces a part at most
    const int pw = warp - GATES - 1, q = pw / (POLLERS / 2), wl = pw % (POLLERS / 2);
    const int row = lane % ROWS, p0 = (q ? 8 * KT0 : 0) + wl * PER + lane / ROWS, p_end = q ? fwd_waited_units(a.H) / 8 : 8 * KT0;
    constexpr int STEP = PER * POLLERS / 2;
    uint32_t want = 0;
#pragma unroll
    for (int x = 0; x < N; ++x)
      if (p0 + x * STEP < p_end) want |= 1u << x;
    uint8_t* const to = sH + p0 * PIECE + row * 16;
    {
      // the state the run starts from, rows past the batch as zeros
      const char* h0 = a.ws + (size_t)a.ops[0].h_src * 16;
      uint4 v[N];
#pragma unroll
      for (int x = 0; x < N; ++x) {
        v[x] = make_uint4(0, 0, 0, 0);
        if ((want >> x & 1) && brow + row < a.B && p0 + x * STEP < a.H / 8) v[x] = *reinterpret_cast<const uint4*>(h0 + ((size_t)(brow + row) * a.H + 8 * (p0 + x * STEP)) * 2);
      }
#pragma unroll
      for (int x = 0; x < N; ++x)
        if (want >> x & 1) *reinterpret_cast<uint4*>(to + x * STEP * PIECE) = v[x];
    }
    const char* const from = g.ring + (size_t)grp * group_bytes + (size_t)p0 * (RB * 16) + row * 16;
    for (int i = 0; i < a.n; ++i) {
      if (i > 0) {
        if (!poll_pieces<N>(from + (size_t)(i & (RING_SLOTS - 1)) * slot_bytes, STEP * RB * 16, to + (i & 1) * h_buf, STEP * PIECE, want, &failed, g.poll_limit)) break;
        if (g.fault && pw == 0 && !poll_pieces<1>(g.never, 0, to, 0, 1u, &failed, g.poll_limit)) break;
      }
      fence_proxy_async_shared();
      __syncwarp();
      if (lane == 0) mbar_arrive(&hfull[i & 1][q]);
      fence_gpu();   // (what was seen here comes before what is polled next)
    }
  } else {
    // ---- gates: warp w has the units 8 (w mod 4) .. + 7 of the CTA and the rows 8 (w / 4) .. + 7 of the group -------------
    // Lane l holds gate row 32 (w mod 4) + l of the accumulators (gate l % 4 of unit l / 4); through the warp's stage it
    // gets the four gates of that unit for two rows.  States leave in pieces of 16 bytes: the warp's units of one row.
    RingFwdStage& st = reinterpret_cast<RingFwdStage*>(sm + Shape::out(KT))[warp];
    const int wq = warp & 3, half = warp >> 2;
    const int u = lane >> 2, r0 = lane & 3;
    const int jw = cta * CU + 8 * wq, j = jw + u;            // the warp's first unit, the lane's
    const bool wvalid = jw < a.H;
    const int b0 = brow + 8 * half, prow = lane & 7;         // first row of the warp; the row whose pieces this lane stores
    const bool pvalid = wvalid && b0 + prow < a.B;
    const size_t ep = (size_t)(b0 + prow) * a.H + jw;
    const DevOp op0 = a.ops[0];
    bool rvalid[2];
    size_t er[2];
    float c[2];
    float4 zx[2];
    uint4 hprev = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int b = b0 + r0 + 4 * v;
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
    // this lane's piece in a slot
    const uint32_t mine = (uint32_t)grp * group_bytes + (uint32_t)(jw / 8) * (RB * 16) + (uint32_t)(8 * half + prow) * 16;
    if (lane < 8)
      for (int s = 0; s < RING_SLOTS; ++s) store_piece(g.other + (size_t)s * slot_bytes + mine, ones());
    weights_move(wt, KT, sm + Shape::stages(KT), tmem, warp, lane, Shape::G, &failed);
    __syncwarp();
    if (lane == 0) mbar_arrive(&ready);

    for (int i = 0; i < a.n; ++i) {
      const DevOp op = a.ops[i];
      const bool got = wait_or_fail(&acc[i & 1], (uint32_t)(i >> 1) & 1, &failed) && !*(volatile int*)&failed;
      tc_fence_after_sync();
      uint32_t p[8], q[8];
      const uint32_t at = tmem + ((uint32_t)(32 * wq) << 16) + ACC + (uint32_t)(2 * (i & 1) * CB + 8 * half);
      tmem_ld_32x8(at, p);
      tmem_ld_32x8(at + CB, q);
      tmem_ld_wait();
      tc_fence_before_sync();
#pragma unroll
      for (int n = 0; n < 8; ++n) {
        st.z[0][n][lane] = __uint_as_float(p[n]);
        st.z[1][n][lane] = __uint_as_float(q[n]);
      }
      __syncwarp();
      float cin[2], gate[2][4];
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const float4 x = *reinterpret_cast<const float4*>(&st.z[0][r0 + 4 * v][4 * u]);
        const float4 y = *reinterpret_cast<const float4*>(&st.z[1][r0 + 4 * v][4 * u]);
        const float iv = sigmoid_fast((zx[v].x + x.x) + y.x), fv = sigmoid_fast((zx[v].y + x.y) + y.y);
        const float gv = tanh_fast((zx[v].z + x.z) + y.z), ov = sigmoid_fast((zx[v].w + x.w) + y.w);
        cin[v] = c[v];
        c[v] = fmaf(fv, c[v], iv * gv);
        st.v[0][r0 + 4 * v][u] = __float2bfloat16_rn(ov * tanh_fast(c[v]));
        gate[v][0] = iv; gate[v][1] = fv; gate[v][2] = gv; gate[v][3] = ov;
      }
      __syncwarp();
      const uint4 hnew = *reinterpret_cast<const uint4*>(&st.v[0][prow][0]);   // (past the last unit: as in fwd_run_cluster)
      if (got && lane < 8) {
        if (i + 1 < a.n) store_piece(g.ring + (size_t)((i + 1) & (RING_SLOTS - 1)) * slot_bytes + mine, hnew);
        if (i >= 1) store_piece(g.ring + (size_t)((i - 1) & (RING_SLOTS - 1)) * slot_bytes + mine, ones());
      }
      // the rest of the state, off the critical path
      if (got) {
        if (pvalid && lane < 8) {
          *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.h_dst * 16) + ep) = hnew;
          if (op.stage) *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.stage * 16) + ep) = hnew;
        }
        if (op.gates) {
#pragma unroll
          for (int v = 0; v < 2; ++v)
#pragma unroll
            for (int x = 0; x < 4; ++x) st.v[1 + x][r0 + 4 * v][u] = __float2bfloat16_rn(gate[v][x]);
          __syncwarp();
          if (pvalid)
            *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.gates * 16) + ep + (size_t)(lane >> 3) * a.plane16 * 8) =
                *reinterpret_cast<const uint4*>(&st.v[1 + (lane >> 3)][prow][0]);
        }
        if (op.in_copy && pvalid && lane < 8)
          *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(a.ws + (size_t)op.in_copy * 16) + ep) = hprev;
        hprev = hnew;
        float* cd = reinterpret_cast<float*>(a.ws + (size_t)op.c_dst * 16);
        float* ci = op.in_copy ? reinterpret_cast<float*>(a.ws + ((size_t)op.in_copy + a.hsz16) * 16) : nullptr;
#pragma unroll
        for (int v = 0; v < 2; ++v)
          if (rvalid[v]) {
            cd[er[v]] = c[v];
            if (ci) ci[er[v]] = cin[v];
            if (i + 1 < a.n) zx[v] = *reinterpret_cast<const float4*>(a.zx + 4 * ((size_t)(i + 1) * a.B * a.H + er[v]));
          }
      }
      fence_gpu();    // the cleared piece comes before what is pushed next
      __syncwarp();   // the stage is free again
    }
  }

  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (grp == 0 && cta == 0) a.counters[0] += a.n;
  }
  if (warp == GATES) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------
// backward run
// ------------------------------------------------------------------------------------------
// Warps 0 .. 4 G - 1: gates; then copies and MMAs; inputs; loss terms; then those that poll.
template <int RB>
struct BwdShape {
  static constexpr int G = RB / 8, GATES = 4 * G, THREADS = 32 * (GATES + 3 + POLLERS);
  static constexpr uint32_t SLOT = recv_slot(RB);
  // KT: tiles of 64 gate columns in a quarter of the contraction index
  static __host__ __device__ uint32_t stay(int) { return 0; }
  static __host__ __device__ uint32_t stages(int KT) { return (uint32_t)(KT > TM_TILES ? KT - TM_TILES : 0) * W_TILE; }
  static __host__ __device__ uint32_t dz(int KT) { return stages(KT) + STG * W_TILE; }
  static __host__ __device__ uint32_t recv(int KT) { return dz(KT) + 2 * (uint32_t)KT * 8 * PIECE; }
  static __host__ __device__ uint32_t in(int KT) { return recv(KT) + 2 * RING_CLUSTER * SLOT; }
  static __host__ __device__ uint32_t total(int KT) { return in(KT) + 2 * (uint32_t)sizeof(GateStage<RB>) + 1024; }
};

template <int RB>
__global__ void __launch_bounds__(BwdShape<RB>::THREADS, 1) bwd_run_ring(const __grid_constant__ CUtensorMap tm_wt, const ClusterBwdArgs a,
                                                                         const RingArgs g, int ncta) {
  typedef BwdShape<RB> Shape;
  constexpr int GATES = Shape::GATES;
  constexpr uint32_t SLOT = Shape::SLOT;
  extern __shared__ uint8_t smem_raw[];
  __shared__ Weights wt;
  __shared__ uint64_t ready, zfull[2][2], acc[2], full[2], inready[2], used[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;

  uint8_t* const sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int per = ncta / RING_CLUSTER;             // CTAs whose dz a CTA of the cluster takes
  const int KT = 2 * per;
  uint8_t* const sZ = sm + Shape::dz(KT);          // [2][8 KT] pieces of dz
  uint8_t* const sR = sm + Shape::recv(KT);        // [2][4] partial sums received
  GateStage<RB>* const sI = reinterpret_cast<GateStage<RB>*>(sm + Shape::in(KT));
  const uint32_t z_buf = (uint32_t)KT * 8 * PIECE;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = g.first + (int)blockIdx.x / ncta, cta = (int)blockIdx.x % ncta, groups = (a.B + RB - 1) / RB;
  const int rank = cta % RING_CLUSTER, cl = cta / RING_CLUSTER;
  const int half0 = 8 * (KT / 2);                  // pieces of two units in a half of the CTA's quarter
  // a slot: the groups one after the other, [2 units][RB rows][16 bytes] each
  const uint32_t cta_bytes = 4 * CU * RB * 2, group_bytes = (uint32_t)ncta * cta_bytes, slot_bytes = group_bytes * groups;

  if (tid == 0) {
    weights_init(wt);
    mbar_init(&ready, GATES);
    for (int b = 0; b < 2; ++b) {
      for (int q = 0; q < 2; ++q) mbar_init(&zfull[b][q], POLLERS / 2);
      mbar_init(&acc[b], 1);
      mbar_init(&full[b], 1);
      mbar_init(&inready[b], 32);
      mbar_init(&used[b], GATES);
    }
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tm_wt);
  }
  for (uint32_t e = tid; e < 2 * z_buf / 16; e += Shape::THREADS) reinterpret_cast<uint4*>(sZ)[e] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_shared();
  if (warp == GATES) tmem_alloc(&tmem_slot, 512);
  tc_fence_before_sync();
  cluster_sync();                                  // peers push onto each other's barriers: all must be initialised
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();

  const int brow = grp * RB, rows = a.B - brow;    // the group's batch rows (RB of them, or fewer)
  const int unit0 = cta * CU, units = a.H - unit0; // the CTA's hidden units (likewise, or none)
  const int s_hi = (a.ops[0].k - 1) % a.S;         // row block of the run's first step; those after it descend
  const uint32_t bytes = RING_CLUSTER * SLOT;

  if (warp == GATES) {
    constexpr uint32_t idesc = make_idesc(1, 128, CB, false, false);
    if (lane == 0) {
      mbar_arrive_expect_tx(&full[0], bytes);
      if (a.n > 1) mbar_arrive_expect_tx(&full[1], bytes);
      // tile t: 64 gate columns t of the CTA's quarter by the cluster's columns of dh
      weights_request(wt, &tm_wt, KT, sm + Shape::stages(KT), sm + Shape::stay(KT),
                      [&](int t) { return make_int2(rank * per * 4 * CU + 64 * t, cl * RING_CLUSTER * CU); }, &failed);
    }
    __syncwarp();
    bool ok = __all_sync(0xffffffffu, wait_or_fail(&ready, 0, &failed));
    if (ok && KT > TM_TILES) ok = __all_sync(0xffffffffu, wait_or_fail(&wt.rest, 0, &failed));
    const uint64_t w_desc = make_desc_sw128(smem_u32(sm + Shape::stay(KT)), 16, 1024);
    for (int i = 0; i < a.n; ++i) {
      const int b = i & 1;
      const uint64_t z_desc = make_desc_plain(smem_u32(sZ + b * z_buf), PIECE, 128);
      for (int q = 0; q < 2; ++q) {
        if (ok) ok = __all_sync(0xffffffffu, wait_or_fail(&zfull[b][q], (uint32_t)(i >> 1) & 1, &failed));
        if (!ok) break;
        tc_fence_after_sync();
        if (elect_one()) {
          // (two sets of accumulators: dz of the next step may be here before this CTA's gates have read those of this one)
          mma_tiles(tmem + ACC + (uint32_t)b * CB, tmem, w_desc, z_desc, q ? KT / 2 : 0, q ? KT : KT / 2, idesc, (uint32_t)q);
        }
        __syncwarp();
      }
      if (elect_one()) mma_commit(&acc[b]);
      __syncwarp();
      if (i == a.n - 1 && lane == 0) grid_dep_launch();
    }
    if (failed && lane == 0) {
      if (KT > TM_TILES) (void)mbar_wait(&wt.rest, 0);
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
    }
  } else if (warp == GATES + 1) {
    const size_t e0 = (size_t)brow * a.H + unit0, bh = (size_t)a.B * a.H;
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
      // The gates have used the inputs of step i and the partial sums of step i - 1.  (Two barriers: the gates may be a step
      // ahead, not two, for the inputs of that one are asked for below.)
      if (!wait_or_fail(&used[i & 1], (uint32_t)(i >> 1) & 1, &failed)) break;
      if (lane == 0 && i >= 1 && i + 1 < a.n && !*(volatile int*)&failed) mbar_arrive_expect_tx(&full[(i + 1) & 1], bytes);
      if (i + 2 < a.n) {
        const DevOp op = next;
        if (i + 3 < a.n) next = a.ops[i + 3];
        fill(op, i + 2);
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp == GATES + 2) {
    // loss terms of the run: the partial sums of a step in a fixed order
    if (grp == 0 && cta == 0)
      for (int i = lane; i < a.n; i += 32) {
        float sum = 0.f;
        for (int p = 0; p < a.loss_parts; ++p) sum += a.loss_part[(s_hi - i) * a.loss_parts + p];
        a.loss_t[a.ops[0].k - 1 - i] = sum;
      }
  } else if (warp > GATES) {
    // ---- polling: the dz of `per` CTAs, 16 pieces of two units each and RB rows ------------------------------------------
    constexpr int PER = 32 / RB, STEP = PER * POLLERS / 2, N = 64 / STEP;   // 64 pieces a half at most
    const int pw = warp - GATES - 3, q = pw / (POLLERS / 2), wl = pw % (POLLERS / 2);
    const int row = lane % RB, p0 = q * half0 + wl * PER + lane / RB;
    uint32_t want = 0;
#pragma unroll
    for (int x = 0; x < N; ++x) {
      if (p0 + x * STEP < (q + 1) * half0) want |= 1u << x;
    }
    uint8_t* const to = sZ + p0 * PIECE + row * 16;
    const char* const from = g.ring + (size_t)grp * group_bytes + (size_t)(rank * per) * cta_bytes + (size_t)p0 * (RB * 16) + row * 16;
    for (int i = 0; i < a.n; ++i) {
      if (!poll_pieces<N>(from + (size_t)(i & (RING_SLOTS - 1)) * slot_bytes, STEP * RB * 16, to + (i & 1) * z_buf, STEP * PIECE, want, &failed, g.poll_limit)) break;
      if (g.fault && pw == 0 && !poll_pieces<1>(g.never, 0, to, 0, 1u, &failed, g.poll_limit)) break;
      fence_proxy_async_shared();
      __syncwarp();
      if (lane == 0) mbar_arrive(&zfull[i & 1][q]);
      fence_gpu();
    }
  } else {
    // ---- gates: warp w has the units 8 (w mod 4) .. + 7 of the CTA and the rows 8 (w / 4) .. + 7 of the group; lane l the
    // unit l % 8 of those and two rows -------------------------------------------------------------------------------------
    constexpr int NV = 2;
    const int wq = warp & 3, half = warp >> 2;
    const int u = 8 * wq + (lane & 7), r0 = 8 * half + NV * (lane >> 3);
    const bool leaf = a.zleaf != nullptr;
    const size_t e = (size_t)(brow + r0) * a.H + unit0 + u;
    bool valid[NV];
    float dh[NV], dc[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      valid[v] = u < units && r0 + v < rows;
      dh[v] = valid[v] ? a.dh[e + (size_t)v * a.H] : 0.f;
      dc[v] = valid[v] ? a.dc[e + (size_t)v * a.H] : 0.f;
    }
    // dz leaves in pieces of two units: an even lane takes them from its neighbour for its first row, an odd one for its second
    const int odd = lane & 1, prow = r0 + odd;
    const uint32_t mine = (uint32_t)grp * group_bytes + (uint32_t)cta * cta_bytes + (uint32_t)(u >> 1) * (RB * 16) + (uint32_t)prow * 16;
    const bool store_ok = u < units && prow < rows;   // (units is a multiple of 8)
    __nv_bfloat16* dzp = reinterpret_cast<__nv_bfloat16*>(a.dz) + 4 * ((size_t)s_hi * a.B * a.H + (size_t)(brow + prow) * a.H + unit0 + (u & ~1));
    const size_t dz_step = (size_t)4 * a.B * a.H;
    for (int s = 0; s < RING_SLOTS; ++s) store_piece(g.other + (size_t)s * slot_bytes + mine, ones());
    // partial sums: lane l holds column 32 wq + l of the cluster's, which CTA wq owns
    const uint32_t to = map_rank(smem_u32(sR) + (uint32_t)rank * SLOT + (uint32_t)(2 * half) * (CU * 16) + (uint32_t)lane * 16, (uint32_t)wq);
    const uint32_t tb = map_rank(smem_u32(&full[0]), (uint32_t)wq);
    const float* const sums = reinterpret_cast<const float*>(sR) + (r0 >> 2) * 4 * CU + 4 * u + (r0 & 3);
    auto receive = [&](int it) {
      const bool got = wait_pushed(&full[it & 1], (uint32_t)(it >> 1) & 1, &failed, a.poll_limit);
      if (!got) return;
      const float* src = sums + (it & 1) * (RING_CLUSTER * (SLOT / 4));
      float s0 = 0.f, s1 = 0.f;
#pragma unroll
      for (int p = 0; p < RING_CLUSTER; ++p) {
        const float2 x = *reinterpret_cast<const float2*>(src + p * (SLOT / 4));
        s0 += x.x; s1 += x.y;
      }
      dh[0] = s0; dh[1] = s1;
    };

    weights_move(wt, KT, sm + Shape::stages(KT), tmem, warp, lane, Shape::G, &failed);
    __syncwarp();
    if (lane == 0) mbar_arrive(&ready);
    GateIn<NV> in;
    (void)wait_or_fail(&inready[0], 0, &failed);
    pick_out<NV, RB>(leaf, sI[0], u, r0, in);
    for (int i = 0; i < a.n; ++i, dzp -= dz_step) {
      if (i > 0) receive(i - 1);
      uint2 out[NV];
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
        out[v] = valid[v] ? make_uint2(pack_bf16x2(zi, zf), pack_bf16x2(zg, zo)) : make_uint2(0, 0);
      }
      const uint2 send = odd ? out[0] : out[1], keep = odd ? out[1] : out[0];
      const uint2 get = make_uint2(__shfl_xor_sync(0xffffffffu, send.x, 1), __shfl_xor_sync(0xffffffffu, send.y, 1));
      const uint4 piece = odd ? make_uint4(get.x, get.y, keep.x, keep.y) : make_uint4(keep.x, keep.y, get.x, get.y);
      const bool live = !*(volatile int*)&failed;
      if (live) store_piece(g.ring + (size_t)(i & (RING_SLOTS - 1)) * slot_bytes + mine, piece);
      __syncwarp();
      if (lane == 0) mbar_arrive(&used[i & 1]);
      // beside the exchange: dz to its stage, the piece of two steps ago cleared, the inputs of the next (earlier) step
      if (live) {
        if (store_ok) *reinterpret_cast<uint4*>(dzp) = piece;
        if (i >= 2) store_piece(g.ring + (size_t)((i - 2) & (RING_SLOTS - 1)) * slot_bytes + mine, ones());
      }
      if (i + 1 < a.n) {
        (void)wait_or_fail(&inready[(i + 1) & 1], (uint32_t)((i + 1) >> 1) & 1, &failed);
        pick_out<NV, RB>(leaf, sI[(i + 1) & 1], u, r0, in);
      }
      fence_gpu();
      const bool got = wait_or_fail(&acc[i & 1], (uint32_t)(i >> 1) & 1, &failed) && !*(volatile int*)&failed;
      tc_fence_after_sync();
      uint32_t r[8];
      tmem_ld_32x8(tmem + ((uint32_t)(32 * wq) << 16) + ACC + (uint32_t)((i & 1) * CB + 8 * half), r);
      tmem_ld_wait();
      tc_fence_before_sync();
      if (got) {
        const uint32_t obuf = (uint32_t)(i & 1) * (RING_CLUSTER * SLOT), bbuf = (uint32_t)(i & 1) * 8;
#pragma unroll
        for (int v = 0; v < 2; ++v) push16(to + obuf + v * (CU * 16), make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]), tb + bbuf);
      }
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
  cluster_sync();     // no CTA leaves while a peer may still push to it
  if (tid == 0) {
    if (failed) *a.status = MEBPTT_ERR_TIMEOUT;
    else if (grp == 0 && cta == 0) a.counters[1] += a.n;
  }
  if (warp == GATES) tmem_dealloc(tmem, 512);
}

const void* kernel(bool bwd, int RB) {
  if (bwd) return RB == 8 ? (const void*)bwd_run_ring<8> : (const void*)bwd_run_ring<16>;
  return RB == 8 ? (const void*)fwd_run_ring<8> : (const void*)fwd_run_ring<16>;
}
int threads(bool bwd, int RB) {
  if (bwd) return RB == 8 ? BwdShape<8>::THREADS : BwdShape<16>::THREADS;
  return RB == 8 ? FwdShape<8>::THREADS : FwdShape<16>::THREADS;
}
int smem_bytes(bool bwd, int RB, int H) {
  const int KT = bwd ? 2 * ring_ctas(H) / RING_CLUSTER : (H + 63) / 64;
  if (bwd) return lone_smem((int)(RB == 8 ? BwdShape<8>::total(KT) : BwdShape<16>::total(KT)));
  return lone_smem((int)(RB == 8 ? FwdShape<8>::total(KT) : FwdShape<16>::total(KT)));
}
int fwd_ctas(int H) { return (H + CU - 1) / CU; }

}  // namespace

RingArgs ring_args(char* rings, int H, int B, bool backward, int id, bool fault, uint32_t poll_limit) {
  const size_t rows = (size_t)ring_slot_rows(B), row = (size_t)ring_ctas(H) * CU * 2;
  const size_t fwd = RING_SLOTS * rows * row, bwd = 4 * fwd;      // bytes of a set
  char* const first = rings + (backward ? 2 * fwd : 0);
  const size_t set = backward ? bwd : fwd;
  return RingArgs{first + (size_t)(id & 1) * set, first + (size_t)(~id & 1) * set, rings + 2 * fwd + 2 * bwd, fault ? 1u : 0u, poll_limit, 0};
}

RingFit ring_fit(int B, int H) {
  const int sms = run_sms();
  RingFit best{0, 0};
  for (int RB : {8, 16}) {
    const int groups = (B + RB - 1) / RB;
    int at_once = sms / fwd_ctas(H);
    for (int dir = 0; dir < 2; ++dir) {
      const void* fn = kernel(dir != 0, RB);
      if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes(dir != 0, RB, 32 * CU)) != cudaSuccess) { cudaGetLastError(); return RingFit{0, 0}; }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ring_ctas(H)); cfg.blockDim = dim3((unsigned)threads(true, RB)); cfg.dynamicSmemBytes = (size_t)smem_bytes(true, RB, H);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = RING_CLUSTER; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel(true, RB), &cfg) != cudaSuccess) { cudaGetLastError(); return RingFit{0, 0}; }
    if (n * RING_CLUSTER > sms) n = sms / RING_CLUSTER;
    if (n * RING_CLUSTER / ring_ctas(H) < at_once) at_once = n * RING_CLUSTER / ring_ctas(H);
    if (at_once >= groups) return RingFit{RB, groups};
    if (at_once > 0) best = RingFit{RB, at_once};   // in turns: of more rows, fewer
  }
  return best;
}

int ring_smem(bool backward, int H, int rows) { return smem_bytes(backward, rows, H); }

cudaError_t ring_forward(const CUtensorMap& tm_w, const ClusterFwdArgs& a, const RingArgs& r, RingFit fit, cudaStream_t s) {
  int ncta = fwd_ctas(a.H), KT0 = ring_first_part_blocks(a.H);
  const int groups = (a.B + fit.rows - 1) / fit.rows;
  cudaError_t e = cudaSuccess;
  RingArgs g = r;
  for (g.first = 0; g.first < groups && e == cudaSuccess; g.first += fit.groups) {
    const int n = groups - g.first < fit.groups ? groups - g.first : fit.groups;
    void* args[] = {(void*)&tm_w, (void*)&a, (void*)&g, (void*)&ncta, (void*)&KT0};
    e = launch_coop(kernel(false, fit.rows), n * ncta, threads(false, fit.rows), (size_t)smem_bytes(false, fit.rows, a.H), s, args, 1);
  }
  return e;
}

cudaError_t ring_backward(const CUtensorMap& tm_wt, const ClusterBwdArgs& a, const RingArgs& r, RingFit fit, cudaStream_t s) {
  int ncta = ring_ctas(a.H);
  const int groups = (a.B + fit.rows - 1) / fit.rows;
  cudaError_t e = cudaSuccess;
  RingArgs g = r;
  for (g.first = 0; g.first < groups && e == cudaSuccess; g.first += fit.groups) {
    const int n = groups - g.first < fit.groups ? groups - g.first : fit.groups;
    void* args[] = {(void*)&tm_wt, (void*)&a, (void*)&g, (void*)&ncta};
    e = launch_coop(kernel(true, fit.rows), n * ncta, threads(true, fit.rows), (size_t)smem_bytes(true, fit.rows, a.H), s, args, RING_CLUSTER, false);
  }
  return e;
}

}  // namespace tc
}  // namespace mebptt
