// Batched-over-time contractions on the tensor cores: C[M][N] (+)= sum_k A(m,k) B(n,k) with
// bfloat16 operands and float32 accumulation in TMEM.
//
// These are the parts of the training step that do not sit on the recurrence and can therefore
// be run for many time steps at once:
//   input projection   Zx[(s,b)][g]  = sum_i x[(s,b)][i] W_ih[g][i] + bias[g]         (A, B K-major)
//   readout            y[(s,b)][o]   = sum_j h[(s,b)][j] W_out[o][j]                 (A, B K-major)
//   readout backward   dha[(s,b)][j] = sum_o dy[(s,b)][o] W_out^T[j][o]              (A, B K-major)
//   weight gradients   dW[g][c]     += sum_(s,b) dz[(s,b)][g] in[(s,b)][c]           (A, B MN-major)
// "K-major" means the operand is stored with the contraction index contiguous; "MN-major" that it
// is stored [k][m] (rows are contraction indices), which is how dz and the layer inputs lie in
// memory for the weight gradient, so no transposed copies are made.
//
// One CTA computes one 128 x 128 tile (128 x 32 where C is short and wide: see gemm_bf16).  A single thread feeds a ring of
// 128-byte swizzled shared-memory tiles by TMA (64 contraction indices per tile, one or three tiles per stage); a single thread issues
// tcgen05.mma (M = 128, N = 128, K = 16, four per tile) into a 128-column TMEM accumulator and
// releases ring slots with tcgen05.commit; then all four warps read the accumulator with
// tcgen05.ld (warp w owns TMEM lanes 32w .. 32w+31 = tile rows) and write the tile.
// Out-of-range parts of a tile are zero-filled by TMA on the way in and masked on the way out.
// The sum over k runs in one fixed order, so results do not depend on how callers batch steps.
#include <cstdlib>
#include <type_traits>

#include "launch.hpp"
#include "sm100.cuh"
#include "tc.hpp"
#include "tmap.hpp"

namespace mebptt {
namespace tc {

namespace {

using namespace sm100;

constexpr int BM = 128, BK = 64, MAX_STAGES = 6;
constexpr int DEEP_TILES = 3;                  // tiles of a stage of the deep rings
constexpr int BN_WIDE = 128, BN_NARROW = 32;   // tile widths; narrow tiles spread a short-and-wide C over more SMs
constexpr int A_BYTES = BM * BK * 2;
constexpr int gemm_smem(int stages, int bn, int tps) { return stages * tps * (A_BYTES + bn * BK * 2) + 1024; }  // + slack to align the ring to 1024 B

// HALVES with K-major operands: an instance whose loss epilogue writes dy in halves.  (Its registers and instructions in the
// other instances' epilogue cost bf16 training steps 0.4 %; an instance of its own for the bf16 loss, too, costs 1 %:
// its loads of the targets are then fewer in flight.)
// Four CTAs an SM would be more than shared memory holds: the bound lets the compiler keep up to 128 registers,
// so that more of an epilogue's loads are in flight, and the instances with an MN-major operand (the gradients)
// have no loss epilogue (H = 1024, full memory with dx: 12.30 -> 12.22 ms; MSM m = 100: 18.13 -> 18.03 ms).
// HALVES with MN-major operands: both lie in halves, and the contraction is walked three times, mid hi, hi mid,
// hi hi, each a shift of the columns that the copies start at.  What bounds a weight gradient of few rows is not
// the products but a launch's filling of its ring and its pass over C, of which there were three (H = 1024, t = 4000,
// ISM m = 50: 122.9 -> 119.6 ms).  The small products come first, so that the accumulator holds no more than before
// while hi hi is added up.
// TPS: tiles of 64 contraction indices per stage.  A grid of at most one wave has an SM for each tile of C, and one tile a
// stage then passes at 60 to 100 GB/s an SM, however many stages there are: what takes the time is a stage's way
// through its two barriers and the requests of its copies.  Three tiles a stage, requested together, come near what an
// SM takes in (120 GB/s); us, one, two and three tiles a stage in 192 KB (narrow tiles of C: 120): 288 x 256, K = 3072
// 16.7, 12.0, 10.1; 128 x 8192, K = 2048 14.7, 12.1, 11.2; 4096 x 256, MN-major, K = 2048 17.4, 13.4, 12.5.  (Two
// threads that request: no change.)  More tiles of C than SMs: one a stage, so that two CTAs share an SM and one's epilogue overlaps the other's products (2048 x 4096, K = 256: 13.4
// against 20.7; 8192 x 8192, K = 4096: 489 against 629).
// `blocks`: bit 0 (1): the map of A (B) sees 64 columns as a block of its own (make_tmap_blocks64), and one copy brings
// all tiles of a stage; without it, where the columns are no whole number of blocks, one copy each.
template <bool A_MN, bool B_MN, int BN = BN_WIDE, bool HALVES = false, int TPS = 1>
__global__ void __launch_bounds__(128, 4) gemm_bf16_kernel(const __grid_constant__ CUtensorMap tma,
                                                        const __grid_constant__ CUtensorMap tmb, GemmOut out,
                                                        int M, int N, int K, int STAGES, int* status,
                                                        float* partial, int fault, int blocks, GemmHalves halves) {
  constexpr bool SEGMENTS = HALVES && A_MN && B_MN;
  constexpr int B_BYTES = BN * BK * 2, STAGE_BYTES = TPS * (A_BYTES + B_BYTES);
  static_assert(BN == BN_WIDE || (!A_MN && !B_MN), "narrow tiles exist for K-major operands only");
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[MAX_STAGES], empty[MAX_STAGES], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int failed;

  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  // this CTA's part of the contraction index: blocks [kb_lo, kb_lo + nk) of 64 (in halves: all of them, three times)
  const int splits = gridDim.z;
  const int nk_all = (K + BK - 1) / BK;
  const int kb_lo = (int)((int64_t)nk_all * blockIdx.z / splits);
  const int nk = (int)((int64_t)nk_all * (blockIdx.z + 1) / splits) - kb_lo;
  const int n_one = (nk + TPS - 1) / TPS, n_st = SEGMENTS ? 3 * n_one : n_one;   // stages: of one walk, in all
  const int tile = blockIdx.y * gridDim.x + blockIdx.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(&done, 1);
    failed = 0;
    mbar_fence_init();
    tma_prefetch_desc(&tma);
    tma_prefetch_desc(&tmb);
  }
  if (warp == 1) tmem_alloc(&tmem_slot, BN);
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  grid_dep_wait();     // operands (and, when accumulating, C) come from the kernels before this one
  grid_dep_launch();

  if (warp == 0 && lane == 0) {
    // ---- producer -----------------------------------------------------------------------
    int armed = 0;  // stages whose full barrier still awaits bytes (for the failure path)
    for (int st = 0; st < n_st; ++st) {
      const int s = st % STAGES;
      if (st >= STAGES && !mbar_wait(&empty[s], ((st / STAGES) - 1) & 1)) { failed = 1; break; }
      uint8_t* sA = ring + s * STAGE_BYTES;
      uint8_t* sB = sA + TPS * A_BYTES;
      // (fault: a testing aid -- the first stage is told to expect 16 bytes that never come, so the
      // issuer's bounded wait runs out and the kernel leaves through its failure path)
      mbar_arrive_expect_tx(&full[s], STAGE_BYTES + ((fault && st == 0) ? 16u : 0u));
      ++armed;
      const int seg = SEGMENTS ? st / n_one : 2;
      const int k0 = kb_lo + (st - (SEGMENTS ? seg * n_one : 0)) * TPS;       // first tile of the stage
      const int ma = m0 + (seg == 0 ? halves.a : 0), nb = n0 + (seg == 1 ? halves.b : 0);
      if (A_MN) {
        if (blocks & 1) tma_load_3d(sA, &tma, 0, k0 * BK, ma / 64, &full[s]);
        else for (int q = 0; q < 2; ++q) tma_load_2d(sA + q * TPS * 8192, &tma, ma + 64 * q, k0 * BK, &full[s]);
      } else if (TPS > 1 && (blocks & 1)) {
        tma_load_3d(sA, &tma, 0, m0, k0, &full[s]);
      } else {
        for (int t = 0; t < TPS; ++t) tma_load_2d(sA + t * A_BYTES, &tma, (k0 + t) * BK, m0, &full[s]);
      }
      if (B_MN) {
        if (blocks & 2) tma_load_3d(sB, &tmb, 0, k0 * BK, nb / 64, &full[s]);
        else for (int q = 0; q < 2; ++q) tma_load_2d(sB + q * TPS * 8192, &tmb, nb + 64 * q, k0 * BK, &full[s]);
      } else if (TPS > 1 && (blocks & 2)) {
        tma_load_3d(sB, &tmb, 0, n0, k0, &full[s]);
      } else {
        for (int t = 0; t < TPS; ++t) tma_load_2d(sB + t * B_BYTES, &tmb, (k0 + t) * BK, n0, &full[s]);
      }
    }
    (void)armed;
  } else if (warp == 1) {
    // ---- MMA issuer: the whole warp walks the loop (descriptors stay in uniform registers), one
    // elected lane issues --------------------------------------------------------------------------
    constexpr uint32_t idesc = make_idesc(1, BM, BN, A_MN, B_MN);
    // K-major: 16 contraction indices = 32 B along the row; MN-major: 16 rows of 128 B
    constexpr uint32_t A_STEP = A_MN ? (2048 >> 4) : (32 >> 4), B_STEP = B_MN ? (2048 >> 4) : (32 >> 4);
    // tiles of a stage: K-major side by side, MN-major 64 rows apart
    constexpr uint32_t A_TILE = (A_MN ? 8192 : A_BYTES) >> 4, B_TILE = (B_MN ? 8192 : B_BYTES) >> 4;
    const uint32_t ring0 = smem_u32(ring);
    const uint64_t a_desc0 = A_MN ? make_desc_sw128(ring0, TPS * 8192, 1024) : make_desc_sw128(ring0, 16, 1024);
    const uint64_t b_desc0 = B_MN ? make_desc_sw128(ring0 + TPS * A_BYTES, TPS * 8192, 1024) : make_desc_sw128(ring0 + TPS * A_BYTES, 16, 1024);
    bool ok = true;
    for (int st = 0; st < n_st && ok; ++st) {
      const int s = st % STAGES;
      if (!mbar_wait(&full[s], (st / STAGES) & 1)) { failed = 1; ok = false; break; }
      tc_fence_after_sync();
      const int live = nk - (SEGMENTS ? st % n_one : st) * TPS;     // tiles from this stage's first on (the last stage may have fewer than TPS)
      if (elect_one()) {
        const uint64_t da = a_desc0 + (uint64_t)(s * (STAGE_BYTES >> 4)), db = b_desc0 + (uint64_t)(s * (STAGE_BYTES >> 4));
#pragma unroll
        for (int t = 0; t < TPS; ++t) {
          if (TPS > 1 && t >= live) break;
#pragma unroll
          for (int k4 = 0; k4 < BK / 16; ++k4)
            mma_f16(tmem, da + (uint64_t)(t * A_TILE + k4 * A_STEP), db + (uint64_t)(t * B_TILE + k4 * B_STEP), idesc,
                    (st > 0 || t > 0 || k4 > 0) ? 1u : 0u);
        }
        mma_commit(&empty[s]);  // the slot may be refilled once these MMAs have read it
      }
      __syncwarp();
    }
    if (elect_one()) mma_commit(&done);
    __syncwarp();
  }

  // ---- epilogue: all four warps ---------------------------------------------------------
  __syncwarp();
  bool ok = mbar_wait(&done, 0);
  tc_fence_after_sync();
  bool finish = ok && !failed;
  if (finish && splits > 1) {
    // a part of a contraction split along K: the raw float32 tile goes to the scratch, and a
    // second kernel adds the parts in index order
    float* mine = partial + (((size_t)tile * splits + blockIdx.z) * BM + (size_t)(warp * 32 + lane)) * BN;
#pragma unroll 1
    for (int c = 0; c < BN / 32; ++c) {
      uint32_t r[32];
      tmem_ld_32x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), r);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *(reinterpret_cast<float4*>(mine + c * 32) + j) =
            make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                        __uint_as_float(r[4 * j + 3]));
    }
    finish = false;
  }
  auto load_acc = [&](int c, uint32_t (&r)[32]) {
    tmem_ld_32x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), r);
    tmem_ld_wait();
  };
  if (finish) {
    // Float32 tiles whose rows can be written as aligned float4: each warp parks its 32 x 128
    // block of the accumulator in the (now idle) operand ring, then writes -- or adds to -- one
    // whole 512-byte row of C per instruction.  Everything else takes the per-thread path below.
    const bool wide = BN == BN_WIDE && out.kind != GemmOut::STORE_BF16 && out.kind != GemmOut::LOSS_DY && (out.ld % 4 == 0) &&
                      ((reinterpret_cast<uintptr_t>(out.ptr) & 15) == 0) && (n0 % 4 == 0) &&
                      ((reinterpret_cast<uintptr_t>(out.bias) & 15) == 0);
    if (wide) {
      constexpr int PITCH = BN + 4;   // floats; keeps both the parking and the row reads conflict-free
      float* park = reinterpret_cast<float*>(ring) + (size_t)warp * 32 * PITCH;
#pragma unroll 1
      for (int c = 0; c < BN / 32; ++c) {
        uint32_t r[32];
        load_acc(c, r);
        float4* dst = reinterpret_cast<float4*>(park + (size_t)lane * PITCH + c * 32);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          dst[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]),
                               __uint_as_float(r[4 * j + 3]));
      }
      __syncwarp();
      const int col = n0 + lane * 4;
      const bool col_ok = col + 3 < N;       // N % 4 == 0 is implied by ld % 4 == 0 only for ld == N: check
      float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
      if (out.bias && col_ok) bv = *reinterpret_cast<const float4*>(out.bias + col);
      float* base = reinterpret_cast<float*>(out.ptr);
#pragma unroll 1
      for (int r0 = 0; r0 < 32; r0 += 8) {
        float4 old[8];
        size_t off[8];
        bool live[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int row = m0 + warp * 32 + r0 + j;
          const int row_o = out.perm_h ? ((row & 3) * out.perm_h + (row >> 2)) : row;
          live[j] = row < M && col_ok;
          off[j] = (size_t)row_o * out.ld + col;
          old[j] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (live[j] && out.kind == GemmOut::ACCUM_F32) old[j] = *reinterpret_cast<const float4*>(base + off[j]);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (!live[j]) continue;
          const float4 v = *reinterpret_cast<const float4*>(park + (size_t)(r0 + j) * PITCH + lane * 4);
          *reinterpret_cast<float4*>(base + off[j]) =
              make_float4(v.x + bv.x + old[j].x, v.y + bv.y + old[j].y, v.z + bv.z + old[j].z, v.w + bv.w + old[j].w);
        }
      }
      // columns of a ragged right edge (N not a multiple of 4 inside this tile)
      if (!col_ok && col < N) {
        for (int r0 = 0; r0 < 32; ++r0) {
          const int row = m0 + warp * 32 + r0;
          if (row >= M) break;
          const int row_o = out.perm_h ? ((row & 3) * out.perm_h + (row >> 2)) : row;
          for (int j = 0; j < 4 && col + j < N; ++j) {
            float v = park[(size_t)r0 * PITCH + lane * 4 + j];
            if (out.bias) v += out.bias[col + j];
            float* q = base + (size_t)row_o * out.ld + col + j;
            if (out.kind == GemmOut::ACCUM_F32) v += *q;
            *q = v;
          }
        }
      }
    } else {
    const int row = m0 + warp * 32 + lane;
    const int row_o = out.perm_h ? ((row & 3) * out.perm_h + (row >> 2)) : row;
#pragma unroll 1
    for (int c = 0; c < BN / 32; ++c) {
      uint32_t r[32];
      load_acc(c, r);
      const int col0 = n0 + c * 32;
      if (!A_MN && !B_MN && out.kind == GemmOut::LOSS_DY) {
        // squared-error loss fused into the readout: this lane's row against its targets, columns in
        // ascending order, then the 32 rows of the warp in a fixed butterfly order
        float sq = 0.f;
        if (row < M) {
          const float* tp = out.target + (size_t)row * out.ld + col0;
          // halves: a row is [hi | hi | mid], each as wide as C
          __nv_bfloat16* dp = HALVES ? reinterpret_cast<__nv_bfloat16*>(out.dy3) + (size_t)row * 3 * out.ld + col0
                                     : reinterpret_cast<__nv_bfloat16*>(out.ptr) + (size_t)row * out.ld + col0;
          const float two = 2.f * out.scale;
          if (col0 + 32 <= N && ((reinterpret_cast<uintptr_t>(tp) & 15) == 0) && ((reinterpret_cast<uintptr_t>(dp) & 15) == 0) &&
              ((reinterpret_cast<uintptr_t>(out.bias) & 15) == 0) && (!HALVES || out.ld % 8 == 0)) {
            float4 t4[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) t4[j] = *reinterpret_cast<const float4*>(tp + 4 * j);
            uint32_t packed[16];
            [[maybe_unused]] uint32_t rest[16];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float4 bv = make_float4(0.f, 0.f, 0.f, 0.f);
              if (out.bias) bv = *reinterpret_cast<const float4*>(out.bias + col0 + 4 * j);
              const float d0 = (__uint_as_float(r[4 * j]) + bv.x) - t4[j].x;
              const float d1 = (__uint_as_float(r[4 * j + 1]) + bv.y) - t4[j].y;
              const float d2 = (__uint_as_float(r[4 * j + 2]) + bv.z) - t4[j].z;
              const float dd = (__uint_as_float(r[4 * j + 3]) + bv.w) - t4[j].w;
              sq = fmaf(d0, d0, sq); sq = fmaf(d1, d1, sq); sq = fmaf(d2, d2, sq); sq = fmaf(dd, dd, sq);
              packed[2 * j] = pack_bf16x2(d0 * two, d1 * two);
              packed[2 * j + 1] = pack_bf16x2(d2 * two, dd * two);
              if constexpr (HALVES) {
                const float2 h0 = unpack_bf16x2(packed[2 * j]), h1 = unpack_bf16x2(packed[2 * j + 1]);
                rest[2 * j] = pack_bf16x2(d0 * two - h0.x, d1 * two - h0.y);
                rest[2 * j + 1] = pack_bf16x2(d2 * two - h1.x, dd * two - h1.y);
              }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint4 v = make_uint4(packed[4 * j], packed[4 * j + 1], packed[4 * j + 2], packed[4 * j + 3]);
              *reinterpret_cast<uint4*>(dp + 8 * j) = v;
              if constexpr (HALVES) {
                *reinterpret_cast<uint4*>(dp + out.ld + 8 * j) = v;
                *reinterpret_cast<uint4*>(dp + 2 * out.ld + 8 * j) = make_uint4(rest[4 * j], rest[4 * j + 1], rest[4 * j + 2], rest[4 * j + 3]);
              }
            }
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (col0 + j < N) {
                const float d = (__uint_as_float(r[j]) + (out.bias ? out.bias[col0 + j] : 0.f)) - tp[j];
                sq = fmaf(d, d, sq);
                const __nv_bfloat16 hi = __float2bfloat16_rn(d * two);
                dp[j] = hi;
                if constexpr (HALVES) {
                  dp[out.ld + j] = hi;
                  dp[2 * out.ld + j] = __float2bfloat16_rn(d * two - __bfloat162float(hi));
                }
              }
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (lane == 0 && m0 + warp * 32 < M && col0 < N)
          out.loss_part[(size_t)((m0 + warp * 32) / 32) * out.parts + col0 / 32] = sq * out.scale;
      } else if (row < M) {
        if (out.kind == GemmOut::STORE_BF16) {
          __nv_bfloat16* p = reinterpret_cast<__nv_bfloat16*>(out.ptr) + (size_t)row_o * out.ld + col0;
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (col0 + j < N) p[j] = __float2bfloat16_rn(__uint_as_float(r[j]));
        } else {
          float* p = reinterpret_cast<float*>(out.ptr) + (size_t)row_o * out.ld + col0;
          const bool vec = (col0 + 32 <= N) && ((reinterpret_cast<uintptr_t>(p) & 15) == 0) &&
                           ((reinterpret_cast<uintptr_t>(out.bias) & 15) == 0);
          if (vec) {
            // all eight loads of the old values first, so that their latencies overlap
            float4 o[8];
            if (out.kind == GemmOut::ACCUM_F32) {
#pragma unroll
              for (int j = 0; j < 8; ++j) o[j] = *reinterpret_cast<const float4*>(p + 4 * j);
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) o[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float4 v = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                     __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
              if (out.bias) {
                const float4 bv = *reinterpret_cast<const float4*>(out.bias + col0 + 4 * j);
                v.x += bv.x; v.y += bv.y; v.z += bv.z; v.w += bv.w;
              }
              v.x += o[j].x; v.y += o[j].y; v.z += o[j].z; v.w += o[j].w;
              *reinterpret_cast<float4*>(p + 4 * j) = v;
            }
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (col0 + j < N) {
                float v = __uint_as_float(r[j]);
                if (out.bias) v += out.bias[col0 + j];
                if (out.kind == GemmOut::ACCUM_F32) v += p[j];
                p[j] = v;
              }
          }
        }
      }
    }
    }
  } else if ((!ok || failed) && status && threadIdx.x == 0) {
    *status = MEBPTT_ERR_TIMEOUT;
  }
  // On the failure path the producer may still have loads in flight: give them a bounded
  // chance to land before the shared memory goes away.
  if (failed && warp == 0 && lane == 0)
    for (int s = 0; s < STAGES; ++s) (void)mbar_wait(&full[s], 0);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, BN);
}

// C[m][n] = sum over the parts, in index order, of a contraction that was split along K.
// partial: [tile][part][128][bn] with tile = (m / 128) * tiles_x + n / bn.  One thread per four
// adjacent columns.
__global__ void splitk_reduce(const float* partial, int splits, int M, int N, int tiles_x, int bn, float* out, int64_t ld) {
  grid_dep_wait();
  grid_dep_launch();
  const int n4 = (N + 3) / 4;
  const size_t total = (size_t)M * n4;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(e / n4), n = (int)(e % n4) * 4;
    const int tile = (m / BM) * tiles_x + n / bn;
    const float* p = partial + (((size_t)tile * splits) * BM + (size_t)(m % BM)) * bn + (n % bn);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z = 0; z < splits; ++z) {
      const float4 v = *reinterpret_cast<const float4*>(p + (size_t)z * BM * bn);
      acc.x += v.x; acc.y += v.y; acc.z += v.z; acc.w += v.w;
    }
    float* q = out + (size_t)m * ld + n;
    if (n + 3 < N) *reinterpret_cast<float4*>(q) = acc;
    else {
      const float a[4] = {acc.x, acc.y, acc.z, acc.w};
      for (int j = 0; j < 4 && n + j < N; ++j) q[j] = a[j];
    }
  }
}

}  // namespace

// Few tiles and a long contraction index: split K so that about a wave of CTAs streams the
// operands, each part at least 8 blocks of 64 long; a second kernel adds the parts.  Only where at
// least four parts come out of it: below that the extra pass costs more than it saves.
int gemm_split_count(bool a_mn, bool b_mn, int M, int N, int K, size_t partial_floats) {
  if (env::no_splitk()) return 1;
  const int wide_tiles = ((N + BN_WIDE - 1) / BN_WIDE) * ((M + BM - 1) / BM);
  const bool narrow = !a_mn && !b_mn && wide_tiles <= 37 && N >= 2 * BN_NARROW;
  const int BN = narrow ? BN_NARROW : BN_WIDE;
  const int tiles = ((N + BN - 1) / BN) * ((M + BM - 1) / BM);
  const int nk = (K + BK - 1) / BK;
  int want = 148 / tiles;
  if (want > nk / 8) want = nk / 8;
  if (want > 16) want = 16;
  while (want > 1 && (size_t)tiles * want * BM * BN > partial_floats) --want;
  return want >= 4 ? want : 1;
}

int gemm_split_count_deferred(int M, int N, int K) {
  if (env::no_splitk()) return 1;
  const int tiles = ((N + BN_WIDE - 1) / BN_WIDE) * ((M + BM - 1) / BM);
  const int nk = (K + BK - 1) / BK;
  int want = 148 / tiles;
  if (want > nk / 8) want = nk / 8;
  if (want > 16) want = 16;
  return want >= 2 ? want : 1;
}

int gemm_bf16(const void* A, int64_t lda, bool a_mn, const void* B, int64_t ldb, bool b_mn, const GemmOut& out,
              int M, int N, int K, int* status, cudaStream_t s, bool early, const SplitWs* split, int force_splits,
              SplitParts* defer, const GemmHalves* halves) {
  if (M <= 0 || N <= 0 || K <= 0) return MEBPTT_ERR_ARG;
  if (halves && !(a_mn && b_mn && out.kind == GemmOut::ACCUM_F32 && !split && halves->a % 8 == 0 && halves->b % 8 == 0))
    return MEBPTT_ERR_ARG;
  const bool loss = out.kind == GemmOut::LOSS_DY;
  if (loss && (a_mn || b_mn || !(out.dy3 || out.ptr))) return MEBPTT_ERR_ARG;
  // A short-and-wide product over K-major operands (a few steps' worth of rows against a whole
  // weight matrix) gives few 128-wide tiles, each streaming all of K through one SM: 32-wide tiles
  // put four times as many SMs to work on the same bytes.
  const int wide_tiles = ((N + BN_WIDE - 1) / BN_WIDE) * ((M + BM - 1) / BM);
  const bool narrow = !a_mn && !b_mn && wide_tiles <= 37 && N >= 2 * BN_NARROW && !(defer && force_splits > 1);
  const int BN = narrow ? BN_NARROW : BN_WIDE;
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
  int splits = 1;
  if (split && split->partial && (out.kind == GemmOut::STORE_F32 || (defer && out.kind == GemmOut::ACCUM_F32)) &&
      !out.bias && !out.perm_h && out.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(out.ptr) & 15) == 0)
    splits = force_splits > 0 ? force_splits : gemm_split_count(a_mn, b_mn, M, N, K, split->partial_floats);
  else if (force_splits > 1)
    return MEBPTT_ERR_ARG;
  if (splits > 1 && (size_t)grid.x * grid.y * splits * BM * BN > split->partial_floats) return MEBPTT_ERR_WORKSPACE;
  grid.z = splits;
  // Grids of at most one wave: two stages of three tiles (a contraction that is longer than both) or six of one, one CTA
  // an SM.  Six as well where both operands are K-major rows of no whole blocks of 64 and the tiles wide: three tiles then take a
  // copy each, six in a row, and nothing is gained (us, one and three a stage: 1024 x 1024, K = 456 8.8, 9.0; 520 x 2080,
  // K = 600 9.8, 10.1 and K = 1992 18.2, 18.5; narrow tiles, 288 x 256, K = 1992 14.1, 12.3).  Larger grids: three stages of
  // one tile, two CTAs per SM, so that one's epilogue overlaps the other's main loop.
  const bool one_wave = grid.x * grid.y * grid.z <= 148;
  const int nk = (halves ? 3 : 1) * (((K + BK - 1) / BK + splits - 1) / splits);
  const bool copy_each = !a_mn && !b_mn && K % 64 != 0;
  const int tps = one_wave && nk > MAX_STAGES && (narrow || !copy_each) ? DEEP_TILES : 1;
  const int stages = tps > 1 ? MAX_STAGES / DEEP_TILES : one_wave ? MAX_STAGES : 3;
  CUtensorMap ta, tb;
  int blocks = 0;
  // K-major: tensor is [M][K], box 64 (k) x tile rows, `tps` of them.  MN-major: tensor is [K][M], box 64 (m) x 64 tps rows, two of
  // them.  In halves the map spans the whole row; what a tile at the edge takes from the neighbouring half goes only
  // into rows and columns that are not written.
  auto encode = [&](CUtensorMap* t, const void* p, bool mn, int rows, int off, int64_t ld, int tile, int bit) {
    const uint64_t cols = mn ? (uint64_t)(rows + off) : (uint64_t)K, n = mn ? (uint64_t)K : (uint64_t)rows;
    const uint32_t high = (uint32_t)(mn ? BK * tps : tile);
    if ((mn || tps > 1) && cols % 64 == 0 && off % 64 == 0) {
      blocks |= bit;
      return make_tmap_blocks64(t, p, cols, n, (uint64_t)ld * 2, high, mn ? 2u : (uint32_t)tps);
    }
    return make_tmap_2d(t, p, 2, cols, n, (uint64_t)ld * 2, 64, high);
  };
  if (!encode(&ta, A, a_mn, M, halves ? halves->a : 0, lda, BM, 1) || !encode(&tb, B, b_mn, N, halves ? halves->b : 0, ldb, BN, 2))
    return MEBPTT_ERR_UNSUPPORTED;
  const int smem = gemm_smem(stages, BN, tps);
  const bool loss3 = loss && out.dy3;
  auto pick = [&](auto t) {
    constexpr int T = decltype(t)::value;
    return halves ? gemm_bf16_kernel<true, true, BN_WIDE, true, T>
           : loss3 ? (narrow ? gemm_bf16_kernel<false, false, BN_NARROW, true, T> : gemm_bf16_kernel<false, false, BN_WIDE, true, T>)
           : narrow ? gemm_bf16_kernel<false, false, BN_NARROW, false, T>
           : a_mn ? (b_mn ? gemm_bf16_kernel<true, true, BN_WIDE, false, T> : gemm_bf16_kernel<true, false, BN_WIDE, false, T>)
                  : (b_mn ? gemm_bf16_kernel<false, true, BN_WIDE, false, T> : gemm_bf16_kernel<false, false, BN_WIDE, false, T>);
  };
  auto* fn = tps > 1 ? pick(std::integral_constant<int, DEEP_TILES>()) : pick(std::integral_constant<int, 1>());
  static const bool attrs = [] {
    auto set = [](auto t) {
      constexpr int T = decltype(t)::value;
      const int wide = gemm_smem(MAX_STAGES, BN_WIDE, 1), narrow = gemm_smem(MAX_STAGES, BN_NARROW, 1);
      const cudaFuncAttribute most = cudaFuncAttributeMaxDynamicSharedMemorySize;
      cudaFuncSetAttribute(gemm_bf16_kernel<true, true, BN_WIDE, false, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<true, true, BN_WIDE, true, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<false, false, BN_WIDE, false, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<true, false, BN_WIDE, false, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<false, true, BN_WIDE, false, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<false, false, BN_NARROW, false, T>, most, narrow);
      cudaFuncSetAttribute(gemm_bf16_kernel<false, false, BN_WIDE, true, T>, most, wide);
      cudaFuncSetAttribute(gemm_bf16_kernel<false, false, BN_NARROW, true, T>, most, narrow);
    };
    set(std::integral_constant<int, 1>());
    set(std::integral_constant<int, DEEP_TILES>());
    return true;
  }();
  (void)attrs;
  const cudaError_t e = launch_on(early, fn, grid, dim3(128), (size_t)smem, s, ta, tb, out, M, N, K, stages, status,
                                  splits > 1 ? split->partial : nullptr, (wait_fault_mask() & 4) ? 1 : 0, blocks,
                                  halves ? *halves : GemmHalves{});
  if (e != cudaSuccess) {
    cudaGetLastError();
    return MEBPTT_ERR_CUDA;
  }
  if (defer) *defer = splits > 1 ? SplitParts{split->partial, splits, (int)grid.x, BN} : SplitParts{};
  if (splits > 1 && !defer) {
    const size_t quads = (size_t)M * ((N + 3) / 4);
    const int blocks = (int)((quads + 255) / 256 > 1184 ? 1184 : (quads + 255) / 256);
    const cudaError_t e2 = launch_on(early, splitk_reduce, dim3(blocks), dim3(256), 0, s, (const float*)split->partial,
                                     splits, M, N, (int)grid.x, BN, reinterpret_cast<float*>(out.ptr), out.ld);
    if (e2 != cudaSuccess) {
      cudaGetLastError();
      return MEBPTT_ERR_CUDA;
    }
  }
  return MEBPTT_OK;
}

}  // namespace tc
}  // namespace mebptt
