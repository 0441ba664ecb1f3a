// The pod kernel (pod.hpp has the scheme).
//
// A phase: wait for the pushes of the phase before; gradients of the own units (B); products, over warps;
// states of the own units (F) and readouts (R), a thread per unit and batch row; pushes; fetch what the
// next phase needs from memory.  What bounds it is that chain: the contraction of a phase is a few
// hundred instructions of a warp, so the number of instructions in a row counts, and the trip of a push
// to another SM and back into a register.
//
// The bytes that arrive are all the CTAs have to agree on: each knows how many a phase brings, and every
// CTA also sends a word to every other once it has read its operands.  A CTA that has everything of phase
// p therefore knows that nobody reads operands of phase p any more: what is pushed in phase p + 1 may
// take the place of anything last read in phase p.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "launch.hpp"
#include "layout.hpp"
#include "pod.hpp"
#include "pod_run.hpp"
#include "sm100.cuh"
#include "team_dev.cuh"

namespace mebptt {
namespace pod {

using bf16 = __nv_bfloat16;
using team::cell_backward;
using team::cell_forward;
using team::lane_sums;
using team::load4;
using team::part;
using team::States;
using team::store;
using team::to_f;

namespace {

__device__ __forceinline__ uint32_t remote(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void push(uint32_t addr, uint32_t a, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(a), "r"(bar) : "memory");
}
__device__ __forceinline__ void push2(uint32_t addr, uint32_t a, uint32_t b, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(addr), "r"(a), "r"(b), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void push4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(a), "r"(b),
               "r"(c), "r"(d), "r"(bar)
               : "memory");
}
// (The hint lets the hardware hold the warp until the barrier turns, for 20 us a time, instead of having it
// poll: sixteen polling warps take issue slots from the ones that still work.)
__device__ __forceinline__ bool wait_for(uint32_t bar, uint32_t parity, uint32_t polls) {
  for (uint32_t i = 0; i < polls; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(20000u) : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// ---- products ------------------------------------------------------------------------------

// F and R on FMA: four weight rows against NB operand rows over the 128-wide slices [lo, hi) of [input | h].
// Lanes split the contraction index; the sums of unit / row group g, part s go to red[(g ns + s)][NB][4].
template <int NB>
__device__ __forceinline__ void rows_fma(const float* in, int pin, int nin, const float* h, int ph, int nh, const float* w, int ldw, int groups,
                                         int lg, float* red, int wk, int lane) {
  const int ns = 1 << lg, ia = (nin + 31) >> 5, its = ia + ((nh + 31) >> 5);
  for (; wk < groups * ns; wk += kWarps) {
    const int g = wk >> lg, s = wk & (ns - 1);
    const int lo = its * s >> lg, hi = its * (s + 1) >> lg;
    const float* wg = w + (size_t)g * 4 * ldw;
    float acc[NB * 4];
#pragma unroll
    for (int q = 0; q < NB * 4; ++q) acc[q] = 0.f;
#pragma unroll 1
    for (int i = lo; i < hi; ++i) {
      const bool first = i < ia;
      const int v = (first ? i : i - ia) * 32 + lane;
      if (v < (first ? nin : nh)) {
        const float* a = (first ? in : h) + 4 * v;
        const int pitch = first ? pin : ph;
        const float* wp = wg + 4 * v + (first ? 0 : 4 * nin);
        float4 wr[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) wr[r] = *reinterpret_cast<const float4*>(wp + (size_t)r * ldw);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
          const float4 x = *reinterpret_cast<const float4*>(a + b * pitch);
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            float t = acc[b * 4 + r];
            t = fmaf(x.x, wr[r].x, t);
            t = fmaf(x.y, wr[r].y, t);
            t = fmaf(x.z, wr[r].z, t);
            acc[b * 4 + r] = fmaf(x.w, wr[r].w, t);
          }
        }
      }
    }
    const float v = lane_sums<NB * 4>(acc, lane);
    constexpr int per = 32 / (NB * 4);
    if (lane % per == 0) red[(g * ns + s) * NB * 4 + lane / per] = v;
  }
}

// F on the tensor cores: 8 units a group; gates i, f are the rows of one 16-row tile, g, o those of
// another, so that a thread ends with the four gates of its unit for two batch rows.
template <int NB>
__device__ __forceinline__ void units_mma(uint32_t in, int nin, uint32_t h, int nh, uint32_t pin, uint32_t ph, uint32_t w, uint32_t ldw, int U,
                                          int lg, float* red, int wk, int lane) {
  const int ns = 1 << lg, steps = nin + nh, works = ((U + 7) >> 3) * ns;   // nin, nh: 16-wide steps
  for (; wk < works; wk += kWarps) {
    const int g = wk >> lg, s = wk & (ns - 1), ng = min(8, U - 8 * g);
    const int lo = steps * s >> lg, hi = steps * (s + 1) >> lg;
    const int row = 32 * g + ((lane >> 3) & 1) * ng + min(lane & 7, ng - 1);
    const uint32_t wa = w + row * ldw + (lane >> 4) * 16, wb = wa + 2 * ng * ldw;
    const uint32_t brow = (lane & 7) % NB, bk = ((lane >> 3) & 1) * 16;
    const uint32_t ia = in + brow * pin + bk, ih = h + brow * ph + bk - nin * 32;
    float c0[4] = {}, c1[4] = {};
#pragma unroll 4
    for (int k = lo; k < hi; ++k) {
      uint32_t a0[4], a1[4], b[2];
      ldsm2(b, (k < nin ? ia : ih) + k * 32);
      ldsm4(a0, wa + k * 32);
      ldsm4(a1, wb + k * 32);
      mma(c0, a0, b);
      mma(c1, a1, b);
    }
    const int u = 8 * g + (lane >> 2), b0 = 2 * (lane & 3);
    if (u < U && b0 < NB) {
      float4* d = reinterpret_cast<float4*>(red + ((size_t)(u * ns + s) * NB + b0) * 4);
      d[0] = make_float4(c0[0], c0[2], c1[0], c1[2]);
      if (NB > 1) d[1] = make_float4(c0[1], c0[3], c1[1], c1[3]);
    }
  }
}

// R on the tensor cores: 16 readout rows a tile; red[(tile ns + s)][16][NB].
template <int NB>
__device__ __forceinline__ void readout_mma(uint32_t h, uint32_t ph, int steps, uint32_t w, uint32_t ldw, int rows, int lg, float* red, int wk,
                                            int lane) {
  const int ns = 1 << lg, works = ((rows + 15) >> 4) * ns;
  for (; wk < works; wk += kWarps) {
    const int g = wk >> lg, s = wk & (ns - 1), lo = steps * s >> lg, hi = steps * (s + 1) >> lg;
    const int row = min(16 * g + ((lane >> 3) & 1) * 8 + (lane & 7), rows - 1);
    const uint32_t wa = w + row * ldw + (lane >> 4) * 16, ib = h + ((lane & 7) % NB) * ph + ((lane >> 3) & 1) * 16;
    float c[4] = {};
#pragma unroll 4
    for (int k = lo; k < hi; ++k) {
      uint32_t a[4], b[2];
      ldsm2(b, ib + k * 32);
      ldsm4(a, wa + k * 32);
      mma(c, a, b);
    }
    const int b0 = 2 * (lane & 3);
    if (b0 < NB) {
      float* d = red + ((size_t)(g * ns + s) * 16 + (lane >> 2)) * NB + b0;
      d[0] = c[0]; d[8 * NB] = c[2];
      if (NB > 1) { d[1] = c[1]; d[8 * NB + 1] = c[3]; }
    }
  }
}

// Shares: the products of the own rows' gradients d with columns of their weights (w points at the first),
// pushed to the owners of the units the columns belong to.  to[column]: where the owner keeps this CTA's
// first share of the unit, less the receiving buffer's offset, and where its shared memory begins;
// columns of no unit have zeros there.
struct Share {
  const uint2* to;
  uint32_t dst0, dst1, bar;   // offsets from the start of shared memory: receiving buffers of the first nc and of the next nc columns
  int nc;                 // columns of one buffer
};
template <int NB>
__device__ __forceinline__ void shares_fma(const float* d, const float* w, int ldw, int rows, int cols, int lg, int step, const Share& s, int tid) {
  for (int job = tid; job < cols << lg; job += kThreads) {
    int col = job, q = 0;
    while (col >= cols) { col -= cols; ++q; }
    const bool own = col >= s.nc;
    const uint2 to = s.to[own ? col - s.nc : col];
    if (!to.y) continue;
    const int lo = rows * q >> lg, hi = rows * (q + 1) >> lg;
    float acc[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) acc[b] = 0.f;
    const float* wp = w + (size_t)lo * ldw + col;
#pragma unroll 4
    for (int g = lo; g < hi; ++g, wp += ldw) {
      const float x = *wp;
      float v[NB];
      if (NB == 1) v[0] = d[g];
      else if (NB == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(d + 2 * g);
      else {
#pragma unroll
        for (int b = 0; b < NB; b += 4) *reinterpret_cast<float4*>(v + b) = *reinterpret_cast<const float4*>(d + NB * g + b);
      }
#pragma unroll
      for (int b = 0; b < NB; ++b) acc[b] = fmaf(x, v[b], acc[b]);
    }
    const uint32_t at = to.x + (own ? s.dst1 : s.dst0) + q * step, bar = to.y + s.bar;
    if (NB == 1) push(at, __float_as_uint(acc[0]), bar);
    else if (NB == 2) push2(at, __float_as_uint(acc[0]), __float_as_uint(acc[1]), bar);
    else {
#pragma unroll
      for (int b = 0; b < NB; b += 4)
        push4(at + 4 * b, __float_as_uint(acc[b]), __float_as_uint(acc[b + 1]), __float_as_uint(acc[b + 2]), __float_as_uint(acc[b + 3]), bar);
    }
  }
}
// The same on the tensor cores: columns are the rows of a tile (the weights are read transposed), two
// tiles a warp; the float32 gradients come as PL bfloat16 planes whose sum they are.
template <int NB, int PL>
__device__ __forceinline__ void shares_mma(uint32_t d, uint32_t pitch, uint32_t w, uint32_t ldw, int rows, int cols, const Share& s, int wk, int lane) {
  const int steps = (rows + 15) >> 4;
  const uint32_t ib = d + ((lane & 7) % NB) * pitch + ((lane >> 3) & 1) * 16;
  const int r0 = (lane >> 4) * 8 + (lane & 7);
  for (int t = wk; t < cols >> 5; t += kWarps) {
    float c[PL][8] = {};
    const uint32_t wc = w + t * 64 + ((lane >> 3) & 1) * 16;
#pragma unroll 2
    for (int k = 0; k < steps; ++k) {
      uint32_t a0[4], a1[4], b[PL][2];
      const uint32_t wa = wc + min(k * 16 + r0, rows - 1) * ldw;
#pragma unroll
      for (int p = 0; p < PL; ++p) ldsm2(b[p], ib + p * NB * pitch + k * 32);
      ldsm4t(a0, wa);
      ldsm4t(a1, wa + 32);
#pragma unroll
      for (int p = 0; p < PL; ++p) {
        mma(*reinterpret_cast<float (*)[4]>(c[p]), a0, b[p]);
        mma(*reinterpret_cast<float (*)[4]>(c[p] + 4), a1, b[p]);
      }
    }
#pragma unroll
    for (int p = 1; p < PL; ++p)
#pragma unroll
      for (int q = 0; q < 8; ++q) c[0][q] += c[p][q];
    const int b0 = 2 * (lane & 3);
    if (b0 >= NB) continue;
    int col = t * 32 + (lane >> 2);
    const bool own = col >= s.nc;        // (nc is a multiple of 32: the same for all of the tile)
    if (own) col -= s.nc;
    const uint32_t dst = (own ? s.dst1 : s.dst0) + b0 * 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint2 to = s.to[col + 8 * q];
      if (!to.y) continue;
      if (NB == 1) push(to.x + dst, __float_as_uint(c[0][2 * q]), to.y + s.bar);
      else push2(to.x + dst, __float_as_uint(c[0][2 * q]), __float_as_uint(c[0][2 * q + 1]), to.y + s.bar);
    }
  }
}

// A float32 value as PL bfloat16 values that add up to it (three hold all 24 bits).
template <int PL>
__device__ __forceinline__ void put_planes(bf16* p, int stride, float v) {
#pragma unroll
  for (int i = 0; i < PL; ++i) {
    const bf16 h = __float2bfloat16_rn(v);
    p[i * stride] = h;
    v -= __bfloat162float(h);
  }
}

// WIDE: a pod's states pass 4 GB, or locations count parts of a block.  The sums are the same.
template <class T, bool GRU, int NB, int PL, bool WIDE>
__global__ void __launch_bounds__(kThreads, 1) pod_walk(const __grid_constant__ Args A) {
  constexpr bool MMA = std::is_same<T, bf16>::value;
  extern __shared__ __align__(128) unsigned char smem[];
  const Config& C = A.c;
  uint4* const windows = reinterpret_cast<uint4*>(smem);                    // records of 32 bytes
  unsigned char* const ctl = smem + kWindows * kWindow * sizeof(Task);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(ctl);                  // even and odd phases
  uint32_t* const peer = reinterpret_cast<uint32_t*>(ctl + 64);             // where each CTA's shared memory begins
  // a wait of an even or odd phase gave up (a thread may be a phase ahead of one that has yet to look)
  volatile int* const dead = reinterpret_cast<volatile int*>(ctl + 128);
  unsigned char* const area = ctl + 1024;
  uint2* const to = reinterpret_cast<uint2*>(area + C.at_map);              // Share::to
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pod = blockIdx.x / C.T, rank = blockIdx.x - pod * C.T, NT = C.T;
  const int H = A.H, L = A.L, U = C.U, up = C.up;
  const int valid = min(NB, A.B - pod * NB);
  const uint32_t base = sm100::smem_u32(smem), bar0 = sm100::smem_u32(bars), area0 = sm100::smem_u32(area) - base;
  auto units_of = [&](int r) { return max(0, min(U, H - r * U)); };
  const int u = units_of(rank);

  if (tid == 0) {
    dead[0] = dead[1] = 0;
    sm100::mbar_init(bars, 1);
    sm100::mbar_init(bars + 1, 1);
    sm100::mbar_fence_init();
  }
  if (tid < NT) peer[tid] = remote(base, tid);
  for (int i = tid; i < C.at_w / 4; i += kThreads) reinterpret_cast<uint32_t*>(area)[i] = 0;
  auto load_window = [&](int w) {
    if (tid < kWindow * 2) windows[(w & (kWindows - 1)) * kWindow * 2 + tid] = __ldg(reinterpret_cast<const uint4*>(A.tasks + (size_t)w * kWindow) + tid);
  };
  const int n_windows = A.n_tasks / kWindow;
  load_window(0);
  if (n_windows > 1) load_window(1);
  __syncthreads();
  for (int i = tid; i < C.kh; i += kThreads) {
    const int r = i / up, j = i - r * up;
    const bool on = r < NT && j < units_of(r);
    to[i] = on ? make_uint2(peer[r] + ((rank * C.ns_b) * U + j) * NB * 4, peer[r]) : make_uint2(0, 0);
  }
  // weights: layer by layer, then the readout
  const int w0 = 4 * U * C.pitch_w(0), w1 = 4 * U * C.pitch_w(1);
  T* const held = reinterpret_cast<T*>(area + C.at_w);
  // weight `at` (counted from the start of the CTA's weights) where they are not held
  auto slice = [&](int l, uint32_t at) -> const T* {   // l == L: readout
    return reinterpret_cast<const T*>(A.ws + (l == L ? A.off_wr : A.off_wf[l])) + (size_t)rank * (l == L ? C.op * C.pitch_r() : l ? w1 : w0) +
           (at - (l ? w0 + (l - 1) * w1 : 0));
  };
  if (C.resident)
    for (int l = 0; l <= L; ++l) {
      const int n = l == L ? C.op * C.pitch_r() : l ? w1 : w0;
      const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const T*>(A.ws + (l == L ? A.off_wr : A.off_wf[l])) + (size_t)rank * n);
      uint4* dst = reinterpret_cast<uint4*>(held + (l ? w0 + (l - 1) * w1 : 0));
      for (int i = tid; i < n * (int)sizeof(T) / 16; i += kThreads) dst[i] = __ldcg(src + i);
    }

  // ---- the thread's elements ----
  // a unit of a layer in a batch row: rows fastest, so that four units in a row are lanes NB apart
  const int eb = tid & (NB - 1), eju = (tid / NB) % up, el = (tid / NB) / up;
  const bool has = el < L && eju < u && eb < valid;
  const bool sends = el < L && (eju & ~3) < u && eb < valid;   // (its group of four has a unit)
  const int row = pod * NB + eb, ej = rank * U + eju, lay = has ? el : 0;
  const size_t e = has ? (size_t)row * H + ej : 0;
  // offsets of this element: h, c and gates from the pod's states, dz and h stages and carried dz from the start
  // of the stages (under 4 GB by the rule of choose_config)
  using St = States<T>;
  const St S(A.ws + A.off_states, A.n_blocks, WIDE ? A.parts : 1, pod, NB, A.B, H);
  const uint32_t le = eb * H + ej, hs_ = S.hs, part_ = S.part;
  const uint32_t o_h = lay * (1 + St::CR) * hs_ + le * (uint32_t)sizeof(T), o_c = (lay * (1 + St::CR) + 1) * hs_ + le * 4;
  const uint32_t o_g = (L * (1 + St::CR) + 4 * lay) * hs_ + le * (uint32_t)sizeof(T), o_in = (L * (1 + St::CR) + 4 * L) * hs_;
  const uint32_t bh = (uint32_t)A.B * H;                         // elements of a row block of the h stage, a quarter of those of dz
  const uint32_t o_dz = (uint32_t)((lay * (size_t)A.S * bh + e) * 16);
  const uint32_t o_cy = (uint32_t)(A.off_carry - A.off_dz + ((size_t)lay * bh + e) * 16);
  const uint32_t o_st = (uint32_t)(A.off_hk - A.off_dz + (lay * (size_t)(A.S + 1) * bh + e) * sizeof(T));
  auto dc_at = [&]() { return reinterpret_cast<float*>(A.ws + A.off_dc + ((size_t)lay * bh + e) * 4); };
  float dc = has ? *dc_at() : 0.f;
  float bias[4] = {0.f, 0.f, 0.f, 0.f};
  if (has)
#pragma unroll
    for (int q = 0; q < (GRU ? 3 : 4); ++q) bias[q] = __ldg(A.bias + ((size_t)el * (GRU ? 3 : 4) + q) * H + ej);
  const int grp = 8 * (eju >> 3), gn = min(8, U - grp);          // mma: rows of a unit's gates are gn apart
  const int zrow = MMA ? 4 * grp + (eju & 7) : 4 * eju, zstep = MMA ? gn : 1;
  const uint32_t at_push = (uint32_t)(eb * C.pitch_h + (rank * up + (eju & ~3)) * (int)sizeof(T));
  // readout rows and groups of four inputs: further back in the block
  const int ri = (tid + kThreads - (L * up * NB) % kThreads) % kThreads, rb = ri & (NB - 1), rj = ri / NB, ro = rank * C.rows_o + rj;
  const bool has_r = rj < C.rows_o && ro < A.O && rb < valid;
  const int rrow = pod * NB + rb;
  const float r_bias = has_r ? __ldg(A.b_out + ro) : 0.f;
  const int i_r = has_r ? rrow * A.O + ro : 0;
  const float dy_scale = 1.f / ((float)A.B * (float)A.O);
  int xg0, xg1;
  part((A.I + 3) >> 2, NT, rank, xg0, xg1);
  const int xi = (ri + kThreads - (C.op * NB) % kThreads) % kThreads, xb = xi & (NB - 1), xg = xg0 + xi / NB;
  const bool has_x = xg < xg1 && xb < valid;
  const int i_x = has_x ? (pod * NB + xb) * A.I + 4 * xg : 0;
  const int x_n = has_x ? min(4, A.I - 4 * xg) : 0;

  // bytes of the pushes a CTA receives: h of a layer, x, shares
  int gh = 0;
  for (int r = 0; r < NT; ++r) gh += (units_of(r) + 3) >> 2;
  const uint32_t by_h = valid * gh * 4 * (uint32_t)sizeof(T), by_x = valid * ((A.I + 3) >> 2) * 4 * (uint32_t)sizeof(T);
  const uint32_t by_p = NT * C.ns_b * u * NB * 4;
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // ---- fetched one phase ahead ----
  // Records are read as two 16-byte words; these pick fields of a task out of them.
  auto rec = [&](int i) { return windows[i]; };               // i: 2 x record (+ 1 for the second half)
  auto k_of = [](const uint4& a) { return (int)a.y; };
  auto sidx_of = [](const uint4& b) { return b.x & 0xffff; };
  auto sa_of = [](const uint4& b) { return (b.x >> 16) * 16; };
  auto sb_of = [](const uint4& b) { return (b.y & 0xffff) * 16; };
  auto so_of = [](const uint4& b) { return (b.y >> 16) * 16; };
  auto red_of = [](const uint4& b) { return (b.w & 0xffff) * 16; };
  auto flags_of = [](const uint4& a) { return a.x >> 16; };
  constexpr uint32_t no_slot = (uint32_t)kNone * 16;
  // whether any thread of the warp has an element of the kind: the others have nothing to do but products
  const bool warp_s = __any_sync(0xffffffffu, sends), warp_r = __any_sync(0xffffffffu, has_r), warp_x = __any_sync(0xffffffffu, has_x);
  const int sh = has ? 4 * el : 28;                           // this layer's place in the header's index words (28: never used)
  const int shs = sends ? 4 * el : 28;
  float om[7];
  float ol = 0.f, o_target = 0.f;
  float4 ox = make_float4(0.f, 0.f, 0.f, 0.f), oz = ox;
  // The states of a generous budget pass 4 GB, and a plan over byte sizes counts in parts of a block.  Where
  // neither is so, an offset of 32 bits from a base that is the same for all threads takes no instruction to
  // add; with 64 bits throughout, the two-layer GRU of 256 units took 1 % longer (2864 -> 2891 us), with parts
  // 0.4 % more.
  auto at = [&](uint32_t o, uint32_t loc) { return WIDE ? S.base + (uint64_t)loc * part_ + o : S.base + (o + loc * part_); };
  // h0: n cells sums n_h | n_p n_x r x | products - | main     h1: load carry bwd -
  auto ahead = [&](int cur, const uint4& h0, const uint4& h1) {
    if (warp_s) {
    const int im = (h0.w >> sh) & 15, il = (h1.x >> sh) & 15, iz = (h1.y >> sh) & 15;
    if (im) {
      const uint4 a = rec(cur + 2 * im);
      if ((h1.z >> sh) & 15) {
        const char* g = at(o_g, a.z);
#pragma unroll
        for (int q = 0; q < 4; ++q) om[q] = to_f(*reinterpret_cast<const T*>(g + q * hs_));
        om[4] = to_f(*reinterpret_cast<const T*>(at(o_h, a.w)));
        if (!GRU) {
          om[5] = *reinterpret_cast<const float*>(at(o_c, a.z));
          om[6] = *reinterpret_cast<const float*>(at(o_c, a.w));
        }
      } else {
        om[4] = GRU ? to_f(*reinterpret_cast<const T*>(at(o_h, a.z))) : *reinterpret_cast<const float*>(at(o_c, a.z));
        if (!GRU && (flags_of(a) & COPY_IN)) om[5] = to_f(*reinterpret_cast<const T*>(at(o_h, a.z)));
      }
    }
    if (il) ol = to_f(*reinterpret_cast<const T*>(at(o_h, rec(cur + 2 * il).z)));
    if (iz) {
      const int k = k_of(rec(cur + 2 * iz));
      const uint32_t sidx = sidx_of(rec(cur + 2 * iz + 1));
      oz = *reinterpret_cast<const float4*>(A.stages + (sidx == kNone ? o_cy + ((k + 1) & 1) * L * bh * 16 : o_dz + sidx * bh * 16));
    }
    }
    const uint32_t ir = (h0.y >> 16) & 0xff, ix = h0.y >> 24;
    if (warp_r && ir && has_r) o_target = __ldg(A.targets + i_r + (size_t)(k_of(rec(cur + 2 * ir)) - 1) * A.B * A.O);
    if (warp_x && ix && has_x) {
      const T* x = reinterpret_cast<const T*>(A.x) + i_x + (size_t)(k_of(rec(cur + 2 * ix)) - 1) * A.B * A.I;
      ox.x = to_f(x[0]);
      ox.y = x_n > 1 ? to_f(x[1]) : 0.f;
      ox.z = x_n > 2 ? to_f(x[2]) : 0.f;
      ox.w = x_n > 3 ? to_f(x[3]) : 0.f;
    }
  };
  // four consecutive units of one batch row: their values in every lane of the group
  auto gather4 = [&](float v) {
    float4 r;
    const bool o1 = eju & 1, o2 = eju & 2;
    const float a = __shfl_xor_sync(0xffffffffu, v, NB);
    const float lo = o1 ? a : v, hi = o1 ? v : a;
    const float lo2 = __shfl_xor_sync(0xffffffffu, lo, 2 * NB), hi2 = __shfl_xor_sync(0xffffffffu, hi, 2 * NB);
    r.x = o2 ? lo2 : lo; r.y = o2 ? hi2 : hi; r.z = o2 ? lo : lo2; r.w = o2 ? hi : hi2;
    return r;
  };
  auto push_quad = [&](uint32_t to, uint32_t off, const float4& v, uint32_t bar) {
    if (MMA) push2(to + off, sm100::pack_bf16x2(v.x, v.y), sm100::pack_bf16x2(v.z, v.w), to + bar);
    else push4(to + off, __float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), __float_as_uint(v.w), to + bar);
  };

  // one phase's operand of F and B per layer: the same for every layer but the first
  const int ldw0 = C.pitch_w(0), ldw1 = C.pitch_w(1), ldr = C.pitch_r();
  const int step = U * NB * 4;
  int w = 0, i0 = 0, ph = 0;
  bool entered = true;       // first phase of a window
  int cur = 0;               // the phase's header: 2 x record
  uint4 h0 = rec(0), h1 = rec(1);
  ahead(cur, h0, h1);
  for (; ph < A.phases; ++ph) {
    const uint32_t bar = bar0 - base + 8 * (ph & 1);
    const bool cells = (h0.x >> 8) & 0xff, sums = (h0.x >> 16) & 0xff;
    unsigned char* const dz_buf = area + C.at_dz + (ph & 1) * L * C.dz_buf;
    const uint32_t red_par = (ph & 1) * C.red_bytes;
    if (ph > 0 && !wait_for(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1, A.polls)) dead[ph & 1] = 1;

    // ---- gradients of the own units ----
    if (cells && warp_s) {
      const int ib = (h1.z >> sh) & 15, iz = (h1.y >> sh) & 15;
      if (ib | iz) {
        float d[4];
        if (ib) {
          const uint4 a = rec(cur + 2 * ib), b = rec(cur + 2 * ib + 1);
          const uint32_t fl = flags_of(a), sidx = sidx_of(b);
          float s0 = 0.f, s1 = 0.f;
          const float* p0 = reinterpret_cast<const float*>(area + sa_of(b)) + eju * NB + eb;
          const float* p1 = reinterpret_cast<const float*>(area + sb_of(b)) + eju * NB + eb;
          const int n = (fl & FIRST) ? 0 : NT * C.ns_b;
#pragma unroll 4
          for (int i = 0; i < NT * C.ns_b; ++i, p0 += U * NB, p1 += U * NB) {
            const float v0 = *p0;
            s1 += *p1;
            if (i < n) s0 += v0;
          }
          const float g[4] = {om[0], om[1], om[2], om[3]};
          cell_backward<GRU>(s0 + s1, g, om[4], om[5], om[6], dc, d);
          const float4 quad = make_float4(d[0], d[1], d[2], d[3]);
          *reinterpret_cast<float4*>(A.stages + (o_dz + sidx * bh * 16)) = quad;
          T* const hs = reinterpret_cast<T*>(A.stages + (o_st + sidx * bh * (uint32_t)sizeof(T)));
          store(hs, om[4]);
          if (fl & CLOSE) *reinterpret_cast<float4*>(A.stages + (o_cy + (k_of(a) & 1) * L * bh * 16)) = quad;
          if (fl & OPEN) store(hs + bh, to_f(*reinterpret_cast<const T*>(at(o_h, a.z))));
        } else {
          d[0] = oz.x; d[1] = oz.y; d[2] = oz.z; d[3] = oz.w;
        }
        unsigned char* const my = dz_buf + el * C.dz_buf;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (MMA) put_planes<PL>(reinterpret_cast<bf16*>(my) + eb * (C.dz_pitch / 2) + zrow + q * zstep, NB * (C.dz_pitch / 2), d[q]);
          else reinterpret_cast<float*>(my)[(zrow + q) * NB + eb] = d[q];
        }
      }
    }
    if (cells || !sums) {
      __syncthreads();
      if (dead[ph & 1]) break;
    }

    // ---- products ----
#pragma unroll 1
    for (int i = 1; i <= (int)(h0.z & 0xff); ++i) {
      const uint4 a = rec(cur + 2 * i);
      const uint32_t kind = a.x & 0xff, l = (a.x >> 8) & 0xff;
      const int wk = (warp - (int)(a.x >> 24)) & (kWarps - 1);
      if (kind == FWD && wk >= (l ? C.works_f1 : C.works_f0)) continue;
      if (kind == READ && wk >= C.works_r) continue;
      const uint4 b = rec(cur + 2 * i + 1);
      if (MMA && wk >= (int)(b.w >> 21) && kind != FWD && kind != READ) continue;   // cols / 32
      const T* wp = MMA || C.resident ? held + b.z : slice(kind == READ || kind == DHA ? L : (int)l, b.z);
      if (kind == FWD) {
        float* const r = reinterpret_cast<float*>(area + red_of(b) + red_par);
        if constexpr (MMA)
          units_mma<NB>(sm100::smem_u32(area + sa_of(b)), l ? C.kh / 16 : C.kx / 16, sm100::smem_u32(area + sb_of(b)), C.kh / 16, l ? C.pitch_h : C.pitch_x, C.pitch_h,
                        sm100::smem_u32(wp), (l ? ldw1 : ldw0) * 2, U, l ? C.lg_f1 : C.lg_f0, r, wk, lane);
        else
          rows_fma<NB>(reinterpret_cast<const float*>(area + sa_of(b)), (l ? C.pitch_h : C.pitch_x) / 4, (l ? C.kh : C.kx) / 4, reinterpret_cast<const float*>(area + sb_of(b)),
                       C.pitch_h / 4, C.kh / 4, wp, l ? ldw1 : ldw0, U, l ? C.lg_f1 : C.lg_f0, r, wk, lane);
      } else if (kind == READ) {
        float* const r = reinterpret_cast<float*>(area + red_of(b) + red_par);
        if constexpr (MMA) readout_mma<NB>(sm100::smem_u32(area + sb_of(b)), C.pitch_h, C.kh / 16, sm100::smem_u32(wp), ldr * 2, C.op, C.lg_r, r, wk, lane);
        else rows_fma<NB>(nullptr, 0, 0, reinterpret_cast<const float*>(area + sb_of(b)), C.pitch_h / 4, C.kh / 4, wp, ldr, C.op / 4, C.lg_r, r, wk, lane);
      } else {   // B, Z, D
        const bool out = kind == DHA;
        const Share sr{to, area0 + red_of(b), area0 + so_of(b), bar, C.kh};
        unsigned char* const d = out ? area + sa_of(b) : dz_buf + l * C.dz_buf;
        const int ld = out ? ldr : l ? ldw1 : ldw0, rows = out ? C.op : 4 * U, cols = b.w >> 16;
        if constexpr (MMA) shares_mma<NB, PL>(sm100::smem_u32(d), out ? C.dy_pitch : C.dz_pitch, sm100::smem_u32(wp), ld * 2, rows, cols, sr, wk, lane);
        else shares_fma<NB>(reinterpret_cast<const float*>(d), wp, ld, rows, cols, C.lg_b, step, sr, tid);
      }
    }
    if (sums) {
      __syncthreads();
      if (dead[ph & 1]) break;
    }
    if (warp == kWarps - 1) {   // the operands have been read: a word to everybody, and what to expect oneself
      if (lane < NT) push(peer[lane] + area0 + C.at_dummy + 4 * rank, 0, peer[lane] + bar);
      if (lane == 31) sm100::mbar_arrive_expect_tx(bars + (ph & 1), (h0.x >> 24) * by_h + (h0.y & 0xff) * by_p + ((h0.y >> 8) & 0xff) * by_x + 4 * NT + A.extra_bytes);
    }

    // ---- states, readouts, loads ----
    const uint32_t fwd = h0.w & ~h1.z;       // index words of the F tasks alone (a layer has an F or a B)
    if (fwd && warp_s) {
      const int f = (fwd >> sh) & 15;
      uint4 a{}, b{};
      float hv = 0.f;
      if (f) {
        a = rec(cur + 2 * f); b = rec(cur + 2 * f + 1);
        const int ns = 1 << (el ? C.lg_f1 : C.lg_f0);
        const float4* p = reinterpret_cast<const float4*>(area + red_of(b) + red_par) + eju * ns * NB + eb;
        float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
        for (int q = 0; q < ns; ++q, p += NB) {
          const float4 r = *p;
          z[0] += r.x; z[1] += r.y; z[2] += r.z; z[3] += r.w;
        }
        float g[4], cv;
        cell_forward<GRU>(z, bias, om[4], g, hv, cv);
        T stored;
        store(&stored, hv);
        *reinterpret_cast<T*>(at(o_h, a.w)) = stored;
        hv = to_f(stored);       // the others read what was stored
        if (!GRU) *reinterpret_cast<float*>(at(o_c, a.w)) = cv;
        if (flags_of(a) & GATES) {
          char* gp = at(o_g, a.w);
#pragma unroll
          for (int q = 0; q < 4; ++q) store(reinterpret_cast<T*>(gp + q * hs_), g[q]);
        }
        if (flags_of(a) & COPY_IN) {
          store(reinterpret_cast<T*>(at(o_h, a.w) + o_in), GRU ? om[4] : om[5]);
          if (!GRU) *reinterpret_cast<float*>(at(o_c, a.w) + o_in) = om[4];
        }
      }
      // (a group of four may hold units past the last one: their lanes send with it all the same)
      const int gi = (fwd >> shs) & 15;
      const uint32_t so = gi ? so_of(rec(cur + 2 * gi + 1)) : no_slot;
      const float4 q = gather4(hv);
      if (so != no_slot)
        for (int r = eju & 3; r < NT; r += 4) push_quad(peer[r], area0 + so + at_push, q, bar);
    }
    if (h1.x && warp_s) {
      const int gi = (h1.x >> shs) & 15;
      const float4 q = gather4(has ? ol : 0.f);
      if (gi) {
        const uint32_t so = so_of(rec(cur + 2 * gi + 1));
        for (int r = eju & 3; r < NT; r += 4) push_quad(peer[r], area0 + so + at_push, q, bar);
      }
    }
    const uint32_t ir = (h0.y >> 16) & 0xff, ix = h0.y >> 24;
    if (warp_r && ir && has_r) {
      const uint4 b = rec(cur + 2 * ir + 1);
      const int ns = 1 << C.lg_r;
      const float* p = reinterpret_cast<const float*>(area + red_of(b) + red_par) +
                       (MMA ? ((rj >> 4) * ns * 16 + (rj & 15)) * NB + rb : (rj >> 2) * ns * NB * 4 + rb * 4 + (rj & 3));
      float z = 0.f;
      for (int q = 0; q < ns; ++q, p += MMA ? 16 * NB : NB * 4) z += *p;
      const float dy = 2.f * (z + r_bias - o_target) * dy_scale;
      reinterpret_cast<float*>(A.ws + A.off_dy)[i_r + sidx_of(b) * A.B * A.O] = dy;
      unsigned char* const d = area + so_of(b);
      if (MMA) put_planes<PL>(reinterpret_cast<bf16*>(d) + rb * (C.dy_pitch / 2) + rj, NB * (C.dy_pitch / 2), dy);
      else reinterpret_cast<float*>(d)[rj * NB + rb] = dy;
    }
    if (warp_x && ix && has_x) {
      const uint32_t off = area0 + so_of(rec(cur + 2 * ix + 1)) + xb * C.pitch_x + 4 * xg * (uint32_t)sizeof(T);
      for (int r = 0; r < NT; ++r) push_quad(peer[r], off, ox, bar);
    }
    if (entered && w + 2 < n_windows) load_window(w + 2);
    entered = false;
    if (ph + 1 < A.phases) {
      const int nx = i0 + 1 + (h0.x & 0xff);
      i0 = nx;
      cur = ((w & (kWindows - 1)) * kWindow + i0) * 2;
      if (i0 < kWindow) h0 = rec(cur);
      if (i0 >= kWindow || (h0.x & 0xff) == 0) {
        ++w; i0 = 0; entered = true;
        cur = (w & (kWindows - 1)) * kWindow * 2;
        h0 = rec(cur);
      }
      h1 = rec(cur + 1);
      ahead(cur, h0, h1);
    }
  }
  bool ok = ph == A.phases;
  if (ok && ph > 0) ok = wait_for(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1, A.polls);
  if (!ok) *A.status = MEBPTT_ERR_TIMEOUT;
  if (has) *dc_at() = dc;
  // nobody leaves while pushes to its shared memory may be under way: all of them have arrived, or the wait for
  // them gave up; then nobody pushes any more behind this barrier, and what is still under way gets time to land
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (!ok)
    for (int i = 0; i < 1024; ++i) __nanosleep(200);
  if (tid == 0 && blockIdx.x == 0 && ok) {
    A.counters[0] += A.fwd_ops;
    A.counters[1] += A.bwd_ops;
  }
}

// One warp per packed row.
template <class T, bool GRU>
__global__ void __launch_bounds__(256) pod_pack(const __grid_constant__ PackArgs P) {
  const Config& C = P.c;
  const int H = P.H, L = P.L, lane = threadIdx.x & 31;
  const size_t first = blockIdx.x * 256 + threadIdx.x, all = (size_t)gridDim.x * 256;
  for (size_t i = first; i < P.n_zero; i += all) P.zero[i] = 0.f;
  if (blockIdx.x == 0 && threadIdx.x < 8) P.counters[threadIdx.x] = 0;
  const size_t bh = (size_t)P.B * H;
  for (int l = 0; l < L; ++l)
    for (size_t i = first; i < bh; i += all) {
      const int b = (int)(i / H), g = b / C.nb;
      const States<T> S(P.states, P.n_blocks, P.parts, g, C.nb, P.B, H);
      const size_t le = i - (size_t)g * C.nb * H;
      S.h((uint32_t)P.init, l)[le] = reinterpret_cast<const T*>(P.h0)[l * bh + i];
      S.c((uint32_t)P.init, l)[le] = P.c0[l * bh + i];
    }
  const int per = 4 * C.U, rows = C.T * (L * per + C.op);
  const T zero = T(0.f);
  for (int n = blockIdx.x * 8 + (threadIdx.x >> 5); n < rows; n += gridDim.x * 8) {
    // column c of the h part: the owner's units in `up` columns each
    auto unit = [&](int c) {
      const int r = c / C.up, j = c - r * C.up;
      return r < C.T && j < C.U && r * C.U + j < H ? r * C.U + j : -1;
    };
    if (n >= C.T * L * per) {
      const int m = n - C.T * L * per, r = m / C.op, o = r * C.rows_o + m - r * C.op;
      T* out = reinterpret_cast<T*>(P.wr) + (size_t)m * C.pitch_r();
      const bool on = m - r * C.op < C.rows_o && o < P.O;
      for (int c = lane; c < C.pitch_r(); c += 32) {
        const int j = c < C.kh ? unit(c) : -1;
        out[c] = on && j >= 0 ? reinterpret_cast<const T*>(P.W_out)[(size_t)o * H + j] : zero;
      }
      continue;
    }
    const int l = n / (C.T * per), m = n - l * C.T * per, r = m / per, p = m - r * per;
    int ju, q;
    if (C.mma) {
      const int g = p >> 5, ng = min(8, C.U - 8 * g), rem = p - 32 * g;
      q = rem / ng;
      ju = 8 * g + rem - q * ng;
    } else {
      ju = p >> 2; q = p & 3;
    }
    const int j = r * C.U + ju, I = l ? H : P.I, kin_ = l ? C.kh : C.kx;
    const T* W = reinterpret_cast<const T*>(P.W) + P.w_off[l] + (size_t)((GRU && q == 3 ? 2 : q) * H + min(j, H - 1)) * (I + H);
    T* out = reinterpret_cast<T*>(P.wf[l]) + (size_t)m * C.pitch_w(l);
    for (int c = lane; c < C.pitch_w(l); c += 32) {
      int col = -1;
      if (c < kin_) {
        col = l ? unit(c) : c < P.I ? c : -1;
        if (GRU && q == 3) col = -1;
      } else if (c < kin_ + C.kh) {
        col = unit(c - kin_);
        if (GRU && q == 2) col = -1;
        if (col >= 0) col += I;
      }
      out[c] = j < H && col >= 0 ? W[col] : zero;
    }
  }
}

template <class T, bool GRU, int PL, bool WIDE>
Fn by_rows(int nb) {
  return nb == 1   ? pod_walk<T, GRU, 1, PL, WIDE>
         : nb == 2 ? pod_walk<T, GRU, 2, PL, WIDE>
         : nb == 4 ? pod_walk<T, GRU, 4, PL, WIDE>
                   : pod_walk<T, GRU, 8, PL, WIDE>;
}
template <class T, int PL>
Fn by_core(bool gru, int nb, bool wide) {
  if (gru) return wide ? by_rows<T, true, PL, true>(nb) : by_rows<T, true, PL, false>(nb);
  return wide ? by_rows<T, false, PL, true>(nb) : by_rows<T, false, PL, false>(nb);
}

}  // namespace

Fn kernel(int dtype, bool gru, int nb, bool wide) {
  return dtype == MEBPTT_BF16 ? by_core<bf16, 3>(gru, nb, wide) : by_core<float, 1>(gru, nb, wide);
}

void launch_pack(int dtype, bool gru, const PackArgs& p, cudaStream_t s) {
  if (dtype == MEBPTT_BF16) {
    if (gru) pod_pack<bf16, true><<<592, 256, 0, counted(s)>>>(p); else pod_pack<bf16, false><<<592, 256, 0, counted(s)>>>(p);
  } else {
    if (gru) pod_pack<float, true><<<592, 256, 0, counted(s)>>>(p); else pod_pack<float, false><<<592, 256, 0, counted(s)>>>(p);
  }
}

}  // namespace pod
}  // namespace mebptt
