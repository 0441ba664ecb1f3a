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
__device__ __forceinline__ bool wait_for(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < sm100::kSpinLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if (i > 1024) __nanosleep(64);
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
__device__ __forceinline__ int log2i(int v) { return 31 - __clz(v); }

// ---- products ------------------------------------------------------------------------------

// F and R on FMA: four weight rows against NB operand rows over the 128-wide slices [lo, hi) of [input | h].
// Lanes split the contraction index; the sums of unit / row group g, part s go to red[(g ns + s)][NB][4].
template <int NB>
__device__ __forceinline__ void rows_fma(const float* in, int pin, int nin, const float* h, int ph, int nh, const float* w, int ldw, int groups,
                                         int ns, float* red, int wk, int lane) {
  const int lg = log2i(ns), ia = (nin + 31) >> 5, its = ia + ((nh + 31) >> 5);
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
                                          int ns, float* red, int wk, int lane) {
  const int lg = log2i(ns), steps = nin + nh, works = ((U + 7) >> 3) * ns;   // nin, nh: 16-wide steps
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
__device__ __forceinline__ void readout_mma(uint32_t h, uint32_t ph, int steps, uint32_t w, uint32_t ldw, int rows, int ns, float* red, int wk,
                                            int lane) {
  const int lg = log2i(ns), works = ((rows + 15) >> 4) * ns;
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
__device__ __forceinline__ void shares_fma(const float* d, const float* w, int ldw, int rows, int cols, int ns, int step, const Share& s, int tid) {
  const int lg = log2i(ns);
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

struct Main { float v[7]; };   // what a cell needs from memory: see ahead()

template <class T, bool GRU, int NB, int PL>
__global__ void __launch_bounds__(kThreads, 1) pod_walk(const __grid_constant__ Args A) {
  constexpr bool MMA = std::is_same<T, bf16>::value;
  extern __shared__ __align__(128) unsigned char smem[];
  const Config& C = A.c;
  uint4* const windows = reinterpret_cast<uint4*>(smem);                    // records of 32 bytes
  unsigned char* const ctl = smem + kWindows * kWindow * sizeof(Task);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(ctl);                  // even and odd phases
  uint32_t* const peer = reinterpret_cast<uint32_t*>(ctl + 64);             // where each CTA's shared memory begins
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
  // weights: layer by layer, then the readout.  (Where they lie is worked out again at each use: an array of
  // pointers would live in local memory, and with this much shared memory taken there is no L1 to hold it.)
  const int w0 = 4 * U * C.pitch_w(0), w1 = 4 * U * C.pitch_w(1);
  T* const held = reinterpret_cast<T*>(area + C.at_w);
  auto weights = [&](int l) -> const T* {     // l == L: readout
    if (MMA || C.resident) return held + (l ? w0 + (l - 1) * w1 : 0);
    return reinterpret_cast<const T*>(A.ws + (l == L ? A.off_wr : A.off_wf[l])) + (size_t)rank * (l == L ? C.op * C.pitch_r() : l ? w1 : w0);
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
  // offsets into the workspace (under 4 GB here): state, gates, dz and h stages, carried dz, of this element
  const uint32_t o_h = (uint32_t)(lay * A.hc + e * sizeof(T)), o_c = (uint32_t)(lay * A.hc + A.csz_off + e * 4);
  const uint32_t o_g = (uint32_t)(A.rec_gates + lay * A.gsz + e * sizeof(T));
  const uint32_t bh = (uint32_t)A.B * H;                         // elements of a row block of the h stage, a quarter of those of dz
  const uint32_t o_dz = (uint32_t)(A.off_dz + (lay * (size_t)A.S * bh + e) * 16);
  const uint32_t o_cy = (uint32_t)(A.off_carry + ((size_t)lay * bh + e) * 16);
  const uint32_t o_st = (uint32_t)(A.off_hk + (lay * (size_t)(A.S + 1) * bh + e) * sizeof(T));
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
  // where F(l) and R leave their partial sums, and the warp that starts with each
  auto red_f = [&](int l) {
    int o = 0;
    for (int i = 0; i < l; ++i) o += (MMA ? (U + 7) / 8 * 8 : U) * C.ns_f[i] * NB * 4;
    return o;
  };
  const int my_red = red_f(lay), red_r = red_f(L);
  const uint32_t p_area = area0 + C.at_p;
  auto p_at = [&](int l, int above, int par) { return p_area + (uint32_t)(((l * 2 + above) * 2 + par) * C.p_slot); };

  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // ---- fetched one phase ahead ----
  Main om;
  float4 ol = make_float4(0.f, 0.f, 0.f, 0.f), ox = ol, oz = ol;
  float o_target = 0.f;
  auto at = [&](uint32_t o, uint32_t loc) { return A.ws + (o + (loc << 8)); };
  auto task = [&](const uint4* ph, int i) { return reinterpret_cast<const Task*>(ph + 2 * i); };   // i: 1 + index
  auto ahead = [&](const uint4* ph, const uint4& h0, const uint4& h1) {
    const uint32_t r_x = h0.y >> 16;   // h0: n cells sums n_h | n_p n_x r d | x pad | main; h1: load carry
    if (has) {
      const int im = (h0.w >> (4 * el)) & 15, il = (h1.x >> (4 * el)) & 15, iz = (h1.y >> (4 * el)) & 15;
      if (im) {
        const Task& k = *task(ph, im);
        if (k.kind == FWD) {
          om.v[4] = GRU ? to_f(*reinterpret_cast<const T*>(at(o_h, k.src))) : *reinterpret_cast<const float*>(at(o_c, k.src));
          if (!GRU && (k.flags & COPY_IN)) om.v[5] = to_f(*reinterpret_cast<const T*>(at(o_h, k.src)));
        } else {
          const char* g = at(o_g, k.src);
#pragma unroll
          for (int q = 0; q < 4; ++q) om.v[q] = to_f(*reinterpret_cast<const T*>(g + q * A.plane));
          om.v[4] = to_f(*reinterpret_cast<const T*>(at(o_h, k.dst)));
          if (!GRU) {
            om.v[5] = *reinterpret_cast<const float*>(at(o_c, k.src));
            om.v[6] = *reinterpret_cast<const float*>(at(o_c, k.dst));
          }
        }
      }
      if (il) ol.x = to_f(*reinterpret_cast<const T*>(at(o_h, task(ph, il)->src)));
      if (iz) {
        const Task& k = *task(ph, iz);
        oz = *reinterpret_cast<const float4*>(A.ws + (k.sidx == kNone ? o_cy + ((k.k + 1) & 1) * L * bh * 16 : o_dz + k.sidx * bh * 16));
      }
    }
    if (has_r && (r_x & 0xff)) o_target = __ldg(A.targets + i_r + (size_t)(task(ph, r_x & 0xff)->k - 1) * A.B * A.O);
    if (has_x && (h0.z & 0xff)) {
      const T* x = reinterpret_cast<const T*>(A.x) + i_x + (size_t)(task(ph, h0.z & 0xff)->k - 1) * A.B * A.I;
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

  int w = 0, i0 = 0, ph = 0;
  bool entered = true;       // first phase of a window
  const uint4* cur = windows;
  uint4 h0 = cur[0], h1 = cur[1];
  ahead(cur, h0, h1);
  for (; ph < A.phases; ++ph) {
    const uint32_t bar = bar0 - base + 8 * (ph & 1);
    const bool cells = (h0.x >> 8) & 0xff, sums = (h0.x >> 16) & 0xff;
    unsigned char* const dz_buf = area + C.at_dz + (size_t)(ph & 1) * L * C.dz_buf;
    float* const red = reinterpret_cast<float*>(area + C.at_red + (size_t)(ph & 1) * C.red_bytes);
    bool ok = true;
    if (ph > 0) ok = wait_for(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1);

    const int im = has ? (h0.w >> (4 * el)) & 15 : 0;
    const Task* const mt = task(cur, im);
    if (cells && has) {
      const int iz = (h1.y >> (4 * el)) & 15;
      float d[4];
      bool on = false;
      if (im && mt->kind == BWD) {
        on = true;
        float s0 = 0.f, s1 = 0.f;
        const int par = mt->k & 1, n = NT * C.ns_b, step = U * NB;
        const float* a = reinterpret_cast<const float*>(smem + p_at(el, 0, par)) + eju * NB + eb;
        const float* b = reinterpret_cast<const float*>(smem + p_at(el, 1, par)) + eju * NB + eb;
        if (!(mt->flags & FIRST))
#pragma unroll 4
          for (int i = 0; i < n; ++i) s0 += a[i * step];
#pragma unroll 4
        for (int i = 0; i < n; ++i) s1 += b[i * step];
        const float g[4] = {om.v[0], om.v[1], om.v[2], om.v[3]};
        cell_backward<GRU>(s0 + s1, g, om.v[4], om.v[5], om.v[6], dc, d);
        const float4 quad = make_float4(d[0], d[1], d[2], d[3]);
        *reinterpret_cast<float4*>(A.ws + (o_dz + mt->sidx * bh * 16)) = quad;
        if (mt->flags & CLOSE) *reinterpret_cast<float4*>(A.ws + (o_cy + (mt->k & 1) * L * bh * 16)) = quad;
        T* const hs = reinterpret_cast<T*>(A.ws + (o_st + mt->sidx * bh * (uint32_t)sizeof(T)));
        store(hs, om.v[4]);
        if (mt->flags & OPEN) store(hs + bh, to_f(*reinterpret_cast<const T*>(at(o_h, mt->src))));
      } else if (iz) {
        on = true;
        d[0] = oz.x; d[1] = oz.y; d[2] = oz.z; d[3] = oz.w;
      }
      if (on) {
        unsigned char* const my = dz_buf + el * C.dz_buf;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (MMA) put_planes<PL>(reinterpret_cast<bf16*>(my) + eb * (C.dz_pitch / 2) + zrow + q * zstep, NB * (C.dz_pitch / 2), d[q]);
          else reinterpret_cast<float*>(my)[(zrow + q) * NB + eb] = d[q];
        }
      }
    }
    bool stop = false;
    if (cells || !sums) stop = __syncthreads_or(!ok);

    // ---- products ----
    {
      Share sh{to, 0, 0, bar, C.kh};
      int first = 0;           // warp that takes the first piece of the next class
      const int step = U * NB * 4;
      auto back = [&](int l, bool input, bool own, int k) {
        const int ldw = C.pitch_w(l), skip = input ? 0 : l ? C.kh : C.kx, cols = (input ? C.kh : 0) + (own ? C.kh : 0);
        unsigned char* const d = dz_buf + l * C.dz_buf;
        sh.dst1 = p_at(l, 0, (k - 1) & 1);
        sh.dst0 = input ? p_at(l - 1, 1, k & 1) : sh.dst1;
        if constexpr (MMA) {
          shares_mma<NB, PL>(sm100::smem_u32(d), C.dz_pitch, sm100::smem_u32(weights(l) + skip), ldw * 2, 4 * U, cols, sh, (warp - first) & (kWarps - 1), lane);
          first += cols >> 5;
        } else {
          shares_fma<NB>(reinterpret_cast<const float*>(d), weights(l) + skip, ldw, 4 * U, cols, C.ns_b, step, sh, tid);
        }
      };
#pragma unroll 1
      for (int l = 0; l < L; ++l) {
        const int i = (h0.w >> (4 * l)) & 15, z = (h1.y >> (4 * l)) & 15;
        if (z) back(l, false, true, task(cur, z)->k + 1);
        if (!i) continue;
        const Task& k = *task(cur, i);
        if (k.kind == BWD) {
          back(l, l > 0, !(k.flags & CLOSE), k.k);
        } else {
          const int wk = (warp - first) & (kWarps - 1), ldw = C.pitch_w(l), nin = l ? C.kh : C.kx, pin = l ? C.pitch_h : C.pitch_x;
          float* const r = red + red_f(l);
          unsigned char* const in = area + k.sa * 16;
          unsigned char* const hs = area + k.sb * 16;
          if constexpr (MMA) units_mma<NB>(sm100::smem_u32(in), nin / 16, sm100::smem_u32(hs), C.kh / 16, pin, C.pitch_h, sm100::smem_u32(weights(l)), ldw * 2, U, C.ns_f[l], r, wk, lane);
          else rows_fma<NB>(reinterpret_cast<const float*>(in), pin / 4, nin / 4, reinterpret_cast<const float*>(hs), C.pitch_h / 4, C.kh / 4, weights(l), ldw, U, C.ns_f[l], r, wk, lane);
          first += (MMA ? (U + 7) / 8 : U) * C.ns_f[l];
        }
      }
      if (const int i = (h0.y >> 16) & 0xff) {       // R
        const int wk = (warp - first) & (kWarps - 1);
        unsigned char* const hs = area + task(cur, i)->sb * 16;
        first += MMA ? ((C.op + 15) >> 4) * C.ns_r : 0;
        if constexpr (MMA) readout_mma<NB>(sm100::smem_u32(hs), C.pitch_h, C.kh / 16, sm100::smem_u32(weights(L)), C.pitch_r() * 2, C.op, C.ns_r, red + red_r, wk, lane);
        else rows_fma<NB>(nullptr, 0, 0, reinterpret_cast<const float*>(hs), C.pitch_h / 4, C.kh / 4, weights(L), C.pitch_r(), C.op / 4, C.ns_r, red + red_r, wk, lane);
      }
      if (const int i = h0.y >> 24) {                // D
        const int k = task(cur, i)->k;
        unsigned char* const d = area + C.at_dy + (k & 1) * C.dy_buf;
        sh.dst0 = p_at(L - 1, 1, k & 1);
        if constexpr (MMA) shares_mma<NB, PL>(sm100::smem_u32(d), C.dy_pitch, sm100::smem_u32(weights(L)), C.pitch_r() * 2, C.op, C.kh, sh, (warp - first) & (kWarps - 1), lane);
        else shares_fma<NB>(reinterpret_cast<const float*>(d), weights(L), C.pitch_r(), C.op, C.kh, C.ns_b, step, sh, tid);
      }
    }
    if (sums) stop |= __syncthreads_or(!ok);
    if (stop) break;
    if (warp == kWarps - 1) {   // the operands have been read: a word to everybody, and what to expect oneself
      if (lane < NT) push(peer[lane] + area0 + C.at_dummy + 4 * rank, 0, peer[lane] + bar);
      if (lane == 31) sm100::mbar_arrive_expect_tx(bars + (ph & 1), (h0.x >> 24) * by_h + (h0.y & 0xff) * by_p + ((h0.y >> 8) & 0xff) * by_x + 4 * NT);
    }

    // ---- states, readouts, loads ----
    if (h0.x >> 24 || sums) {
      float hv = 0.f;
      const bool f = im && mt->kind == FWD;
      if (f) {
        const int ns = C.ns_f[el];
        const float4* p = reinterpret_cast<const float4*>(red + my_red) + eju * ns * NB + eb;
        float z[4] = {0.f, 0.f, 0.f, 0.f};
        for (int q = 0; q < ns; ++q, p += NB) {
          const float4 r = *p;
          z[0] += r.x; z[1] += r.y; z[2] += r.z; z[3] += r.w;
        }
        float g[4], cv;
        cell_forward<GRU>(z, bias, om.v[4], g, hv, cv);
        T stored;
        store(&stored, hv);
        *reinterpret_cast<T*>(at(o_h, mt->dst)) = stored;
        hv = to_f(stored);       // the others read what was stored
        if (!GRU) *reinterpret_cast<float*>(at(o_c, mt->dst)) = cv;
        if (mt->flags & GATES) {
          char* gp = at(o_g, mt->dst);
#pragma unroll
          for (int q = 0; q < 4; ++q) store(reinterpret_cast<T*>(gp + q * A.plane), g[q]);
        }
        if (mt->flags & COPY_IN) {
          store(reinterpret_cast<T*>(at(o_h, mt->dst) + A.rec_in), GRU ? om.v[4] : om.v[5]);
          if (!GRU) *reinterpret_cast<float*>(at(o_c, mt->dst) + A.rec_in) = om.v[4];
        }
      }
      auto send = [&](float v, uint32_t so, bool on) {
        const float4 q = gather4(v);
        if (on)
          for (int r = eju & 3; r < NT; r += 4) push_quad(peer[r], area0 + so * 16 + at_push, q, bar);
      };
      if (h0.w) {
        // (a group of four may hold units past the last one: their tasks are those of the group)
        const int gi = sends ? (h0.w >> (4 * el)) & 15 : 0;
        const Task* const gt = task(cur, gi);
        const bool on = gi && gt->kind == FWD && gt->so != kNone;
        send(hv, on ? gt->so : 0, on);
      }
      if (h1.x) {
        const int gi = sends ? (h1.x >> (4 * el)) & 15 : 0;
        send(has ? ol.x : 0.f, gi ? task(cur, gi)->so : 0, gi != 0);
      }
    }
    if (has_r && ((h0.y >> 16) & 0xff)) {
      const Task& k = *task(cur, (h0.y >> 16) & 0xff);
      const float* p = red + red_r + (MMA ? ((rj >> 4) * C.ns_r * 16 + (rj & 15)) * NB + rb : (rj >> 2) * C.ns_r * NB * 4 + rb * 4 + (rj & 3));
      float z = 0.f;
      for (int q = 0; q < C.ns_r; ++q, p += MMA ? 16 * NB : NB * 4) z += *p;
      const float dy = 2.f * (z + r_bias - o_target) * dy_scale;
      reinterpret_cast<float*>(A.ws + A.off_dy)[i_r + k.sidx * A.B * A.O] = dy;
      unsigned char* const d = area + C.at_dy + (k.k & 1) * C.dy_buf;
      if (MMA) put_planes<PL>(reinterpret_cast<bf16*>(d) + rb * (C.dy_pitch / 2) + rj, NB * (C.dy_pitch / 2), dy);
      else reinterpret_cast<float*>(d)[rj * NB + rb] = dy;
    }
    if (has_x && (h0.z & 0xff)) {
      const uint32_t off = area0 + task(cur, h0.z & 0xff)->so * 16 + xb * C.pitch_x + 4 * xg * (uint32_t)sizeof(T);
      for (int r = 0; r < NT; ++r) push_quad(peer[r], off, ox, bar);
    }
    if (entered && w + 2 < n_windows) load_window(w + 2);
    entered = false;
    i0 += 1 + (h0.x & 0xff);
    if (ph + 1 < A.phases) {
      cur = windows + ((w & (kWindows - 1)) * kWindow + i0) * 2;
      if (i0 >= kWindow || (reinterpret_cast<const uint32_t*>(cur)[0] & 0xff) == 0) {
        ++w; i0 = 0; entered = true;
        cur = windows + (w & (kWindows - 1)) * kWindow * 2;
      }
      h0 = cur[0]; h1 = cur[1];
      ahead(cur, h0, h1);
    }
  }
  bool ok = ph == A.phases;
  if (ok && ph > 0) ok = wait_for(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1);
  if (!ok) *A.status = MEBPTT_ERR_TIMEOUT;
  if (has) *dc_at() = dc;
  // nobody leaves while pushes to its shared memory may be under way
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
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
      reinterpret_cast<T*>(P.init + l * P.hc)[i] = reinterpret_cast<const T*>(P.h0)[l * bh + i];
      reinterpret_cast<float*>(P.init + l * P.hc + P.csz_off)[i] = P.c0[l * bh + i];
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

template <class T, bool GRU, int PL>
Fn by_rows(int nb) {
  return nb == 1 ? pod_walk<T, GRU, 1, PL> : nb == 2 ? pod_walk<T, GRU, 2, PL> : nb == 4 ? pod_walk<T, GRU, 4, PL> : pod_walk<T, GRU, 8, PL>;
}

}  // namespace

Fn kernel(int dtype, bool gru, int nb) {
  if (dtype == MEBPTT_BF16) return gru ? by_rows<bf16, true, 3>(nb) : by_rows<bf16, false, 3>(nb);
  return gru ? by_rows<float, true, 1>(nb) : by_rows<float, false, 1>(nb);
}

void launch_pack(int dtype, bool gru, const PackArgs& p, cudaStream_t s) {
  if (dtype == MEBPTT_BF16) {
    if (gru) pod_pack<bf16, true><<<592, 256, 0, s>>>(p); else pod_pack<bf16, false><<<592, 256, 0, s>>>(p);
  } else {
    if (gru) pod_pack<float, true><<<592, 256, 0, s>>>(p); else pod_pack<float, false><<<592, 256, 0, s>>>(p);
  }
}

}  // namespace pod
}  // namespace mebptt
