// Kernels and launches of the team path (team.hpp has the scheme).
//
// One persistent kernel walks the phases of a chunk: float32 FMA arithmetic whatever the storage type
// (operands are widened, all sums are float32 in a fixed order), weights of the CTA's hidden units in
// shared memory.  What bounds it is the chain of phases: at the sizes it serves the arithmetic of a
// phase is a fraction of a microsecond, and the rest is the trip of the new states through the L2 and
// the meeting of the team.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <type_traits>
#include <vector>

#include "env.hpp"
#include "kernels.hpp"
#include "launch.hpp"
#include "layout.hpp"
#include "plan.hpp"
#include "sm100.cuh"
#include "pod.hpp"
#include "pod_run.hpp"
#include "team.hpp"
#include "team_dev.cuh"
#include "team_run.hpp"

namespace mebptt {
namespace team {

namespace {

struct Args {
  int L, I, H, O, B, S;
  int T, rows;
  Dims d;
  int ns_f[kMaxLayers], ns_b[kMaxLayers], ns_r;
  uint64_t resident;
  int pool_floats;
  size_t off_states;                   // states, by team
  int64_t n_blocks;
  int parts;
  char* ws;
  size_t off_wf[kMaxLayers], off_wb[kMaxLayers], off_wr;
  size_t off_dz, off_hk, off_dy, off_carry, off_dc;
  const void* x;
  const float *bias, *b_out, *targets;
  const Task* tasks;
  int n_tasks;
  unsigned* sync;                      // one 128-byte line per team
  unsigned sync_base;                  // arrivals before this launch, per team
  unsigned polls;                      // a wait gives up after so many polls
  int* status;
  int64_t* counters;
};

// Four weight rows (ld apart) against NB operand rows (lda apart) over the 128-wide slices [i0, i1) of
// the contraction index (nv float4 in all).  Each lane takes four consecutive elements of a slice.
template <class T, int NB>
__device__ __forceinline__ void four_rows(const float* a, int lda, const T* w, int ldw, int i0, int i1, int nv, int lane,
                                          float (&acc)[NB * 4]) {
  for (int i = i0; i < i1; ++i) {
    const int v = i * 32 + lane;
    if (v < nv) {
      float4 wr[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) wr[r] = load4(w + (size_t)r * ldw + 4 * v);
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float4 x = *reinterpret_cast<const float4*>(a + (size_t)b * lda + 4 * v);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float s = acc[b * 4 + r];
          s = fmaf(x.x, wr[r].x, s);
          s = fmaf(x.y, wr[r].y, s);
          s = fmaf(x.z, wr[r].z, s);
          acc[b * 4 + r] = fmaf(x.w, wr[r].w, s);
        }
      }
    }
  }
}

// Four values as float32.
__device__ __forceinline__ float4 widen(float4 v) { return v; }
__device__ __forceinline__ float4 widen(uint2 v) {
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}

// ---- operands -------------------------------------------------------------------------------

// Four consecutive elements p[0..3] of which the first n exist, from the L2.
__device__ __forceinline__ float4 piece(const float* p, int n, bool whole) {
  if (whole && n >= 4) return __ldcg(reinterpret_cast<const float4*>(p));
  return make_float4(n > 0 ? __ldcg(p) : 0.f, n > 1 ? __ldcg(p + 1) : 0.f, n > 2 ? __ldcg(p + 2) : 0.f, n > 3 ? __ldcg(p + 3) : 0.f);
}
__device__ __forceinline__ uint2 piece(const __nv_bfloat16* p, int n, bool whole) {
  if (whole && n >= 4) return __ldcg(reinterpret_cast<const uint2*>(p));
  const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
  uint2 r = make_uint2(0, 0);
  if (n > 0) r.x = __ldcg(q);
  if (n > 1) r.x |= (uint32_t)__ldcg(q + 1) << 16;
  if (n > 2) r.y = __ldcg(q + 2);
  if (n > 3) r.y |= (uint32_t)__ldcg(q + 3) << 16;
  return r;
}
// Brings NB rows of `len` elements (`padded` with zeros, ld apart in memory) to wherever put(row, element,
// piece) wants them.  A warp has one row; its loads are under way together.
template <int NB, class T, class Put>
__device__ __forceinline__ void stage(const T* src, size_t ld, int len, int padded, int valid, int warp, int lane, Put put) {
  const bool whole = ((ld | (size_t)len) & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & (4 * sizeof(T) - 1)) == 0;
  const int b = warp & (NB - 1), stride = (kWarps / NB) * 32;
  const T* row = src + (size_t)b * ld;
  const int lim = b < valid ? len : 0;
  for (int v = (warp / NB) * 32 + lane; v < padded >> 2; v += 4 * stride) {
    decltype(piece(row, 0, true)) x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = piece(row + 4 * (v + i * stride), lim - 4 * (v + i * stride), whole);
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (v + i * stride < padded >> 2) put(b, 4 * (v + i * stride), x[i]);
  }
}

// A group of 16 weight rows in the order of the tensor cores' fragments against up to 8 operand rows in PL
// bfloat16 planes, steps [lo, hi) of 16; c[0], c[1]: row lane / 4, batch rows 2 (lane & 3), + 1; c[2], c[3]: row + 8.
template <int NB, int PL>
__device__ __forceinline__ void sixteen_rows(uint32_t a, uint32_t pitch, const uint4* w, int lo, int hi, int lane, float (&c)[4]) {
  const uint32_t at = a + ((lane & 7) % NB) * pitch + ((lane >> 3) & 1) * 16;
#pragma unroll 4
  for (int k = lo; k < hi; ++k) {
    const uint4 f = w[k * 32 + lane];
#pragma unroll
    for (int p = 0; p < PL; ++p) {
      uint32_t b0, b1;
      asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(b0), "=r"(b1) : "r"(at + p * NB * pitch + k * 32) : "memory");
      asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                   : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(f.x), "r"(f.y), "r"(f.z), "r"(f.w), "r"(b0), "r"(b1));
    }
  }
}

// What a task's element needs from memory beside its sums; fetched while the operands are staged.
struct Operands { float v[9]; };

template <class T, bool GRU>
__device__ __forceinline__ void fetch(const Args& A, const States<T>& S, const Task& t, size_t row, int lr, int j, Operands& o) {
  const int H = A.H, l = t.layer;
  const size_t e = row * H + j, le = (size_t)lr * H + j;   // among all rows, among the team's
  if (t.kind == FWD) {
    const float* bias = A.bias + (size_t)l * (GRU ? 3 : 4) * H + j;
#pragma unroll
    for (int q = 0; q < (GRU ? 3 : 4); ++q) o.v[q] = __ldg(bias + (size_t)q * H);
    if (GRU) {
      o.v[4] = to_f(ld_l2(S.h(t.src, l) + le));
    } else {
      o.v[4] = ld_l2(S.c(t.src, l) + le);
      if (t.flags & COPY_IN) o.v[5] = to_f(ld_l2(S.h(t.src, l) + le));
    }
  } else if (t.kind == READ) {
    o.v[0] = __ldg(A.b_out + j);
    o.v[1] = __ldg(A.targets + ((size_t)(t.k - 1) * A.B + row) * A.O + j);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) o.v[q] = to_f(ld_l2(S.gate(t.src, A.L, l, q) + le));
    o.v[4] = ld_l2(reinterpret_cast<const float*>(A.ws + A.off_dc) + (size_t)l * A.B * H + e);
    o.v[5] = to_f(ld_l2(S.h(t.dst, l) + le));   // h_{k-1}
    if (t.flags & CARRY_IN) o.v[6] = to_f(ld_l2(S.h(t.src, l) + le));   // h_k
    if (!GRU) {
      o.v[7] = ld_l2(S.c(t.src, l) + le);
      o.v[8] = ld_l2(S.c(t.dst, l) + le);
    }
  }
}

// z: the element's sums (four gates; one value for R and B).
template <class T, bool GRU>
__device__ __forceinline__ void apply(const Args& A, const States<T>& S, const Task& t, size_t row, int lr, int j, const Operands& o, const float (&z)[4]) {
  const int H = A.H, l = t.layer;
  const size_t e = row * H + j, le = (size_t)lr * H + j;
  if (t.kind == FWD) {
    const float bias[4] = {o.v[0], o.v[1], o.v[2], o.v[3]}, cp = o.v[4];
    float gv[4], h, cv;
    cell_forward<GRU>(z, bias, cp, gv, h, cv);
    store(S.h(t.dst, l) + le, h);
    if (!GRU) S.c(t.dst, l)[le] = cv;
    if (t.flags & GATES) {
#pragma unroll
      for (int q = 0; q < 4; ++q) store(S.gate(t.dst, A.L, l, q) + le, gv[q]);
    }
    if (t.flags & COPY_IN) {
      const uint32_t in = S.input(t.dst, A.L);
      store(S.h(in, l) + le, GRU ? cp : o.v[5]);
      if (!GRU) S.c(in, l)[le] = cp;
    }
  } else if (t.kind == READ) {
    const float d = z[0] + o.v[0] - o.v[1];
    reinterpret_cast<float*>(A.ws + A.off_dy)[((size_t)t.sidx * A.B + row) * A.O + j] = 2.f * d * (1.f / ((float)A.B * (float)A.O));
  } else {
    const size_t G = (size_t)4 * H, srow = ((size_t)l * A.S + t.sidx) * A.B + row;
    float* dc_p = reinterpret_cast<float*>(A.ws + A.off_dc) + (size_t)l * A.B * H + e;
    const float gv[4] = {o.v[0], o.v[1], o.v[2], o.v[3]};
    float d4[4], carry = o.v[4];
    cell_backward<GRU>(z[0], gv, o.v[5], o.v[7], o.v[8], carry, d4);
    *dc_p = carry;
    const float4 quad = make_float4(d4[0], d4[1], d4[2], d4[3]);   // the four gates of a unit side by side
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(A.ws + A.off_dz) + srow * G + 4 * j) = quad;
    if (t.flags & CARRY_OUT)
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(A.ws + A.off_carry) + (((size_t)(t.k & 1) * A.L + l) * A.B + row) * G + 4 * j) = quad;
    T* hs = reinterpret_cast<T*>(A.ws + A.off_hk) + (((size_t)l * (A.S + 1) + t.sidx) * A.B + row) * H + j;
    store(hs, o.v[5]);                                                    // h_{k-1}
    if (t.flags & CARRY_IN) store(hs + (size_t)A.B * H, o.v[6]);          // the chunk's last step: h_k too
  }
}

// Meeting of the team's CTAs: everything written before it is visible after it.
__device__ __forceinline__ bool meet(const Args& A, unsigned* line, unsigned target, volatile int* flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(line) : "memory");
    bool ok = false;
    for (uint32_t i = 0; i < sm100::kSpinLimit; ++i) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(line) : "memory");
      if ((int)(v - target) >= 0) { ok = true; break; }
      if (i > 256) {
        if (i >= A.polls) break;
        __nanosleep(32);
      }
    }
    if (!ok) { *A.status = MEBPTT_ERR_TIMEOUT; *flag = 1; }
  }
  __syncthreads();
  return *flag == 0;
}

template <class T, bool GRU, int NB, bool MMA>
__global__ void __launch_bounds__(kThreads, 1) walk(const __grid_constant__ Args A) {
  constexpr int RPG = MMA ? 16 : 4, UPG = RPG / 4;                    // rows of a group, units of a forward group
  extern __shared__ __align__(128) unsigned char smem[];
  Task* window = reinterpret_cast<Task*>(smem);                       // two windows of tasks
  volatile int& s_flag = *reinterpret_cast<volatile int*>(smem + 2 * kTaskWindow * sizeof(Task));
  float* pool = reinterpret_cast<float*>(smem + 2 * kTaskWindow * sizeof(Task) + 256);
  T* held = reinterpret_cast<T*>(pool + A.pool_floats);               // resident weights
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int team = blockIdx.x / A.T, rank = blockIdx.x - team * A.T;
  const int H = A.H, L = A.L;
  const int row0 = team * A.rows, rows = min(A.rows, A.B - row0);
  const States<T> S(A.ws + A.off_states, A.n_blocks, A.parts, team, A.rows, A.B, H);
  if (tid == 0) s_flag = *A.status;   // an earlier launch gave up: do nothing
  int f0, f1, b0, b1, r0g, r1g;       // groups of this CTA
  part(A.d.gf, A.T, rank, f0, f1);
  part(A.d.gb, A.T, rank, b0, b1);
  part(A.d.gr, A.T, rank, r0g, r1g);
  // first column (unit, readout row) and number of columns of the CTA by kind of task
  auto cols_at = [&](int kind) { return kind == FWD ? f0 * UPG : (kind == READ ? r0g : b0) * RPG; };
  auto cols_of = [&](int kind) {
    return max(0, kind == FWD ? min(f1 * UPG, H) - f0 * UPG : kind == READ ? min(r1g * RPG, A.O) - r0g * RPG : min(b1 * RPG, H) - b0 * RPG);
  };
  auto groups_of = [&](int kind) { return kind == FWD ? f1 - f0 : kind == READ ? r1g - r0g : b1 - b0; };
  auto splits_of = [&](const Task& k) { return k.kind == FWD ? A.ns_f[k.layer] : k.kind == READ ? A.ns_r : A.ns_b[k.layer]; };
  auto width_of = [&](const Task& k) { return k.kind == FWD ? A.d.kf[k.layer] : k.kind == READ ? A.d.hp : A.d.kb[k.layer]; };

  // resident weights, in the order of their bits; offsets in elements
  const int nf = (f1 - f0) * RPG, nbk = (b1 - b0) * RPG, nr = (r1g - r0g) * RPG;
  auto f_at = [&](int l) { int o = 0; for (int i = 0; i < l; ++i) if (A.resident >> (2 * i) & 1) o += nf * A.d.kf[i]; return o; };
  auto b_at = [&](int l) {
    int o = f_at(L);
    for (int i = 0; i < l; ++i) if (A.resident >> (2 * i + 1) & 1) o += nbk * A.d.kb[i];
    return o;
  };
  auto copy_in = [&](T* dst, const T* src, size_t n) {   // n is a multiple of 8, both sides are 16-byte aligned
    const uint4* s4 = reinterpret_cast<const uint4*>(src);
    uint4* d4 = reinterpret_cast<uint4*>(dst);
    const int q = (int)(n * sizeof(T) / 16);
    for (int i = tid; i < q; i += kThreads) d4[i] = __ldcg(s4 + i);
  };
  for (int l = 0; l < L; ++l) {
    const T* wf = reinterpret_cast<const T*>(A.ws + A.off_wf[l]) + (size_t)f0 * RPG * A.d.kf[l];
    const T* wb = reinterpret_cast<const T*>(A.ws + A.off_wb[l]) + (size_t)b0 * RPG * A.d.kb[l];
    if (A.resident >> (2 * l) & 1) copy_in(held + f_at(l), wf, (size_t)nf * A.d.kf[l]);
    if (A.resident >> (2 * l + 1) & 1) copy_in(held + b_at(l), wb, (size_t)nbk * A.d.kb[l]);
  }
  if (A.resident >> 63) copy_in(held + b_at(L), reinterpret_cast<const T*>(A.ws + A.off_wr) + (size_t)r0g * RPG * A.d.hp, (size_t)nr * A.d.hp);

  auto load_window = [&](int w) {
    if (tid < kTaskWindow * 2)
      reinterpret_cast<uint4*>(window + (w & 1) * kTaskWindow)[tid] =
          __ldg(reinterpret_cast<const uint4*>(A.tasks + (size_t)w * kTaskWindow) + tid);
  };
  const int windows = A.n_tasks / kTaskWindow;
  load_window(0);
  __syncthreads();
  if (s_flag != 0) return;

  int64_t fwd_ops = 0, bwd_ops = 0;
  unsigned target = A.sync_base;
  int w = 0, i0 = 0;
  if (windows > 1) load_window(1);
  while (w < windows) {
    const Task* t = window + (w & 1) * kTaskWindow + i0;
    if (i0 >= kTaskWindow || t[0].kind == NOP) {   // next window; the one after it is fetched meanwhile
      ++w; i0 = 0;
      __syncthreads();
      if (w + 1 < windows) load_window(w + 1);
      continue;
    }
    int n = 1;
    while (!(t[n - 1].flags & LAST)) ++n;
    i0 += n;
    for (int sub = 0; sub * NB < rows; ++sub) {
      const int r0 = row0 + sub * NB, valid = min(NB, rows - sub * NB);
      int works = 0, elems = 0;
      // operands of every task of the phase
      for (int i = 0; i < n; ++i) {
        const Task& k = t[i];
        const int l = k.layer, width = width_of(k);
        float* const a = pool + k.a_off;
        // values as they are stored: float32, or bfloat16 rows width + 8 apart
        auto plain = [&](const T* src, int first, int len, int padded, int at) {
          stage<NB>(src + (size_t)first * len, (size_t)len, len, padded, valid, warp, lane, [&](int b, int e, auto x) {
            if constexpr (MMA) *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a) + b * (width + 8) + at + e) = x;
            else *reinterpret_cast<float4*>(a + b * width + at + e) = widen(x);
          });
        };
        // float32 gradients, on the tensor cores as three bfloat16 planes that add up to them
        auto gradient = [&](const float* src, int len, int padded, int at) {
          stage<NB>(src + (size_t)r0 * len, (size_t)len, len, padded, valid, warp, lane, [&](int b, int e, float4 v) {
            if constexpr (MMA) {
              __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(a) + b * (width + 8) + at + e;
#pragma unroll
              for (int q = 0; q < 3; ++q) {
                const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
                *reinterpret_cast<uint2*>(d + q * NB * (width + 8)) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
                v.x -= __low2float(lo); v.y -= __high2float(lo); v.z -= __low2float(hi); v.w -= __high2float(hi);
              }
            } else {
              *reinterpret_cast<float4*>(a + b * width + at + e) = v;
            }
          });
        };
        if (k.kind == FWD) {
          plain(l ? S.h(k.dst, l - 1) : reinterpret_cast<const T*>(A.x) + (size_t)(k.k - 1) * A.B * A.I, l ? sub * NB : r0, l ? H : A.I, A.d.ip[l], 0);
          plain(S.h(k.src, l), sub * NB, H, A.d.hp, A.d.ip[l]);
        } else if (k.kind == READ) {
          plain(S.h(k.src, l), sub * NB, H, A.d.hp, 0);
        } else {
          const int G = 4 * H;
          const float* const dz = reinterpret_cast<const float*>(A.ws + A.off_dz);
          gradient((k.flags & CARRY_IN) ? reinterpret_cast<const float*>(A.ws + A.off_carry) + ((size_t)((k.k + 1) & 1) * L + l) * A.B * G
                                        : dz + ((size_t)l * A.S + k.sidx + 1) * A.B * G,
                   G, A.d.gp, 0);
          if (l + 1 < L) gradient(dz + ((size_t)(l + 1) * A.S + k.sidx) * A.B * G, G, A.d.gp, A.d.gp);
          else gradient(reinterpret_cast<const float*>(A.ws + A.off_dy) + (size_t)k.sidx * A.B * A.O, A.O, width - A.d.gp, A.d.gp);
        }
        works += groups_of(k.kind) * splits_of(k);
        elems += cols_of(k.kind) * NB;
      }
      // element f of the phase: its task, batch row (the fast index) and column
      auto locate = [&](int f, const Task*& k, int& b, int& j) {
        for (int i = 0; i < n; ++i) {
          k = t + i;
          const int m = cols_of(k->kind) * NB;
          if (f < m) { b = f & (NB - 1); j = f / NB; return; }
          f -= m;
        }
      };
      Operands o;
      const Task* ek = nullptr;
      int eb = 0, ej = 0;
      if (tid < elems) {
        locate(tid, ek, eb, ej);
        if (eb < valid) fetch<T, GRU>(A, S, *ek, (size_t)(r0 + eb), sub * NB + eb, cols_at(ek->kind) + ej, o);
      }
      __syncthreads();
      // partial sums
      for (int wk = warp; wk < works; wk += kWarps) {
        int rem = wk, i = 0, ns = 1;
        for (;; ++i) {
          ns = splits_of(t[i]);
          const int m = groups_of(t[i].kind) * ns;
          if (rem < m) break;
          rem -= m;
        }
        const Task& k = t[i];
        const int l = k.layer, g = rem / ns, s = rem - g * ns, ld = width_of(k);
        const int bit = k.kind == FWD ? 2 * l : k.kind == READ ? 63 : 2 * l + 1;
        const bool res = A.resident >> bit & 1;
        const T* wg;
        if (res) {
          wg = held + (k.kind == FWD ? f_at(l) : k.kind == READ ? b_at(L) : b_at(l)) + (size_t)g * RPG * ld;
        } else {
          const size_t off = k.kind == FWD ? A.off_wf[l] : k.kind == READ ? A.off_wr : A.off_wb[l];
          wg = reinterpret_cast<const T*>(A.ws + off) + (size_t)((k.kind == FWD ? f0 : k.kind == READ ? r0g : b0) + g) * RPG * ld;
        }
        float* const red = pool + k.red_off + (size_t)(g * ns + s) * NB * RPG;
        if constexpr (MMA) {
          const int steps = ld >> 4, lo = steps * s / ns, hi = steps * (s + 1) / ns;
          float c[4] = {};
          const uint32_t a = sm100::smem_u32(pool + k.a_off), pitch = (ld + 8) * 2;
          if (k.kind == BWD) sixteen_rows<NB, 3>(a, pitch, reinterpret_cast<const uint4*>(wg), lo, hi, lane, c);
          else sixteen_rows<NB, 1>(a, pitch, reinterpret_cast<const uint4*>(wg), lo, hi, lane, c);
          const int c0 = 2 * (lane & 3), r = lane >> 2;
          if (c0 < NB) {   // [batch row][16]
            red[c0 * 16 + r] = c[0]; red[c0 * 16 + r + 8] = c[2];
            if (NB > 1) { red[(c0 + 1) * 16 + r] = c[1]; red[(c0 + 1) * 16 + r + 8] = c[3]; }
          }
        } else {
          const int nv = ld >> 2, its = (nv + 31) >> 5;
          float acc[NB * 4];
#pragma unroll
          for (int q = 0; q < NB * 4; ++q) acc[q] = 0.f;
          four_rows<T, NB>(pool + k.a_off, ld, wg, ld, its * s / ns, its * (s + 1) / ns, nv, lane, acc);
          const float v = lane_sums<NB * 4>(acc, lane);
          constexpr int per = 32 / (NB * 4);
          if (lane % per == 0) red[lane / per] = v;   // [batch row][4]
        }
      }
      __syncthreads();
      for (int f = tid; f < elems; f += kThreads) {
        if (f != tid) {
          locate(f, ek, eb, ej);
          if (eb < valid) fetch<T, GRU>(A, S, *ek, (size_t)(r0 + eb), sub * NB + eb, cols_at(ek->kind) + ej, o);
        }
        if (eb >= valid) continue;
        const Task& k = *ek;
        const int ns = splits_of(k), per = k.kind == FWD ? UPG : RPG, g = ej / per, in = ej - g * per;
        const float* p = pool + k.red_off + (size_t)g * ns * NB * RPG + eb * RPG;
        float z[4] = {0.f, 0.f, 0.f, 0.f};
        if (k.kind == FWD) {
          p += in * 4;
          for (int s = 0; s < ns; ++s, p += NB * RPG) {
            const float4 v = *reinterpret_cast<const float4*>(p);
            z[0] += v.x; z[1] += v.y; z[2] += v.z; z[3] += v.w;
          }
        } else {
          p += in;
          for (int s = 0; s < ns; ++s, p += NB * RPG) z[0] += *p;
        }
        apply<T, GRU>(A, S, k, (size_t)(r0 + eb), sub * NB + eb, cols_at(k.kind) + ej, o, z);
      }
      if ((sub + 1) * NB < rows) __syncthreads();
    }
    if (tid == 0 && blockIdx.x == 0)
      for (int i = 0; i < n; ++i)
        if (t[i].flags & COUNT) { if (t[i].kind == FWD) ++fwd_ops; else ++bwd_ops; }
    target += (unsigned)A.T;
    if (!meet(A, A.sync + (size_t)team * 32, target, &s_flag)) return;
  }
  if (tid == 0 && blockIdx.x == 0) {
    A.counters[0] += fwd_ops;
    A.counters[1] += bwd_ops;
  }
}

// ---- what surrounds the walk ---------------------------------------------------------------

// Packed weights, zeroed carries and counters.  Blocks of 32 x 32 elements; the transposed matrices
// go through shared memory so that both sides are read and written along rows.
template <class T>
struct PackArgs {
  int L, I, H, O;
  Dims d;
  const T *W, *W_out;
  size_t w_off[kMaxLayers];
  T *wf[kMaxLayers], *wb[kMaxLayers], *wr;
  char* states; int64_t n_blocks, init; int parts, R;   // the caller's initial state goes to block `init` of each group's states
  const void* h0; const float* c0;
  int B;
  float* zero; size_t n_zero;     // carried gradients, sync lines, status
  int64_t* counters;
};

// Where element (row, column) of a matrix of rows of `width` goes: row after row, or in the order of the
// tensor cores' fragments, 16 rows a tile: [tile][16 columns][lane][8].
template <bool MMA>
__device__ __forceinline__ size_t place(int row, int col, int width) {
  if (!MMA) return (size_t)row * width + col;
  const int r = row & 15, c = col & 15, lane = (r & 7) * 4 + ((c & 7) >> 1), reg = (r >> 3) + 2 * (c >> 3);
  return (((size_t)(row >> 4) * (width >> 4) + (col >> 4)) * 32 + lane) * 8 + reg * 2 + (c & 1);
}

template <class T, bool GRU, bool MMA>
__global__ void __launch_bounds__(256) pack(const PackArgs<T> P) {
  const int rf = P.d.gf * P.d.rpg, rb = P.d.gb * P.d.rpg, rr = P.d.gr * P.d.rpg;   // rows with the padding
  __shared__ float tile[32][33];
  const int x = threadIdx.x & 31, y0 = threadIdx.x >> 5, H = P.H;
  for (size_t i = blockIdx.x * 256 + threadIdx.x; i < P.n_zero; i += (size_t)gridDim.x * 256) P.zero[i] = 0.f;
  if (blockIdx.x == 0 && threadIdx.x < 8) P.counters[threadIdx.x] = 0;
  const size_t bh = (size_t)P.B * H;
  for (int l = 0; l < P.L; ++l)
    for (size_t i = blockIdx.x * 256 + threadIdx.x; i < bh; i += (size_t)gridDim.x * 256) {
      const int b = (int)(i / H), g = b / P.R;
      const States<T> S(P.states, P.n_blocks, P.parts, g, P.R, P.B, H);
      const size_t le = i - (size_t)g * P.R * H;
      S.h((uint32_t)P.init, l)[le] = reinterpret_cast<const T*>(P.h0)[l * bh + i];
      S.c((uint32_t)P.init, l)[le] = P.c0[l * bh + i];
    }
  auto tiles = [](int rows, int cols) { return ((rows + 31) / 32) * ((cols + 31) / 32); };
  int total = tiles(rr, P.d.hp);
  for (int l = 0; l < P.L; ++l) total += tiles(rf, P.d.kf[l]) + tiles(rb, P.d.kb[l]);
  for (int b = blockIdx.x; b < total; b += gridDim.x) {
    int t = b, l = 0, what = 0;   // 0: forward rows, 1: transposed, 2: readout
    for (; l < P.L; ++l) {
      int n = tiles(rf, P.d.kf[l]);
      if (t < n) { what = 0; break; }
      t -= n;
      n = tiles(rb, P.d.kb[l]);
      if (t < n) { what = 1; break; }
      t -= n;
    }
    if (l == P.L) what = 2;
    if (what == 0) {
      const int kf = P.d.kf[l], nx = (kf + 31) / 32, r0 = (t / nx) * 32, c = (t % nx) * 32 + x;
      const int I = l ? H : P.I, K = I + H, ip = P.d.ip[l];
      const T* W = P.W + P.w_off[l];
      for (int r = r0 + y0; r < r0 + 32 && r < rf; r += 8) {
        if (c >= kf) continue;
        const int j = r >> 2, q = r & 3;
        const bool rec = c >= ip;
        const int col = rec ? c - ip + I : c;
        bool on = rec ? c - ip < H : c < I;
        int row = q * H + j;
        if (GRU && q >= 2) { on = on && (rec == (q == 3)); row = 2 * H + j; }
        P.wf[l][place<MMA>(r, c, kf)] = on && j < H ? W[(size_t)row * K + col] : T(0.f);
      }
    } else if (what == 2) {
      const int hp = P.d.hp, nx = (hp + 31) / 32, r0 = (t / nx) * 32, c = (t % nx) * 32 + x;
      for (int r = r0 + y0; r < r0 + 32 && r < rr; r += 8)
        if (c < hp) P.wr[place<MMA>(r, c, hp)] = (r < P.O && c < H) ? P.W_out[(size_t)r * H + c] : T(0.f);
    } else {
      // out[j][g]: tile rows j0.., columns g0..; read with j fastest
      const int kb = P.d.kb[l], nx = (kb + 31) / 32, j0 = (t / nx) * 32, g0 = (t % nx) * 32;
      const bool top = l + 1 == P.L;
      for (int yy = y0; yy < 32; yy += 8) {
        const int g = g0 + yy, j = j0 + x;
        float v = 0.f;
        if (j < H && g < kb) {
          if (g < P.d.gp) {
            if (g < 4 * H) {
              const int c = g & 3, u = g >> 2, row = (GRU && c == 3 ? 2 : c) * H + u, I = l ? H : P.I;
              if (!(GRU && c == 2)) v = to_f(P.W[P.w_off[l] + (size_t)row * (I + H) + I + j]);
            }
          } else if (top) {
            const int o = g - P.d.gp;
            if (o < P.O) v = to_f(P.W_out[(size_t)o * H + j]);
          } else {
            const int gu = g - P.d.gp, c = gu & 3, u = gu >> 2;
            if (u < H && !(GRU && c == 3)) v = to_f(P.W[P.w_off[l + 1] + (size_t)(c * H + u) * (2 * H) + j]);
          }
        }
        tile[yy][x] = v;
      }
      __syncthreads();
      for (int yy = y0; yy < 32; yy += 8) {
        const int j = j0 + yy, g = g0 + x;
        if (j < rb && g < kb) store(P.wb[l] + place<MMA>(j, g, kb), tile[x][yy]);
      }
      __syncthreads();
    }
  }
}

// The contractions of a finished chunk: weight gradients and dx, all in one launch, 64 x 64 tiles.
// C[m][n] (+)= sum_k A(m, k) B[k][n]; A is stored [k][m] (a_mn) or [m][k].  The contraction index is summed in
// blocks, each by itself, and the blocks are added to C from the last to the first: with blocks of a fixed
// number of time steps the result does not depend on how many steps a chunk has.
struct Product {
  const float* A; const void* B; float* C;
  int lda, ldb, ldc, M, N, K, block, a_mn, accumulate, tile0;
  int H, skip, last;   // H > 0: gate rows 4 u + q of A (a_mn) or of the contraction belong to rows q H + u of the weights;
                       // rows with q == skip to none, and those with q == 3 to block `last`
};
constexpr int kMaxProducts = 2 * kMaxLayers + 2;
struct Products { int n, tiles; Product p[kMaxProducts]; };

// Row of the weights that gate row r of a stage belongs to; -1: none.
__device__ __forceinline__ int gate_row(const Product& p, int r) {
  if (!p.H) return r;
  const int q = r & 3;
  return q == p.skip ? -1 : (q == 3 ? p.last : q) * p.H + (r >> 2);
}

// A tile of a product is formed by two groups of 128 threads, each over every other slice of a block
// of the contraction index, so that the loads of one hide behind the arithmetic of the other (a chunk
// has few tiles: with one group an SM held eight warps that waited for one another); the second group's
// sums are added to the first's at the end of a block.  (Whole blocks to each group, an exchange for two
// of them: the second group is idle where a short sequence has one, up to 5 % of a step.)  Operands come
// in 16-byte pieces where their rows allow it.
constexpr int kTileThreads = 256;
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory"); }

// 4 consecutive values p[0..3], of which the first n exist.
__device__ __forceinline__ float4 load_some(const float* p, int n, bool whole) {
  if (whole && n >= 4) return *reinterpret_cast<const float4*>(p);
  return make_float4(n > 0 ? p[0] : 0.f, n > 1 ? p[1] : 0.f, n > 2 ? p[2] : 0.f, n > 3 ? p[3] : 0.f);
}
__device__ __forceinline__ uint2 load_some(const __nv_bfloat16* p, int n, bool whole) {
  if (whole && n >= 4) return *reinterpret_cast<const uint2*>(p);
  const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
  uint2 r = make_uint2(0, 0);
  if (n > 0) r.x = q[0];
  if (n > 1) r.x |= (uint32_t)q[1] << 16;
  if (n > 2) r.y = q[2];
  if (n > 3) r.y |= (uint32_t)q[3] << 16;
  return r;
}

// The pieces of a slice of TK steps that a thread brings: N = TK / 8 of A and of B.
template <class T, int TK>
struct Slice {
  static constexpr int N = TK / 8;
  using Piece = typename std::conditional<std::is_same<T, float>::value, float4, uint2>::type;
  float4 a[N];
  Piece b[N];
  // t: thread of the group.  Operands stored [k][*]: piece (t & 15) of step (t >> 4) + 8 e; A stored
  // [m][k]: piece t % (TK / 4) of row t / (TK / 4) + e * 512 / TK.
  // Steps from k1 on count as zero.
  __device__ __forceinline__ void fetch(const Product& p, int m0, int n0, int k0, int k1, int t) {
    const bool wa = (p.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(p.A) & 15) == 0;
    const bool wb = (p.ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(p.B) & (4 * sizeof(T) - 1)) == 0;
    const int c = (t & 15) * 4;
#pragma unroll
    for (int e = 0; e < N; ++e) {
      const int k = k0 + (t >> 4) + 8 * e;
      const bool on = k < k1;
      if (p.a_mn) {
        a[e] = load_some(p.A + (size_t)(on ? k : 0) * p.lda + m0 + c, on ? p.M - m0 - c : 0, wa);
      } else {
        const int m = m0 + t / (TK / 4) + e * (512 / TK), kk = k0 + (t % (TK / 4)) * 4;
        a[e] = load_some(p.A + (size_t)(m < p.M ? m : 0) * p.lda + kk, m < p.M ? k1 - kk : 0, wa);
      }
      const int row = !on ? -1 : p.a_mn ? k : gate_row(p, k);
      b[e] = load_some(reinterpret_cast<const T*>(p.B) + (size_t)(row < 0 ? 0 : row) * p.ldb + n0 + c, row < 0 ? 0 : p.N - n0 - c, wb);
    }
  }
};

// The slices of TK steps that group g takes of a product, block by block from the last: take(next, end) uses the
// fetched slice and fetches the one at `next` (of the block that ends at `end`; none if next < 0); done() adds a
// block up.
template <int TK, class First, class Take, class Done>
__device__ __forceinline__ void blocks_of(const Product& p, int g, First first, Take take, Done done) {
  const int blocks = (p.K + p.block - 1) / p.block;
  auto end = [&](int b) { return min(p.K, (b + 1) * p.block); };
  auto fetch = [&](int b, auto f) {   // the group's first slice of block b or of the next one that has one
    for (; b >= 0; --b)
      if (b * p.block + g * TK < end(b)) { f(b * p.block + g * TK, end(b)); return; }
    f(-1, 0);
  };
  fetch(blocks - 1, [&](int k, int e) { if (k >= 0) first(k, e); });
  for (int b = blocks - 1; b >= 0; --b) {
    for (int k = b * p.block + g * TK; k < end(b); k += 2 * TK) {
      if (k + 2 * TK < end(b)) take(k + 2 * TK, end(b));
      else fetch(b - 1, take);
    }
    done();
  }
}

// FMA, 8 x 4 results a thread.
template <class T>
__device__ __forceinline__ void product_fma(const Product& p, int m0, int n0, float* smem) {
  constexpr int TK = 16, LD = 68;
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127, tx = t & 15, ty = t >> 4;
  float (*As)[LD] = reinterpret_cast<float (*)[LD]>(smem + g * 2 * TK * LD);
  float (*Bs)[LD] = As + TK;
  float* const x = smem + 4 * TK * LD + t;     // the second group's sums
  Slice<T, TK> s;
  float acc[8][4] = {}, sum[8][4];
  auto at = [&](int r, int q) -> float* {      // null: no element of C
    const int m = m0 + ty * 8 + r, n = n0 + tx * 4 + q, row = m < p.M ? (p.a_mn ? gate_row(p, m) : m) : -1;
    return row < 0 || n >= p.N ? nullptr : p.C + (size_t)row * p.ldc + n;
  };
  bool any = p.accumulate;
  if (g == 0 && any)
#pragma unroll
    for (int i = 0; i < 32; ++i) { const float* o = at(i >> 2, i & 3); sum[i >> 2][i & 3] = o ? *o : 0.f; }
  blocks_of<TK>(
      p, g, [&](int k0, int k1) { s.fetch(p, m0, n0, k0, k1, t); },
      [&](int next0, int next1) {
#pragma unroll
        for (int e = 0; e < s.N; ++e) {
          if (p.a_mn) {
            *reinterpret_cast<float4*>(&As[(t >> 4) + 8 * e][(t & 15) * 4]) = s.a[e];
          } else {
            const int m = t / (TK / 4) + e * (512 / TK), k = (t % (TK / 4)) * 4;
            As[k][m] = s.a[e].x; As[k + 1][m] = s.a[e].y; As[k + 2][m] = s.a[e].z; As[k + 3][m] = s.a[e].w;
          }
          *reinterpret_cast<float4*>(&Bs[(t >> 4) + 8 * e][(t & 15) * 4]) = widen(s.b[e]);
        }
        group_sync(g);
        if (next0 >= 0) s.fetch(p, m0, n0, next0, next1, t);
#pragma unroll
        for (int k = 0; k < TK; ++k) {
          const float4 a0 = *reinterpret_cast<const float4*>(&As[k][ty * 8]), a1 = *reinterpret_cast<const float4*>(&As[k][ty * 8 + 4]);
          const float4 b = *reinterpret_cast<const float4*>(&Bs[k][tx * 4]);
          const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
          for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(av[r], bv[q], acc[r][q]);
        }
        group_sync(g);
      },
      [&]() {
        if (g == 1)
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i * 128] = acc[i >> 2][i & 3];
        __syncthreads();
        if (g == 0)
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float v = acc[i >> 2][i & 3] + x[i * 128];
            sum[i >> 2][i & 3] = any ? sum[i >> 2][i & 3] + v : v;
          }
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i >> 2][i & 3] = 0.f;
        any = true;
        __syncthreads();
      });
  if (g == 1) return;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (float* o = at(i >> 2, i & 3)) *o = sum[i >> 2][i & 3];
}

// Bfloat16 storage: A (float32 gradients) as three bfloat16 planes that add up to it, on mma.sync; a warp
// has 32 x 32 results.
__device__ __forceinline__ void product_mma(const Product& p, int m0, int n0, float* smem) {
  constexpr int TK = 32, LM = 72, LK = 40;   // row lengths of [k][m] and [m][k] tiles: no bank conflicts for ldmatrix
  constexpr int plane = 64 * LK;
  const int g = threadIdx.x >> 7, t = threadIdx.x & 127, lane = t & 31, warp = t >> 5, wm = (warp & 1) * 32, wn = (warp >> 1) * 32;
  __nv_bfloat16* const As = reinterpret_cast<__nv_bfloat16*>(smem) + g * (3 * plane + TK * LM);   // [plane][TK][LM] or [plane][64][LK]
  __nv_bfloat16* const Bs = As + 3 * plane;                                                      // [TK][LM]
  Slice<__nv_bfloat16, TK> s;
  float acc[2][4][4] = {};
  auto put_tile = [&]() {
#pragma unroll
    for (int e = 0; e < s.N; ++e) {
      __nv_bfloat16* d = As + (p.a_mn ? ((t >> 4) + 8 * e) * LM + (t & 15) * 4 : (t / (TK / 4) + e * (512 / TK)) * LK + (t % (TK / 4)) * 4);
      float4 v = s.a[e];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
        *reinterpret_cast<uint2*>(d + q * plane) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        v.x -= __low2float(lo); v.y -= __high2float(lo); v.z -= __low2float(hi); v.w -= __high2float(hi);
      }
      *reinterpret_cast<uint2*>(Bs + ((t >> 4) + 8 * e) * LM + (t & 15) * 4) = s.b[e];
    }
  };
  auto ldsm = [](uint32_t (&r)[4], uint32_t addr, bool trans) {
    if (trans) asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
    else asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
  };
  const uint32_t a0 = sm100::smem_u32(As), b0 = sm100::smem_u32(Bs);
  const int l8 = lane & 7, q8 = lane >> 3;   // row inside an 8 x 8 block, block
  // the second group's sums, over its tiles (read before: the barrier behind each slice)
  float* const x = reinterpret_cast<float*>(reinterpret_cast<__nv_bfloat16*>(smem) + 3 * plane + TK * LM) + t;
  float sum[32];
  auto at = [&](int i) -> float* {           // i: fragment of 16 rows, 8 columns, half of the rows, column; null: no element of C
    const int m = m0 + wm + (i >> 4) * 16 + ((i >> 1) & 1) * 8 + (lane >> 2), n = n0 + wn + ((i >> 2) & 3) * 8 + 2 * (lane & 3) + (i & 1);
    const int row = m < p.M ? (p.a_mn ? gate_row(p, m) : m) : -1;
    return row < 0 || n >= p.N ? nullptr : p.C + (size_t)row * p.ldc + n;
  };
  bool any = p.accumulate;
  if (g == 0 && any)
#pragma unroll
    for (int i = 0; i < 32; ++i) { const float* o = at(i); sum[i] = o ? *o : 0.f; }
  blocks_of<TK>(
      p, g, [&](int k0, int k1) { s.fetch(p, m0, n0, k0, k1, t); },
      [&](int next0, int next1) {
        put_tile();
        group_sync(g);
        if (next0 >= 0) s.fetch(p, m0, n0, next0, next1, t);
#pragma unroll
        for (int k = 0; k < TK; k += 16) {
          uint32_t b[2][4];
#pragma unroll
          for (int j = 0; j < 2; ++j)   // blocks (k, n), (k + 8, n), (k, n + 8), (k + 8, n + 8)
            ldsm(b[j], b0 + ((k + (q8 & 1) * 8 + l8) * LM + wn + j * 16 + (q8 >> 1) * 8) * 2, true);
#pragma unroll
          for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              uint32_t a[4];             // blocks (m, k), (m + 8, k), (m, k + 8), (m + 8, k + 8)
              if (p.a_mn) ldsm(a, a0 + (q * plane + (k + (q8 >> 1) * 8 + l8) * LM + wm + i * 16 + (q8 & 1) * 8) * 2, true);
              else ldsm(a, a0 + (q * plane + (wm + i * 16 + (q8 & 1) * 8 + l8) * LK + k + (q8 >> 1) * 8) * 2, false);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float (&d)[4] = acc[i][j];
                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                             : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                             : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[j >> 1][(j & 1) * 2]), "r"(b[j >> 1][(j & 1) * 2 + 1]));
              }
            }
        }
        group_sync(g);
      },
      [&]() {
        if (g == 1)
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i * 128] = acc[i >> 4][(i >> 2) & 3][i & 3];
        __syncthreads();
        if (g == 0)
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float v = acc[i >> 4][(i >> 2) & 3][i & 3] + x[i * 128];
            sum[i] = any ? sum[i] + v : v;
          }
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i >> 4][(i >> 2) & 3][i & 3] = 0.f;
        any = true;
        __syncthreads();
      });
  if (g == 1) return;
#pragma unroll
  for (int i = 0; i < 32; ++i)
    if (float* o = at(i)) *o = sum[i];
}

// MMA: the caller has not forbidden tensor cores.
template <class T, bool MMA>
__global__ void __launch_bounds__(kTileThreads) chunk_products(const __grid_constant__ Products P) {
  __shared__ __align__(16) float smem[MMA ? 3 * 64 * 40 + 32 * 72 : 4 * 16 * 68 + 32 * 128];
  int i = P.n - 1;
  while ((int)blockIdx.x < P.p[i].tile0) --i;
  const Product& p = P.p[i];
  const int t = blockIdx.x - p.tile0, nx = (p.N + 63) / 64, m0 = (t / nx) * 64, n0 = (t % nx) * 64;
  if constexpr (MMA) product_mma(p, m0, n0, smem);
  else product_fma<T>(p, m0, n0, smem);
}

// Bias gradients (column sums of a chunk's dz and dy) and the loss terms of its steps.  dy = 2 d / (B O),
// so the mean of d * d over a step is the sum of dy * dy times B O / 4.
struct Sums {
  const float *dz, *dy; float *db, *db_out, *loss_t;
  int L, NG, H, O, B, S, steps, block, accumulate;   // block: rows summed by themselves, as in Product
};
__global__ void __launch_bounds__(1024) chunk_sums(const Sums q) {
  __shared__ float part_s[2][32][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5, G = 4 * q.H, nh = (G + 31) / 32, no = (q.O + 31) / 32;
  const int rows = q.steps * q.B;
  int b = blockIdx.x;
  if (b < q.L * nh + no) {
    const bool out = b >= q.L * nh;
    const int l = b / nh, n = (out ? b - q.L * nh : b - l * nh) * 32 + x, N = out ? q.O : G, ld = out ? q.O : G;
    const float* v = out ? q.dy : q.dz + (size_t)l * q.S * q.B * G;
    float* const o = out ? q.db_out + n : q.db + (size_t)l * q.NG * q.H + (size_t)(n & 3) * q.H + (n >> 2);
    const bool mine = y == 0 && n < N && (out || (n & 3) < q.NG);   // (a GRU's d q belongs to no bias)
    bool any = q.accumulate;
    float sum = mine && any ? *o : 0.f;
    for (int blk = (rows - 1) / q.block; blk >= 0; --blk) {
      float (*part)[33] = part_s[blk & 1];
      const int end = min(rows, (blk + 1) * q.block);
      float a0 = 0.f, a1 = 0.f;
      if (n < N) {
        int r = blk * q.block + y;
        for (; r + 32 < end; r += 64) { a0 += v[(size_t)r * ld + n]; a1 += v[(size_t)(r + 32) * ld + n]; }
        if (r < end) a0 += v[(size_t)r * ld + n];
      }
      part[y][x] = a0 + a1;
      __syncthreads();
      if (mine) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i) s += part[i][x];
        sum = any ? sum + s : s;
        any = true;
      }
    }
    if (mine) *o = sum;
  } else {
    const int k = b - q.L * nh - no;
    const float* v = q.dy + (size_t)k * q.B * q.O;
    float a = 0.f;
    for (int e = threadIdx.x; e < q.B * q.O; e += 1024) a = fmaf(v[e], v[e], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if (x == 0) part_s[0][0][y] = a;
    __syncthreads();
    if (y == 0) {
      a = part_s[0][0][x];
      for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
      if (x == 0) q.loss_t[k] = a * ((float)q.B * (float)q.O * 0.25f);
    }
  }
}

using WalkFn = void (*)(const Args);
template <class T, bool GRU, bool MMA>
WalkFn walk_nb(int nb) {
  return nb == 1 ? walk<T, GRU, 1, MMA> : nb == 2 ? walk<T, GRU, 2, MMA> : nb == 4 ? walk<T, GRU, 4, MMA> : walk<T, GRU, 8, MMA>;
}
WalkFn walk_fn(const Layout& y, int nb) {
  if (y.dtype != MEBPTT_BF16) return y.gru ? walk_nb<float, true, false>(nb) : walk_nb<float, false, false>(nb);
  if (y.tensor_cores) return y.gru ? walk_nb<__nv_bfloat16, true, true>(nb) : walk_nb<__nv_bfloat16, false, true>(nb);
  return y.gru ? walk_nb<__nv_bfloat16, true, false>(nb) : walk_nb<__nv_bfloat16, false, false>(nb);
}

}  // namespace

// ------------------------------------------------------------------------------------------
// host
// ------------------------------------------------------------------------------------------
namespace {

// The kernels take nearly a whole SM's shared memory and clusters of up to 16 CTAs.
cudaError_t allow(const void* fn) {
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

}  // namespace

DeviceFacts facts() {
  static std::mutex mu;
  static DeviceFacts table[64];
  static bool known[64];
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return DeviceFacts{}; }
  std::lock_guard<std::mutex> lock(mu);
  DeviceFacts& f = table[dev];
  if (known[dev]) return f;
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return DeviceFacts{}; }
  if (sms < f.sms) {
    f.sms = sms;
    const pod::Fn fn = pod::kernel(MEBPTT_FP32, false, 1, false);
    const bool may = allow(reinterpret_cast<const void*>(fn)) == cudaSuccess;
    for (int i = 0; i <= 4; ++i) {
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 1u << i; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(sms >> i) << i); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = kSmemMax - 1024;
      cfg.attrs = at; cfg.numAttrs = 1;
      int n = 0;
      if (!may || cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) n = 0;
      f.clusters[i] = n;
    }
    cudaGetLastError();
  }
  known[dev] = true;
  return f;
}

namespace {

// The schedule of a plan for one problem on one device, kept from step to step (eight of them, most
// recently used first); its tasks lie in page-locked memory where that can be had.
struct Kept {
  uint64_t plan_id = 0;
  Layout y;
  bool pageable = false;
  Route route;
  std::vector<Launch> launches;
  char* tasks = nullptr;       // 32 bytes each
  bool pinned = false;
  Kept() = default;
  Kept(const Kept&) = delete;
  Kept& operator=(const Kept&) = delete;
  ~Kept() {
    if (tasks && pinned) cudaFreeHost(tasks);
    else free(tasks);
  }
};
std::mutex g_mu;
std::vector<std::shared_ptr<Kept>> g_kept;
constexpr size_t kKeep = 8, kMaxPinned = (size_t)64 << 20;
int64_t g_built = 0, g_reused = 0, g_pinned = 0;   // (under g_mu)

bool same_problem(const Layout& a, const Layout& b) {
  return a.L == b.L && a.I == b.I && a.H == b.H && a.O == b.O && a.B == b.B && a.dtype == b.dtype && a.t == b.t && a.gru == b.gru && a.tensor_cores == b.tensor_cores &&
         a.S == b.S && a.tape_bytes == b.tape_bytes;
}

// Null, and a status, where there is none.
std::shared_ptr<Kept> schedule_for(const Layout& y, const Plan* p, bool pageable, int& status) {
  const Route r = route(y);
  status = MEBPTT_ERR_UNSUPPORTED;
  if (!r.ok) return nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    for (size_t i = 0; i < g_kept.size(); ++i) {
      Kept& k = *g_kept[i];
      if (k.plan_id == p->id && same_problem(k.y, y) && (k.pageable || !pageable) && k.route.pod == r.pod && k.route.c.T == r.c.T && k.route.c.teams == r.c.teams && k.route.pc.T == r.pc.T && k.route.pc.nb == r.pc.nb) {
        std::shared_ptr<Kept> hit = g_kept[i];
        g_kept.erase(g_kept.begin() + (long)i);
        g_kept.insert(g_kept.begin(), hit);
        ++g_reused;
        return hit;
      }
    }
  }
  std::shared_ptr<Kept> k = std::make_shared<Kept>();
  k->plan_id = p->id; k->y = y; k->route = r; k->pageable = pageable;
  Records rec;
  if (!build_records(y, p, r, y.tape_bytes / sizeof(Task), rec)) return nullptr;
  k->launches = rec.launches;
  void* mem = nullptr;
  if (!pageable && rec.bytes.size() <= kMaxPinned && cudaHostAlloc(&mem, rec.bytes.size(), cudaHostAllocDefault) == cudaSuccess) {
    k->pinned = true;
  } else {
    cudaGetLastError();
    mem = malloc(rec.bytes.size());
    status = MEBPTT_ERR_OOM;
    if (!mem) return nullptr;
  }
  k->tasks = static_cast<char*>(mem);
  memcpy(k->tasks, rec.bytes.data(), rec.bytes.size());
  std::lock_guard<std::mutex> lock(g_mu);
  ++g_built;
  g_pinned += k->pinned;
  g_kept.insert(g_kept.begin(), k);
  if (g_kept.size() > kKeep) g_kept.pop_back();
  return k;
}

// cluster: CTAs per cluster, or 0 for a cooperative grid
int launch(const void* fn, int grid, int cluster, int smem, void** args, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = counted(s);
  cudaLaunchAttribute at[1];
  if (cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args) == cudaSuccess ? MEBPTT_OK : MEBPTT_ERR_CUDA;
}

template <class T>
void launch_pack(const Layout& y, const Dims& d, int rows, const tc::StepPtrs& io, cudaStream_t s) {
  PackArgs<T> P{};
  P.L = y.L; P.I = y.I; P.H = y.H; P.O = y.O; P.d = d;
  P.W = reinterpret_cast<const T*>(io.W); P.W_out = reinterpret_cast<const T*>(io.W_out);
  for (int l = 0; l < y.L; ++l) {
    P.w_off[l] = y.w_layer_offset(l);
    P.wf[l] = reinterpret_cast<T*>(io.ws + y.off_wf[l]);
    P.wb[l] = reinterpret_cast<T*>(io.ws + y.off_wb[l]);
  }
  P.wr = reinterpret_cast<T*>(io.ws + y.off_wr);
  P.states = io.ws + y.off_arena; P.n_blocks = y.n_blocks; P.parts = y.parts; P.init = y.blk_init; P.R = rows; P.h0 = io.h0; P.c0 = io.c0; P.B = y.B;
  P.zero = reinterpret_cast<float*>(io.ws + y.off_dc);
  P.n_zero = (y.off_zero_end - y.off_dc) / 4;
  P.counters = io.counters;
  constexpr bool half = !std::is_same<T, float>::value;
  if (half && d.mma) {
    if (y.gru) pack<T, true, half><<<592, 256, 0, counted(s)>>>(P); else pack<T, false, half><<<592, 256, 0, counted(s)>>>(P);
  } else {
    if (y.gru) pack<T, true, false><<<592, 256, 0, counted(s)>>>(P); else pack<T, false, false><<<592, 256, 0, counted(s)>>>(P);
  }
}

// The products of chunk `chunk` (steps [k0, k0 + steps), 0-based).
void fill_products(Products& P, const Layout& y, const tc::StepPtrs& io, bool want_dx, int64_t k0, int steps, bool accumulate) {
  const int H = y.H, G = 4 * H, rows = steps * y.B;
  const size_t SB = (size_t)y.S * y.B;
  const float* dz = reinterpret_cast<const float*>(io.ws + y.off_dz);
  // a layer's h: row block i is h_{k-1} of the step in block i of dz, block i + 1 its h_k
  auto h_rows = [&](int l, int block) {
    return (const void*)(io.ws + y.off_st_h + (((size_t)l * (y.S + 1) + block) * y.B * H) * y.esz);
  };
  P.n = 0; P.tiles = 0;
  auto add = [&](const float* A, int lda, bool a_mn, const void* B, int ldb, float* C, int ldc, int M, int N, int K, bool acc,
                 int hidden, int skip, int last) {
    const int block = a_mn ? sum_steps(y.B) * y.B : K;   // (dx is summed over the gates)
    P.p[P.n++] = Product{A, B, C, lda, ldb, ldc, M, N, K, block, a_mn ? 1 : 0, acc ? 1 : 0, P.tiles, hidden, skip, last};
    P.tiles += ((M + 63) / 64) * ((N + 63) / 64);
  };
  for (int l = 0; l < y.L; ++l) {
    const int I = l ? H : y.I, K = I + H;
    const float* z = dz + (size_t)l * SB * G;
    const void* in = l ? h_rows(l - 1, 1) : (const void*)(io.x + (size_t)k0 * y.B * I * y.esz);
    float* dW = io.dW + y.w_layer_offset(l);
    // (GRU: the rows of n meet the input through d n_pre and the state through d q)
    add(z, G, true, in, I, dW, K, G, I, rows, accumulate, H, y.gru ? 3 : -1, 3);
    add(z, G, true, h_rows(l, 0), H, dW + I, K, G, H, rows, accumulate, H, y.gru ? 2 : -1, y.gru ? 2 : 3);
  }
  add(reinterpret_cast<const float*>(io.ws + y.off_dy), y.O, true, h_rows(y.L - 1, 1), H, io.dW_out, H, y.O, H,
      rows, accumulate, 0, -1, 3);
  if (want_dx) add(dz, G, false, io.W, y.I + H, io.dx + (size_t)k0 * y.B * y.I, y.I, rows, y.I, G, false, H, y.gru ? 3 : -1, 3);
}

}  // namespace

void forget_plan(uint64_t plan_id) {
  std::lock_guard<std::mutex> lock(g_mu);
  for (size_t i = g_kept.size(); i-- > 0;)
    if (g_kept[i]->plan_id == plan_id) g_kept.erase(g_kept.begin() + (long)i);
}

int prepare_host(const Layout& y, const Plan* p) {
  int status = MEBPTT_OK;
  return schedule_for(y, p, false, status) ? MEBPTT_OK : status;
}

void prepare_stats(int64_t* out) {
  std::lock_guard<std::mutex> lock(g_mu);
  out[0] += g_built; out[1] += g_reused; out[2] += g_pinned; out[3] += (int64_t)g_kept.size();
}

int64_t run_step(const Layout& y, const Plan* p, const tc::StepPtrs& io, bool want_dx, cudaStream_t s, bool dry) {
  int status = MEBPTT_OK;
  const std::shared_ptr<Kept> kept = schedule_for(y, p, io.pageable_tape, status);
  if (!kept) return dry ? -1 : status;
  const Config& c = kept->route.c;
  const pod::Config& pc = kept->route.pc;
  const bool pods = kept->route.pod;
  if (dry) {
    int64_t n = 2;   // packing, finalisation
    for (const Launch& g : kept->launches) n += g.chunk >= 0 ? 3 : 1;
    return n;
  }
  const Dims d = dims(y);
  if (pods) {
    pod::PackArgs q{};
    q.L = y.L; q.I = y.I; q.H = y.H; q.O = y.O; q.B = y.B; q.c = pc;
    q.W = io.W; q.W_out = io.W_out; q.h0 = io.h0; q.c0 = io.c0;
    for (int l = 0; l < y.L; ++l) { q.wf[l] = io.ws + y.off_wf[l]; q.w_off[l] = y.w_layer_offset(l); }
    q.wr = io.ws + y.off_wr; q.states = io.ws + y.off_arena; q.n_blocks = y.n_blocks; q.parts = y.parts; q.init = y.blk_init;
    q.zero = reinterpret_cast<float*>(io.ws + y.off_dc); q.n_zero = (y.off_zero_end - y.off_dc) / 4;
    q.counters = io.counters;
    pod::launch_pack(y.dtype, y.gru, q, s);
  } else if (y.dtype == MEBPTT_BF16) {
    launch_pack<__nv_bfloat16>(y, d, c.rows, io, s);
  } else {
    launch_pack<float>(y, d, c.rows, io, s);
  }

  Args a{};
  unsigned met = 0;            // arrivals of a team before a launch
  pod::Args pa{};
  WalkFn fn = nullptr;
  pod::Fn pf = nullptr;
  auto common = [&](auto& q) {
    q.L = y.L; q.I = y.I; q.H = y.H; q.O = y.O; q.B = y.B; q.S = y.S;
    for (int l = 0; l < y.L; ++l) q.off_wf[l] = y.off_wf[l];
    q.off_wr = y.off_wr;
    q.off_states = y.off_arena; q.n_blocks = y.n_blocks; q.parts = y.parts;
    q.ws = io.ws;
    q.off_dz = y.off_dz; q.off_hk = y.off_st_h; q.off_dy = y.off_dy; q.off_carry = y.off_carry; q.off_dc = y.off_dc;
    q.x = io.x; q.bias = io.b; q.b_out = io.b_out; q.targets = io.targets;
    q.status = reinterpret_cast<int*>(io.ws + y.off_status);
    q.counters = io.counters;
  };
  if (pods) {
    common(pa);
    pa.stages = io.ws + y.off_dz;
    const bool fault = tc::wait_fault_mask() & 8;
    pa.polls = fault ? 64 : 1u << 16;
    pa.extra_bytes = fault ? 16 : 0;
    pa.c = pc;
    const size_t states = (size_t)y.n_blocks * (block_bytes(pc.nb, y.H, y.esz, y.parts) / y.parts);
    pf = pod::kernel(y.dtype, y.gru, pc.nb, states >> 32 != 0 || y.parts > 1);
    if (allow(reinterpret_cast<const void*>(pf)) != cudaSuccess) { cudaGetLastError(); return MEBPTT_ERR_CUDA; }
  } else {
    common(a);
    a.d = d; a.T = c.T; a.rows = c.rows;
    for (int l = 0; l < y.L; ++l) { a.ns_f[l] = c.ns_f[l]; a.ns_b[l] = c.ns_b[l]; a.off_wb[l] = y.off_wb[l]; }
    a.ns_r = c.ns_r; a.resident = c.resident; a.pool_floats = c.pool_floats;
    a.sync = reinterpret_cast<unsigned*>(io.ws + y.off_sync);
    const bool fault = tc::wait_fault_mask() & 16;
    a.polls = fault ? tc::fault_poll_limit : sm100::kSpinLimit;
    met = fault ? 1 : 0;   // (arrivals that nobody makes)
    fn = walk_fn(y, c.nb);
    if (allow(reinterpret_cast<const void*>(fn)) != cudaSuccess) { cudaGetLastError(); return MEBPTT_ERR_CUDA; }
  }

  float* loss_t = reinterpret_cast<float*>(io.ws + y.off_loss_t);
  Task* region = reinterpret_cast<Task*>(io.ws + y.off_tape);
  const std::vector<Launch>& ls = kept->launches;
  const size_t room = y.tape_bytes / sizeof(Task);
  size_t up_lo = 0, up_hi = 0;   // tasks that lie in the region
  bool first = true;
  Products P;
  for (size_t i = 0; i < ls.size(); ++i) {
    const Launch& g = ls[i];
    if (g.task0 + g.ntasks > up_hi) {   // the tasks of this launch and of as many after it as fit
      up_lo = g.task0;
      up_hi = up_lo;
      for (size_t j = i; j < ls.size() && ls[j].task0 + ls[j].ntasks - up_lo <= room; ++j) up_hi = ls[j].task0 + ls[j].ntasks;
      cudaMemcpyAsync(region, kept->tasks + up_lo * sizeof(Task), (up_hi - up_lo) * sizeof(Task), cudaMemcpyHostToDevice, s);
    }
    if (g.ntasks) {
      int rc;
      if (pods) {
        pa.tasks = reinterpret_cast<const pod::Task*>(region + (g.task0 - up_lo));
        pa.n_tasks = (int)g.ntasks; pa.phases = g.phases; pa.fwd_ops = g.fwd_ops; pa.bwd_ops = g.bwd_ops;
        void* args[1] = {&pa};
        rc = launch(reinterpret_cast<const void*>(pf), pc.pods * pc.T, pc.T, pc.smem, args, s);
      } else {
        a.tasks = region + (g.task0 - up_lo);
        a.n_tasks = (int)g.ntasks;
        a.sync_base = met;
        met += (unsigned)g.phases * (unsigned)c.T;
        void* args[1] = {&a};
        rc = launch(reinterpret_cast<const void*>(fn), c.teams * c.T, 0, c.smem, args, s);
      }
      if (rc != MEBPTT_OK) return rc;
    }
    if (g.chunk >= 0) {
      const int64_t k0 = (int64_t)g.chunk * y.S;
      const int steps = (int)std::min<int64_t>(y.S, y.t - k0);
      fill_products(P, y, io, want_dx, k0, steps, !first);
      if (y.dtype != MEBPTT_BF16) chunk_products<float, false><<<P.tiles, kTileThreads, 0, counted(s)>>>(P);
      else if (y.tensor_cores) chunk_products<__nv_bfloat16, true><<<P.tiles, kTileThreads, 0, counted(s)>>>(P);
      else chunk_products<__nv_bfloat16, false><<<P.tiles, kTileThreads, 0, counted(s)>>>(P);
      const Sums q{reinterpret_cast<const float*>(io.ws + y.off_dz), reinterpret_cast<const float*>(io.ws + y.off_dy), io.db, io.db_out,
                   loss_t + k0, y.L, y.NG, y.H, y.O, y.B, y.S, steps, sum_steps(y.B) * y.B, first ? 0 : 1};
      chunk_sums<<<y.L * ((4 * y.H + 31) / 32) + (y.O + 31) / 32 + steps, 1024, 0, counted(s)>>>(q);
      first = false;
    }
  }
  generic::finalize_step(loss_t, y.t, io.loss, io.counters, p->peak_units, reinterpret_cast<int*>(io.ws + y.off_status), s);
  return cudaGetLastError() == cudaSuccess ? MEBPTT_OK : MEBPTT_ERR_CUDA;
}

}  // namespace team
}  // namespace mebptt
