// The pod kernel (pod.hpp has the scheme): one thread-block cluster walks the tape for NB batch rows.
//
// A phase: wait until every CTA's pushes of the phase before have arrived; partial sums of the CTA's
// units over warps; one CTA-wide barrier; cell arithmetic, a thread per unit and batch row, whose
// result goes to memory for later and into the operand slots of all CTAs of the pod at once; fetch
// what the next phase needs from memory.
//
// What bounds it is that chain.  The arrival counts of a phase (one arrival per CTA and the bytes it
// sends) are the only thing the CTAs have to agree on: a CTA that has all arrivals of phase p knows
// that nobody reads operands of phase p - 1 or earlier any more, so slots need no other protection.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "layout.hpp"
#include "pod.hpp"
#include "pod_run.hpp"
#include "sm100.cuh"
#include "team_dev.cuh"

namespace mebptt {
namespace pod {

using team::cell_backward;
using team::cell_forward;
using team::lane_sums;
using team::load4;
using team::part;
using team::store;
using team::to_f;

namespace {

// One class of contraction of this CTA: F(l), B(l) or the readout.
struct Tab {
  int groups, ns;        // groups of 4 weight rows, parts the contraction index is cut into
  int na, nb;            // 16-byte operand vectors of the two segments (na is padded to a whole number of slices for the part arithmetic)
  int ia, its;           // 128-element slices of the first segment, of both
  int lda, ldb, ldw;     // row lengths in floats / elements
  int held;              // element offset of resident weights, or -1
  const void* w;         // weights in memory
};

__device__ __forceinline__ uint32_t remote(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void push1(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void push4(uint32_t addr, float4 v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)), "r"(__float_as_uint(v.w)), "r"(bar)
               : "memory");
}
__device__ __forceinline__ bool wait_cluster(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < sm100::kSpinLimit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if (i > 1024) __nanosleep(64);
  }
  return false;
}

template <class T, int NB>
__device__ __forceinline__ void segment(const float* a, int lda, const T* w, int ldw, int i0, int i1, int nv, int lane, float (&acc)[NB * 4]) {
#pragma unroll 2
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

// One state element of a thread: unit j (global) of layer l, batch row b of the pod.
struct Elem { int l, b, j, jl; bool on; };

// What an element's arithmetic needs from memory.
struct Main { float v[9]; };

template <class T, bool GRU>
struct Walk {
  const Args& A;
  int row0;

  __device__ __forceinline__ const T* h_at(uint32_t loc, int l) const {
    return loc == team::kInit ? reinterpret_cast<const T*>(A.h0) + (size_t)l * A.B * A.H
                              : reinterpret_cast<const T*>(A.ws + ((size_t)loc << 8) + (size_t)l * A.hc);
  }
  __device__ __forceinline__ const float* c_at(uint32_t loc, int l) const {
    return loc == team::kInit ? A.c0 + (size_t)l * A.B * A.H
                              : reinterpret_cast<const float*>(A.ws + ((size_t)loc << 8) + (size_t)l * A.hc + A.csz_off);
  }
  __device__ __forceinline__ T* gates_at(uint32_t rec, int l) const {
    return reinterpret_cast<T*>(A.ws + ((size_t)rec << 8) + A.rec_gates + (size_t)l * A.gsz);
  }
  __device__ __forceinline__ float* dc_at(int l) const { return reinterpret_cast<float*>(A.ws + A.off_dc) + (size_t)l * A.B * A.H; }

  __device__ __forceinline__ void fetch(const Task& t, const Elem& s, Main& o) const {
    const int l = s.l;
    const size_t e = (size_t)(row0 + s.b) * A.H + s.j;
    if (t.kind == FWD) {
      o.v[4] = GRU ? to_f(h_at(t.src, l)[e]) : c_at(t.src, l)[e];
      if (!GRU && (t.flags & COPY_IN)) o.v[5] = to_f(h_at(t.src, l)[e]);
    } else {
      const T* g = gates_at(t.src, l) + e;
      const size_t pl = A.plane / sizeof(T);
#pragma unroll
      for (int q = 0; q < 4; ++q) o.v[q] = to_f(g[q * pl]);
      o.v[4] = dc_at(l)[e];
      o.v[5] = to_f(h_at(t.dst, l)[e]);
      o.v[6] = to_f(h_at(t.src, l)[e]);
      if (!GRU) { o.v[7] = c_at(t.src, l)[e]; o.v[8] = c_at(t.dst, l)[e]; }
    }
  }
  // the value a load task sends: h, or the four gate gradients of a unit
  __device__ __forceinline__ float4 fetch_load(const Task& t, const Elem& s) const {
    const size_t row = row0 + s.b;
    if (t.kind == LOAD_H) return make_float4(to_f(h_at(t.src, s.l)[row * A.H + s.j]), 0.f, 0.f, 0.f);
    const float* p = (t.flags & CARRY)
                         ? reinterpret_cast<const float*>(A.ws + A.off_carry) + (((size_t)(t.k & 1) * A.L + s.l) * A.B + row) * 4 * A.H
                         : reinterpret_cast<const float*>(A.ws + A.off_dz) + (((size_t)s.l * A.S + t.sidx) * A.B + row) * 4 * A.H;
    return *reinterpret_cast<const float4*>(p + 4 * s.j);
  }
  // returns the value to push: h (in x), or the four gate gradients
  __device__ __forceinline__ float4 apply(const Task& t, const Elem& s, const Main& o, const float (&z)[4], const float (&bias)[4]) const {
    const int l = s.l, H = A.H;
    const size_t row = row0 + s.b, e = row * H + s.j;
    if (t.kind == FWD) {
      float g[4], h, c;
      cell_forward<GRU>(z, bias, o.v[4], g, h, c);
      char* dst = A.ws + ((size_t)t.dst << 8);
      T* hp = reinterpret_cast<T*>(dst + (size_t)l * A.hc) + e;
      store(hp, h);
      if (!GRU) reinterpret_cast<float*>(dst + (size_t)l * A.hc + A.csz_off)[e] = c;
      if (t.flags & GATES) {
        T* gp = gates_at(t.dst, l) + e;
        const size_t pl = A.plane / sizeof(T);
#pragma unroll
        for (int q = 0; q < 4; ++q) store(gp + q * pl, g[q]);
      }
      if (t.flags & COPY_IN) {
        char* in = dst + A.rec_gates + (size_t)A.L * A.gsz;
        store(reinterpret_cast<T*>(in + (size_t)l * A.hc) + e, GRU ? o.v[4] : o.v[5]);
        if (!GRU) reinterpret_cast<float*>(in + (size_t)l * A.hc + A.csz_off)[e] = o.v[4];
      }
      T r;
      store(&r, h);   // the others read what was stored
      return make_float4(to_f(r), 0.f, 0.f, 0.f);
    }
    const float g[4] = {o.v[0], o.v[1], o.v[2], o.v[3]};
    float d[4], carry = o.v[4];
    cell_backward<GRU>(z[0], g, o.v[5], o.v[7], o.v[8], carry, d);
    dc_at(l)[e] = carry;
    const float4 quad = make_float4(d[0], d[1], d[2], d[3]);
    const size_t srow = ((size_t)l * A.S + t.sidx) * A.B + row;
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(A.ws + A.off_dz) + srow * 4 * H + 4 * s.j) = quad;
    if (t.flags & CARRY_OUT)
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(A.ws + A.off_carry) + (((size_t)(t.k & 1) * A.L + l) * A.B + row) * 4 * H + 4 * s.j) = quad;
    store(reinterpret_cast<T*>(A.ws + A.off_hp) + srow * H + s.j, o.v[5]);
    store(reinterpret_cast<T*>(A.ws + A.off_hk) + srow * H + s.j, o.v[6]);
    return quad;
  }
};

template <class T, bool GRU, int NB>
__global__ void __launch_bounds__(kThreads, 1) pod_walk(const __grid_constant__ Args A) {
  extern __shared__ __align__(128) unsigned char smem[];
  Task* const windows = reinterpret_cast<Task*>(smem);
  unsigned char* const ctl = smem + kWindows * kWindow * sizeof(Task);
  uint64_t* const bars = reinterpret_cast<uint64_t*>(ctl);             // arrivals of even and odd phases
  uint32_t* const peer = reinterpret_cast<uint32_t*>(ctl + 16);        // where each CTA's shared memory begins
  Tab* const tab = reinterpret_cast<Tab*>(ctl + 128);                  // F(0..L-1), B(0..L-1), readout
  float* const slots = reinterpret_cast<float*>(ctl + 2048);
  float* const sums = slots + A.slot_floats;
  T* const held = reinterpret_cast<T*>(sums + 2 * A.red_floats);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pod = blockIdx.x / A.T, rank = blockIdx.x - pod * A.T;
  const int H = A.H, L = A.L;
  const Walk<T, GRU> W{A, pod * NB};
  const int valid = min(NB, A.B - pod * NB);
  const uint32_t base = sm100::smem_u32(smem), bar0 = sm100::smem_u32(bars), slots0 = sm100::smem_u32(slots);
  int u0, u1, go0, go1, x0, x1;
  part(H, A.T, rank, u0, u1);
  part(A.d.groups_o, A.T, rank, go0, go1);
  part(A.I, A.T, rank, x0, x1);
  const int u = u1 - u0, gb = (u + 3) >> 2, ro = max(0, min(go1 * 4, A.O) - go0 * 4), xo = x1 - x0;

  if (tid == 0) {
    sm100::mbar_init(bars, (uint32_t)A.T);
    sm100::mbar_init(bars + 1, (uint32_t)A.T);
    sm100::mbar_fence_init();
    int at = 0;
    for (int i = 0; i <= 2 * L; ++i) {
      Tab& t = tab[i];
      const bool f = i < L, r = i == 2 * L;
      const int l = f ? i : r ? L - 1 : i - L;
      const int ka = f ? A.d.ip[l] : r ? A.d.hp : A.d.gp, k = f ? A.d.kf[l] : r ? A.d.hp : A.d.kb[l];
      t.groups = f ? u : r ? go1 - go0 : gb;
      t.ns = f ? A.ns_f[l] : r ? A.ns_r : A.ns_b[l];
      t.na = ka >> 2; t.nb = (k - ka) >> 2;
      t.ia = (t.na + 31) >> 5; t.its = t.ia + ((t.nb + 31) >> 5);
      t.lda = ka; t.ldb = k - ka; t.ldw = k;
      const T* w = reinterpret_cast<const T*>(A.ws + (f ? A.off_wf[l] : r ? A.off_wr : A.off_wb[l]));
      t.w = w + (size_t)(f ? u0 * 4 : r ? go0 * 4 : u0) * k;
      t.held = -1;
    }
    // resident weights in the order F, B, readout
    for (int i = 0; i <= 2 * L; ++i) {
      const int bit = i < L ? 2 * i : i == 2 * L ? 63 : 2 * (i - L) + 1;
      if (A.resident >> bit & 1) { tab[i].held = at; at += tab[i].groups * 4 * tab[i].ldw; }
    }
  }
  if (tid < A.T) peer[tid] = remote(base, tid);
  for (int i = tid; i < A.slot_floats; i += kThreads) slots[i] = 0.f;
  auto load_window = [&](int w) {
    if (tid < kWindow * 2)
      reinterpret_cast<uint4*>(windows + (w & (kWindows - 1)) * kWindow)[tid] =
          __ldg(reinterpret_cast<const uint4*>(A.tasks + (size_t)w * kWindow) + tid);
  };
  const int n_windows = A.n_tasks / kWindow;
  load_window(0);
  if (n_windows > 1) load_window(1);
  __syncthreads();
  for (int i = 0; i <= 2 * L; ++i)
    if (tab[i].held >= 0) {
      uint4* d = reinterpret_cast<uint4*>(held + tab[i].held);
      const uint4* s = reinterpret_cast<const uint4*>(tab[i].w);
      const int n = tab[i].groups * 4 * tab[i].ldw * (int)sizeof(T) / 16;
      for (int k = tid; k < n; k += kThreads) d[k] = __ldcg(s + k);
    }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // the thread's elements: states from the front of the block, readouts and inputs from its back
  const int per_l = NB * u, all_s = L * per_l, all_r = NB * ro, all_x = NB * xo, back = kThreads - 1 - tid;
  auto state_elem = [&](int e) {
    Elem s;
    s.l = e / max(1, per_l);
    const int r = e - s.l * per_l;
    s.b = r / max(1, u);
    s.jl = r - s.b * u;
    s.j = u0 + s.jl;
    s.on = s.b < valid;
    return s;
  };
  const bool has_s = tid < all_s;
  const Elem mine = state_elem(has_s ? tid : 0);
  float bias[4] = {0.f, 0.f, 0.f, 0.f};
  auto load_bias = [&](int l, int j, float (&b)[4]) {
#pragma unroll
    for (int q = 0; q < (GRU ? 3 : 4); ++q) b[q] = __ldg(A.bias + ((size_t)l * (GRU ? 3 : 4) + q) * H + j);
  };
  if (has_s) load_bias(mine.l, mine.j, bias);
  const int rb = ro ? back / ro : 0, rj = ro ? go0 * 4 + back - rb * ro : 0;     // first readout element
  const int xb = xo ? back / xo : 0, xj = xo ? x0 + back - xb * xo : 0;          // first input element
  const float r_bias = (back < all_r && rb < valid) ? __ldg(A.b_out + rj) : 0.f;
  const float dy_scale = 1.f / ((float)A.B * (float)A.O);

  // fetched one phase ahead: the first cell task, load task, readout and input load that concern the thread
  Main om;
  float4 ol = make_float4(0.f, 0.f, 0.f, 0.f);
  float o_target = 0.f, o_x = 0.f;
  int im = -1, il = -1;
  auto ahead = [&](const Task* t) {
    const int n = t[0].n;
    im = il = -1;
    bool got_r = false, got_x = false;
    for (int i = 0; i < n; ++i) {
      const Task& k = t[i];
      if (has_s && mine.on && k.layer == mine.l && k.kind != READ && k.kind != LOAD_X && k.kind != NOP) {
        if (k.kind <= BWD) { if (im < 0) { im = i; W.fetch(k, mine, om); } }
        else if (il < 0) { il = i; ol = W.fetch_load(k, mine); }
      }
      if (k.kind == READ && !got_r) {
        got_r = true;
        if (back < all_r && rb < valid) o_target = __ldg(A.targets + ((size_t)(k.k - 1) * A.B + pod * NB + rb) * A.O + rj);
      }
      if (k.kind == LOAD_X && !got_x) {
        got_x = true;
        if (back < all_x && xb < valid)
          o_x = to_f(reinterpret_cast<const T*>(A.x)[((size_t)(k.k - 1) * A.B + pod * NB + xb) * A.I + xj]);
      }
    }
  };

  int64_t fwd_ops = 0, bwd_ops = 0;
  int w = 0, i0 = 0;
  bool entered = true;      // first phase of a window
  const Task* t = windows;
  ahead(t);
  int ph = 0;
  for (; ph < A.phases; ++ph) {
    const int n = t[0].n;
    const uint32_t bar = bar0 + 8 * (ph & 1);
    bool ok = true;
    if (ph > 0) ok = wait_cluster(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1);
    float* const red = sums + (ph & 1) * A.red_floats;
    // partial sums
    {
      int i = 0, first = 0, works = 0;
      const Tab* b = nullptr;
      for (int wk = warp;; wk += kWarps) {
        while (i < n && wk >= first + works) {      // the task this piece of work belongs to
          first += works;
          const Task& k = t[i++];
          works = 0;
          if (k.kind >= FWD && k.kind <= BWD) {
            b = tab + (k.kind == FWD ? k.layer : k.kind == READ ? 2 * L : L + k.layer);
            works = b->groups * b->ns;
          }
        }
        if (wk >= first + works) break;
        const Task& k = t[i - 1];
        const int rem = wk - first, ns = b->ns, g = rem / ns, s = rem - g * ns;
        const int lo = b->its * s / ns, hi = b->its * (s + 1) / ns, ia = b->ia;
        float acc[NB * 4];
#pragma unroll
        for (int q = 0; q < NB * 4; ++q) acc[q] = 0.f;
        const float* pa = slots + (size_t)k.sa * 16;
        const float* pb = slots + (size_t)k.sb * 16;
        const int ldw = b->ldw;
        if (b->held >= 0) {
          const T* wp = held + b->held + (size_t)g * 4 * ldw;
          if (lo < ia) segment<T, NB>(pa, b->lda, wp, ldw, lo, min(hi, ia), b->na, lane, acc);
          if (hi > ia) segment<T, NB>(pb, b->ldb, wp + b->lda, ldw, max(lo - ia, 0), hi - ia, b->nb, lane, acc);
        } else {
          const T* wp = reinterpret_cast<const T*>(b->w) + (size_t)g * 4 * ldw;
          if (lo < ia) segment<T, NB>(pa, b->lda, wp, ldw, lo, min(hi, ia), b->na, lane, acc);
          if (hi > ia) segment<T, NB>(pb, b->ldb, wp + b->lda, ldw, max(lo - ia, 0), hi - ia, b->nb, lane, acc);
        }
        const float v = lane_sums<NB * 4>(acc, lane);
        constexpr int per = 32 / (NB * 4);
        if (lane % per == 0) red[k.red * 4 + (g * ns + s) * NB * 4 + lane / per] = v;
      }
    }
    if (__syncthreads_or(!ok)) break;
    if (tid < A.T) {
      uint32_t bytes = 0;
      for (int i = 0; i < n; ++i) {
        const Task& k = t[i];
        if (k.so == kNone || k.kind == NOP) continue;
        bytes += k.kind == READ ? ro * 4 : k.kind == LOAD_X ? xo * 4 : (k.kind == BWD || k.kind == LOAD_DZ) ? u * 16 : u * 4;
      }
      asm volatile("mbarrier.arrive.expect_tx.release.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(peer[tid] + (bar - base)),
                   "r"(bytes * (uint32_t)valid) : "memory");
    }
    // cells
    for (int e = tid; e < all_s; e += kThreads) {
      const bool first = e == tid;
      const Elem s = first ? mine : state_elem(e);
      if (!s.on) continue;
      for (int i = 0; i < n; ++i) {
        const Task& k = t[i];
        if (k.layer != s.l || k.kind == NOP || k.kind == READ || k.kind == LOAD_X) continue;
        float4 v;
        bool quad = k.kind == LOAD_DZ;
        if (k.kind <= BWD) {
          if (!first || i != im) W.fetch(k, s, om);
          float z[4] = {0.f, 0.f, 0.f, 0.f};
          if (k.kind == FWD) {
            const int ns = tab[s.l].ns;
            const float* p = red + k.red * 4 + s.jl * ns * NB * 4 + s.b * 4;
            for (int q = 0; q < ns; ++q, p += NB * 4) {
              const float4 r = *reinterpret_cast<const float4*>(p);
              z[0] += r.x; z[1] += r.y; z[2] += r.z; z[3] += r.w;
            }
          } else {
            const int ns = tab[L + s.l].ns;
            const float* p = red + k.red * 4 + (s.jl >> 2) * ns * NB * 4 + s.b * 4 + (s.jl & 3);
            for (int q = 0; q < ns; ++q, p += NB * 4) z[0] += *p;
            quad = true;
          }
          float bs[4] = {bias[0], bias[1], bias[2], bias[3]};
          if (!first) load_bias(s.l, s.j, bs);
          v = W.apply(k, s, om, z, bs);
        } else {
          v = (first && i == il) ? ol : W.fetch_load(k, s);
        }
        if (k.so != kNone) {
          const uint32_t off = slots0 - base + k.so * 64, bo = bar - base;
          if (quad) {
            const uint32_t at = off + (uint32_t)(s.b * A.d.gp + 4 * s.j) * 4;
            for (int r = 0; r < A.T; ++r) push4(peer[r] + at, v, peer[r] + bo);
          } else {
            const uint32_t at = off + (uint32_t)(s.b * A.d.hp + s.j) * 4;
            for (int r = 0; r < A.T; ++r) push1(peer[r] + at, v.x, peer[r] + bo);
          }
        }
      }
    }
    // readouts and inputs
    bool got_r = false, got_x = false;
    for (int i = 0; i < n; ++i) {
      const Task& k = t[i];
      const uint32_t off = slots0 - base + k.so * 64, bo = bar - base;
      if (k.kind == READ) {
        const int ns = tab[2 * L].ns, op = (A.O + 7) & ~7;
        for (int e = back; e < all_r; e += kThreads) {
          const int b = e / ro, j = go0 * 4 + e - b * ro, jl = j - go0 * 4;
          if (b >= valid) continue;
          const float target = (e == back && !got_r) ? o_target : __ldg(A.targets + ((size_t)(k.k - 1) * A.B + pod * NB + b) * A.O + j);
          const float bo_ = e == back ? r_bias : __ldg(A.b_out + j);
          const float* p = red + k.red * 4 + (jl >> 2) * ns * NB * 4 + b * 4 + (jl & 3);
          float z = 0.f;
          for (int q = 0; q < ns; ++q, p += NB * 4) z += *p;
          const float dy = 2.f * (z + bo_ - target) * dy_scale;
          reinterpret_cast<float*>(A.ws + A.off_dy)[((size_t)k.sidx * A.B + pod * NB + b) * A.O + j] = dy;
          const uint32_t at = off + (uint32_t)(b * op + j) * 4;
          for (int r = 0; r < A.T; ++r) push1(peer[r] + at, dy, peer[r] + bo);
        }
        got_r = true;
      } else if (k.kind == LOAD_X) {
        for (int e = back; e < all_x; e += kThreads) {
          const int b = e / xo, j = x0 + e - b * xo;
          if (b >= valid) continue;
          const float v = (e == back && !got_x)
                              ? o_x
                              : to_f(reinterpret_cast<const T*>(A.x)[((size_t)(k.k - 1) * A.B + pod * NB + b) * A.I + j]);
          const uint32_t at = off + (uint32_t)(b * A.d.ip[0] + j) * 4;
          for (int r = 0; r < A.T; ++r) push1(peer[r] + at, v, peer[r] + bo);
        }
        got_x = true;
      }
    }
    if (tid == 0 && blockIdx.x == 0)
      for (int i = 0; i < n; ++i)
        if (t[i].flags & COUNT) { if (t[i].kind == FWD) ++fwd_ops; else if (t[i].kind == BWD) ++bwd_ops; }
    if (entered && w + 2 < n_windows) load_window(w + 2);
    entered = false;
    i0 += n;
    if (ph + 1 < A.phases) {
      if (i0 >= kWindow || windows[(w & (kWindows - 1)) * kWindow + i0].n == 0) { ++w; i0 = 0; entered = true; }
      t = windows + (w & (kWindows - 1)) * kWindow + i0;
      ahead(t);
    }
  }
  bool ok = ph == A.phases;
  if (ok && ph > 0) ok = wait_cluster(bar0 + 8 * ((ph - 1) & 1), ((ph - 1) >> 1) & 1);
  if (!ok) *A.status = MEBPTT_ERR_TIMEOUT;
  // nobody leaves while pushes to its shared memory may be under way
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (tid == 0 && blockIdx.x == 0) {
    A.counters[0] += fwd_ops;
    A.counters[1] += bwd_ops;
  }
}

template <class T, bool GRU>
Fn by_rows(int nb) {
  return nb == 1 ? pod_walk<T, GRU, 1> : nb == 2 ? pod_walk<T, GRU, 2> : nb == 4 ? pod_walk<T, GRU, 4> : pod_walk<T, GRU, 8>;
}

}  // namespace

Fn kernel(int dtype, bool gru, int nb) {
  if (dtype == MEBPTT_BF16) return gru ? by_rows<__nv_bfloat16, true>(nb) : by_rows<__nv_bfloat16, false>(nb);
  return gru ? by_rows<float, true>(nb) : by_rows<float, false>(nb);
}

}  // namespace pod
}  // namespace mebptt
