// Device helpers shared by the kernels of the team path.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mebptt {
namespace team {

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void store(float* p, float v) { *p = v; }
__device__ __forceinline__ void store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
__device__ __forceinline__ float sigmoid(float a) { return 1.0f / (1.0f + expf(-a)); }
// States and stages are written by other SMs between phases: read them from the L2.
__device__ __forceinline__ float ld_l2(const float* p) { return __ldcg(p); }
__device__ __forceinline__ __nv_bfloat16 ld_l2(const __nv_bfloat16* p) {
  const unsigned short v = __ldcg(reinterpret_cast<const unsigned short*>(p));
  return __ushort_as_bfloat16(v);
}
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}

// Sums the N per-lane partial values over the warp; lane i ends with value i * N / 32 (every group of
// 32 / N lanes holds the same one).  Fixed order, N - 1 + log2(32 / N) exchanges.
template <int N>
__device__ __forceinline__ float lane_sums(float (&v)[N], int lane) {
  int off = 16;
#pragma unroll
  for (int n = N; n > 1; n >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float send = up ? v[i] : v[i + n / 2];
      const float keep = up ? v[i + n / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (int o = 16 / N; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

// The states of one group of batch rows (row R i and on, of group i): blocks of `hs` bytes -- one layer's h
// of the group -- with a cell state in the CR blocks behind its h, layer after layer, then four gate blocks a
// layer, then the input state.  Locations count parts of a block, `parts` to a block.
template <class T>
struct States {
  static constexpr int CR = (int)(4 / sizeof(T));
  char* base;
  uint32_t hs, part;
  int parts;
  __host__ __device__ static uint32_t block(int rows, int H, int parts) {
    const uint32_t a = 16 * (uint32_t)parts;
    return ((uint32_t)rows * H * (uint32_t)sizeof(T) + a - 1) / a * a;
  }
  // n: parts of a group's states
  __host__ __device__ States(char* all, int64_t n, int parts_, int group, int R, int B, int H)
      : base(all + (size_t)group * n * (block(R, H, parts_) / parts_)), hs(block(R < B - group * R ? R : B - group * R, H, parts_)), part(hs / parts_),
        parts(parts_) {}
  __host__ __device__ char* at(uint32_t loc, int blocks) const { return base + (size_t)(loc + (uint32_t)(blocks * parts)) * part; }
  __host__ __device__ T* h(uint32_t loc, int l) const { return reinterpret_cast<T*>(at(loc, l * (1 + CR))); }
  __host__ __device__ float* c(uint32_t loc, int l) const { return reinterpret_cast<float*>(at(loc, l * (1 + CR) + 1)); }
  __host__ __device__ T* gate(uint32_t loc, int L, int l, int q) const { return reinterpret_cast<T*>(at(loc, L * (1 + CR) + 4 * l + q)); }
  __host__ __device__ uint32_t input(uint32_t loc, int L) const { return loc + (L * (1 + CR) + 4 * L) * parts; }
};

__device__ __forceinline__ void part(int n, int T, int r, int& lo, int& hi) {   // CTA r's share of n things
  lo = (int)((int64_t)n * r / T);
  hi = (int)((int64_t)n * (r + 1) / T);
}

// One unit of the cell.  z: pre-activations without bias (GRU: z[2] the input part of n, z[3] the
// recurrent part); g: what the internal state keeps; cp: c_{k-1} (LSTM) or h_{k-1} (GRU).
template <bool GRU>
__device__ __forceinline__ void cell_forward(const float (&z)[4], const float (&bias)[4], float cp, float (&g)[4], float& h, float& c) {
  if (GRU) {
    g[0] = sigmoid(z[0] + bias[0]);
    g[1] = sigmoid(z[1] + bias[1]);
    g[3] = z[3];
    g[2] = tanhf(fmaf(g[0], g[3], z[2] + bias[2]));
    h = fmaf(g[1], cp - g[2], g[2]);   // (1 - z) n + z h
    c = 0.f;
  } else {
    g[0] = sigmoid(z[0] + bias[0]);
    g[1] = sigmoid(z[1] + bias[1]);
    g[2] = tanhf(z[2] + bias[2]);
    g[3] = sigmoid(z[3] + bias[3]);
    c = fmaf(g[1], cp, g[0] * g[2]);
    h = g[3] * tanhf(c);
  }
}
// Its derivatives.  dh: the gradient of h_k without what is carried; carry in: dc of the step after
// (LSTM), or the part of dh that bypassed its gates (GRU); carry out likewise.  h_prev is used by the
// GRU, c and c_prev by the LSTM.
template <bool GRU>
__device__ __forceinline__ void cell_backward(float dh, const float (&g)[4], float h_prev, float c, float c_prev, float& carry, float (&d)[4]) {
  if (GRU) {
    dh += carry;
    const float dn = dh * (1.f - g[1]) * (1.f - g[2] * g[2]);
    d[0] = dn * g[3] * g[0] * (1.f - g[0]);
    d[1] = dh * (h_prev - g[2]) * g[1] * (1.f - g[1]);
    d[2] = dn;
    d[3] = dn * g[0];
    carry = dh * g[1];
  } else {
    const float th = tanhf(c);
    const float dc = fmaf(dh * g[3], 1.f - th * th, carry);
    d[0] = dc * g[2] * g[0] * (1.f - g[0]);
    d[1] = dc * c_prev * g[1] * (1.f - g[1]);
    d[2] = dc * g[0] * (1.f - g[2] * g[2]);
    d[3] = dh * th * g[3] * (1.f - g[3]);
    carry = dc * g[1];
  }
}

}  // namespace team
}  // namespace mebptt
