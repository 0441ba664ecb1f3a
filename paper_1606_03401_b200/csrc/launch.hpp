// Kernel launches with programmatic stream serialization: the launched kernel may become
// resident (and run its prologue: barrier set-up, TMEM allocation) while the previous kernel of
// the stream is still running.  Every kernel launched through here calls grid_dep_wait before
// its first access to global memory.  MEBPTT_NO_PDL in the environment turns the attribute off.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstdlib>

#include "env.hpp"

namespace mebptt {

// Kernels launched by the process, counted where they are (a testing aid: what launch counts are compared with).
inline std::atomic<int64_t> g_launches{0};
inline cudaStream_t counted(cudaStream_t s) {
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return s;
}

inline bool pdl_enabled() { return !env::no_pdl(); }

// Dynamic shared memory of a kernel whose CTAs wait for one another while they hold tensor memory: more than half of an
// SM's 228 KB (a CTA takes 1 KB beside what it asks for), so that no SM ever has two such CTAs, of one kernel or of
// steps on different streams.  tcgen05.alloc blocks until its columns are free, and the scheduler, which places CTAs by
// shared memory, registers and threads, knows nothing of them: a CTA of kernel A could hold an SM where one of kernel B
// waits for columns, and one of B another where A waits, each kernel waiting for its own CTA for good.  CTAs that hold
// tensor memory and wait for nobody (the contractions) end by themselves, whatever they share an SM with.
// What it costs is that such CTAs no longer share SMs: with one layer up to 320 units wide, two steps on two streams.
constexpr int LONE_SMEM = 228 * 1024 / 2 - 1024 + 16;
inline int lone_smem(int bytes) { return bytes > LONE_SMEM ? bytes : LONE_SMEM; }

// CTAs that wait for one another the current device keeps resident (one an SM, as above); 0 if it cannot be asked.
inline int run_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return env::run_sms() > 0 && env::run_sms() < sms ? env::run_sms() : sms;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_on(bool pdl, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = counted(s);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = (pdl && pdl_enabled()) ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args) {
  return launch_on(true, kernel, grid, block, smem, s, static_cast<Args&&>(args)...);
}

// Cooperative launch (all CTAs co-resident), optionally in clusters of `cluster` CTAs, with
// programmatic stream serialization if the driver accepts the combination: the first refusal
// turns the attribute off for every later cooperative launch of the process.
inline cudaError_t launch_coop(const void* fn, int grid, int block, size_t smem, cudaStream_t s, void** args,
                               int cluster, bool early = true) {
  static std::atomic<int> pdl_state{-1};   // -1 untried, 0 refused, 1 accepted
  for (;;) {
    const bool pdl = early && pdl_enabled() && pdl_state.load() != 0;
    cudaLaunchAttribute at[3];
    int n = 0;
    at[n].id = cudaLaunchAttributeCooperative;
    at[n].val.cooperative = 1;
    ++n;
    if (cluster > 1) {
      at[n].id = cudaLaunchAttributeClusterDimension;
      at[n].val.clusterDim.x = (unsigned)cluster; at[n].val.clusterDim.y = 1; at[n].val.clusterDim.z = 1;
      ++n;
    }
    if (pdl) {
      at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[n].val.programmaticStreamSerializationAllowed = 1;
      ++n;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3((unsigned)block); cfg.dynamicSmemBytes = smem; cfg.stream = s;
    cfg.attrs = at; cfg.numAttrs = (unsigned)n;
    const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
    if (e == cudaSuccess) {
      (void)counted(s);
      if (pdl) pdl_state.store(1);
      return e;
    }
    if (!pdl || pdl_state.load() == 1) return e;
    cudaGetLastError();
    pdl_state.store(0);
  }
}

}  // namespace mebptt
