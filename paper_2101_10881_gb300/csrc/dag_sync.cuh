// dag_sync.cuh -- how the jobs of a persistent launch wait for one another: completion
// flags set to the call's epoch, bounded waits, a global abort flag.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.hpp"

namespace pes {

namespace {

constexpr int kStatusTimeout = 5;  // PES_ETIMEOUT

__device__ __forceinline__ unsigned long long global_timer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int ld_acquire(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(int32_t* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void set_error(Ctrl* ctrl, int code, long long d0, long long d1) {
  if (atomicCAS(&ctrl->status, 0, code) == 0) {
    ctrl->diag[0] = d0;
    ctrl->diag[1] = d1;
  }
  atomicExch(&ctrl->abort, 1);
}

// Parts of every job of the launch (a split of 0 reads as 1).
__device__ __forceinline__ int parts(const DagArgs& a) { return a.split > 1 ? a.split : 1; }

// Every part of job `dep` of this call has completed (dep < 0: an input series).
__device__ __forceinline__ bool is_done(const DagArgs& a, int dep, int epoch) {
  if (dep < 0) return true;
  const int s = parts(a);
  for (int p = 0; p < s; ++p)
    if (ld_acquire(a.flags + dep * s + p) != epoch) return false;
  return true;
}

// Bounded wait until sub-job `f` (a flag index) of this call has completed.
__device__ bool wait_flag(const DagArgs& a, int f, int epoch, int job) {
  if (ld_acquire(a.flags + f) == epoch) return true;
  unsigned long long t0 = global_timer();
  for (;;) {
    if (ld_acquire(a.flags + f) == epoch) return true;
    if (*reinterpret_cast<volatile int32_t*>(&a.ctrl->abort)) return false;
    if (static_cast<long long>(global_timer() - t0) > a.timeout_ns) {
      set_error(a.ctrl, kStatusTimeout, f, job);
      return false;
    }
    __nanosleep(200);
  }
}

// Bounded wait until every part of job `dep` of this call has completed.
__device__ bool wait_done(const DagArgs& a, int dep, int epoch, int job) {
  if (dep < 0) return true;
  const int s = parts(a);
  for (int p = 0; p < s; ++p)
    if (!wait_flag(a, dep * s + p, epoch, job)) return false;
  return true;
}

}  // namespace

}  // namespace pes
