// Device-side building blocks shared by the solver kernels: warp / block
// reductions, L2-coherent loads, and the bounded grid barrier.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mlg {

// Host-side count of kernels this library has launched (all handles); the
// launch sites call note_launches() right after each launch.
void note_launches(long long k);
long long launches_so_far();

constexpr int kErrNone = 0;
constexpr int kErrTimeout = -4;
constexpr int kErrNonfinite = -5;
constexpr int kErrConfig = -6;  // launch parameters inconsistent with a task (reported as ERR_CUDA)

// Loads of data that another CTA wrote before a grid barrier go through L2
// (ld.global.cg) so a stale L1 line can never be read.
template <typename T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const void* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u64(void* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_relaxed_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// 16-byte words, each read and written as one (single-copy atomic b128 accesses).
__device__ __forceinline__ void st_relaxed_b128(void* p, uint4 v) {
  asm volatile(
      "{\n .reg .b128 w;\n .reg .b64 lo, hi;\n mov.b64 lo, {%1, %2};\n mov.b64 hi, {%3, %4};\n"
      " mov.b128 w, {lo, hi};\n st.relaxed.gpu.global.b128 [%0], w;\n}" ::"l"(p),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
      : "memory");
}
__device__ __forceinline__ uint4 ld_relaxed_b128(const void* p) {
  uint4 v;
  asm volatile(
      "{\n .reg .b128 w;\n .reg .b64 lo, hi;\n ld.relaxed.gpu.global.b128 w, [%4];\n"
      " mov.b128 {lo, hi}, w;\n mov.b64 {%0, %1}, lo;\n mov.b64 {%2, %3}, hi;\n}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p)
      : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier over a group of `nblocks` co-resident CTAs sharing the monotonically
// increasing counter *ctr (zeroed before the launch).  Every wait is bounded:
// after timeout_ns the waiting CTA raises *err = kErrTimeout and every CTA
// leaves its wait as soon as it sees a raised *err.  Returns false when the
// group must abandon the solve.  `epoch` is the caller's count of barriers
// passed (only thread 0's copy is used).
struct GroupBarrier {
  unsigned long long* ctr;
  int* err;
  unsigned nblocks;
  unsigned long long timeout_ns;
};

// Thread 0's half of the group barrier: arrive (release) and wait (acquire,
// bounded); returns 0 on a timeout or a raised error flag.  RELAXED: neither
// releases nor acquires -- it only says when the group has arrived, for data
// that carries its own tags (the release's wait for the CTA's stores to be
// performed is then off the critical path).
template <bool RELAXED = false>
__device__ __forceinline__ int group_arrive_wait(const GroupBarrier& gb, unsigned long long& epoch) {
  epoch += 1;
  const unsigned long long target = epoch * (unsigned long long)gb.nblocks;
  if (RELAXED)
    red_relaxed_add_u64(gb.ctr, 1ull);
  else
    red_release_add_u64(gb.ctr, 1ull);
  auto poll = [&]() { return RELAXED ? ld_relaxed_u64(gb.ctr) : ld_acquire_u64(gb.ctr); };
  int ok = 1;
  if (poll() < target) {
    const unsigned long long t0 = globaltimer_ns();
    unsigned it = 0;
    while (poll() < target) {
      // the error flag and the clock every eighth poll: a poll is one load
      if ((++it & 7u) != 0) continue;
      if (*(volatile int*)gb.err != kErrNone) { ok = 0; break; }
      if (globaltimer_ns() - t0 > gb.timeout_ns) {
        atomicCAS(gb.err, kErrNone, kErrTimeout);
        ok = 0;
        break;
      }
    }
  }
  if (ok && *(volatile int*)gb.err != kErrNone) ok = 0;
  return ok;
}

// One round of a bounded spin on tagged data: false once the group must give up
// (a raised error flag, or the limit passed since the first round).
struct SpinLimit {
  unsigned it = 0;
  unsigned long long t0 = 0;
  __device__ __forceinline__ bool more(const GroupBarrier& gb) {
    if ((++it & 15u) != 0) return true;
    if (*(volatile int*)gb.err != kErrNone) return false;
    const unsigned long long t = globaltimer_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > gb.timeout_ns) {
      atomicCAS(gb.err, kErrNone, kErrTimeout);
      return false;
    }
    return true;
  }
};

// side() runs on warp 1 while thread 0 waits at the barrier (work that would
// otherwise sit on the critical path between two barriers).
template <typename Side>
__device__ __forceinline__ bool group_sync_with(const GroupBarrier& gb,
                                                unsigned long long& epoch, int* s_flag,
                                                Side side) {
  __syncthreads();
  if ((threadIdx.x >> 5) == 1) side();
  if (gb.nblocks == 1) {  // a one-CTA group only needs the CTA barrier
    if (threadIdx.x == 0) *s_flag = (*(volatile int*)gb.err == kErrNone);
    __syncthreads();
    return *s_flag != 0;
  }
  if (threadIdx.x == 0) {
    // the CTA's writes are ordered before this release by the CTA barrier
    // above; the acquire loads order the other CTAs' writes before the CTA
    // barrier that ends the wait (release/acquire at gpu scope, cumulative
    // through bar.sync), so no separate fences are needed
    *s_flag = group_arrive_wait(gb, epoch);
  }
  __syncthreads();
  return *s_flag != 0;
}

struct NoSide {
  __device__ void operator()() const {}
};

__device__ __forceinline__ bool group_sync(const GroupBarrier& gb, unsigned long long& epoch,
                                           int* s_flag) {
  return group_sync_with(gb, epoch, s_flag, NoSide());
}

}  // namespace mlg
