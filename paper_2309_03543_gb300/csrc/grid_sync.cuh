// Grid synchronisation of the persistent solves (one cooperative launch, all
// blocks resident): release / acquire flags, bounded waits and the halo flags
// between neighbouring blocks.
#pragma once

#include "cps_internal.cuh"

#include <cstdint>

namespace cps {
namespace {

constexpr int kPBlock = 1024;
constexpr long long kSpinCap = 1LL << 26;           // polls; each one an L2 round trip
constexpr unsigned long long kWaitNs = 1000000000ull;
constexpr int kFlagStride = 16;                      // one 128-byte line per block flag
constexpr int kMaxDeps = 8;
constexpr int kPartialSlots = 4;                     // quantities per reduction buffer

struct GridSync {
    unsigned long long count;   // arrivals since the launch
    int timeout;
    int pad[29];
    unsigned long long flag[kMaxGrid * kFlagStride];   // per-block iteration flags
};

__device__ __forceinline__ void red_release_add(unsigned long long* p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Hint: fetch the line holding p into this SM's L1 (no register result).
__device__ __forceinline__ void prefetch_l1(const void* p) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait until *p >= target (one thread).  False if it ran out, or if
// another block has already recorded a timeout.
__device__ bool wait_geq(const unsigned long long* p, unsigned long long target, GridSync* gs) {
    if (ld_acquire(p) < target) {
        const unsigned long long t0 = global_ns();
        for (long long spins = 1;; ++spins) {
            if (ld_acquire(p) >= target) break;
            if (spins > kSpinCap || ((spins & 255) == 0 && global_ns() - t0 > kWaitNs)) {
                atomicExch(&gs->timeout, 1);
                return false;
            }
        }
    }
    return *(volatile int*)&gs->timeout == 0;
}

// This block has finished phase `slot` (0: direction update, 1: the reduced
// system's red phase) `it` times.
__device__ __forceinline__ void halo_post(GridSync* gs, unsigned long long it, int slot = 0) {
    __syncthreads();
    if (threadIdx.x == 0) st_release(&gs->flag[blockIdx.x * kFlagStride + slot], it);
}

// Wait until the blocks [dlo, dhi] (other than this one) have posted `it`
// in `slot`.
__device__ bool halo_wait(GridSync* gs, int dlo, int dhi, unsigned long long it, int slot = 0) {
    __shared__ int s_ok;
    if (threadIdx.x == 0) {
        int ok = 1;
        for (int d = dlo; d <= dhi && ok; ++d)
            if (d != (int)blockIdx.x && !wait_geq(&gs->flag[d * kFlagStride + slot], it, gs))
                ok = 0;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace
}  // namespace cps
