// What the kernels that hand data from CTA to CTA share: bounded waits and loads that see other
// SMs' stores.
#pragma once

#include "mma_tiles.cuh"

namespace {

constexpr int kCopies = 8;     // of the logit words (expert_chain.cu)

__device__ __forceinline__ unsigned long long clock_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// A bound for a spin: expired() is called once per turn and looks at the clock every 32nd.
// P: parameters with hold, wait_ns and status.
struct SpinBound {
  unsigned long long t0 = 0;
  unsigned n = 0;
  template <class P>
  __device__ __forceinline__ bool expired(const P& p) {
    if (++n & 31u) return false;
    const unsigned long long now = clock_ns();
    if (t0 == 0) t0 = now;
    const unsigned long long el = now - t0;
    if (el > (p.hold ? 2000000ull : p.wait_ns)) return true;
    // once a wait has run out on this handle the later ones give up quickly, until the caller has
    // read and cleared the status word
    return el > 1000000ull &&
           (*reinterpret_cast<volatile uint32_t*>(p.status) & BLOCKFFN_DEV_WAIT_EXPIRED) != 0;
  }
};
// 32 bytes, 32-byte aligned: 16 consecutive k of a row. (Four lanes then take a whole line of a
// row with one instruction; with two 16-byte loads the eight rows' lines are looked up twice.)
__device__ __forceinline__ void ld_relaxed_v8(Frag64& f, const void* p) {
  asm volatile("ld.relaxed.gpu.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(f.lo.x), "=r"(f.lo.y), "=r"(f.lo.z), "=r"(f.lo.w), "=r"(f.hi.x), "=r"(f.hi.y),
                 "=r"(f.hi.z), "=r"(f.hi.w)
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_cg128(const void* p) {
  uint4 v;
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
// whether one of the eight words has not been written (a word is written as a whole, and its upper
// half is never 0xffff then)
__device__ __forceinline__ bool unwritten(const Frag64& f) {
  const uint32_t a = max(max(f.lo.x, f.lo.y), max(f.lo.z, f.lo.w));
  const uint32_t b = max(max(f.hi.x, f.hi.y), max(f.hi.z, f.hi.w));
  return max(a, b) >= 0xffff0000u;
}

}  // namespace
