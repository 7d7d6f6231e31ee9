// The waits of the panels that hold their rows in shared memory (panel_cluster.cu),
// both bounded: a cluster's transaction barrier, and words in global memory that
// carry the column's stamp beside their data.
#pragma once

#include "common.cuh"

namespace gb {

__device__ __forceinline__ bool pc_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// wait for the phase of a transaction barrier; *abort_flag (shared memory) is set
// when the wait runs out, and seen by every thread after the CTA's next barrier
__device__ __forceinline__ void pc_wait(uint32_t bar, uint32_t parity, int* abort_flag, int* status) {
  if (pc_try(bar, parity)) return;
  const uint64_t t0 = gtimer();
  while (!pc_try(bar, parity)) {
    if (*(volatile int*)abort_flag) return;
    if (gtimer() - t0 > GB_SPIN_LIMIT_NS) {
      atomicOr(status, ST_TIMEOUT);
      *(volatile int*)abort_flag = 1;
      return;
    }
  }
}

// A value between its stamps: a double as two 8-byte words {low half, stamp},
// {high half, stamp}, a float as one; relaxed loads and stores (each 8-byte word
// is read and written whole).
__device__ __forceinline__ ulonglong2 pr_load(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void pr_store(ulonglong2* p, ulonglong2 v) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v.x), "l"(v.y) : "memory");
}
template <typename T>
struct PrWord;
template <>
struct PrWord<double> {
  using type = ulonglong2;
  static __device__ __forceinline__ void put(type* p, double v, unsigned stamp) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    pr_store(p, make_ulonglong2((b << 32) | stamp, (b & 0xffffffff00000000ull) | stamp));
  }
  static __device__ __forceinline__ bool get(const type* p, double& v, unsigned stamp) {
    const ulonglong2 x = pr_load(p);
    v = __longlong_as_double((long long)((x.y & 0xffffffff00000000ull) | (x.x >> 32)));
    return (unsigned)x.x == stamp && (unsigned)x.y == stamp;
  }
};
template <>
struct PrWord<float> {
  using type = unsigned long long;
  static __device__ __forceinline__ void put(type* p, float v, unsigned stamp) {
    const unsigned long long x = ((unsigned long long)__float_as_uint(v) << 32) | stamp;
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
  }
  static __device__ __forceinline__ bool get(const type* p, float& v, unsigned stamp) {
    unsigned long long x;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
    v = __uint_as_float((unsigned)(x >> 32));
    return (unsigned)x == stamp;
  }
};

// wait for a stamped value; *abort_flag is set when the wait runs out
template <typename T>
__device__ __forceinline__ void pr_fetch(const typename PrWord<T>::type* q, T& v, unsigned stamp, int* abort_flag,
                                         int* status) {
  if (PrWord<T>::get(q, v, stamp)) return;
  const uint64_t t0 = gtimer();
  while (!PrWord<T>::get(q, v, stamp)) {
    if (*(volatile int*)abort_flag) return;
    if (gtimer() - t0 > GB_SPIN_LIMIT_NS) {
      atomicOr(status, ST_TIMEOUT);
      *(volatile int*)abort_flag = 1;
      return;
    }
  }
}

}  // namespace gb
