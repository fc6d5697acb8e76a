// Device helpers of the Krylov kernels: warp sums, the exchange of partial
// sums between resident blocks, and division by one divisor.
#pragma once

#include <cuda_runtime.h>

namespace silu {

constexpr unsigned long long kArnWaitNs = 2000000000ull;  // 2 s bound on any wait

__device__ __forceinline__ unsigned long long arn_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ double arn_warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

__device__ __forceinline__ void publish(ulonglong2* e, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned long long t = (unsigned long long)tag << 32;
  const unsigned long long lo = t | (b & 0xffffffffull), hi = t | (b >> 32);
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(e), "l"(lo), "l"(hi) : "memory");
}

__device__ __forceinline__ bool peek(const ulonglong2* e, unsigned tag, double& v) {
  unsigned long long lo, hi;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(lo), "=l"(hi) : "l"(e) : "memory");
  if ((unsigned)(lo >> 32) != tag || (unsigned)(hi >> 32) != tag) return false;
  v = __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
  return true;
}

// The K values at e[0], e[stride], ... (those with k < cnt), once all are there.
template <int K>
__device__ __forceinline__ void collect(const ulonglong2* e, int stride, int cnt, unsigned tag, double (&v)[K],
                                        bool& alive, int* err) {
  unsigned missing = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    v[k] = 0.0;
    if (k < cnt && !peek(e + k * stride, tag, v[k])) missing |= 1u << k;
  }
  if (!missing || !alive) return;
  const unsigned long long t0 = arn_ns();
  for (unsigned spins = 1; missing; ++spins) {
    __nanosleep(100);
#pragma unroll
    for (int k = 0; k < K; ++k)
      if ((missing >> k) & 1u)
        if (peek(e + k * stride, tag, v[k])) missing &= ~(1u << k);
    if ((spins & 255u) == 0 && arn_ns() - t0 > kArnWaitNs) {
      atomicOr(err, 16);
      alive = false;
      return;
    }
  }
}

// w / h for many w: correctly rounded, five FP64 operations instead of the
// division's twelve or so (which made normalising 1.9 M rows 48 us of FP64
// work).  r = RN(1/h); q0 = RN(w r), within two units in the last place; the
// first step q + RN(w - q h) r makes q faithful, whatever its remainder loses
// to rounding; the second starts from a faithful q, whose remainder an FMA
// gives exactly, and rounds correctly (Markstein, "IA-64 and Elementary
// Functions", Sec. 8.1: a correctly rounded reciprocal and a faithful quotient
// give the rounded one).  That holds while
// nothing over- or underflows, so operands outside the middle of the exponent
// range (zeros, infinities and NaN among them) are divided.
struct Divider {
  double h, r;
  bool fast;
  __device__ __forceinline__ explicit Divider(double d) : h(d), r(1.0 / d) {
    const int e = (__double2hiint(d) >> 20) & 0x7ff;
    fast = e > 1023 - 300 && e < 1023 + 300;
  }
  __device__ __forceinline__ double operator()(double w) const {
    const int e = (__double2hiint(w) >> 20) & 0x7ff;
    if (!(fast && e > 1023 - 600 && e < 1023 + 600)) return w / h;
    double q = w * r;
    q = fma(fma(-q, h, w), r, q);
    return fma(fma(-q, h, w), r, q);
  }
};

}  // namespace silu
