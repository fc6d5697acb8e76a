// Device helpers shared by the sweep kernels: L2 policies, vector accesses
// that keep the iterates in L2, and the epilogues.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "device.cuh"

namespace silu {
namespace {

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint64_t policy_evict_normal() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Vector accesses that keep the iterates resident in L2 across sweeps.  A sweep
// may be resident while the kernel before it still writes these vectors: the
// loads stay behind griddepcontrol.wait (volatile, memory clobber) and are
// ordinary ones (an .nc load is for data that nobody writes meanwhile).
__device__ __forceinline__ double ld_keep(const double* p, uint64_t pol) {
  double v;
  asm volatile("ld.global.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol) : "memory");
  return v;
}
__device__ __forceinline__ float ld_keep(const float* p, uint64_t pol) {
  float v;
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol) : "memory");
  return v;
}
__device__ __forceinline__ void st_keep(double* p, double v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(p), "d"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void st_keep(float* p, float v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p), "f"(v), "l"(pol) : "memory");
}

// Epilogue operands (dinv_row, x_row) are read after the accumulation; a
// prefetch into L1 issued before it takes their memory latency off the end
// of the tile without holding registers through the gathers.
__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}
__device__ __forceinline__ void prefetch_epilogue(int epi, int row, size_t o, const double* dinv, const double* x) {
  switch (epi) {
    case EPI_SCALE:
      prefetch_l1(dinv + row);
      break;
    case EPI_SCALE_ADDX:
    case EPI_JAC_ADDX:
      prefetch_l1(dinv + row);
      prefetch_l1(x + o);
      break;
    case EPI_SCALE_SETX:
    case EPI_JAC:
    case EPI_JAC_SETX:
      prefetch_l1(dinv + row);
      break;
    case EPI_ADDX:
    case EPI_RICH_ADDX:
      prefetch_l1(x + o);
      break;
    default:
      break;
  }
}

// t = c_row - (T in)_row, already formed by the accumulation
template <class MT, class VI, class VO>
__device__ __forceinline__ void epilogue(int epi, int row, MT t, const VI* in, VO* out, const double* dinv,
                                         double* x, uint64_t keep) {
  switch (epi) {
    case EPI_STORE: st_keep(out + row, (VO)t, keep); break;
    case EPI_SCALE: st_keep(out + row, (VO)(dinv[row] * (double)t), keep); break;
    case EPI_ADDX: x[row] += (double)t; break;
    case EPI_SETX: x[row] = (double)t; break;
    case EPI_SCALE_ADDX: x[row] += dinv[row] * (double)t; break;
    case EPI_SCALE_SETX: x[row] = dinv[row] * (double)t; break;
    case EPI_JAC: st_keep(out + row, (VO)((MT)in[row] + (MT)dinv[row] * t), keep); break;
    case EPI_JAC_ADDX: x[row] += (double)((MT)in[row] + (MT)dinv[row] * t); break;
    case EPI_JAC_SETX: x[row] = (double)((MT)in[row] + (MT)dinv[row] * t); break;
    case EPI_RICH: st_keep(out + row, (VO)(t + (MT)in[row]), keep); break;
    case EPI_RICH_ADDX: x[row] += (double)(t + (MT)in[row]); break;
    case EPI_RICH_SETX: x[row] = (double)(t + (MT)in[row]); break;
    default: break;
  }
}

// The same epilogues for column k of R interleaved right-hand sides: vector
// entries at o = row * ldx + k, dinv at row.
template <class MT, class VI, class VO>
__device__ __forceinline__ void epilogue_col(int epi, int row, size_t o, MT t, const VI* in, VO* out,
                                             const double* dinv, double* x, uint64_t keep) {
  switch (epi) {
    case EPI_STORE: st_keep(out + o, (VO)t, keep); break;
    case EPI_SCALE: st_keep(out + o, (VO)(dinv[row] * (double)t), keep); break;
    case EPI_ADDX: x[o] += (double)t; break;
    case EPI_SETX: x[o] = (double)t; break;
    case EPI_SCALE_ADDX: x[o] += dinv[row] * (double)t; break;
    case EPI_SCALE_SETX: x[o] = dinv[row] * (double)t; break;
    case EPI_JAC: st_keep(out + o, (VO)((MT)in[o] + (MT)dinv[row] * t), keep); break;
    case EPI_JAC_ADDX: x[o] += (double)((MT)in[o] + (MT)dinv[row] * t); break;
    case EPI_JAC_SETX: x[o] = (double)((MT)in[o] + (MT)dinv[row] * t); break;
    case EPI_RICH: st_keep(out + o, (VO)(t + (MT)in[o]), keep); break;
    case EPI_RICH_ADDX: x[o] += (double)(t + (MT)in[o]); break;
    case EPI_RICH_SETX: x[o] = (double)(t + (MT)in[o]); break;
    case EPI_SPMV: st_keep(out + o, (VO)t, keep); break;
    default: break;
  }
}

}  // namespace
}  // namespace silu
