// The sliced sweep (sm_103a): out = epilogue(c - T in) for R = 1..4
// interleaved right-hand sides, one warp per slice of 32 rows, one lane per
// row, on the padded slices of `Slices` (device.cuh).
//
// What bounds it: FP64 sweeps run at the rate of the FP64 pipe (one warp-wide
// fused multiply-add per padded entry and column takes 19 clocks of an SM's
// FP64 unit, whatever lanes are active: 500 to 530 G lane-FMAs/s); FP32
// sweeps at HBM.  So the slices carry the fewest bytes (10 per FP64 entry and
// 6 per FP32 entry against 12 and 8 in CSR, no row pointers) and the kernel
// keeps the FP64 pipe fed: no shared memory, hence the whole L1 for the
// gathers and as many warps as the registers allow; the loads of a warp's
// next chunk of entries (of the same slice or of its next one) are issued
// after the current chunk's gathers and before its multiply-adds, so a warp
// always has one chunk in flight.  Measured against the tiled CSR sweeps
// (k_sweep_rows, k_sweep_staged, k_sweep_multi): 128^3 cut-cell ILUT FP64
// lower / upper sweep 45.9 / 49.6 -> 43.9 / 43.9 us (20.9 M slots: 477 G/s),
// 24^3 ILUT 10+10 application 83 -> 38 us, 160^3 27-point FP64 residual 290 -> 232 us,
// three columns of the 101 x 97 x 89 box 1111 -> 507 us per application.
//
// Each lane accumulates c_i - sum t_ij in_j in column order with one FMA per
// entry, in LN partial sums for rows that the tiled sweep gives to LN lanes
// (entry k into sum k mod LN, then the sums added as that sweep's lanes add
// theirs), so results are the tiled sweep's bits; a padded entry multiplies 0 by 0,
// which leaves the accumulator as it is (its column is not read, so an
// infinite or NaN entry of `in` reaches only the rows that refer to it).
//
// The next launch is released (its blocks become resident and read their
// first entries) only once this one may start: were it released at once, the
// blocks of three and more later launches would fill the SMs, and a launch
// would start wherever room happened to be left, two blocks on some SMs and
// none on others (24^3 ILUT 5+5 application 24.2 -> 19 us, 42^3 ILUT 10+10
// 62.8 -> 59.5 us, 128^3 823 -> 819 us).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "device.cuh"
#include "sweep_ptx.cuh"

namespace silu {
namespace {

// Loads of the matrix stream: not kept in L1, which is left to the gathers.
__device__ __forceinline__ void ld_pair(const double* p, uint64_t pol, double& a, double& b) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;" : "=d"(a), "=d"(b) : "l"(p), "l"(pol));
}
__device__ __forceinline__ void ld_pair(const float* p, uint64_t pol, float& a, float& b) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(a), "=f"(b) : "l"(p), "l"(pol));
}
__device__ __forceinline__ void ld_one(const double* p, uint64_t pol, double& a) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(a) : "l"(p), "l"(pol));
}
__device__ __forceinline__ void ld_one(const float* p, uint64_t pol, float& a) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(a) : "l"(p), "l"(pol));
}

// The columns of CP pairs of entries of one lane.
template <class CT, int CP>
struct SliceCols;

template <int CP>
struct SliceCols<uint16_t, CP> {
  unsigned o[CP];
  __device__ __forceinline__ void pair(int q, const uint16_t* p, uint64_t pol) {
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(o[q]) : "l"(p), "l"(pol));
  }
  __device__ __forceinline__ void one(int q, const uint16_t* p, uint64_t pol) {
    uint16_t v;
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(v) : "l"(p), "l"(pol));
    o[q] = 0xffff0000u | v;
  }
  __device__ __forceinline__ void none(int q) { o[q] = 0xffffffffu; }
  __device__ __forceinline__ unsigned at(int k) const { return (k & 1) ? o[k >> 1] >> 16 : o[k >> 1] & 0xffffu; }
  static __device__ __forceinline__ bool padded(unsigned c) { return c == 0xffffu; }
};

template <int CP>
struct SliceCols<int, CP> {
  unsigned o[2 * CP];
  __device__ __forceinline__ void pair(int q, const int* p, uint64_t pol) {
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.u32 {%0, %1}, [%2], %3;"
        : "=r"(o[2 * q]), "=r"(o[2 * q + 1])
        : "l"(p), "l"(pol));
  }
  __device__ __forceinline__ void one(int q, const int* p, uint64_t pol) {
    asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(o[2 * q]) : "l"(p), "l"(pol));
    o[2 * q + 1] = 0xffffffffu;
  }
  __device__ __forceinline__ void none(int q) { o[2 * q] = o[2 * q + 1] = 0xffffffffu; }
  __device__ __forceinline__ unsigned at(int k) const { return o[k]; }
  static __device__ __forceinline__ bool padded(unsigned c) { return c == 0xffffffffu; }
};

// R adjacent vector entries (ordered as ld_keep's).  VEC: in 16-byte (or, two floats, 8-byte) loads,
// for pointers and leading dimensions that keep every row's entries aligned.
template <class MT, int R, bool VEC>
__device__ __forceinline__ void ld_cols(const double* p, uint64_t pol, MT (&v)[R]) {
  if constexpr (VEC) {
#pragma unroll
    for (int k = 0; k < R; k += 2) {
      double a, b;
      asm volatile("ld.global.L2::cache_hint.v2.f64 {%0, %1}, [%2], %3;"
                   : "=d"(a), "=d"(b)
                   : "l"(p + k), "l"(pol)
                   : "memory");
      v[k] = (MT)a;
      v[k + 1] = (MT)b;
    }
  } else {
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = (MT)ld_keep(p + k, pol);
  }
}
template <class MT, int R, bool VEC>
__device__ __forceinline__ void ld_cols(const float* p, uint64_t pol, MT (&v)[R]) {
  if constexpr (VEC && R == 4) {
    float a, b, c, d;
    asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(a), "=f"(b), "=f"(c), "=f"(d)
                 : "l"(p), "l"(pol)
                 : "memory");
    v[0] = a;
    v[1] = b;
    v[2] = c;
    v[3] = d;
  } else if constexpr (VEC && R == 2) {
    float a, b;
    asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;"
                 : "=f"(a), "=f"(b)
                 : "l"(p), "l"(pol)
                 : "memory");
    v[0] = a;
    v[1] = b;
  } else {
#pragma unroll
    for (int k = 0; k < R; ++k) v[k] = (MT)ld_keep(p + k, pol);
  }
}

constexpr int kSliceThreads = 256;

// The epilogues that read dinv, and those that read x.
constexpr unsigned kEpiDinv = 1u << EPI_SCALE | 1u << EPI_SCALE_ADDX | 1u << EPI_SCALE_SETX | 1u << EPI_JAC |
                              1u << EPI_JAC_ADDX | 1u << EPI_JAC_SETX;
constexpr unsigned kEpiX = 1u << EPI_ADDX | 1u << EPI_SCALE_ADDX | 1u << EPI_JAC_ADDX | 1u << EPI_RICH_ADDX;

// Launch flag beside the L2 flags: block b of B walks the slices
// [b ns / B, (b + 1) ns / B) (of few per warp: B ns fits 32 bits) instead of
// every (B W)-th group of W.
constexpr int kFlagSpread = 8;

// CP pairs of entries per chunk, at least MINB blocks of (up to) 8 warps per SM,
// LN partial sums per row.
template <class MT, class VI, class VO, class CT, int R, int CP, int MINB, bool VEC, int LN>
__global__ void __launch_bounds__(kSliceThreads, MINB)
    k_slices(int ns, int n, const int2* __restrict__ hdr, const CT* __restrict__ ci, const MT* __restrict__ va,
             const VI* c, const VI* in, VO* __restrict__ out, int ldx,
             const double* __restrict__ dinv, double* __restrict__ x, int epi, int flags) {
  static_assert(2 * CP % LN == 0, "a chunk starts at the first partial sum");
  const int W = blockDim.x >> 5;
  const int ld = R == 1 ? 1 : ldx;
  const int lane = threadIdx.x & 31;
  const bool spread = (flags & kFlagSpread) != 0;
  const int nw = spread ? W : gridDim.x * W;
  int s = blockIdx.x * W + (threadIdx.x >> 5), end = ns;
  if (spread) {
    s = (int)((unsigned)blockIdx.x * (unsigned)ns / gridDim.x) + (threadIdx.x >> 5);
    end = (int)(((unsigned)blockIdx.x + 1u) * (unsigned)ns / gridDim.x);
  }
  const bool rev = (flags & kFlagReverse) != 0;
  const uint64_t stream = (flags & kFlagFactorNormal) ? policy_evict_normal() : policy_evict_first();
  const uint64_t keep = (flags & kFlagVectorNormal) ? policy_evict_normal() : policy_evict_last();
  if (s >= end) {
    grid_wait_prior();
    return;
  }
  MT v[2 * CP];
  SliceCols<CT, CP> col;
  // the chunk of entries [p, min(p + 64 CP, pe)) of a slice, p and pe multiples of 32
  auto load = [&](int p, int pe) {
#pragma unroll
    for (int q = 0; q < CP; ++q) {
      const int a = p + 64 * q;
      if (a + 64 <= pe) {
        ld_pair(va + a + 2 * lane, stream, v[2 * q], v[2 * q + 1]);
        col.pair(q, ci + a + 2 * lane, stream);
      } else if (a < pe) {
        ld_one(va + a + lane, stream, v[2 * q]);
        v[2 * q + 1] = MT(0);
        col.one(q, ci + a + lane, stream);
      } else {
        v[2 * q] = v[2 * q + 1] = MT(0);
        col.none(q);
      }
    }
  };
  // the row's constant term, and its epilogue operands into L1
  auto start_row = [&](int row, MT (&a)[R]) {
#pragma unroll
    for (int k = 0; k < R; ++k) a[k] = MT(0);
    if (row < n) {
      const size_t o = (size_t)row * (size_t)ld;
      if (c) ld_cols<MT, R, VEC>(c + o, keep, a);
      if ((kEpiDinv >> epi) & 1u) prefetch_l1(dinv + row);
      if ((kEpiX >> epi) & 1u) prefetch_l1(x + o);
    }
  };
  int sl = rev ? ns - 1 - s : s;
  int2 h = __ldg(hdr + sl);
  int p = h.x, pe = __ldg(&hdr[sl + 1].x);
  load(p, pe);  // the matrix is never written by a sweep: its first entries need not wait
  s += nw;
  int nsl = 0, npe = 0;
  int2 nh = make_int2(0, 0);
  if (s < end) {
    nsl = rev ? ns - 1 - s : s;
    nh = __ldg(hdr + nsl);
    npe = __ldg(&hdr[nsl + 1].x);
  }
  grid_wait_prior();  // c, in, out and x below belong to the previous kernel until it completes
  grid_launch_dependents();
  int row = sl * 32 + lane;
  MT acc[LN][R];  // acc[0] starts at c
  auto clear_rest = [&]() {
#pragma unroll
    for (int l = 1; l < LN; ++l)
#pragma unroll
      for (int k = 0; k < R; ++k) acc[l][k] = MT(0);
  };
  start_row(row, acc[0]);
  clear_rest();
  for (;;) {
    const VI* ib = in;
    if constexpr (sizeof(CT) == 2) ib = in + (size_t)h.y * (size_t)ld;
    MT xv[2 * CP][R], w[2 * CP];
#pragma unroll
    for (int q = 0; q < 2 * CP; ++q) {
      const unsigned j = col.at(q);
      w[q] = v[q];
      if (!SliceCols<CT, CP>::padded(j)) {
        ld_cols<MT, R, VEC>(ib + (size_t)j * (size_t)ld, keep, xv[q]);
      } else {
#pragma unroll
        for (int k = 0; k < R; ++k) xv[q][k] = MT(0);
      }
    }
    const int left = (pe - p) >> 5;  // entries of the slice's longest row from this chunk on
    p += 64 * CP;
    const bool last = p >= pe;
    const int orow = row;
    bool more = true;
    MT nacc[R];
    if (!last) {
      load(p, pe);
    } else {
      more = s < end;
      if (more) {
        h = nh;
        p = h.x;
        pe = npe;
        row = nsl * 32 + lane;
        load(p, pe);
        start_row(row, nacc);
        s += nw;
        if (s < end) {
          nsl = rev ? ns - 1 - s : s;
          nh = __ldg(hdr + nsl);
          npe = __ldg(&hdr[nsl + 1].x);
        }
      }
    }
    // warp-uniform exit: a padded multiply-add would still occupy the FP64 pipe
#pragma unroll
    for (int q = 0; q < 2 * CP; ++q) {
      if (q >= left) break;
#pragma unroll
      for (int k = 0; k < R; ++k) acc[q % LN][k] = fma(-w[q], xv[q][k], acc[q % LN][k]);
    }
    if (last) {
#pragma unroll
      for (int off = LN / 2; off > 0; off >>= 1)
#pragma unroll
        for (int l = 0; l < off; ++l)
#pragma unroll
          for (int k = 0; k < R; ++k) acc[l][k] += acc[l + off][k];
      if (orow < n) {
        const size_t o = (size_t)orow * (size_t)ld;
#pragma unroll
        for (int k = 0; k < R; ++k) {
          if (epi == EPI_SPMV)
            st_keep(out + o + k, (VO)(MT(0) - acc[0][k]), keep);  // summed as 0 - T in, the same roundings
          else
            epilogue_col<MT, VI, VO>(epi, orow, o + k, acc[0][k], in, out, dinv, x, keep);
        }
      }
      if (!more) break;
#pragma unroll
      for (int k = 0; k < R; ++k) acc[0][k] = nacc[k];
      clear_rest();
    }
  }
}

// Matrices of at most 16 slices per SM: a launch is a chain of latencies, so a
// chunk takes a whole row (one round of gathers), whatever registers it needs,
// and the slices are split evenly over one block per SM (two beyond eight
// slices per SM), each of no more warps than its share: blocks of eight warps
// leave SMs idle while the four FP64 partitions of others queue (24^3 ILUT
// 10+10 application 60 us that way, 38.3 us this way).  The line: 5+5
// applications at 10 slices per SM (36^3), 1 / 2 / 4 columns, this way
// against the large matrices' way: ILU(0) 27.0 / 36.3 / 52.5 and 27.7 / 46.6 /
// 67.5 us, ILUT 34.5 / 57.4 / 89.6 and 52.7 / 78 / 111 us; at 25 slices per SM
// (50^3), where several rounds per warp are needed either way, ILUT four
// columns 122 us the large way.
constexpr int kSliceSmall = 16;
inline bool slice_small(int ns, int sms) { return ns <= kSliceSmall * sms; }

// Large matrices: every (B W)-th group of W slices to a block, all blocks
// resident, so that neighbouring slices are swept at the same time.  In the
// second and third round of the warps this leaves SMs of unequal loads where
// a round is partly full (5+5 applications, 7-point ILU(0), rounds / us with
// the slices dealt evenly: one column at 64^3 1.12 / 41.4 (45.6), 67^3 1.29 /
// 47.3 (48.1), 70^3 1.47 / 56.2 (48.8), 73^3 1.67 / 57.5 (51.9), 86^3 2.73 /
// 76.9 (73.4), 90^3 3.12 / 82 (90); two columns at 64^3 1.35 / 80.4 (70.8),
// 73^3 2.00 / 91.6 (92.5)), so the slices are dealt evenly from 0.3 of a round.
// Not with int32 columns, whose far gathers want all blocks in one window of
// the vector (27-point 260 x 260 x 4 FP32 2.32 / 68 us (80)).
constexpr double kSliceUneven = 0.3, kSliceFull = 0.97;

struct SlicePlan {
  int warps, blocks, flags;
};
inline SlicePlan slice_plan(int ns, int sms, int most, bool wide) {
  constexpr int W = kSliceThreads / 32;
  if (!slice_small(ns, sms)) {
    const int want = (ns + W - 1) / W, grid = want < sms * most ? want : sms * most;
    const double rounds = (double)ns / (sms * most * W), last = rounds - (int)rounds;
    const bool even = !wide && rounds > 1 && rounds < 3 && last >= kSliceUneven && last < kSliceFull;
    return {W, grid, even ? kFlagSpread : 0};
  }
  const int full = ns > W * sms && most > 1 ? 2 * sms : sms;
  const int blocks = ns < full ? ns : full, share = (ns + blocks - 1) / blocks;
  return {share < W ? share : W, blocks, kFlagSpread};
}

template <class MT, class VI, class VO, class CT, int R, int CP, int MINB, bool VEC, int LN = 1>
struct SliceKernel {
  static cudaError_t prepare() {
    // no shared memory: all of it as L1
    return cudaFuncSetAttribute(k_slices<MT, VI, VO, CT, R, CP, MINB, VEC, LN>,
                                cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxL1);
  }
  static cudaError_t launch(const DevCsr& T, const LaunchEnv& env, int ldx, const void* c, const void* in, void* out,
                            const double* dinv, double* x, int epi, cudaStream_t s) {
    const Slices& S = *T.sl;
    if (S.ns == 0) return cudaSuccess;
    const SlicePlan plan = slice_plan(S.ns, env.sms, MINB, sizeof(CT) == 4);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan.blocks);
    cfg.blockDim = dim3((unsigned)(plan.warps * 32));
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = env.overlap ? 1 : 0;
    // consecutive launches alternate their direction, so each starts on the
    // rows that the previous one touched last, while they are still in L2
    int flags = plan.flags | (env.l2 & (kFlagFactorNormal | kFlagVectorNormal));
    if ((env.l2 & kFlagReverse) && (env.flips++ & 1u)) flags |= kFlagReverse;
    return cudaLaunchKernelEx(&cfg, k_slices<MT, VI, VO, CT, R, CP, MINB, VEC, LN>, S.ns, T.n, (const int2*)S.hdr,
                              (const CT*)S.ci, (const MT*)S.va, (const VI*)c, (const VI*)in, (VO*)out, ldx, dinv, x,
                              epi, flags);
  }
};

}  // namespace
}  // namespace silu
