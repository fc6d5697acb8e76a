// The sliced sweep with its matrix stream staged through shared memory
// (sm_103a), one right-hand side, slices of at most 16 entries per row.
//
// What bounds it: HBM.  FP32 entries (6 bytes each) ask for four times the
// rows in flight that FP64 entries do before the FP64 pipe or the issue slots
// matter, and k_slices, whose next chunk waits in registers, then runs at the
// latency of DRAM: 77 us per lower sweep of the 160^3 27-point FP32 factor
// (316 MB), as long as the tiled CSR sweep takes for its 420 MB.  Here every
// warp streams its own sequence of units through a private ring of stages
// filled by bulk asynchronous copies (one of values, one of columns), so the
// bytes in flight do not depend on its registers; it gathers for a whole unit
// before the first multiply-add.
//
// A unit is G consecutive slices with at most KW entries per row each
// (G KW = 16): four slices of short rows (7-point ILU(0) factors), two, or
// one.  Sums, order and results are k_slices': one lane per row, column order.
#include "bulk.cuh"
#include "slices.cuh"

namespace silu {
namespace {

template <class MT>
struct RingStage {
  static constexpr int kRows = 16;  // 32-lane rows of entries a stage holds
  static constexpr size_t kVal = kRows * 32 * sizeof(MT);
  static constexpr size_t kBytes = kVal + kRows * 32 * sizeof(uint16_t);
};

template <class MT, class VI, class VO, int G, int W, int D>
__global__ void __launch_bounds__(W * 32, 1)
    k_slices_ring(int ns, int n, const int2* __restrict__ hdr, const uint16_t* __restrict__ ci,
                  const MT* __restrict__ va, const VI* c, const VI* in,
                  VO* __restrict__ out, const double* __restrict__ dinv, double* __restrict__ x, int epi, int flags,
                  int* __restrict__ err) {
  using S = RingStage<MT>;
  constexpr int KW = S::kRows / G;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[W][D];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int w = 0; w < W; ++w)
      for (int s = 0; s < D; ++s) mbar_init(&full[w][s], 1);
    fence_mbar_init();
  }
  __syncthreads();
  const int nu = (ns + G - 1) / G;
  const int gw = blockIdx.x * W + warp;
  const int nw = gridDim.x * W;
  unsigned char* ring = smem + (size_t)warp * D * S::kBytes;
  const bool rev = (flags & kFlagReverse) != 0;
  const uint64_t stream = (flags & kFlagFactorNormal) ? policy_evict_normal() : policy_evict_first();
  const uint64_t keep = (flags & kFlagVectorNormal) ? policy_evict_normal() : policy_evict_last();
  grid_launch_dependents();
  // lane l <= G holds the header of slice u G + l of unit t (past the last slice: the end)
  auto header = [&](int t) {
    const int u = rev ? nu - 1 - t : t;
    int2 h = make_int2(0, 0);
    if (lane <= G) h = __ldg(hdr + min(u * G + lane, ns));
    return h;
  };
  // lane 0 issues the copies of a unit (header h) into stage s
  auto issue = [&](int2 h, int s) {
    const int p1 = __shfl_sync(0xffffffffu, h.x, G);
    if (lane == 0) {
      const uint32_t slots = (uint32_t)(p1 - h.x);
      unsigned char* st = ring + s * S::kBytes;
      fence_proxy_async();
      mbar_expect_tx(&full[warp][s], slots * (uint32_t)(sizeof(MT) + sizeof(uint16_t)));
      if (slots) {
        bulk_g2s(st, va + h.x, slots * (uint32_t)sizeof(MT), &full[warp][s], stream);
        bulk_g2s(st + S::kVal, ci + h.x, slots * (uint32_t)sizeof(uint16_t), &full[warp][s], stream);
      }
    }
  };
  // headers of the unit in hand and of the D - 1 units after it, whose copies are in flight
  int2 hq[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const int t = gw + d * nw;
    hq[d] = t < nu ? header(t) : make_int2(0, 0);
    if (t < nu) issue(hq[d], d);
  }
  grid_wait_prior();  // c, in, out and x below belong to the previous kernel until it completes
  int k = 0;
  for (int t = gw; t < nu; t += nw, ++k) {
    const int u = rev ? nu - 1 - t : t;
    const int tn = t + D * nw;
    const int2 hn = tn < nu ? header(tn) : make_int2(0, 0);
    MT acc[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int row = (u * G + g) * 32 + lane;
      acc[g] = (row < n && c) ? (MT)ld_keep(c + row, keep) : MT(0);
      if (row < n && ((kEpiDinv >> epi) & 1u)) prefetch_l1(dinv + row);
      if (row < n && ((kEpiX >> epi) & 1u)) prefetch_l1(x + row);
    }
    const int s = k % D;
    const bool ok = mbar_wait_bounded(&full[warp][s], (uint32_t)(k / D) & 1u);
    if (!__all_sync(0xffffffffu, ok)) {
      // a copy did not land in time: report, let the other stages' copies land, leave
      if (lane == 0) {
        atomicOr(err, 1);
        for (int d = 1; d < D; ++d) {
          const int kd = k + d;
          if (t + d * nw < nu) mbar_wait_bounded(&full[warp][kd % D], (uint32_t)(kd / D) & 1u);
        }
      }
      return;
    }
    const int2 h = hq[0];
    const MT* sv = (const MT*)(ring + s * S::kBytes);
    const uint16_t* sc = (const uint16_t*)(ring + s * S::kBytes + S::kVal);
    const int p0 = __shfl_sync(0xffffffffu, h.x, 0);
    MT v[G][KW], xv[G][KW];
    int width[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int a = __shfl_sync(0xffffffffu, h.x, g), b = __shfl_sync(0xffffffffu, h.x, g + 1);
      const VI* ib = in + __shfl_sync(0xffffffffu, h.y, g);
      width[g] = (b - a) >> 5;
      const int o = a - p0;
#pragma unroll
      for (int q = 0; q < KW; q += 2) {
        unsigned cc = 0xffffffffu;
        v[g][q] = v[g][q + 1] = MT(0);
        if (q + 2 <= width[g]) {
          cc = *(const unsigned*)(sc + o + 32 * q + 2 * lane);
          v[g][q] = sv[o + 32 * q + 2 * lane];
          v[g][q + 1] = sv[o + 32 * q + 2 * lane + 1];
        } else if (q < width[g]) {
          cc = 0xffff0000u | sc[o + 32 * q + lane];
          v[g][q] = sv[o + 32 * q + lane];
        }
        const unsigned c0 = cc & 0xffffu, c1 = cc >> 16;
        xv[g][q] = c0 != 0xffffu ? (MT)ld_keep(ib + c0, keep) : MT(0);
        xv[g][q + 1] = c1 != 0xffffu ? (MT)ld_keep(ib + c1, keep) : MT(0);
      }
    }
    __syncwarp();  // the stage is read: its next unit may land
    if (tn < nu) issue(hn, s);
#pragma unroll
    for (int g = 0; g < G; ++g) {
#pragma unroll
      for (int q = 0; q < KW; ++q) {
        if (q >= width[g]) break;  // warp-uniform
        acc[g] = fma(-v[g][q], xv[g][q], acc[g]);
      }
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int row = (u * G + g) * 32 + lane;
      if (row < n) {
        if (epi == EPI_SPMV)
          st_keep(out + row, (VO)(MT(0) - acc[g]), keep);
        else
          epilogue<MT, VI, VO>(epi, row, acc[g], in, out, dinv, x, keep);
      }
    }
#pragma unroll
    for (int d = 0; d + 1 < D; ++d) hq[d] = hq[d + 1];
    hq[D - 1] = hn;
  }
}

template <class MT, class VI, class VO, int G, int W, int D>
struct RingKernel {
  static constexpr size_t kSmem = (size_t)W * D * RingStage<MT>::kBytes;
  static cudaError_t prepare() {
    return cudaFuncSetAttribute(k_slices_ring<MT, VI, VO, G, W, D>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kSmem);
  }
  static cudaError_t launch(const DevCsr& T, const LaunchEnv& env, const void* c, const void* in, void* out,
                            const double* dinv, double* x, int epi, cudaStream_t s) {
    const Slices& S = *T.sl;
    if (S.ns == 0) return cudaSuccess;
    const int nu = (S.ns + G - 1) / G;
    const int want = (nu + W - 1) / W;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(want < env.sms ? want : env.sms));
    cfg.blockDim = dim3(W * 32);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = env.overlap ? 1 : 0;
    int flags = env.l2 & (kFlagFactorNormal | kFlagVectorNormal);
    if ((env.l2 & kFlagReverse) && (env.flips++ & 1u)) flags |= kFlagReverse;
    return cudaLaunchKernelEx(&cfg, k_slices_ring<MT, VI, VO, G, W, D>, S.ns, T.n, (const int2*)S.hdr,
                              (const uint16_t*)S.ci, (const MT*)S.va, (const VI*)c, (const VI*)in, (VO*)out, dinv, x,
                              epi, flags, env.err);
  }
};

// 32 warps of two stages (196 KB) with 56 to 64 registers a thread.  Lower
// sweep of the 160^3 27-point FP32 factor and application of the 48-system
// FP32 batch, by warps x stages: 20 x 2 65.5 us / 174 us, 24 x 2 59.4 / 162,
// 24 x 3 60.0 / 164, 16 x 4 76.4 / 186, 32 x 2 56.6 / 153 (k_slices: 76.5 / 177).
template <int G>
using FloatRing = RingKernel<float, float, float, G, 32, 2>;

}  // namespace

cudaError_t slices_prepare_ring() {
  cudaError_t e = FloatRing<1>::prepare();
  if (e == cudaSuccess) e = FloatRing<2>::prepare();
  if (e == cudaSuccess) e = FloatRing<4>::prepare();
  return e;
}

// FP32 sweeps with at least 64 slices per SM, rows of at most 16 entries and
// 16-bit columns.  Below, a launch is mostly latency and k_slices, which has no
// barriers to set up, is shorter (2.4 us a sweep against 4.1 on 32^3 cut-cell
// rows); they meet at 8192 slices with one slice per unit (27-point 64^3: 8.7 /
// 8.5 us) and between 8192 and 16000 with four (cut-cell 64^3: 3.5 / 4.2 us,
// 80^3: 5.0 / 4.5 us).  FP64 sweeps gain nothing here (the FP64 pipe bounds
// them: 128^3 ILUT 43.9 us either way, ILU(0) 19.7 us against 25.3).
bool slices_ring_fits(const DevCsr& T, Mode mode, int sms) {
  return mode == MODE_F && !T.sl->wide && T.sl->widest <= RingStage<float>::kRows && T.sl->ns >= 64 * sms;
}

cudaError_t launch_slices_ring(const DevCsr& T, const LaunchEnv& env, const void* c, const void* in, void* out,
                               const double* dinv, double* x, int epi, cudaStream_t s) {
  if (T.sl->widest <= 4) return FloatRing<4>::launch(T, env, c, in, out, dinv, x, epi, s);
  if (T.sl->widest <= 8) return FloatRing<2>::launch(T, env, c, in, out, dinv, x, epi, s);
  return FloatRing<1>::launch(T, env, c, in, out, dinv, x, epi, s);
}

}  // namespace silu
