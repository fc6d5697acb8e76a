// Building the sliced copy of a matrix on the device, and the sliced sweep
// for one right-hand side (see slices.cuh).
#include "slices.cuh"

#include <algorithm>
#include <new>
#include <vector>

namespace silu {

void Slices::release() {
  if (buf) device_free(buf, bytes);
  buf = nullptr;
}

namespace {

// A sliced copy is made where padding adds at most two fifths to the entries
// (and for any matrix of a few slices).  Padding costs FP64 sweeps issue time
// and every sweep bytes: the 128^3 cut-cell ILUT lower factor (1.26 slots per
// entry) takes 44.0 us sliced against 45.9 us tiled; of the AMG operators of
// the 128^3 cut-cell matrix, those within 1.4 gain (V-cycle 743 -> 732 us
// against a limit of 1.2) and taking those up to 1.7 as well, rows of 30 and
// more entries of uneven length, loses (843 us).
constexpr double kSlicePadMax = 1.4;
constexpr double kSlicePadFree = 2048.0;
constexpr int64_t kMaxSlots = (int64_t)INT32_MAX - 65536;  // slot numbers (and a chunk beyond the last) fit an int

// Smallest column of every slice into its header, largest span of any slice
// into *span (at least 0).  One warp per slice.
__global__ void k_slice_span(int ns, int n, const int* __restrict__ rp, const int* __restrict__ ci,
                             int2* __restrict__ hdr, int* __restrict__ span) {
  const int s = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (s >= ns) return;
  const int r0 = s * 32, r1 = min(n, r0 + 32);
  int lo = INT32_MAX, hi = -1;
  for (int p = rp[r0] + lane; p < rp[r1]; p += 32) {
    lo = min(lo, ci[p]);
    hi = max(hi, ci[p]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    hdr[s].y = hi < 0 ? 0 : lo;
    if (hi >= 0) atomicMax(span, hi - lo);
  }
}

// Fill the slices from the CSR arrays: one warp per slice, one lane per row.
template <class MT, class CT>
__global__ void k_slice_fill(int ns, int n, const int* __restrict__ rp, const int* __restrict__ ci,
                             const MT* __restrict__ va, const int2* __restrict__ hdr, CT* __restrict__ sci,
                             MT* __restrict__ sva) {
  const int s = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (s >= ns) return;
  const int2 h = hdr[s];
  const int width = (hdr[s + 1].x - h.x) >> 5;
  const int r = s * 32 + lane;
  const int b = r < n ? rp[r] : 0;
  const int len = r < n ? rp[r + 1] - b : 0;
  for (int k = 0; k < width; ++k) {
    const int at = (k | 1) < width ? h.x + 64 * (k >> 1) + 2 * lane + (k & 1) : h.x + 32 * k + lane;
    CT c = (CT)~(CT)0;
    MT v = MT(0);
    if (k < len) {
      c = (CT)(sizeof(CT) == 2 ? ci[b + k] - h.y : ci[b + k]);
      v = va[b + k];
    }
    sci[at] = c;
    sva[at] = v;
  }
}

template <class MT>
cudaError_t fill(const DevCsr& d, const Slices& S, cudaStream_t s) {
  const unsigned blocks = (unsigned)((S.ns + 7) / 8);
  if (S.wide)
    k_slice_fill<MT, int><<<blocks, 256, 0, s>>>(S.ns, d.n, d.rp, d.ci, (const MT*)d.va, S.hdr, (int*)S.ci,
                                                 (MT*)S.va);
  else
    k_slice_fill<MT, uint16_t><<<blocks, 256, 0, s>>>(S.ns, d.n, d.rp, d.ci, (const MT*)d.va, S.hdr, (uint16_t*)S.ci,
                                                      (MT*)S.va);
  return cudaGetLastError();
}

// FP64 for one right-hand side: one pair per chunk and 48 warps per SM (128^3
// ILUT application 820 us; two pairs and 32 or 40 warps 896 / 893, three and
// 32 830; 160^3 27-point residual 232 us against 236 / 227 / 240), which no
// register spills; four partial sums need a chunk of four entries.
template <class VO, class CT, int LN>
using Double1 = SliceKernel<double, double, VO, CT, 1, LN == 4 ? 2 : 1, LN == 4 ? 4 : 6, false, LN>;

// The same for small matrices of 16-bit columns: a whole row per chunk where
// the registers of one block per SM (two beyond eight slices per SM) allow.
template <class VO, int LN, int CP, int MINB>
using DoubleSmall = SliceKernel<double, double, VO, uint16_t, 1, CP, MINB, false, LN>;

template <class VO>
cudaError_t double1_small(const DevCsr& T, const LaunchEnv& env, const void* c, const void* in, void* out,
                          const double* dinv, double* x, int epi, cudaStream_t s) {
  const int w = T.sl->widest;
  const bool one = T.sl->ns <= kSliceThreads / 32 * env.sms;  // one block per SM
  auto go = [&](auto k) { return decltype(k)::launch(T, env, 1, c, in, out, dinv, x, epi, s); };
  switch (T.sl->lanes) {
    case 1:
      if (w <= 4) return go(DoubleSmall<VO, 1, 2, 2>());
      return w <= 10 || !one ? go(DoubleSmall<VO, 1, 5, 2>()) : go(DoubleSmall<VO, 1, 7, 1>());
    case 2: return one ? go(DoubleSmall<VO, 2, 7, 1>()) : go(DoubleSmall<VO, 2, 5, 2>());
    case 4: return one ? go(DoubleSmall<VO, 4, 8, 1>()) : go(DoubleSmall<VO, 4, 4, 2>());
  }
  return cudaErrorInvalidValue;
}

template <class F, class VO>
cudaError_t each_small(F f) {
  cudaError_t e = f(DoubleSmall<VO, 1, 2, 2>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 1, 5, 2>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 1, 7, 1>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 2, 7, 1>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 2, 5, 2>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 4, 8, 1>());
  if (e == cudaSuccess) e = f(DoubleSmall<VO, 4, 4, 2>());
  return e;
}

template <class VO, class CT>
cudaError_t double1(const DevCsr& T, const LaunchEnv& env, const void* c, const void* in, void* out,
                    const double* dinv, double* x, int epi, cudaStream_t s) {
  switch (T.sl->lanes) {
    case 1: return Double1<VO, CT, 1>::launch(T, env, 1, c, in, out, dinv, x, epi, s);
    case 2: return Double1<VO, CT, 2>::launch(T, env, 1, c, in, out, dinv, x, epi, s);
    case 4: return Double1<VO, CT, 4>::launch(T, env, 1, c, in, out, dinv, x, epi, s);
  }
  return cudaErrorInvalidValue;
}

// Every instance that launch_sweep_slices picks for one right-hand side.
template <class F>
cudaError_t for_each_shape(F f) {
  cudaError_t e = cudaSuccess;
  auto add = [&](cudaError_t r) {
    if (e == cudaSuccess) e = r;
  };
  add(f(Double1<double, uint16_t, 1>()));
  add(f(Double1<double, uint16_t, 2>()));
  add(f(Double1<double, uint16_t, 4>()));
  add(f(Double1<double, int, 1>()));
  add(f(Double1<double, int, 2>()));
  add(f(Double1<double, int, 4>()));
  add(f(Double1<float, uint16_t, 1>()));
  add(f(Double1<float, uint16_t, 2>()));
  add(f(Double1<float, uint16_t, 4>()));
  add(f(Double1<float, int, 1>()));
  add(f(Double1<float, int, 2>()));
  add(f(Double1<float, int, 4>()));
  add(each_small<F, double>(f));
  add(each_small<F, float>(f));
  add(f(SliceKernel<float, float, float, uint16_t, 1, 2, 5, false>()));
  add(f(SliceKernel<float, float, float, uint16_t, 1, 4, 3, false>()));
  add(f(SliceKernel<float, float, float, uint16_t, 1, 7, 3, false>()));
  add(f(SliceKernel<float, float, float, int, 1, 2, 5, false>()));
  add(f(SliceKernel<float, float, float, int, 1, 4, 3, false>()));
  return e;
}

}  // namespace

bool slices_pay(const int64_t* rp, int64_t n, bool fp32, std::vector<int2>& hdr) {
  hdr.clear();
  // FP32 rows of more than 16 entries on average keep the tiled sweep, whose
  // lanes share a row (an FP32 sum in another order differs by 1e-7)
  if (n <= 0 || (fp32 && staged_lanes(rp, n) > 1)) return false;
  const double most = std::min((double)kMaxSlots, kSlicePadMax * (double)rp[n] + kSlicePadFree);
  const int64_t ns = (n + 31) / 32;
  hdr.resize((size_t)ns + 1);
  int64_t slots = 0;
  for (int64_t s = 0; s < ns; ++s) {
    hdr[(size_t)s] = make_int2((int)slots, 0);
    int64_t w = 0;
    for (int64_t r = s * 32; r < std::min<int64_t>(n, s * 32 + 32); ++r) w = std::max<int64_t>(w, rp[r + 1] - rp[r]);
    slots += 32 * w;
    if ((double)slots > most) return false;
  }
  hdr[(size_t)ns] = make_int2((int)slots, 0);
  return true;
}

cudaError_t build_slices(const std::vector<int2>& hdr, int lanes, DevCsr& d, cudaStream_t s) {
  std::shared_ptr<Slices> S;
  S.swap(d.sl);
  if (!S || S.use_count() > 1 || S->sole) S.reset(new (std::nothrow) Slices);
  if (!S) return cudaSuccess;
  S->slots = hdr.back().x;
  S->ns = (int)hdr.size() - 1;
  S->lanes = lanes;
  S->wide = false;
  S->widest = 0;
  for (size_t k = 0; k + 1 < hdr.size(); ++k) S->widest = std::max(S->widest, (hdr[k + 1].x - hdr[k].x) / 32);
  // one allocation: the headers and, past them, one int for the span; values; columns
  const size_t hb = (sizeof(int2) * (hdr.size() + 1) + 255) / 256 * 256;
  const size_t slots = (size_t)std::max<int64_t>(S->slots, 32);
  const size_t vb = ((d.fp32 ? sizeof(float) : sizeof(double)) * slots + 255) / 256 * 256;
  auto allocate = [&](size_t col_bytes) {
    const size_t bytes = hb + vb + col_bytes * slots;
    cudaError_t e = cudaSuccess;
    if (!S->buf || S->bytes != bytes) {  // else the buffer of the values before these
      S->release();
      e = device_alloc(&S->buf, bytes);
    }
    S->bytes = bytes;
    S->hdr = (int2*)S->buf;
    S->va = (char*)S->buf + hb;
    S->ci = (char*)S->buf + hb + vb;
    return e;
  };
  auto give_up = [](cudaError_t e) {
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();  // no room for the copy: the sweeps run on the CSR tiles
    return cudaSuccess;
  };
  cudaError_t e = allocate(sizeof(uint16_t));
  if (e != cudaSuccess) return give_up(e);
  const unsigned blocks = (unsigned)((S->ns + 7) / 8);
  for (;;) {
    int* span = (int*)(S->hdr + hdr.size());
    e = cudaMemcpyAsync(S->hdr, hdr.data(), sizeof(int2) * hdr.size(), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(span, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_slice_span<<<blocks, 256, 0, s>>>(S->ns, d.n, d.rp, d.ci, S->hdr, span);
    e = cudaGetLastError();
    int widest = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&widest, span, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (widest < 65535 || S->wide) break;  // offset 65535 marks padding
    S->wide = true;
    e = allocate(sizeof(int));
    if (e != cudaSuccess) return give_up(e);
  }
  e = d.fp32 ? fill<float>(d, *S, s) : fill<double>(d, *S, s);
  // A sweep reads the slices ahead of the wait for the kernel before it.  With
  // an operation that is no kernel behind the fill, one that follows at once
  // starts only when the fill is complete, without the host waiting for it.
  if (e == cudaSuccess) e = cudaMemsetAsync(S->hdr + hdr.size(), 0, sizeof(int), s);
  if (e == cudaSuccess) d.sl = std::move(S);
  return e;
}

cudaError_t refill_slices(const DevCsr& d, cudaStream_t s) {
  if (!d.sliced()) return cudaSuccess;
  return d.fp32 ? fill<float>(d, *d.sl, s) : fill<double>(d, *d.sl, s);
}

cudaError_t slices_prepare() {
  cudaError_t e = for_each_shape([](auto k) { return decltype(k)::prepare(); });
  if (e == cudaSuccess) e = slices_prepare_ring();
  return e == cudaSuccess ? slices_prepare_multi() : e;
}

cudaError_t launch_sweep_slices(const DevCsr& T, Mode mode, const LaunchEnv& env, int R, int ldx, const void* c,
                                const void* in, void* out, const double* dinv, double* x, int epi, cudaStream_t s) {
  if (!T.sliced() || R < 1 || R > 4 || ldx < R || (R == 1 && ldx != 1)) return cudaErrorInvalidValue;
  if (R > 1) return launch_slices_multi(T, mode, env, R, ldx, c, in, out, dinv, x, epi, s);
  if (slices_ring_fits(T, mode, env.sms)) return launch_slices_ring(T, env, c, in, out, dinv, x, epi, s);
  const bool wide = T.sl->wide;
  // Two blocks per SM (beyond eight slices) with the registers of a whole row
  // leave no room for the launches of other streams.  For rows of up to four
  // entries the large matrices' kernel (40 registers) is as fast alone: 7-point
  // ILU(0) 8+8 applications at 36^3 / 40^3 / 42^3 alone 32.5 / 36.9 / 35.8 us
  // that way, 33.3 / 35.8 / 38.2 us this way, and with eight streams 14.7 /
  // 18.4 / 22.5 and 14.3 / 14.5 / 15.2 us each.  (Rows of seven, the matrix
  // itself, gain nothing more with streams and cost an FGMRES iteration alone
  // 2 us; ILUT rows of ten at 40^3 take 38 us each with eight streams either
  // way.)
  const bool small = !wide && slice_small(T.sl->ns, env.sms) &&
                     !(mode != MODE_F && T.sl->widest <= 4 && T.sl->ns > kSliceThreads / 32 * env.sms);
  // FP32, where the ring does not fit (fewer slices, longer rows, int32
  // columns): a whole row per chunk where rows allow (27-point 32^3 4.5 us a
  // sweep).  Rows of up to four entries at 40 warps per SM and 48 registers:
  // 48 warps spill (cut-cell 50^3 / 54^3 / 58^3 / 64^3 5+5 applications 25.0 /
  // 26.1 / 26.5 / 34.2 us that way, 23.8 / 24.3 / 26.6 / 34.6 this way).
  const double mean = (double)T.sl->slots / (32.0 * (double)T.sl->ns);
  auto go = [&](auto k) { return decltype(k)::launch(T, env, ldx, c, in, out, dinv, x, epi, s); };
  switch (mode) {
    case MODE_D:
      if (small) return double1_small<double>(T, env, c, in, out, dinv, x, epi, s);
      return wide ? double1<double, int>(T, env, c, in, out, dinv, x, epi, s)
                  : double1<double, uint16_t>(T, env, c, in, out, dinv, x, epi, s);
    case MODE_DF:
      if (small) return double1_small<float>(T, env, c, in, out, dinv, x, epi, s);
      return wide ? double1<float, int>(T, env, c, in, out, dinv, x, epi, s)
                  : double1<float, uint16_t>(T, env, c, in, out, dinv, x, epi, s);
    case MODE_F:
      if (mean <= 4.0 && !(small && T.sl->widest > 4))
        return wide ? go(SliceKernel<float, float, float, int, 1, 2, 5, false>())
                    : go(SliceKernel<float, float, float, uint16_t, 1, 2, 5, false>());
      if (wide || mean <= 8.0 || mean > 14.0)
        return wide ? go(SliceKernel<float, float, float, int, 1, 4, 3, false>())
                    : go(SliceKernel<float, float, float, uint16_t, 1, 4, 3, false>());
      return go(SliceKernel<float, float, float, uint16_t, 1, 7, 3, false>());
  }
  return cudaErrorInvalidValue;
}

}  // namespace silu
