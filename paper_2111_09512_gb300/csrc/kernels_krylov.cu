// FP64 Krylov kernels of the flexible GMRES solve (Sec. 6: FGMRES with
// modified Gram-Schmidt, Givens rotations, Eq. relres stopping test).
//
// Reductions are two-stage and deterministic: a fixed grid writes one
// partial sum per block, and every consumer reduces the partials in the same
// fixed order.  The same inputs therefore give bitwise the same results
// whatever else runs on the device.
#include <cmath>

#include "device.cuh"
#include "exchange.cuh"
#include "krylov.cuh"

namespace silu {
namespace {

constexpr int KB = 256;
constexpr int kMaxParts = 1024;
constexpr int kGivensStaged = 1024;  // columns whose Givens update fits in shared memory without opting in

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Block-wide sum in a fixed order; the result is returned to every thread.
__device__ double block_sum(double v) {
  __shared__ double red[KB / 32];
  __shared__ double total;
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < KB / 32; ++i) s += red[i];
    total = s;
  }
  __syncthreads();
  const double out = total;
  __syncthreads();
  return out;
}

__device__ double sum_parts(const double* __restrict__ part, int nparts) {
  double v = 0.0;
  for (int i = threadIdx.x; i < nparts; i += KB) v += part[i];
  return block_sum(v);
}

// The streaming loops below visit a thread's elements i0, i0 + S, i0 + 2S, ...
// (S = the grid's thread count) in that order, as a plain grid-stride loop
// would, but load two of them before using either: twice the bytes in
// flight per thread, the same accumulation order, the same bits.  Indices are
// unsigned 32-bit (n < 2^31, so i + 2S cannot wrap), which keeps each kernel
// within 32 registers: all 1024 blocks of the largest grid are resident at
// once (eight per SM) and none waits for a second wave.
__global__ void __launch_bounds__(KB, 8) k_dot_part(int n, const double* __restrict__ a, const double* __restrict__ b,
                                                    double* __restrict__ part) {
  const unsigned N = (unsigned)n, S = gridDim.x * KB;
  unsigned i = blockIdx.x * KB + threadIdx.x;
  double acc = 0.0;
  for (; i + S < N; i += 2 * S) {
    const double a0 = a[i], a1 = a[i + S];
    const double b0 = b[i], b1 = b[i + S];
    acc += a0 * b0;
    acc += a1 * b1;
  }
  for (; i < N; i += S) acc += a[i] * b[i];
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// U rows are loaded at a time.  U = 4, the first ones before h is summed, for
// grids of at most four blocks per SM, where a step is the latency of its
// loads (FGMRES, 60 iterations: Poisson 48^3 / 64^3 7264 / 8582 -> 7001 / 8285
// us); U = 2 (32 registers, eight blocks per SM) beyond, where it is bandwidth.
template <int U>
__global__ void __launch_bounds__(KB, U > 2 ? 4 : 8) k_mgs_step(int n, const double* __restrict__ part_in, int nparts,
                                                    double* __restrict__ hout, double* __restrict__ w,
                                                    const double* __restrict__ vi, const double* __restrict__ vnext,
                                                    double* __restrict__ part_out) {
  const unsigned N = (unsigned)n, S = gridDim.x * KB;
  unsigned i = blockIdx.x * KB + threadIdx.x;
  double w0[U], v0[U], u0[U];
  auto load = [&]() {
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const bool in = i + (unsigned)k * S < N;
      w0[k] = in ? w[i + (unsigned)k * S] : 0.0;
      v0[k] = in ? vi[i + (unsigned)k * S] : 0.0;
      u0[k] = in && vnext ? vnext[i + (unsigned)k * S] : 0.0;  // none: the partial sums of ||w||^2
    }
  };
  if constexpr (U > 2) load();
  const double h = sum_parts(part_in, nparts);
  if (blockIdx.x == 0 && threadIdx.x == 0 && hout) *hout = h;
  if constexpr (U <= 2) load();
  double acc = 0.0;
  while (i < N) {
#pragma unroll
    for (int k = 0; k < U; ++k)
      if (i + (unsigned)k * S < N) {
        const double wn = w0[k] - h * v0[k];
        w[i + (unsigned)k * S] = wn;
        acc += wn * (vnext ? u0[k] : wn);
      }
    i += U * S;
    if (i < N) load();
  }
  const double s = block_sum(acc);
  if (threadIdx.x == 0) part_out[blockIdx.x] = s;
}

__global__ void __launch_bounds__(KB, 8) k_normalize(int n, const double* __restrict__ part_in, int nparts,
                                                     double* __restrict__ hout, const double* w, double* vout) {
  const double h = sqrt(sum_parts(part_in, nparts));
  if (blockIdx.x == 0 && threadIdx.x == 0 && hout) *hout = h;
  if (h == 0.0) return;
  const Divider by(h);
  const unsigned N = (unsigned)n, S = gridDim.x * KB;
  unsigned i = blockIdx.x * KB + threadIdx.x;
  for (; i + S < N; i += 2 * S) {  // w may be vout: each element is read, then written, by one thread
    const double w0 = w[i], w1 = w[i + S];
    vout[i] = by(w0);
    vout[i + S] = by(w1);
  }
  for (; i < N; i += S) vout[i] = by(w[i]);
}

// The end of Arnoldi step j: h_{j+1,j} and v_{j+1} as k_normalize, and, by one
// thread of block 0, the Givens update of column j (the rows h_0 .. h_j of H):
// the earlier rotations, the new one, the right-hand side g.  Column and
// rotations are read by the whole block first: the update is a chain of
// dependent operations, and reading each operand from memory where it is used
// took 10 us at j = 16.
__global__ void __launch_bounds__(KB, 8) k_normalize_givens(int n, const double* __restrict__ part_in, int nparts,
                                                            const double* w, double* vout, int j, int m, double* H,
                                                            double* cs, double* sn, double* g, double* res) {
  extern __shared__ double sh[];  // block 0: column j (j + 1 entries), cs and sn (j each); none where that is too much
  const bool lead = blockIdx.x == 0;
  const bool staged = j < kGivensStaged;
  double* col = staged ? sh : H + j;  // entry i at col[i * ld]
  const size_t ld = staged ? 1 : (size_t)m;
  const double* c0 = staged ? sh + j + 1 : cs;
  const double* s0 = staged ? sh + 2 * j + 1 : sn;
  if (lead && staged) {
    for (int i = threadIdx.x; i <= j; i += KB) sh[i] = H[(size_t)i * m + j];
    for (int i = threadIdx.x; i < j; i += KB) {
      sh[j + 1 + i] = cs[i];
      sh[2 * j + 1 + i] = sn[i];
    }
  }
  const double h = sqrt(sum_parts(part_in, nparts));
  if (h != 0.0) {
    const Divider by(h);
    const unsigned N = (unsigned)n, S = gridDim.x * KB;
    unsigned i = blockIdx.x * KB + threadIdx.x;
    for (; i + S < N; i += 2 * S) {
      const double w0 = w[i], w1 = w[i + S];
      vout[i] = by(w0);
      vout[i + S] = by(w1);
    }
    for (; i < N; i += S) vout[i] = by(w[i]);
  }
  if (!lead || threadIdx.x != 0) return;
  for (int i = 0; i < j; ++i) {
    const double a = col[i * ld], b = col[(i + 1) * ld];
    const double c = c0[i], s = s0[i];
    H[(size_t)i * m + j] = c * a + s * b;
    col[(i + 1) * ld] = -s * a + c * b;
  }
  const double a = col[j * ld], b = h;
  const double den = hypot(a, b);
  const double c = den != 0.0 ? a / den : 1.0;
  const double s = den != 0.0 ? b / den : 0.0;
  cs[j] = c;
  sn[j] = s;
  H[(size_t)j * m + j] = den;
  H[(size_t)(j + 1) * m + j] = 0.0;
  const double gj = g[j];
  g[j + 1] = -s * gj;
  g[j] = c * gj;
  res[0] = fabs(-s * gj);
  res[1] = b;  // h_{j+1,j}: zero means the Krylov space is exhausted
}

// Minimal-residual step: alpha = sum(part_num) / sum(part_den) (0 when the
// denominator is 0), y = alpha s.
__global__ void __launch_bounds__(KB) k_mr_step(int n, const double* __restrict__ part_num,
                                                const double* __restrict__ part_den, int nparts,
                                                const double* __restrict__ s, double* __restrict__ y) {
  const double num = sum_parts(part_num, nparts);
  const double den = sum_parts(part_den, nparts);
  const double alpha = den != 0.0 ? num / den : 0.0;
  for (long long i = (long long)blockIdx.x * KB + threadIdx.x; i < n; i += (long long)gridDim.x * KB)
    y[i] = alpha * s[i];
}

__global__ void k_norm_final(const double* __restrict__ part_in, int nparts, double* __restrict__ out) {
  const double h = sqrt(sum_parts(part_in, nparts));
  if (threadIdx.x == 0) *out = h;
}

// q = w / h entry by entry, by the division the normalisations use.
__global__ void k_divide(int64_t n, const double* __restrict__ w, const double* __restrict__ h,
                         double* __restrict__ q) {
  const int64_t i = blockIdx.x * (int64_t)KB + threadIdx.x;
  if (i < n) q[i] = Divider(h[i])(w[i]);
}

// Every block solves the small triangle (redundantly, same order) and then
// updates its slice of x with the combination of the preconditioned vectors.
__global__ void __launch_bounds__(KB) k_update_x(int n, int jend, int m, const double* __restrict__ H,
                                                 const double* __restrict__ g, double* __restrict__ yout,
                                                 const double* __restrict__ Z, double* __restrict__ x) {
  extern __shared__ double ys[];
  if (threadIdx.x == 0) {
    for (int i = jend - 1; i >= 0; --i) {
      double s = g[i];
      for (int t = i + 1; t < jend; ++t) s -= H[i * m + t] * ys[t];
      ys[i] = s / H[i * m + i];
    }
    if (blockIdx.x == 0)
      for (int i = 0; i < jend; ++i) yout[i] = ys[i];
  }
  __syncthreads();
  for (long long i = (long long)blockIdx.x * KB + threadIdx.x; i < n; i += (long long)gridDim.x * KB) {
    double acc = x[i];
    for (int k = 0; k < jend; ++k) acc += ys[k] * Z[(size_t)k * (size_t)n + i];
    x[i] = acc;
  }
}

}  // namespace

int krylov_parts(int n) {
  long long p = ((long long)n + 8 * KB - 1) / (8 * KB);
  if (p < 1) p = 1;
  if (p > kMaxParts) p = kMaxParts;
  return (int)p;
}

cudaError_t launch_dot_part(int n, const double* a, const double* b, double* part, cudaStream_t s) {
  k_dot_part<<<krylov_parts(n), KB, 0, s>>>(n, a, b, part);
  return cudaGetLastError();
}

cudaError_t launch_mgs_step(int n, const double* part_in, double* hout, double* w, const double* vi,
                            const double* vnext, double* part_out, int sms, cudaStream_t s) {
  const int np = krylov_parts(n);
  if (np <= 4 * sms)
    k_mgs_step<4><<<np, KB, 0, s>>>(n, part_in, np, hout, w, vi, vnext, part_out);
  else
    k_mgs_step<2><<<np, KB, 0, s>>>(n, part_in, np, hout, w, vi, vnext, part_out);
  return cudaGetLastError();
}

cudaError_t launch_normalize(int n, const double* part_in, double* hout, const double* w, double* vout,
                             cudaStream_t s) {
  const int np = krylov_parts(n);
  k_normalize<<<np, KB, 0, s>>>(n, part_in, np, hout, w, vout);
  return cudaGetLastError();
}

cudaError_t launch_normalize_givens(int n, const double* part_in, const double* w, double* vout, int j, int m,
                                    double* H, double* cs, double* sn, double* g, double* res, cudaStream_t s) {
  const int np = krylov_parts(n);
  const size_t smem = j < kGivensStaged ? sizeof(double) * (size_t)(3 * j + 1) : 0;
  k_normalize_givens<<<np, KB, smem, s>>>(n, part_in, np, w, vout, j, m, H, cs, sn, g,
                                                                         res);
  return cudaGetLastError();
}

cudaError_t launch_mr_step(int n, const double* part_num, const double* part_den, const double* sv, double* y,
                           cudaStream_t s) {
  const int np = krylov_parts(n);
  k_mr_step<<<np, KB, 0, s>>>(n, part_num, part_den, np, sv, y);
  return cudaGetLastError();
}

cudaError_t launch_norm_final(int n, const double* part_in, double* out, cudaStream_t s) {
  k_norm_final<<<1, KB, 0, s>>>(part_in, krylov_parts(n), out);
  return cudaGetLastError();
}

cudaError_t launch_divide(int64_t n, const double* w, const double* h, double* q, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_divide<<<(unsigned)((n + KB - 1) / KB), KB, 0, s>>>(n, w, h, q);
  return cudaGetLastError();
}

cudaError_t launch_update_x(int n, int jend, int m, const double* H, const double* g, double* y, const double* Z,
                            double* x, cudaStream_t s) {
  if (jend <= 0) return cudaSuccess;
  k_update_x<<<krylov_parts(n), KB, sizeof(double) * (size_t)jend, s>>>(n, jend, m, H, g, y, Z, x);
  return cudaGetLastError();
}

}  // namespace silu
