// One Arnoldi step of the flexible GMRES in one launch (sm_103a): w against
// v_0 .. v_j by modified Gram-Schmidt (Sec. 6), h_{j+1,j}, v_{j+1} and the
// Givens update of column j.
//
// Modified Gram-Schmidt needs a global reduction per basis vector, and one
// launch per basis vector (k_mgs_step) pays for each: the launch, every
// block's sum of all partial sums, and w and v_i read and w written again
// (32 bytes per row).  Here one grid, every block resident (cooperative
// launch), keeps its part of w, v_i and v_{i+1} in registers through all
// steps, so that each basis vector is read once (8 bytes per row and step; the
// next one is loaded while the reduction is under way) and w is never written.
// What is left is the FP64 pipe, which issues one warp-wide operation per 64 to
// 76 clocks on each of an SM's four partitions whatever lanes are active (two
// per 32 rows and step, and the adds of the reductions), and one exchange of
// partial sums per step.
//
// The exchange: every block publishes its partial sums and every block reads
// all of them.  An entry is two 8-byte words, each holding half of the FP64
// value and a 32-bit tag that numbers the exchange, so an entry is complete
// when both tags match and no fence or atomic is needed.  The j + 2 exchanges of
// step j have numbers of their own within a restart cycle, known to the host
// (exchange_number), and the entries are zeroed at the start of each cycle
// (arnoldi_reset), so nothing that an earlier cycle or solve left behind, one
// that gave up included, carries a number that is waited for.  Two
// buffers alternate; a block writes a buffer again only after an exchange
// through the other one, which every block enters after leaving the first.
// Every wait is bounded (2 s); one that gives up sets bit 4 (value 16) of the
// error word and no later wait of that thread waits.
//
// The sums are k_dot_part's and k_mgs_step's, in their order and with their
// roundings: rows are dealt to np groups of 256 threads, eight at most to each,
// a thread adds its products in row order, a warp by the same shuffle tree, the
// eight warps of a group one after the other, the np groups as sum_parts adds
// them.  So results are the bits of the launch-per-vector form.  Two layouts:
// k_arnoldi, blocks of one to three whole groups, one block per SM, whose
// reductions pack the trees of a group's eight warps into the lanes of one (9
// adds instead of 40); and, for at most 16 groups, k_arnoldi_cluster, one
// cluster of blocks of a group each, whose warps write their own sums into
// every block's shared memory (no exchange through L2).
//
// Measured per basis vector: the cluster at 16 groups (32^3 rows) 3.0 us, 4.0
// with a launch per vector, 4.9 with the exchange through L2; 152 to 456 groups
// of 2048 rows 5.6 to 7.8 us, 8 to 11 with launches; between them the launches
// (5.0 to 5.8 us with the exchange) are kept.
#include <cmath>

#include "device.cuh"
#include "exchange.cuh"
#include "krylov.cuh"

namespace silu {
namespace {

constexpr int kArnRows = 8;  // rows per thread at most
constexpr int kArnMaxBasis = 1024;
constexpr int kArnMaxGroups = 512;

struct ArnoldiArgs {
  int n, np, j, m;
  const double* w;
  double* V;  // column k at V + k n
  double* H;  // row-major, leading dimension m
  double* cs;
  double* sn;
  double* g;
  double* res;
  ulonglong2* entries;  // two buffers of `cap` entries
  int cap;
  unsigned tag;  // number of this step's first exchange
  int* err;
};

// Number of the first exchange of step j: steps 0 .. j - 1 have i + 2 each, and
// 0 is an entry that nothing has been written to.
__host__ __device__ constexpr unsigned exchange_number(int j) { return 1u + (unsigned)j * ((unsigned)j + 3u) / 2u; }

// r[q] holds lane values of warp q (q < 8): the sum over each warp's lanes by
// the tree of arn_warp_sum, the trees sharing the lanes of one warp (a lane
// keeps one value and sends the other to its partner), and those eight sums
// added one after the other.  Every lane returns the result.
__device__ __forceinline__ double sum_of_eight_warps(double (&r)[8], int lane) {
  auto fold = [lane](double a, double b, int off) {  // a's pairs in lanes without bit `off`, b's in the others
    const bool up = (lane & off) != 0;
    const double send = up ? a : b;
    return (up ? b : a) + __shfl_xor_sync(0xffffffffu, send, off);
  };
  const double s0 = fold(r[0], r[1], 16), s1 = fold(r[2], r[3], 16), s2 = fold(r[4], r[5], 16),
               s3 = fold(r[6], r[7], 16);
  const double t0 = fold(s0, s1, 8), t1 = fold(s2, s3, 8);
  double v = fold(t0, t1, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  // warp q's sum lies in the lanes whose bits 16, 8, 4 are q's bits 1, 2, 4
  double s = __shfl_sync(0xffffffffu, v, 0);
#pragma unroll
  for (int q = 1; q < 8; ++q)
    s += __shfl_sync(0xffffffffu, v, ((q & 1) ? 16 : 0) | ((q & 2) ? 8 : 0) | ((q & 4) ? 4 : 0));
  return s;
}

// Block 0's shared memory: column j of H (m + 1 entries), cs and sn (m each).
__device__ __forceinline__ void load_rotations(const ArnoldiArgs& a, double* sh, int threads) {
  for (int i = threadIdx.x; i < a.j; i += threads) {
    sh[a.m + 1 + i] = a.cs[i];
    sh[2 * a.m + 1 + i] = a.sn[i];
  }
}

// One thread: the earlier rotations on column j (h_0 .. h_j in sh, h its last
// entry), the new one, the right-hand side; k_normalize_givens's arithmetic.
__device__ __forceinline__ void givens_column(const ArnoldiArgs& a, double* hc, double h) {
  const int j = a.j, m = a.m;
  const double* cs = hc + m + 1;
  const double* sn = cs + m;
  hc[j + 1] = h;
  for (int i = 0; i < j; ++i) {
    const double p = hc[i], q = hc[i + 1];
    hc[i] = cs[i] * p + sn[i] * q;
    hc[i + 1] = -sn[i] * p + cs[i] * q;
    a.H[(size_t)i * m + j] = hc[i];
  }
  const double p = hc[j], q = hc[j + 1];
  const double den = hypot(p, q);
  const double c = den != 0.0 ? p / den : 1.0;
  const double s = den != 0.0 ? q / den : 0.0;
  a.cs[j] = c;
  a.sn[j] = s;
  a.H[(size_t)j * m + j] = den;
  a.H[(size_t)(j + 1) * m + j] = 0.0;
  const double gj = a.g[j];
  a.g[j + 1] = -s * gj;
  a.g[j] = c * gj;
  a.res[0] = fabs(-s * gj);
  a.res[1] = q;  // h_{j+1,j}: zero means the Krylov space is exhausted
}

// One thread's share: rows i0, i0 + S, ..., cnt of them.  NARROW: addressed by
// 32-bit offsets, which spares the registers that three groups per block lack
// (and costs one or two groups, and the cluster, 1 to 5% of a step).
template <bool NARROW>
struct ArnoldiRows {
  unsigned i0, S;
  int cnt;
  double w[kArnRows], u[kArnRows], nx[kArnRows];
  __device__ __forceinline__ ArnoldiRows(const ArnoldiArgs& a, int group, int place) {
    S = (unsigned)a.np * 256u;
    i0 = (unsigned)group * 256u + (unsigned)place;
    cnt = group < a.np && i0 < (unsigned)a.n ? (int)(((unsigned)a.n - i0 + S - 1) / S) : 0;
  }
  __device__ __forceinline__ void load(const double* p, double (&v)[kArnRows]) const {
    if constexpr (!NARROW) p += i0;
#pragma unroll
    for (int k = 0; k < kArnRows; ++k)
      if constexpr (NARROW)
        v[k] = k < cnt ? p[i0 + (unsigned)k * S] : 0.0;
      else
        v[k] = k < cnt ? p[(size_t)k * S] : 0.0;
  }
  // this thread's part of <w, v_0>
  __device__ __forceinline__ double first() const {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kArnRows; ++k)
      if (k < cnt) acc += w[k] * u[k];
    return acc;
  }
  // w -= h v_i, and this thread's part of <w, v_{i+1}> (of |w|^2 after the last)
  __device__ __forceinline__ double step(double h, bool more) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < kArnRows; ++k) {
      if (k < cnt) {
        const double wn = w[k] - h * u[k];
        w[k] = wn;
        acc += wn * (more ? nx[k] : wn);
      }
      u[k] = nx[k];
    }
    return acc;
  }
  __device__ __forceinline__ void normalize(double h, double* vout) const {
    if (h == 0.0) return;
    const Divider by(h);
    if constexpr (!NARROW) vout += i0;
#pragma unroll
    for (int k = 0; k < kArnRows; ++k)
      if (k < cnt) {
        if constexpr (NARROW)
          vout[i0 + (unsigned)k * S] = by(w[k]);
        else
          vout[(size_t)k * S] = by(w[k]);
      }
  }
};

// GB groups of 256 threads per block, one block per SM.
template <int GB>
__global__ void __launch_bounds__(GB * 256, 1) k_arnoldi(ArnoldiArgs a) {
  constexpr int T = GB * 256;
  extern __shared__ double sh[];  // column j of H, cs, sn (givens_column)
  __shared__ double lanes[T];
  __shared__ double parts[256];
  __shared__ double total;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = blockIdx.x * GB + (threadIdx.x >> 8);
  const bool lead = blockIdx.x == 0;
  ArnoldiRows<GB == 3> rows(a, group, threadIdx.x & 255);
  bool alive = true;
  unsigned tag = a.tag;
  if (lead) load_rotations(a, sh, T);
  // publish the groups' parts of the sum over all rows of the threads' acc
  auto give = [&](double acc, int step) {
    lanes[threadIdx.x] = acc;
    __syncthreads();
    if ((warp & 7) == 0) {  // one warp per group
      double r[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) r[q] = lanes[(warp + q) * 32 + lane];
      const double s = sum_of_eight_warps(r, lane);
      if (lane == 0 && group < a.np) publish(a.entries + (step & 1) * a.cap + group, s, tag);
    }
  };
  // the whole sum, to every thread: as sum_parts, thread t of 256 adds groups t and t + 256
  auto take = [&](int step) {
    if (threadIdx.x < 256) {
      constexpr int K = kArnMaxGroups / 256;
      double v[K];
      const int t = threadIdx.x;
      const int cnt = t < a.np ? (a.np - t + 255) >> 8 : 0;
      collect<K>(a.entries + (step & 1) * a.cap + t, 256, cnt, tag, v, alive, a.err);
      double s = v[0];
#pragma unroll
      for (int k = 1; k < K; ++k)
        if (k < cnt) s += v[k];
      parts[t] = s;
    }
    __syncthreads();
    if (warp == 0) {
      double r[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) r[q] = parts[q * 32 + lane];
      const double s = sum_of_eight_warps(r, lane);
      if (lane == 0) total = s;
    }
    __syncthreads();
    ++tag;
    return total;
  };
  rows.load(a.w, rows.w);
  rows.load(a.V, rows.u);
  give(rows.first(), 0);
  for (int i = 0; i <= a.j; ++i) {
    const bool more = i < a.j;
    if (more) rows.load(a.V + (size_t)(i + 1) * (size_t)a.n, rows.nx);
    const double h = take(i);
    if (lead && threadIdx.x == 0) sh[i] = h;
    give(rows.step(h, more), i + 1);
  }
  const double h = sqrt(take(a.j + 1));
  rows.normalize(h, a.V + (size_t)(a.j + 1) * (size_t)a.n);
  if (lead && threadIdx.x == 0) givens_column(a, sh, h);
}

__device__ __forceinline__ uint32_t cluster_smem(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(r)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}

// At most 16 groups: one cluster of CT blocks, a group each.  Warps write their
// sums into every block's shared memory; the cluster's barrier takes the place
// of the exchange through L2.
template <int CT>
__global__ void __launch_bounds__(256, 1) k_arnoldi_cluster(ArnoldiArgs a) {
  extern __shared__ double sh[];  // column j of H, cs, sn (givens_column)
  __shared__ double slot[2][8][CT];  // [buffer][warp][group]
  __shared__ double total[2];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = blockIdx.x;  // one cluster: the block's rank
  const bool lead = group == 0;
  ArnoldiRows<false> rows(a, group, threadIdx.x);
  if (lead) load_rotations(a, sh, 256);
  // every block of the cluster runs before another writes into its shared memory
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  auto sum = [&](double acc, int step) {
    const int p = step & 1;
    const double s = arn_warp_sum(acc);
    if (lane < CT) {
      const uint32_t to = cluster_smem(&slot[p][warp][group], (uint32_t)lane);
      asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(s) : "memory");
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 0) {
      double v = 0.0;
      if (lane < CT) {
        v = slot[p][0][lane];
#pragma unroll
        for (int q = 1; q < 8; ++q) v += slot[p][q][lane];
      }
      v = arn_warp_sum(v);  // groups beyond np are zeros, as sum_parts has them
      if (lane == 0) total[p] = v;
    }
    __syncthreads();
    return total[p];
  };
  rows.load(a.w, rows.w);
  rows.load(a.V, rows.u);
  double acc = rows.first();
  for (int i = 0; i <= a.j; ++i) {
    const bool more = i < a.j;
    if (more) rows.load(a.V + (size_t)(i + 1) * (size_t)a.n, rows.nx);
    const double h = sum(acc, i);
    if (lead && threadIdx.x == 0) sh[i] = h;
    acc = rows.step(h, more);
  }
  const double h = sqrt(sum(acc, a.j + 1));
  rows.normalize(h, a.V + (size_t)(a.j + 1) * (size_t)a.n);
  if (lead && threadIdx.x == 0) givens_column(a, sh, h);
  // no block leaves while another may still write into it
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// What a step that gave up may leave behind: a wait that runs out (no exchange
// has this number), then entries numbered as the next cycle's first step
// numbers its own, with values that no sum survives.
__global__ void k_exchange_selftest(ulonglong2* entries, int cap, int* err) {
  bool alive = true;
  double v[1];
  if (threadIdx.x == 0) collect<1>(entries, 1, 1, ~0u, v, alive, err);
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * cap; i += blockDim.x)
    publish(entries + i, __longlong_as_double(0x7ff8000000000000ll), exchange_number(0) + (i < cap ? 0u : 1u));
}

template <int GB>
cudaError_t launch_groups(const ArnoldiArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((a.np + GB - 1) / GB));
  cfg.blockDim = dim3(GB * 256);
  cfg.dynamicSmemBytes = sizeof(double) * (size_t)(3 * a.m + 1);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_arnoldi<GB>, a);
}

template <int CT>
cudaLaunchConfig_t cluster_config(int m, cudaLaunchAttribute* attr, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CT);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = sizeof(double) * (size_t)(3 * m + 1);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CT;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int CT>
cudaError_t launch_cluster(const ArnoldiArgs& a, cudaStream_t s) {
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = cluster_config<CT>(a.m, attr, s);
  return cudaLaunchKernelEx(&cfg, k_arnoldi_cluster<CT>, a);
}

// Clusters of CT blocks that fit on the device (0: none).
template <int CT>
cudaError_t prepare_cluster(int* fit) {
  cudaError_t e = cudaSuccess;
  if (CT > 8) e = cudaFuncSetAttribute(k_arnoldi_cluster<CT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = cluster_config<CT>(kArnMaxBasis, attr, nullptr);
  return cudaOccupancyMaxActiveClusters(fit, k_arnoldi_cluster<CT>, &cfg);
}

// The form for np groups: 16, 8, ... (a cluster of so many blocks), 1 to 3
// groups per block (negative), or 0: launch per vector.
int arnoldi_form(int np, const LaunchEnv& env) {
  if (np <= 16) {
    for (int ct = 1; ct <= 16; ct *= 2)
      if (np <= ct) return ct <= env.arnoldi_cluster ? ct : 0;
  }
  const int gb = (np + env.sms - 1) / env.sms;
  return env.arnoldi && np >= env.sms && np <= kArnMaxGroups && gb <= 3 ? -gb : 0;
}

}  // namespace

size_t arnoldi_bytes(int n) { return 2 * sizeof(ulonglong2) * (size_t)krylov_parts(n); }

cudaError_t arnoldi_reset(int n, int m, void* scratch, const LaunchEnv& env, cudaStream_t s) {
  if (!arnoldi_fits(n, m, env) || arnoldi_form(krylov_parts(n), env) > 0) return cudaSuccess;
  return cudaMemsetAsync(scratch, 0, arnoldi_bytes(n), s);
}

cudaError_t launch_exchange_selftest(int n, void* scratch, int* err, cudaStream_t s) {
  k_exchange_selftest<<<1, 256, 0, s>>>((ulonglong2*)scratch, krylov_parts(n), err);
  return cudaGetLastError();
}

cudaError_t arnoldi_prepare(LaunchEnv& env) {
  const size_t smem = sizeof(double) * (3 * kArnMaxBasis + 1);
  int occ[3] = {0, 0, 0}, fit[5] = {0, 0, 0, 0, 0};
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[0], k_arnoldi<1>, 256, smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[1], k_arnoldi<2>, 512, smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ[2], k_arnoldi<3>, 768, smem);
  env.arnoldi = occ[0] > 0 && occ[1] > 0 && occ[2] > 0;
  if (e == cudaSuccess) e = prepare_cluster<1>(&fit[0]);
  if (e == cudaSuccess) e = prepare_cluster<2>(&fit[1]);
  if (e == cudaSuccess) e = prepare_cluster<4>(&fit[2]);
  if (e == cudaSuccess) e = prepare_cluster<8>(&fit[3]);
  if (e == cudaSuccess) e = prepare_cluster<16>(&fit[4]);
  env.arnoldi_cluster = 0;
  for (int k = 0; k < 5 && fit[k] > 0; ++k) env.arnoldi_cluster = 1 << k;
  return e;
}

bool arnoldi_fits(int n, int m, const LaunchEnv& env) {
  const int np = krylov_parts(n);
  return m <= kArnMaxBasis && (long long)np * 256 * kArnRows >= n && arnoldi_form(np, env) != 0;
}

cudaError_t launch_arnoldi(int n, int j, int m, const double* w, double* V, double* H, double* cs, double* sn,
                           double* g, double* res, void* scratch, const LaunchEnv& env, cudaStream_t s) {
  ArnoldiArgs a;
  a.n = n;
  a.np = krylov_parts(n);
  a.j = j;
  a.m = m;
  a.w = w;
  a.V = V;
  a.H = H;
  a.cs = cs;
  a.sn = sn;
  a.g = g;
  a.res = res;
  a.cap = a.np;
  a.entries = (ulonglong2*)scratch;
  a.tag = exchange_number(j);
  a.err = env.err;
  switch (arnoldi_form(a.np, env)) {
    case -1: return launch_groups<1>(a, s);
    case -2: return launch_groups<2>(a, s);
    case -3: return launch_groups<3>(a, s);
    case 1: return launch_cluster<1>(a, s);
    case 2: return launch_cluster<2>(a, s);
    case 4: return launch_cluster<4>(a, s);
    case 8: return launch_cluster<8>(a, s);
    case 16: return launch_cluster<16>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace silu
