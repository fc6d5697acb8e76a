// The sliced sweep for 2, 3 and 4 interleaved right-hand sides (see
// slices.cuh): each entry read feeds R multiply-adds, so the FP64 pipe bounds
// it; two to four entries per chunk keep R columns of gathers in registers.
#include "slices.cuh"

#include <type_traits>

namespace silu {
namespace {

// Pairs per chunk and blocks per SM by R (FP32 keeps more in registers).
template <class MT, int R>
struct MultiShape {
  static constexpr int CP = sizeof(MT) == 4 ? 2 : 1;
  static constexpr int MINB = sizeof(MT) == 4 ? (R == 2 ? 5 : 4) : (R == 2 ? 5 : 4);
};

template <class MT, class VI, class VO, class CT, int R, bool VEC>
using MultiKernel = SliceKernel<MT, VI, VO, CT, R, MultiShape<MT, R>::CP, MultiShape<MT, R>::MINB, VEC>;

// Small matrices (16-bit columns): rows of up to 4 entries in one chunk, longer
// ones 8 at a time.
template <class MT, class VI, class VO, int R, bool VEC, int CP>
using SmallKernel = SliceKernel<MT, VI, VO, uint16_t, R, CP, 1, VEC>;

template <class MT, class VI, class VO, int R, bool VEC>
cudaError_t prepare_small() {
  const cudaError_t e = SmallKernel<MT, VI, VO, R, VEC, 2>::prepare();
  return e == cudaSuccess ? SmallKernel<MT, VI, VO, R, VEC, 4>::prepare() : e;
}

template <class MT, class VI, class VO>
cudaError_t prepare_small_mode() {
  cudaError_t e = prepare_small<MT, VI, VO, 2, false>();
  if (e == cudaSuccess) e = prepare_small<MT, VI, VO, 2, true>();
  if (e == cudaSuccess) e = prepare_small<MT, VI, VO, 3, false>();
  if (e == cudaSuccess) e = prepare_small<MT, VI, VO, 4, false>();
  if (e == cudaSuccess) e = prepare_small<MT, VI, VO, 4, true>();
  return e;
}

template <class MT, class VI, class VO, class CT>
cudaError_t prepare_mode() {
  cudaError_t e = MultiKernel<MT, VI, VO, CT, 2, false>::prepare();
  if (e == cudaSuccess) e = MultiKernel<MT, VI, VO, CT, 2, true>::prepare();
  if (e == cudaSuccess) e = MultiKernel<MT, VI, VO, CT, 3, false>::prepare();
  if (e == cudaSuccess) e = MultiKernel<MT, VI, VO, CT, 4, false>::prepare();
  if (e == cudaSuccess) e = MultiKernel<MT, VI, VO, CT, 4, true>::prepare();
  return e;
}

template <class MT, class VI, class VO, class CT>
cudaError_t multi(const DevCsr& T, const LaunchEnv& env, int R, int ldx, const void* c, const void* in, void* out,
                  const double* dinv, double* x, int epi, cudaStream_t s) {
  // vector loads need every row's R entries of c and in on a boundary of
  // their width (16 bytes; 8 for two floats)
  const size_t unit = sizeof(VI) * (size_t)(sizeof(VI) == 8 ? 2 : R);
  const bool vec = R != 3 && ldx % (int)(unit / sizeof(VI)) == 0 && (uintptr_t)in % unit == 0 &&
                   (uintptr_t)c % unit == 0;
  auto go = [&](auto k) { return decltype(k)::launch(T, env, ldx, c, in, out, dinv, x, epi, s); };
  if constexpr (sizeof(CT) == 2) {
    if (slice_small(T.sl->ns, env.sms)) {
      auto pick = [&](auto r, auto v) {
        constexpr int RR = decltype(r)::value;
        constexpr bool VV = decltype(v)::value;
        return T.sl->widest <= 4 ? go(SmallKernel<MT, VI, VO, RR, VV, 2>()) : go(SmallKernel<MT, VI, VO, RR, VV, 4>());
      };
      using std::integral_constant;
      switch (R) {
        case 2:
          return vec ? pick(integral_constant<int, 2>(), std::true_type())
                     : pick(integral_constant<int, 2>(), std::false_type());
        case 3: return pick(integral_constant<int, 3>(), std::false_type());
        case 4:
          return vec ? pick(integral_constant<int, 4>(), std::true_type())
                     : pick(integral_constant<int, 4>(), std::false_type());
      }
    }
  }
  switch (R) {
    case 2: return vec ? go(MultiKernel<MT, VI, VO, CT, 2, true>()) : go(MultiKernel<MT, VI, VO, CT, 2, false>());
    case 3: return go(MultiKernel<MT, VI, VO, CT, 3, false>());
    case 4: return vec ? go(MultiKernel<MT, VI, VO, CT, 4, true>()) : go(MultiKernel<MT, VI, VO, CT, 4, false>());
  }
  return cudaErrorInvalidValue;
}

template <class CT>
cudaError_t multi_mode(const DevCsr& T, Mode mode, const LaunchEnv& env, int R, int ldx, const void* c,
                       const void* in, void* out, const double* dinv, double* x, int epi, cudaStream_t s) {
  switch (mode) {
    case MODE_D: return multi<double, double, double, CT>(T, env, R, ldx, c, in, out, dinv, x, epi, s);
    case MODE_F: return multi<float, float, float, CT>(T, env, R, ldx, c, in, out, dinv, x, epi, s);
    case MODE_DF: return multi<double, double, float, CT>(T, env, R, ldx, c, in, out, dinv, x, epi, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t slices_prepare_multi() {
  cudaError_t e = prepare_mode<double, double, double, uint16_t>();
  if (e == cudaSuccess) e = prepare_mode<double, double, double, int>();
  if (e == cudaSuccess) e = prepare_mode<float, float, float, uint16_t>();
  if (e == cudaSuccess) e = prepare_mode<float, float, float, int>();
  if (e == cudaSuccess) e = prepare_mode<double, double, float, uint16_t>();
  if (e == cudaSuccess) e = prepare_mode<double, double, float, int>();
  if (e == cudaSuccess) e = prepare_small_mode<double, double, double>();
  if (e == cudaSuccess) e = prepare_small_mode<float, float, float>();
  if (e == cudaSuccess) e = prepare_small_mode<double, double, float>();
  return e;
}

cudaError_t launch_slices_multi(const DevCsr& T, Mode mode, const LaunchEnv& env, int R, int ldx, const void* c,
                                const void* in, void* out, const double* dinv, double* x, int epi, cudaStream_t s) {
  return T.sl->wide ? multi_mode<int>(T, mode, env, R, ldx, c, in, out, dinv, x, epi, s)
                    : multi_mode<uint16_t>(T, mode, env, R, ldx, c, in, out, dinv, x, epi, s);
}

}  // namespace silu
