// Launches of the population evaluator: one instantiation per (bit planes, slab height, trend
// option), picked from the matrix's layout.
#include "eval_kernel.cuh"

namespace ebic {
namespace {

// The dynamic shared-memory limit of one instantiation, raised on the current device. The
// attribute is a per-device property of the function, so it is set once per device (a bit per
// device index, set after the call succeeded; concurrent first calls may both set it, which is
// harmless). Setting it also loads the function's code on that device under lazy module loading.
template <int NB, int T, bool NEG>
cudaError_t ready_variant() {
  static std::atomic<uint64_t> ready_devices{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit && (ready_devices.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(eval_population_kernel<NB, T, NEG>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemDynMax);
  if (e != cudaSuccess) return e;
  if (bit) ready_devices.fetch_or(bit, std::memory_order_acq_rel);
  return cudaSuccess;
}

struct Launch {
  const EvalArgs* a = nullptr;  // null: only ready the variant
  int grid = 0;
  bool pdl = false;
  cudaStream_t s = nullptr;
};

template <int NB, int T>
cudaError_t apply(const Launch& l, bool negative) {
  cudaError_t e = negative ? ready_variant<NB, T, true>() : ready_variant<NB, T, false>();
  if (e != cudaSuccess || !l.a) return e;
  count_launch();
  return launch_maybe_pdl(l.pdl, negative ? eval_population_kernel<NB, T, true>
                                          : eval_population_kernel<NB, T, false>,
                          dim3(l.grid), dim3(kEvalThreads), l.a->smem_bytes, l.s, *l.a);
}

// The layouts make_layout gives: slabs of 16 words up to 208 columns, 8 up to 369, 4 up to 665,
// 2 beyond.
template <class F>
cudaError_t for_layout(int planes, int t, F f) {
  switch (planes * 100 + t) {
    case 116: return f(std::integral_constant<int, 1>(), std::integral_constant<int, 16>());
    case 216: return f(std::integral_constant<int, 2>(), std::integral_constant<int, 16>());
    case 316: return f(std::integral_constant<int, 3>(), std::integral_constant<int, 16>());
    case 416: return f(std::integral_constant<int, 4>(), std::integral_constant<int, 16>());
    case 516: return f(std::integral_constant<int, 5>(), std::integral_constant<int, 16>());
    case 616: return f(std::integral_constant<int, 6>(), std::integral_constant<int, 16>());
    case 716: return f(std::integral_constant<int, 7>(), std::integral_constant<int, 16>());
    case 816: return f(std::integral_constant<int, 8>(), std::integral_constant<int, 16>());
    case 808: return f(std::integral_constant<int, 8>(), std::integral_constant<int, 8>());
    case 908: return f(std::integral_constant<int, 9>(), std::integral_constant<int, 8>());
    case 904: return f(std::integral_constant<int, 9>(), std::integral_constant<int, 4>());
    case 1004: return f(std::integral_constant<int, 10>(), std::integral_constant<int, 4>());
    case 1002: return f(std::integral_constant<int, 10>(), std::integral_constant<int, 2>());
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t ready_eval() {
  cudaError_t e = cudaSuccess;
  for (int nb = 1; nb <= kMaxPlanes; ++nb)
    for (int t = 2; t <= 16; t *= 2) {
      if (nb < 8 && t != 16) continue;
      const cudaError_t r = for_layout(nb, t, [](auto n, auto h) {
        cudaError_t x = apply<n(), h()>(Launch{}, false);
        return x != cudaSuccess ? x : apply<n(), h()>(Launch{}, true);
      });
      if (r != cudaSuccess && r != cudaErrorInvalidValue && e == cudaSuccess) e = r;
    }
  return e;
}

cudaError_t launch_eval(const EvalArgs& a, bool negative, int grid, bool pdl, cudaStream_t s) {
  return for_layout(a.planes, a.slab_high, [&](auto n, auto h) {
    return apply<n(), h()>(Launch{&a, grid, pdl, s}, negative);
  });
}

}  // namespace ebic
