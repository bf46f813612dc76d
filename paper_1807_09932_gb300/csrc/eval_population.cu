// Launches of the population evaluator: one instantiation per (bit planes, slab height, words per lane,
// trend option), picked from the matrix's layout and the tile.
#include "eval_kernel.cuh"

namespace ebic {
namespace {

// The dynamic shared-memory limit of one instantiation, raised on the current device. The
// attribute is a per-device property of the function, so it is set once per device (a bit per
// device index, set after the call succeeded; concurrent first calls may both set it, which is
// harmless). Setting it also loads the function's code on that device under lazy module loading.
template <int NB, int T, int WPL, bool NEG>
cudaError_t ready_variant() {
  static std::atomic<uint64_t> ready_devices{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? (uint64_t)1 << dev : 0;
  if (bit && (ready_devices.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(eval_population_kernel<NB, T, WPL, NEG>,
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

template <int NB, int T, int WPL>
cudaError_t apply(const Launch& l, bool negative) {
  cudaError_t e = negative ? ready_variant<NB, T, WPL, true>() : ready_variant<NB, T, WPL, false>();
  if (e != cudaSuccess || !l.a) return e;
  count_launch();
  return launch_maybe_pdl(l.pdl, negative ? eval_population_kernel<NB, T, WPL, true>
                                          : eval_population_kernel<NB, T, WPL, false>,
                          dim3(l.grid), dim3(kEvalThreads), l.a->smem_bytes, l.s, *l.a);
}

// The layouts make_layout gives: slabs of 16 words up to 208 columns, 8 up to 369, 4 up to 665, 2
// beyond; and the tiles tile_allowed lets them have: 1, 2 or 4 slabs of 16 words, of which 4 fit up to
// 52 columns and 2 up to 104, else one slab. The walks are kernels of their own: with all three in
// one, calls that take 11 us took 1 us longer, and one-slab tiles lost up to 15 %.
template <int NB, int T>
cudaError_t for_tile(int ts, const Launch& l, bool negative) {
  if constexpr (T == 16 && NB <= 7)
    if (ts == 2) return apply<NB, T, 1>(l, negative);
  if constexpr (T == 16 && NB <= 6)
    if (ts == 4) return apply<NB, T, 2>(l, negative);
  return ts == 1 ? apply<NB, T, 0>(l, negative) : cudaErrorInvalidValue;
}

cudaError_t for_layout(int planes, int t, int ts, const Launch& l, bool negative) {
  switch (planes * 100 + t) {
    case 116: return for_tile<1, 16>(ts, l, negative);
    case 216: return for_tile<2, 16>(ts, l, negative);
    case 316: return for_tile<3, 16>(ts, l, negative);
    case 416: return for_tile<4, 16>(ts, l, negative);
    case 516: return for_tile<5, 16>(ts, l, negative);
    case 616: return for_tile<6, 16>(ts, l, negative);
    case 716: return for_tile<7, 16>(ts, l, negative);
    case 816: return for_tile<8, 16>(ts, l, negative);
    case 808: return for_tile<8, 8>(ts, l, negative);
    case 908: return for_tile<9, 8>(ts, l, negative);
    case 904: return for_tile<9, 4>(ts, l, negative);
    case 1004: return for_tile<10, 4>(ts, l, negative);
    case 1002: return for_tile<10, 2>(ts, l, negative);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t ready_eval() {
  cudaError_t e = cudaSuccess;
  for (int nb = 1; nb <= kMaxPlanes; ++nb)
    for (int t = 2; t <= 16; t *= 2)
      for (int ts = 1; ts <= 4; ts *= 2)
        for (bool negative : {false, true}) {
          if (nb < 8 && t != 16) continue;
          const cudaError_t r = for_layout(nb, t, ts, Launch{}, negative);
          if (r != cudaSuccess && r != cudaErrorInvalidValue && e == cudaSuccess) e = r;
        }
  return e;
}

cudaError_t launch_eval(const EvalArgs& a, bool negative, int grid, bool pdl, cudaStream_t s) {
  return for_layout(a.planes, a.slab_high, a.ts, Launch{&a, grid, pdl, s}, negative);
}

}  // namespace ebic
