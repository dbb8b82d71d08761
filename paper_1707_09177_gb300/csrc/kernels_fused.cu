// Float32 pass kernels compiled for one transform length 2^a 3 or 2^a 9 each,
// at 12 elements per thread (fused radices, plan.h): constant strides instead
// of the general stages' float quotients, no spills. Two translation units
// (GAD_LONG 0: up to 192, 1: longer) that compile in parallel.
#include "launch.h"
#include "passes.cuh"

namespace gad {

template <int L>
static PassKernelF of_length(int kind, const PassArgs<float>& a) {
  if (a.fft.L != L || !ct_matches<L, 12, false>(a.fft)) return nullptr;
  if (kind == PK_FILT) return ct_matches<L, 12, true>(a.fft_inv) ? k_filt<float, 12, L> : nullptr;
  if constexpr (L <= 768) {             // longer x and y tiles take 24 elements per thread
    switch (kind) {
      case PK_XFWD: return k_xfwd<float, 12, L>;
      case PK_XINV: return k_xinv<float, 12, L>;
      case PK_YFWD: return k_yfwd<float, 12, L>;
      case PK_YINV: return k_yinv<float, 12, L>;
      default: break;
    }
  }
  return nullptr;
}

template <int... L>
static PassKernelF find(int kind, const PassArgs<float>& a) {
  PassKernelF fn = nullptr;
  (void)(... || ((fn = of_length<L>(kind, a)) != nullptr));
  return fn;
}

#if GAD_LONG
PassKernelF fused_kernel_long(int kind, const PassArgs<float>& a) {
  return find<288, 384, 576, 768, 1152, 1536, 2304>(kind, a);
}
#else
PassKernelF fused_kernel(int kind, const PassArgs<float>& a) {
  return a.fft.L > 192 ? fused_kernel_long(kind, a) : find<36, 48, 72, 96, 144, 192>(kind, a);
}
#endif

}  // namespace gad
