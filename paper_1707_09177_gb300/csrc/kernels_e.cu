// The FFT pass kernels of one precision (GAD_REAL) and per-thread element
// count (GAD_E): the build compiles this file once per pair, in parallel.
#include "launch.h"
#include "passes.cuh"
#include "spectral.cuh"

namespace gad {

template <typename T, int E>
cudaError_t launch_pass_e(int kind, dim3 grid, int threads, size_t smem, cudaStream_t s,
                                 const PassArgs<T>& a) {
  void (*fn)(PassArgs<T>) = nullptr;
  switch (kind) {
    case PK_XFWD: fn = k_xfwd<T, E>; break;
    case PK_XINV: fn = k_xinv<T, E>; break;
    case PK_FILT: fn = k_filt<T, E>; break;
    case PK_YFWD: fn = k_yfwd<T, E>; break;
    case PK_YINV: fn = k_yinv<T, E>; break;
    case PK_LFWD: fn = k_lfwd<T, E>; break;
    case PK_LINV: fn = k_linv<T, E>; break;
    default: return cudaErrorInvalidValue;
  }
  if constexpr (sizeof(T) == 4 && E == 12) {
    if (auto fk = fused_kernel(kind, a)) fn = fk;
  }
  const cudaError_t e = allow_smem(fn, smem, kPassSmem);
  if (e != cudaSuccess) return e;
  fn<<<grid, threads, smem, s>>>(a);
  return cudaGetLastError();
}

template cudaError_t launch_pass_e<GAD_REAL, GAD_E>(int, dim3, int, size_t, cudaStream_t, const PassArgs<GAD_REAL>&);

}  // namespace gad
