// float32 instantiation of the multi-group pass kernels (k_multi) for one
// per-thread element count (GAD_E): one launch per pass stage over the blocks
// of several shape groups of a batched solve. Compiled once per E, in parallel
// with the single-group kernels.
#include <algorithm>

#include "launch.h"
#include "passes.cuh"

namespace gad {

template <typename T, int E, int KIND>
static cudaError_t launch_multi_k(int blocks, int threads, size_t smem, cudaStream_t s, const PassArgs<T>* args,
                                  const int* start, int ngroups) {
  const cudaError_t e = allow_smem(k_multi<T, E, KIND>, smem, kPassSmem);
  if (e != cudaSuccess) return e;
  k_multi<T, E, KIND><<<blocks, threads, smem, s>>>(args, start, ngroups);
  return cudaGetLastError();
}

template <typename T, int E>
cudaError_t launch_multi_e(int kind, int blocks, int threads, size_t smem, cudaStream_t s,
                                  const PassArgs<T>* args, const int* start, int ngroups) {
  switch (kind) {
    case PK_XFWD: return launch_multi_k<T, E, 0>(blocks, threads, smem, s, args, start, ngroups);
    case PK_XINV: return launch_multi_k<T, E, 1>(blocks, threads, smem, s, args, start, ngroups);
    case PK_FILT: return launch_multi_k<T, E, 2>(blocks, threads, smem, s, args, start, ngroups);
    case PK_YFWD: return launch_multi_k<T, E, 3>(blocks, threads, smem, s, args, start, ngroups);
    case PK_YINV: return launch_multi_k<T, E, 4>(blocks, threads, smem, s, args, start, ngroups);
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_multi_e<float, GAD_E>(int, int, int, size_t, cudaStream_t, const PassArgs<float>*,
                                                  const int*, int);

}  // namespace gad
