// float32 instantiation of the pass kernels.
#define GAD_REAL float
#include "kernels_impl.cuh"

namespace gad {
cudaError_t launch_reset_state(FieldState* st, int batch, cudaStream_t s) {
  k_reset_state<<<(batch + 127) / 128, 128, 0, s>>>(st, batch);
  return cudaGetLastError();
}
template <typename T>
cudaError_t launch_multi(int kind, int E, int blocks, int threads, size_t smem, cudaStream_t s,
                         const PassArgs<T>* args, const int* start, int ngroups) {
  if (E == 16) return launch_multi_e<T, 16>(kind, blocks, threads, smem, s, args, start, ngroups);
  if (E == 24) return launch_multi_e<T, 24>(kind, blocks, threads, smem, s, args, start, ngroups);
  if (E == 4) return launch_multi_e<T, 4>(kind, blocks, threads, smem, s, args, start, ngroups);
  if (E == 12) return launch_multi_e<T, 12>(kind, blocks, threads, smem, s, args, start, ngroups);
  return cudaErrorInvalidValue;
}

template cudaError_t launch_multi<float>(int, int, int, int, size_t, cudaStream_t, const PassArgs<float>*, const int*,
                                         int);
}  // namespace gad
