// Host-side launchers for the pass kernels, instantiated per precision in
// kernels_f32.cu and kernels_f64.cu (compiled in parallel).
#pragma once

#include <cuda_runtime.h>

#include "args.h"

namespace gad {

enum PassKind : int {
  PK_XFWD = 0, PK_XINV = 1, PK_FILT = 2, PK_YFWD = 3, PK_YINV = 4,
  PK_LFWD = 5,   // forward FFT along the last axis, S1 (2D) / S2 (3D) -> spectral vector O1
  PK_LINV = 6,   // inverse FFT along the last axis, spectral vector A (scaled by 1/P) -> S1 / S2
  PK_SPEC = 7,   // spectral-space Krylov pass (SpOp), 256 threads, no shared memory
  PK_STEN = 8,   // preconditioner z = M r with the dot (r, z), W rows per block (stencil.cuh)
};

// Launches pass `kind` with per-thread element count E (4, 12, 16 or 24). Returns the
// launch error (cudaSuccess when enqueued).
template <typename T>
cudaError_t launch_pass(int kind, int E, dim3 grid, int threads, size_t smem, cudaStream_t s,
                        const PassArgs<T>& a);

// The same for one E (kernels_e.cu, one translation unit per precision and E).
template <typename T, int E>
cudaError_t launch_pass_e(int kind, dim3 grid, int threads, size_t smem, cudaStream_t s, const PassArgs<T>& a);

// The float32 pass kernel of 12 elements per thread compiled for the plan's own
// length (kernels_fused.cu), or nullptr when there is none.
using PassKernelF = void (*)(PassArgs<float>);
PassKernelF fused_kernel(int kind, const PassArgs<float>& a);
PassKernelF fused_kernel_long(int kind, const PassArgs<float>& a);

// Dynamic shared memory above 48 KB per block needs an opt-in; the kernels'
// static shared memory (reduction scratch, mbarrier: under 1 KB) counts
// against the same limit, so the opt-in is made with this margin. The limit
// belongs to the kernel and is shared by all host threads, so every launch
// sets the same one, the most that a kernel of its kind may take: a launch that
// set its own size could lower it between another thread's opt-in and launch.
constexpr size_t kStaticSmemMargin = 4096;
constexpr size_t kPassSmem = 104 * 1024;      // tiles: 100 KB and the padding of transposed_ld (plan.h)
constexpr size_t kMaxSmem = 224 * 1024;       // what a block may take beside its static shared memory

template <typename Fn>
cudaError_t allow_smem(Fn* fn, size_t smem, size_t most) {
  if (smem + kStaticSmemMargin <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// A batch of small fields, one cluster of a.csize CTAs each (kernels_cluster.cu).
template <typename T>
cudaError_t launch_cluster(const ClusterArgs<T>& a, int batch, int threads, size_t smem, cudaStream_t s);
// How many such clusters the GPU holds at a time.
template <typename T>
int cluster_room(int csize, int threads, size_t smem);

// One pass kind over several shape groups (k_multi): `args` (device) holds
// each group's PassArgs (vgx, vgy its own launch shape), `start` (device,
// ngroups + 1 entries) the first block of each group; blocks = start[ngroups].
template <typename T>
cudaError_t launch_multi(int kind, int E, int blocks, int threads, size_t smem, cudaStream_t s,
                         const PassArgs<T>* args, const int* start, int ngroups);

template <typename T, int E>
cudaError_t launch_multi_e(int kind, int blocks, int threads, size_t smem, cudaStream_t s, const PassArgs<T>* args,
                           const int* start, int ngroups);

// Ends a deferred dot pass of `nblk` blocks per field and `batch` fields.
template <typename T>
cudaError_t launch_finish(const PassArgs<T>& a, int nblk, int batch, int threads, cudaStream_t s);

template <typename T>
cudaError_t launch_cg_finish(T* u, const T* p, const FieldState* st, long long P, int batch, cudaStream_t s);

cudaError_t launch_reset_state(FieldState* st, int batch, cudaStream_t s);

// Statistics (stats.cuh). X, U, W are half spectra of the field's precision.
template <typename T>
cudaError_t launch_shell(const void* X, int nx, int ny, int nz, long long SP, int batch, int ncomp, int nbins,
                         double scale, double* out, cudaStream_t s);
template <typename T>
cudaError_t launch_hist(const T* x, long long n, double lo, double scale, int nbins, unsigned long long* counts,
                        cudaStream_t s);
template <typename T>
cudaError_t launch_curl(const void* U, void* W, int nx, int ny, int nz, long long SP, int nvel, int ncomp,
                        cudaStream_t s);

}  // namespace gad
