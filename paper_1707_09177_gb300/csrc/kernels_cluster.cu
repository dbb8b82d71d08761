// The cluster solve of small grids (cluster.cuh) for one precision (GAD_REAL).
#include "cluster.cuh"

namespace gad {

template <typename T>
static cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* at, int csize, int batch, int threads, size_t smem,
                                         cudaStream_t s) {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)csize * (unsigned)batch);
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)csize;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}

// The same limits for every launch: they are shared by all host threads.
template <typename T>
static cudaError_t cluster_attributes() {
  cudaError_t e = cudaFuncSetAttribute(k_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClusterSmem);
  return e;
}

template <typename T>
cudaError_t launch_cluster(const ClusterArgs<T>& a, int batch, int threads, size_t smem, cudaStream_t s) {
  cudaError_t e = cluster_attributes<T>();
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at{};
  const cudaLaunchConfig_t c = cluster_config<T>(&at, a.csize, batch, threads, smem, s);
  e = cudaLaunchKernelEx(&c, k_cluster<T>, a);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
int cluster_room(int csize, int threads, size_t smem) {
  int n = 0;
  cudaLaunchAttribute at{};
  const cudaLaunchConfig_t c = cluster_config<T>(&at, csize, 1, threads, smem, nullptr);
  const bool ok = cluster_attributes<T>() == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&n, k_cluster<T>, &c) == cudaSuccess && n > 0;
  if (!ok) cudaGetLastError();
  return ok ? n : 0;
}

template cudaError_t launch_cluster<GAD_REAL>(const ClusterArgs<GAD_REAL>&, int, int, size_t, cudaStream_t);
template int cluster_room<GAD_REAL>(int, int, size_t);

}  // namespace gad
