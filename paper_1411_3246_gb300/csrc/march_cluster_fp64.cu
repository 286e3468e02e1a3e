// Cluster forms of the FP64 march (march_cluster.cuh).
#include "march_cluster.cuh"

namespace wake {

int cluster_max_fp64(bool slab, bool step, int n1, int np, int cn) {
  return ClusterForm<PolFP64>::max_clusters(slab, step, n1, np, cn);
}
cudaError_t launch_march_cluster_fp64(bool slab, const SimDesc *d, const int *order, int count, int n1, int np, int cn,
                                      cudaStream_t stream) {
  void *args[] = {&d, &order};
  return ClusterForm<PolFP64>::launch(slab, false, n1, np, cn, count, args, stream);
}
cudaError_t launch_step_cluster_fp64(const PipeArgs &a, int cn, int clusters, cudaStream_t stream) {
  PipeArgs arg = a;
  void *args[] = {&arg};
  return ClusterForm<PolFP64>::launch(a.d.slab != 0, true, a.d.nr + 1, a.d.np, cn, clusters, args, stream);
}

}  // namespace wake
