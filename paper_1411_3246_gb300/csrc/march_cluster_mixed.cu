// Cluster forms of the mixed pipelined steps (march_cluster.cuh), and the choice between the forms.
#include "march_cluster.cuh"

namespace wake {

using StepClusters = ClusterForm<StepOf<PolMixed>, false>;

int cluster_max(int form, bool slab, bool step, int n1, int np, int cn) {
  if (form == kFormMixed) return StepClusters::max_clusters(slab, step, n1, np, cn);
  return form == kFormFP64 ? cluster_max_fp64(slab, step, n1, np, cn) : 0;
}
cudaError_t launch_march_cluster(int form, bool slab, const SimDesc *d, const int *order, int count, int n1, int np, int cn,
                                 cudaStream_t stream) {
  return form == kFormFP64 ? launch_march_cluster_fp64(slab, d, order, count, n1, np, cn, stream) : cudaErrorInvalidValue;
}
cudaError_t launch_step_cluster(int form, const PipeArgs &a, int cn, int clusters, cudaStream_t stream) {
  if (form == kFormFP64) return launch_step_cluster_fp64(a, cn, clusters, stream);
  PipeArgs arg = a;
  void *args[] = {&arg};
  return StepClusters::launch(a.d.slab != 0, true, a.d.nr + 1, a.d.np, cn, clusters, args, stream);
}

}  // namespace wake
