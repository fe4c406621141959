// Work-queue launches of the cluster form (pc_fused_kernel.cuh): a cluster of K CTAs per work item, for classes
// with too few positions to fill the GPU with one CTA per item (pc_fused_queue.cu).
#include "pc_fused_kernel.cuh"

namespace ptycho {

cudaError_t launch_fused_queue_cluster(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  if (!a.probs || !a.chunks || !a.queue || a.nchunks < 0) return cudaErrorInvalidValue;
  return launch_cluster<QUEUED>(M, a, slots, s);
}
cudaError_t fused_queue_cluster_max_slots(int M, int K, int* slots) { return cluster_slots<QUEUED>(M, K, slots); }

}  // namespace ptycho
