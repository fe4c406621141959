// pc-DM launches of the cluster form (pc_fused_kernel.cuh): a cluster of K CTAs per position, for scans too
// short to fill the GPU with one CTA per position (pc_fused_dm.cu describes the engine).
#include "pc_fused_kernel.cuh"

namespace ptycho {

cudaError_t launch_fused_dm_cluster(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  if (!a.psi) return cudaErrorInvalidValue;
  return launch_cluster<DM>(M, a, slots, s);
}
cudaError_t fused_dm_cluster_max_slots(int M, int K, int* slots) { return cluster_slots<DM>(M, K, slots); }

}  // namespace ptycho
