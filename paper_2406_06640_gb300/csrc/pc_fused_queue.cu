// Work-queue launches of the one-CTA-per-position kernel (pc_fused_seq.cuh): the chunks of several problems
// sharing M, K, geometry and kernel width class. One CTA per chunk needs no cluster barrier and keeps every
// SM busy for any K. Twelve problems of 64^2 to 256^2 in one plan: 5.84 -> 5.58 ms an iteration against a
// cluster of K CTAs per chunk (a third of it is the M <= 128 members' launches). Few positions run as clusters
// (pc_fused_queue_cluster.cu; cluster_form in capi.cu).
#include "pc_fused_seq.cuh"

namespace ptycho {

bool fused_queue_supported(int M) { return M == 8 || M == 16 || M == 32 || M == 64 || M == 128; }

cudaError_t launch_fused_queue(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  if (!a.probs || !a.chunks || !a.queue || a.nchunks < 0) return cudaErrorInvalidValue;
  return launch_seq<QUEUED>(M, a, slots, s);
}
cudaError_t fused_queue_max_slots(int M, int /*K*/, int* slots) { return seq_slots<QUEUED>(M, slots); }

}  // namespace ptycho
