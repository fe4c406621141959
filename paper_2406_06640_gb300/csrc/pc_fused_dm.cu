// pc-DM launches of the one-CTA-per-position kernel (pc_fused_seq.cuh): the difference map of Thibault et
// al. with the pc intensity model in its modulus projection. Per position, the estimate P o_n goes
// through the FFT / blur path for the error E only, then the reflected waves chi = 2 P o_n - psi_n through
// the same path for the modulus ratio, and psi_n <- psi_n + Pi_F(chi) - P o_n (the exit-wave state lives in
// global memory). The overlap projection alternates: the object step of the single-problem path with
// dpsi = psi_n - P o_n, then (update.cu) the probe step from the new object and the state.
// Bound like the other modes by the transforms (4K - 1 per position against the cluster form's 3K plus
// eight cluster barriers): 900 positions of 128^2, four modes, 1.66 ms an iteration as clusters, 1.28 here.
// Few positions run as clusters (pc_fused_dm_cluster.cu; cluster_form in capi.cu).
#include "pc_fused_seq.cuh"

namespace ptycho {

cudaError_t launch_fused_dm(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  if (!a.psi) return cudaErrorInvalidValue;
  return launch_seq<DM>(M, a, slots, s);
}
cudaError_t fused_dm_max_slots(int M, int /*K*/, int* slots) { return seq_slots<DM>(M, slots); }

}  // namespace ptycho
