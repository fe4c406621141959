// Single-problem launches of the one-CTA-per-position kernel (pc_fused_seq.cuh).
#include "pc_fused_seq.cuh"

namespace ptycho {

cudaError_t launch_fused(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  return launch_seq<SINGLE>(M, a, slots, s);
}
cudaError_t fused_max_slots(int M, int /*K*/, int* slots) { return seq_slots<SINGLE>(M, slots); }

}  // namespace ptycho
