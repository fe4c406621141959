// Fused per-position pc-engine kernel in its cluster form, used by mini-batches and difference-map scans too
// small to fill the GPU with one CTA per position (every other launch runs the one-CTA-per-position kernel
// of pc_fused_seq.cuh): one cluster of K CTAs per scan position,
// CTA rank k owns probe mode k and rows [k R, (k + 1) R) of the detector
// (R = ceil(M / K)). Everything between the object gather and the per-position
// contributions stays on chip:
//
//   psi_k   = P_k o_n                                       (Eq. 1, Fig. 1)
//   Psi_k   = centred FFT2 (far field, checkerboard trick)  (Eq. 1)
//           | IFFT2(FFT2(psi_k) H)  (near field, Fresnel transfer function)
//   |Psi_k|^2 is pushed (DSMEM stores) to the rank owning its row; the owner
//   sums the K modes in rank order:  S = sum_k |Psi_k|^2
//   A^G     = sqrt(S) (x) g  (Eq. 6)  or  I_m = S (x) g (Eq. 2), separable and
//             zero padded, g of Eq. 7 normalised; each owner blurs its own
//             rows and receives the x-blurred halo rows it needs from the others
//   R       = sqrt(I_n) / (A^G + eps)   or   sqrt(I_n) / sqrt(I_m + eps^2)
//             (sqrt(I_n) precomputed once per plan; fast 2-ulp divide / rsqrt),
//             pushed by its owner to every rank
//   Psi'_k  = R Psi_k;  psi'_k = inverse propagation;  dpsi_k = psi'_k - psi_k
//   c_n     = sum_k conj(P_k) dpsi_k: pushed to the row owner, summed in rank
//             order, written once per position (the object update gathers it)
//   pacc    += conj(o_n) dpsi_k, dacc += |o_n|^2  (per-slot partials, no atomics)
//   error   : compensated FP32 per thread of sum (Ihat - I_n)^2 over own rows,
//             FP64 across threads, ranks and slots
//
// Persistent: cluster `slot` handles positions slot, slot + slots, ... so the
// per-slot partials are written in a fixed order and the iteration is
// bitwise reproducible. Five cluster barriers per position order the pushes.
#include <cuda_runtime.h>

#include "pc_fused_kernel.cuh"

namespace ptycho {

// Self-test of the bounded wait above (the one the cluster kernels use on their copy barriers):
// one thread waits for phase 0 of a fresh mbarrier with the given budget. With `signal` it arrives
// first and the wait succeeds at once; otherwise nothing ever arrives, the wait gives up after
// `budget_ns` and raises the flag that status-reading calls look at, exactly as a fused kernel does.
__global__ void k_wait_selftest(unsigned long long budget_ns, int signal, volatile int* flag) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x != 0) return;
  const uint32_t b = smem_addr(&bar);
  mbar_init(b, 1);
  if (signal) mbar_arrive_expect_tx(b, 0u);  // the one expected arrival, no transaction bytes
  if (!mbar_wait_bounded(b, 0u, budget_ns)) report_timeout(flag);
}

cudaError_t launch_wait_selftest(unsigned long long budget_ns, bool signal, volatile int* flag, cudaStream_t s) {
  k_wait_selftest<<<1, 32, 0, s>>>(budget_ns, signal ? 1 : 0, flag);
  return cudaGetLastError();
}

size_t fused_smem_bytes(int M) {
  switch (M) {
    case 8: return FusedSmem<8, 15>::BYTES;
    case 16: return FusedSmem<16, 15>::BYTES;
    case 32: return FusedSmem<32, 15>::BYTES;
    case 64: return FusedSmem<64, 15>::BYTES;
    case 128: return FusedSmem<128, 15>::BYTES;
    default: return 0;
  }
}

cudaError_t launch_fused_cluster(int M, const FusedArgs& a, int slots, cudaStream_t s) {
  return launch_cluster<SINGLE>(M, a, slots, s);
}
cudaError_t fused_cluster_max_slots(int M, int K, int* slots) { return cluster_slots<SINGLE>(M, K, slots); }

}  // namespace ptycho
