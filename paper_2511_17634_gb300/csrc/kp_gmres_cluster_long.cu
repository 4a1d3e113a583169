// kp_gmres_cluster_long.cu -- the cluster solvers of kp_gmres_cluster.cu for
// long columns (LONG in kp_gmres_mixed_kernel.cuh).
#include "kp_gmres_mixed_kernel.cuh"

namespace kp {

cudaError_t launch_gmres_cluster_long(const GmresParams& p, int ept, int nt, int cs, size_t smem, cudaStream_t st) {
  if (ept == 16 && nt == 256) {
    if (cs == 4) return launch_mx<16, 256, 4, 2, 2, false, true>(p, smem, st);
    if (cs == 2) return launch_mx<16, 256, 2, 2, 2, false, true>(p, smem, st);
  }
  if (ept == 8 && nt == 256) {
    if (cs == 8) return launch_mx<8, 256, 8, 2, 0, false, true>(p, smem, st);
    if (cs == 4) return launch_mx<8, 256, 4, 2, 0, false, true>(p, smem, st);
    if (cs == 2) return launch_mx<8, 256, 2, 2, 0, false, true>(p, smem, st);
  }
  if (ept == 8 && nt == 128 && cs == 16) return launch_mx<8, 128, 16, 4, 0, false, true>(p, smem, st);
  return cudaErrorInvalidValue;
}

}  // namespace kp
