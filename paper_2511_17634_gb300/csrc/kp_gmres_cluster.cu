// kp_gmres_cluster.cu -- the mixed-precision solver of
// kp_gmres_mixed_kernel.cuh with a thread-block cluster per system: grids too
// large for one SM (128x128 = 16384 unknowns), or any above 1024 points on
// request (kp_options.cluster_size).
#include "kp_gmres_mixed_kernel.cuh"

namespace kp {

cudaError_t launch_gmres_cluster(const GmresParams& p, int ept, int nt, int cs, bool reg, bool long_columns,
                                 size_t smem, cudaStream_t st) {
  if (long_columns) return reg ? cudaErrorInvalidValue : launch_gmres_cluster_long(p, ept, nt, cs, smem, st);
  if (ept == 16 && nt == 256) {                  // the default: 4096 points per CTA
    if (cs == 4) return reg ? launch_mx<16, 256, 4, mixed_reg_blocks(4), 2, true>(p, smem, st) : launch_mx<16, 256, 4, 2, 2, false>(p, smem, st);
    if (cs == 2) return reg ? launch_mx<16, 256, 2, mixed_reg_blocks(2), 2, true>(p, smem, st) : launch_mx<16, 256, 2, 2, 2, false>(p, smem, st);
  }
  if (ept == 8 && nt == 256) {                   // cluster_size 2, 4, 8: 2048 points per CTA
    if (cs == 8) return launch_mx<8, 256, 8, 2, 0, false>(p, smem, st);
    if (cs == 4) return launch_mx<8, 256, 4, 2, 0, false>(p, smem, st);
    if (cs == 2) return launch_mx<8, 256, 2, 2, 0, false>(p, smem, st);
  }
  if (ept == 8 && nt == 128 && cs == 16) return launch_mx<8, 128, 16, 4, 0, false>(p, smem, st);   // 1024 points per CTA
  return cudaErrorInvalidValue;
}

}  // namespace kp
