// kp_gmres_mixed.cu -- the mixed-precision solver of kp_gmres_mixed_kernel.cuh
// with one CTA per system (grids of up to 4096 points).
#include <algorithm>

#include "kp_gmres_mixed_kernel.cuh"

namespace kp {

size_t gmres_mixed_smem_bytes(int nt, int cs, int hmax, int vld, int S, int m, int redv) {
  const size_t nw = nt / 32, f = sizeof(float), f2 = sizeof(float2);
  const size_t fixed = (4 * (size_t)m + 2) * f2 + nw * kMaxV * f2 + 4 * (redv > 0 ? redv : kRedV) * nw * cs * f + kMaxV * f +
                       8 * sizeof(int) + 4 * (size_t)hmax * f;
  const size_t hess = (size_t)m * (m + 1) / 2 * f2;
  // exact Galerkin lays its a x a FP64 matrix over the Hessenberg matrix and the slots
  return fixed + std::max(hess + (size_t)S * vld * f, cs == 1 ? (size_t)(m + 1) * m * sizeof(double) : 0);
}

cudaError_t launch_gmres_mixed(const GmresParams& p, int ept, int nt, bool reg, size_t smem, cudaStream_t st) {
  if (ept == 4 && nt == 256)
    return reg ? launch_mx<4, 256, 1, 4, 0, true>(p, smem, st) : launch_mx<4, 256, 1, 4, 0, false>(p, smem, st);
  if (ept == 8 && nt == 128) return launch_mx<8, 128, 1, 4, 0, false>(p, smem, st);
  if (ept == 16 && nt == 256)
    return reg ? launch_mx<16, 256, 1, mixed_reg_blocks(1), 1, true>(p, smem, st) : launch_mx<16, 256, 1, 2, 1, false>(p, smem, st);
  return cudaErrorInvalidValue;
}

}  // namespace kp
