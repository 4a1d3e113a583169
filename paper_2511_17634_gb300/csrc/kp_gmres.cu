// kp_gmres.cu -- batched restarted GMRES(m) for the five-point Fokker-Planck
// systems of Sec. 2.3 (Eq. 11-13), FP64, one thread block per system: the
// lean instantiations of the kernel in kp_gmres_kernel.cuh, the operator /
// right-hand-side kernel, and the launch helpers of the march.
#include "kp_gmres_kernel.cuh"

namespace kp {
namespace {

// y = A x, b = m^{n-1}/dt - Div_h f or r = b - A x (launch_apply), 1024 points
// of one system per block.  Bound by the FP64 pipe (13 FP64 instructions per
// point of A x with a drift field, 2 lanes per clock and SM), so the constants
// come from the descriptor's quotients (four divisions a thread before), W and
// S coefficients from those of E and N, and the division by dt is a
// multiplication by 1/dt with one exact-remainder correction (Markstein 1990:
// correctly rounded for a correctly rounded 1/dt).  3072 systems of 64x64 with
// drift: A x 0.31 ms as before (87 % of the FP64 pipe), b - A x 0.61 -> 0.35 ms
// (one pass instead of two), b 0.31 -> 0.17 ms.
static __device__ __noinline__ double slow_div(double a, double b) { return a / b; }

template <int MODE>
__global__ void __launch_bounds__(256) apply_rhs_kernel(const SysDesc* sys, int chunks) {
  const SysDesc d = sys[blockIdx.x / chunks];
  const int H = d.H, W = d.W, N = H * W;
  const int p0 = (blockIdx.x % chunks) * 1024 + threadIdx.x;
  if (MODE == kRhs) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int pp = p0 + k * 256;
      if (pp >= N) return;
      const double v = d.b[pp];
      double q = v * d.kd;
      q = fma(fma(-q, d.dt, v), d.kd, q);
      // (an overflow or a NaN on the way: the division itself, out of line so
      // that its instructions are not speculated; tested on the bits)
      if ((__double2hiint(q) & 0x7FF00000) == 0x7FF00000) q = slow_div(v, d.dt);
      if (d.fx || d.fy) {
        const int i = pp / H, j = pp - i * H;
        const double fE = (d.fx && i + 1 < W) ? d.fx[pp + H] : 0.0;
        const double fW = (d.fx && i > 0) ? d.fx[pp - H] : 0.0;
        const double fN = (d.fy && j + 1 < H) ? d.fy[pp + 1] : 0.0;
        const double fS = (d.fy && j > 0) ? d.fy[pp - 1] : 0.0;
        q -= ((fE - fW) + (fN - fS)) * d.ki;
      }
      d.x[pp] = q;
    }
    return;
  }
  const double cc = d.g2 * d.kc, ee = 0.25 * cc, cd = fma(4.0, cc, d.kd), c2 = -2.0 * cc;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int pp = p0 + k * 256;
    if (pp >= N) return;
    const int i = pp / H, j = pp - i * H;
    const bool e = i + 1 < W, w = i > 0, n = j + 1 < H, s = j > 0;
    const double dmx = (e ? d.mt[pp + H] : 0.0) - (w ? d.mt[pp - H] : 0.0);
    const double dmy = (n ? d.mt[pp + 1] : 0.0) - (s ? d.mt[pp - 1] : 0.0);
    const double cE = fma(-ee, dmx, d.fx ? fma(d.fx[pp], d.ki, -cc) : -cc);
    const double cN = fma(-ee, dmy, d.fy ? fma(d.fy[pp], d.ki, -cc) : -cc);
    double y = cd * d.b[pp];
    if (e) y = fma(cE, d.b[pp + H], y);
    if (w) y = fma(c2 - cE, d.b[pp - H], y);
    if (n) y = fma(cN, d.b[pp + 1], y);
    if (s) y = fma(c2 - cN, d.b[pp - 1], y);
    d.x[pp] = MODE == kResidual ? d.score[pp] - y : y;
  }
}

}  // namespace

size_t gmres_fp64_smem_bytes(int ept, int nt, int S, int m) {
  const int npad = ept * nt;
  const size_t doubles = (size_t)S * npad + npad + (nt / 32) * kMaxV + kMaxV +
                         (size_t)(m + 1) * m + (m + 1) + 4 * m + 8;
  return doubles * sizeof(double) + 8 * sizeof(int);
}

cudaError_t launch_gmres_fp64(const GmresParams& p, int ept, int nt, int minb, size_t smem,
                              cudaStream_t st) {
  if (p.bicg && p.capV) return launch_gmres_fp64_bicg(p, ept, nt, minb, smem, st);
  const int nfeat = (p.score_stride != 0) + (p.dense_slots != 0) + (p.picard > 1);
  if (p.x0_mode == X0_GALERKIN || nfeat > 1) return launch_gmres_fp64_feat(p, ept, nt, minb, smem, st);
  if (p.picard > 1) return launch_gmres_fp64_picard(p, ept, nt, minb, smem, st);
  if (p.score_stride) return launch_gmres_fp64_score(p, ept, nt, minb, smem, st);
  if (p.dense_slots) return launch_gmres_fp64_dense(p, ept, nt, minb, smem, st);
  if (ept == 4 && nt == 256 && minb == 2) return launch_one<4, 256, 2, kVarLean>(p, smem, st);
  if (ept == 4 && nt == 256 && minb == 3) return launch_one<4, 256, 3, kVarLean>(p, smem, st);
  if (ept == 8 && nt == 128 && minb == 2) return launch_one<8, 128, 2, kVarLean>(p, smem, st);
  if (ept == 8 && nt == 128 && minb == 3) return launch_one<8, 128, 3, kVarLean>(p, smem, st);
  if (ept == 8 && nt == 128 && minb == 4) return launch_one<8, 128, 4, kVarLean>(p, smem, st);
  if (ept == 16 && nt == 64 && minb == 4) return launch_one<16, 64, 4, kVarLean>(p, smem, st);
  if (ept == 8 && nt == 512) return launch_one<8, 512, 1, kVarLean>(p, smem, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_gmres_fp64_1k_grid(const GmresParams& p, size_t smem, int grid,
                                      cudaStream_t st) {
  auto k = gmres_fp64_kernel<4, 256, 2, kVarLean>;
  cudaError_t e = allow_max_smem(k, smem);
  if (e != cudaSuccess) return e;
  k<<<grid, 256, smem, st>>>(p);
  return cudaGetLastError();
}

__global__ void advance_kernel(int* step, int by, int* zero, int nzero) {
  *step += by;
  for (int k = 0; zero && k < nzero; ++k) zero[k] = 0;
}

cudaError_t launch_advance(int* step, cudaStream_t st, int by, int* zero, int nzero) {
  advance_kernel<<<1, 1, 0, st>>>(step, by, zero, nzero);
  return cudaGetLastError();
}

int gmres_fp64_blocks_per_sm(int ept, int nt, int minb, size_t smem) {
  int n = 0;
  cudaError_t e = cudaErrorInvalidValue;
  auto occ = [&](auto k, int threads) {
    e = allow_max_smem(k, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem);
  };
  if (ept == 4 && nt == 256 && minb == 2) occ(gmres_fp64_kernel<4, 256, 2, kVarLean>, 256);
  else if (ept == 4 && nt == 256 && minb == 3) occ(gmres_fp64_kernel<4, 256, 3, kVarLean>, 256);
  else if (ept == 8 && nt == 128 && minb == 2) occ(gmres_fp64_kernel<8, 128, 2, kVarLean>, 128);
  else if (ept == 8 && nt == 128 && minb == 3) occ(gmres_fp64_kernel<8, 128, 3, kVarLean>, 128);
  else if (ept == 8 && nt == 128 && minb == 4) occ(gmres_fp64_kernel<8, 128, 4, kVarLean>, 128);
  else if (ept == 16 && nt == 64 && minb == 4) occ(gmres_fp64_kernel<16, 64, 4, kVarLean>, 64);
  else if (ept == 8 && nt == 512) occ(gmres_fp64_kernel<8, 512, 1, kVarLean>, 512);
  return e == cudaSuccess ? n : 0;
}

cudaError_t launch_apply(const SysDesc* sys, int nsys, int nmax, int mode, cudaStream_t st) {
  const int chunks = (nmax + 1023) / 1024;
  const unsigned grid = (unsigned)nsys * (unsigned)chunks;
  if (mode == kApply) apply_rhs_kernel<kApply><<<grid, 256, 0, st>>>(sys, chunks);
  else if (mode == kRhs) apply_rhs_kernel<kRhs><<<grid, 256, 0, st>>>(sys, chunks);
  else apply_rhs_kernel<kResidual><<<grid, 256, 0, st>>>(sys, chunks);
  return cudaGetLastError();
}

}  // namespace kp
