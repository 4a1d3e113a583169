// kp_gmres_mixed_kernel.cuh -- mixed-precision solver for the five-point
// systems of Sec. 2.3: iterative refinement around an FP32 restarted GMRES,
// one CTA per system (grids of up to 4096 points, kp_gmres_mixed.cu) or one
// thread-block cluster of CS CTAs per system (kp_gmres_cluster.cu), CTA r
// holding columns [r W/CS, (r+1) W/CS) of every vector (whole columns, so
// north/south neighbours stay local).
//
// Precision.  The Krylov work (stencil, Gram-Schmidt updates, normalisation)
// is FP32 on FP32 vectors.  The refinement's high-precision arithmetic -- the
// solution x, the operator coefficients and the true residual r = b - A x --
// and the small least-squares problem (Hessenberg matrix, Givens rotations,
// back substitution, the projection's triangular solve) are double-float
// (kp_dd.cuh: a pair of floats, about 48 bits).  Inner products of FP32
// vectors are summed in FP32 within a CTA and in double-float across CTAs.
// Outer loop: r = b - A x; inner GMRES(m) on A d = r in FP32 until the
// residual estimate drops by eta = 1e-5 (FP32 cannot resolve much more) or to
// half the outer target (kInnerFloor); x += d.  The outer loop stops on the
// true residual, so every returned solve meets ||b - A x|| <= tol ||b||.  The
// residual's error is a few units of 2^-44 times ||b||, far below every
// tolerance the solver is asked for (>= 1e-12).
//
// No FP64 instruction runs per step.  GB300 issues an FP64 warp instruction
// over 64 cycles of one scheduler, whether one lane or 32 take part, so a
// Givens step of some 60 FP64 instructions on one lane held up its CTA for
// about 2 us per Arnoldi step, and the FP64 pipe of that one scheduler was
// 75 % (64x64) to 86 % (128x128) busy: it bounded the kernel.  In
// double-float the same chain is about 0.2 us.
//
// Barriers.  A reduction's per-warp partials go to every CTA of the cluster
// (distributed shared memory); after one barrier every warp adds all of them
// itself, in the same order, so the coefficients need no second barrier and
// are bit-identical everywhere.  Warp 0 takes the Givens step beside its
// vector work; its stop flag is read at the barrier that v_{j+1} needs in any
// case.  Halos: every CTA keeps its neighbours' edge columns of each Krylov
// vector and of x.  Only w = A v_j crosses the cluster (its edge columns are
// pushed with the partials); v_{j+1} and x on the halo follow from the same
// coefficients by the same operations as in the neighbour, bit for bit.  That
// leaves one cluster barrier per Arnoldi step (without a second Gram-Schmidt
// pass) and one per residual.
//
// Memory.  Shared memory holds the first S Krylov vectors; the others, x and
// q_x, q_y (hi and lo) live in a device workspace per resident CTA (L2).
// During a residual the first three vector slots hold x (hi, lo) and r: the
// Krylov vectors are dead by then.  Resident CTAs (or clusters) claim system
// after system, the next one during the first residual of the one before, so
// neither the workspace nor the last wave grows with the number of systems.
// REG: full CTAs whose threads divide into columns; a thread's points then lie
// in one row, its neighbours at fixed offsets, and three CTAs of 4096 points
// share an SM (two in general), so that one system's barriers and serial work
// overlap the others' vector work.
//
// What bounds it is issue and latency: 45 % of the issue slots are used.  Eight
// timesteps of 3072 channels of 64x64 take 8.2 ms, four of 128x128 18.2 (with
// one CTA per SM, FP64 scalars and halos read across the cluster 16.5 and
// 38.8).  16 points a thread rather than 8 take 170 instead of 235 thousand
// instructions per system; the long loops stay rolled, since unrolled code of
// that length stalls on instruction fetch (10.2 ms against 8.9).  Systems of 30
// and more steps are bound by the Krylov vectors past the window (L2, or memory
// with many systems): 90 of 101x80 with g = 0.5 take 1.5 ms a timestep.
//
// The operator is applied from q_x = f_x/(2h) - e (m~_E - m~_W) and q_y per
// point:
//   A x = cd x_p - c (x_E + x_W + x_N + x_S) + q_x (x_E - x_W) + q_y (x_N - x_S)
// with out-of-grid neighbours zero -- algebraically the coefficients of the
// listing after Eq. 11.  The Arnoldi process runs on A - cd I (same Krylov
// space, H_A = H + cd I), which avoids the cancellation of the large
// diagonal in Gram-Schmidt -- in FP32 it would cost a digit per step.
#pragma once

#include <cooperative_groups.h>

#include "kp_dd.cuh"
#include "kp_internal.cuh"

namespace kp {
namespace {

// Values per reduction round: longer Gram-Schmidt sums take several rounds
// (and barriers), which keeps the partials of 64 warps within 4 KB (two sets).
// Clusters, whose barriers cost more, take as many more as the shared memory
// beside the Krylov window holds (GmresParams::red_v).
constexpr int kRedV = 8;

__device__ __forceinline__ float2 as_f2(dd x) { return make_float2(x.hi, x.lo); }
__device__ __forceinline__ dd as_dd(float2 x) { return {x.x, x.y}; }

// Warp reduce-scatter of 4 FP32 values per lane, each in NH parts: every lane
// ends with the warp sum of value lane >> 3 (NH = 1), or of part lane >> 4 of
// value (lane >> 2) & 3 (NH = 2).
template <int NH>
__device__ __forceinline__ float warp_reduce4f(float (&a)[NH][4], int lane) {
  if (NH == 2) {
    const bool up = lane & 16;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float send = up ? a[0][k] : a[NH - 1][k];
      const float keep = up ? a[NH - 1][k] : a[0][k];
      a[0][k] = keep + __shfl_xor_sync(kFull, send, 16);
    }
  }
  constexpr int o = NH == 2 ? 8 : 16;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool up = lane & o;
    const float send = up ? a[0][k] : a[0][k + 2];
    const float keep = up ? a[0][k + 2] : a[0][k];
    a[0][k] = keep + __shfl_xor_sync(kFull, send, o);
  }
  {
    const bool up = lane & (o / 2);
    const float send = up ? a[0][0] : a[0][1];
    const float keep = up ? a[0][1] : a[0][0];
    a[0][0] = keep + __shfl_xor_sync(kFull, send, o / 2);
  }
#pragma unroll
  for (int q = o / 4; q > 0; q /= 2) a[0][0] += __shfl_xor_sync(kFull, a[0][0], q);
  return a[0][0];
}

// alpha = R^{-1} (G c) in double-float by one warp (the double-float form of
// solve_projected_warp): c in shared memory, a <= 64, the FP64 factors split
// as they are loaded, eight columns of R ahead of their use.  alpha -> out
// (FP32).  Every lane of the warp calls it; ends with __syncwarp.
__device__ __forceinline__ void solve_projected_dd(float2* c, int a, int nrot, const double* R, int ld,
                                                   const double* rot, const double* rinv, float* out, int lane) {
  // rotations: lane l holds pairs l and l + 32, every lane follows the chain
  dd rc[2], rs[2], ri[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int l = lane + 32 * u;
    rc[u] = l < nrot ? dd_from_double(rot[2 * l]) : dd{1.f, 0.f};
    rs[u] = l < nrot ? dd_from_double(rot[2 * l + 1]) : dd{0.f, 0.f};
    ri[u] = l < a ? dd_from_double(rinv[l]) : dd{0.f, 0.f};
  }
  auto bcast = [&](const dd (&v)[2], int j) -> dd {
    const dd s = j < 32 ? v[0] : v[1];
    return {__shfl_sync(kFull, s.hi, j & 31), __shfl_sync(kFull, s.lo, j & 31)};
  };
  dd cur = as_dd(c[0]);
  dd g[2] = {{0.f, 0.f}, {0.f, 0.f}};
  auto put = [&](int j, dd v) {
    if (lane == (j & 31)) g[j >> 5] = v;
  };
  int j = 0;
  for (; j < nrot; ++j) {
    const dd cc = bcast(rc, j), s = bcast(rs, j), nx = as_dd(c[j + 1]);
    put(j, dd_add(dd_mul(cc, cur), dd_mul(s, nx)));
    cur = dd_sub(dd_mul(cc, nx), dd_mul(s, cur));
  }
  if (j < a) put(j, cur);
  for (++j; j < a; ++j) put(j, as_dd(c[j]));
  for (int i0 = a - 1; i0 >= 0; i0 -= 8) {
    double r0[8], r1[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 - u;
      r0[u] = (i >= 0 && lane < i) ? R[lane + (size_t)i * ld] : 0.0;
      r1[u] = (i >= 0 && lane + 32 < i) ? R[lane + 32 + (size_t)i * ld] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 - u;
      if (i < 0) break;
      const dd ai = dd_mul(bcast(g, i), bcast(ri, i));
      if (lane == 0) out[i] = ai.hi;
      if (lane < i) g[0] = dd_sub(g[0], dd_mul(dd_from_double(r0[u]), ai));
      if (lane + 32 < i) g[1] = dd_sub(g[1], dd_mul(dd_from_double(r1[u]), ai));
    }
  }
  __syncwarp();
}

// HALF: a thread's EPT points in two halves, each with its own FP32 sums, so
// that a sum has the bits of twice as many threads (HALF = 1: even and odd k)
// or CTAs (HALF = 2: the two halves of the slice) with EPT / 2 points each;
// 0: one chain.  REG: every system of the launch fills its CTAs (N = CS EPT
// NT) and its columns divide the CTA's threads, so that all of a thread's
// points share one row j: two neighbour flags per thread instead of four bits
// per point, no guards, and zero halo columns beside the grid (the launcher
// decides).  LONG (clusters, columns of more than half a block's threads): the
// halo columns of x and of every v are stored by the neighbour that has them,
// for one cluster barrier more per Arnoldi step; kept up here they would be
// 2 H more points per CTA (100 systems of 1024x16, warm: 9.0 -> 7.2 ms, 50 of
// 2048x8 20.4 -> 8.6).
template <int EPT, int NT, int CS, int MINB, int HALF, bool REG, bool LONG = false>
__global__ void __launch_bounds__(NT, MINB) gmres_mixed_kernel(const GmresParams p) {
  namespace cg = cooperative_groups;
  constexpr int NH = HALF ? 2 : 1;
  constexpr int NWS = NT / 32 * (HALF == 1 ? 2 : 1);   // warps (HALF 1: half-warps' worth) of FP32 partials
  constexpr int VC = CS * (HALF == 2 ? 2 : 1);   // blocks above them, added in double-float
  constexpr int P = NWS * VC;                    // partials of one value
  // four lanes add a value's partials: the lanes take blocks (VC >= 4), a
  // block bit and a warp bit (2), or two warp bits (1)
  constexpr int VL = VC >= 4 ? VC / 4 : 1;       // blocks in a lane
  constexpr int NWL = P / 4 / VL;                // warps of each in a lane
  constexpr bool HALO = CS > 1 || REG;
  extern __shared__ __align__(16) unsigned char smem_mx[];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = CS > 1 ? (int)cluster.block_rank() : 0;
  const int m = p.m;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // shared-memory carve (identical offsets in every CTA of the cluster);
  // gmres_mixed_smem_bytes counts the same pieces
  float2* cs = reinterpret_cast<float2*>(smem_mx);            // [m]
  float2* sn = cs + m;                                        // [m]
  float2* rinv = sn + m;                                      // [m]
  float2* gv = rinv + m;                                      // [m + 2]
  float2* hball = gv + m + 2;                                 // [NT / 32][kMaxV] sums, a copy per warp
  float2* hb = hball + warp * kMaxV;
  float* red = reinterpret_cast<float*>(hball + (NT / 32) * kMaxV);   // [2][redv][P]
  const int redv = CS > 1 ? p.red_v : kRedV;
  float* yf = red + 2 * redv * P;                             // [kMaxV] combination coefficients
  int* fl = reinterpret_cast<int*>(yf + kMaxV);               // [8]
  float* whalo = reinterpret_cast<float*>(fl + 8);            // [2][2 hmax] pushed edge columns (not LONG)
  float2* Hr = reinterpret_cast<float2*>(whalo + (LONG ? 0 : 4 * p.hmax)); // packed columns of R: j at j (j + 1) / 2
  float* V = reinterpret_cast<float*>(Hr + m * (m + 1) / 2);  // [S][vld]
  const int vld = p.vld;
  // workspace of this CTA: x (hi, lo) over the extended slice, q_x and q_y
  // (hi, lo each), then the Krylov vectors past the shared-memory window
  float2* xs = reinterpret_cast<float2*>(p.spill32 + (size_t)blockIdx.x * p.ws_ld);
  float4* qc = reinterpret_cast<float4*>(xs + vld + (vld & 1));
  float* Vg = reinterpret_cast<float*>(qc + EPT * NT);
  auto slot = [&](int i) -> float* {
    return i < p.S ? V + (size_t)i * vld : Vg + (size_t)(i - p.S) * vld;
  };
  int tstep = 0;
  if (p.step) {
    tstep = *p.step + p.step_offset;
    if (tstep >= *p.step_end) return;            // uniform over the whole grid
  }
  const int parity_base = slot_set_base(p, tstep);
  const float kEta = p.inner_eta > 0.0 ? (float)p.inner_eta : 1e-5f;
  int buf = 0, hbuf = 0;                         // parities of the reductions and of the halo pushes
  int geometry = -1, zeroed = 0;                 // slots whose space behind the halo is zero, for these slices

  // resident CTAs claim systems until none is left: the workspace is then as
  // large as the GPU holds CTAs and stays in L2 (a slice per system was 7 GB
  // written back to memory per timestep of 12288 systems of 128x128)
  // The next system is claimed while the current one's first residual runs and
  // reaches the cluster's CTAs with that residual's sums.
  auto tell_claim = [&](int sys) {
    if (CS > 1) {
#pragma unroll
      for (int r = 0; r < CS; ++r) *cluster.map_shared_rank(fl + 4, r) = sys;
    } else {
      fl[4] = sys;
    }
  };
  const bool claimer = rank == 0 && tid == 0;
  if (CS > 1) cluster.sync();                    // every CTA of the cluster runs
  if (claimer) tell_claim(atomicAdd(p.claim, 1));
  if (CS > 1) cluster.sync();
  else __syncthreads();
#pragma unroll 1
  for (;;) {
    const int sysi = fl[4];
    if (sysi >= p.nsys) break;                   // uniform over the cluster
    const SysDesc d = p.sys[sysi];
    const int H = d.H, W = d.W, N = H * W;
    const int SL = N / CS;                       // slice length (whole columns)
    const int SH = SL / 2;                       // its halves (HALF = 2)
    const int base = rank * SL;
    const int hal = HALO ? H : 0;                // halo columns before and after the slice
    // this thread's point k of the slice, whether it lies inside, its chain
    auto lp = [&](int k) { return !REG && HALF == 2 && k >= EPT / 2 ? SH + tid + (k - EPT / 2) * NT : tid + k * NT; };
    auto inside = [&](int k) { return REG || (HALF == 2 ? tid + (k % (EPT / 2)) * NT < SH : tid + k * NT < SL); };
    auto chain = [](int k) { return HALF == 1 ? k & 1 : HALF == 2 ? (k >= EPT / 2) : 0; };
    // points past the slice: w = 0 there.  On one CTA their slots hold zeros.
    // On a cluster that space is the halo's, so stores of short slices are
    // guarded; the sums and updates of Gram-Schmidt read it all the same (a
    // guard per point and vector doubled the instructions of a system of 30
    // steps: 101x80, 270 systems with g = 0.5, 4.73 -> 3.08 ms), which takes
    // finite values behind the halo too
    const bool full = REG || CS == 1 || SL == EPT * NT;
    auto zero_outside = [&](int n) {
      float* v = slot(n);
      for (int q = SL + 2 * H + tid; q < vld; q += NT) v[q] = 0.f;
      for (int q = tid; LONG && q < H; q += NT) {   // (LONG: nobody stores the halo outside the grid)
        if (rank == 0) v[q] = 0.f;
        if (rank == CS - 1) v[H + SL + q] = 0.f;
      }
    };
    if ((LONG || !full) && geometry != SL * 4096 + H) {   // (H <= 2048)
      geometry = SL * 4096 + H;
      zeroed = 0;
      for (; LONG && zeroed < 2; ++zeroed) zero_outside(zeroed);   // x
    }
    // the operator constants c = g^2/(2h^2), e = c/4, c_d = 1/dt + 4c from the
    // descriptor's quotients: a division is a dozen FP64 instructions on
    // every warp.  Solved as (A / s) x = b / s with s = 1/dt in a march, else 1:
    // the scale is in those quotients instead of on every point of b.
    const double g2 = p.step ? p.g2_sched[tstep] : d.g2;
    const double cc = g2 * d.kc;
    const dd ccd = dd_from_double(cc), cdd = dd_from_double(fma(4.0, cc, d.kd));
    const float ccf = ccd.lo + ccd.hi;
    const bool capture = p.capV32 != nullptr;
    const int cidx = p.factor ? parity_base + sysi : sysi;
    float* capV = capture ? p.capV32 + (size_t)cidx * (p.cap_a + 1) * p.cap_ld : nullptr;
    double* capH = capture ? p.capH + (size_t)cidx * (p.cap_a + 1) * p.cap_a : nullptr;

    // put(at, get(at, pp)) over this thread's points of the slice and of its
    // halo columns (at: index in a vector slot, pp: point of the grid or -1
    // outside), values read in groups ahead of their stores
    // (rolled: see the residual below)
    auto each_ext = [&](auto&& get, auto&& put) {
      constexpr int B = !REG ? 2 : EPT < 8 ? EPT : 8;
#pragma unroll 1
      for (int k0 = 0; k0 < EPT; k0 += B) {
        dd v[B];
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (inside(k0 + u)) v[u] = get(hal + lp(k0 + u), base + lp(k0 + u));
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (inside(k0 + u)) put(hal + lp(k0 + u), v[u]);
      }
      if (CS > 1 && !LONG)
        for (int q = tid; q < 2 * H; q += NT) {
          const int pp = q < H ? base - H + q : base + SL + q - H, at = q < H ? q : SL + q;
          put(at, get(at, (unsigned)pp < (unsigned)N ? pp : -1));
        }
    };
    // x (hi, lo) lives in the workspace and, outside the Krylov phases, in the
    // first two vector slots
    float* xh = V;
    float* xl = V + vld;
    // LONG: fn(r, at): point l of the slice is at index at of CTA r's halo
    auto to_neighbours = [&](int l, auto&& fn) {
      if (LONG && rank > 0 && l < H) fn(rank - 1, H + SL + l);
      if (LONG && rank + 1 < CS && l >= SL - H) fn(rank + 1, l - (SL - H));
    };
    auto put_x = [&](int at, dd v) {
      xh[at] = v.hi;
      xl[at] = v.lo;
      xs[at] = as_f2(v);
      to_neighbours(at - hal, [&](int r, int o) {
        float* n = cluster.map_shared_rank(V, r) + o;
        n[0] = v.hi;
        n[vld] = v.lo;
      });
    };
    auto sync_x = [&]() {                        // every CTA's reads or stores of x on the halo are done
      if (LONG) cluster.sync();
      else __syncthreads();
    };
    // x = u + yf-combination of the nc rows U (indexed by grid point)
    auto add_basis = [&](const float* U, int nc, bool from_zero) {
      each_ext([&](int at, int pp) -> dd {
        float xv = 0.f;
        if (pp >= 0)
          for (int i = 0; i < nc; ++i) xv = fmaf(yf[i], U[(size_t)i * p.slot_ld + pp], xv);
        return from_zero ? dd{xv, 0.f} : dd_add_f(dd{xh[at], xl[at]}, xv);
      }, put_x);
    };
    auto load_x = [&](const double* src) {
      each_ext([&](int, int pp) -> dd { return src && pp >= 0 ? dd_from_double(src[pp]) : dd{0.f, 0.f}; }, put_x);
    };
    // zero columns beside the grid, in the shared-memory slots (REG on one CTA)
    auto zero_halo = [&]() {
      if (REG && CS == 1)
        for (int q = tid; q < p.S * 2 * H; q += NT) {
          const int r = q / (2 * H), o = q - r * 2 * H;
          V[(size_t)r * vld + (o < H ? o : SL + o)] = 0.f;
        }
    };

    // neighbours of this thread's points: 1 E, 2 W, 4 N, 8 S per point (REG:
    // N and S of all its points).  With halo columns E and W are always there.
    unsigned long long msk = 0;
    if (REG) {
      const int j = tid % H;
      msk = (j + 1 < H ? 4u : 0u) | (j > 0 ? 8u : 0u);
    } else {
#pragma unroll
      for (int k = 0; k < EPT; ++k)
        if (inside(k)) {
          const int pp = base + lp(k);
          const int i = pp / H, j = pp - i * H;
          msk |= (unsigned long long)((CS > 1 || i + 1 < W ? 1u : 0u) | (CS > 1 || i > 0 ? 2u : 0u) |
                                      (j + 1 < H ? 4u : 0u) | (j > 0 ? 8u : 0u)) << (4 * k);
        }
    }
    const bool rN = msk & 4u, rS = msk & 8u;
    auto nb = [&](int k, unsigned bit) { return ((unsigned)(msk >> (4 * k)) & bit) != 0u; };
    auto nbE = [&](const float* v, int at, int k) { return REG || nb(k, 1u) ? v[at + H] : 0.f; };
    auto nbW = [&](const float* v, int at, int k) { return REG || nb(k, 2u) ? v[at - H] : 0.f; };
    auto nbN = [&](const float* v, int at, int k) {
      if (REG) { const float t = v[at + 1]; return rN ? t : 0.f; }
      return nb(k, 4u) ? v[at + 1] : 0.f;
    };
    auto nbS = [&](const float* v, int at, int k) {
      if (REG) { const float t = v[at - 1]; return rS ? t : 0.f; }
      return nb(k, 8u) ? v[at - 1] : 0.f;
    };

    // the lagged field, then q_x, q_y (hi parts in registers for the Krylov
    // operator, low parts in the workspace for the residual)
    if (CS > 1 && !LONG) {
      // (both buffers whole: nobody pushes the halo outside the grid, and a
      // system before this one may have had longer columns)
      for (int q = tid; q < 4 * p.hmax; q += NT) whalo[q] = 0.f;
    }
    zero_halo();
    load_x(d.mt);
    if (CS == 1) __syncthreads();
    else cluster.sync();                         // (every CTA's halo buffer is zero, and it has read its claim)
    int next_sys = 0;
    if (claimer) next_sys = atomicAdd(p.claim, 1);
    // (kA, kB): the pair u of this thread's points, one of each half where the
    // sums keep two chains
    auto kA = [](int u) { return HALF == 2 ? u : 2 * u; };
    auto kB = [](int u) { return HALF == 2 ? u + EPT / 2 : 2 * u + 1; };
    {
      const dd eed = {0.25f * ccd.hi, 0.25f * ccd.lo};
      const dd i2hd = dd_from_double(d.ki);
      auto coeff = [&](int k) -> float4 {
        const int at = hal + lp(k);
        const dd mE = {nbE(xh, at, k), nbE(xl, at, k)}, mW = {nbW(xh, at, k), nbW(xl, at, k)};
        const dd mN = {nbN(xh, at, k), nbN(xl, at, k)}, mS = {nbS(xh, at, k), nbS(xl, at, k)};
        dd x = dd_mul(eed, dd_sub(mW, mE)), y = dd_mul(eed, dd_sub(mS, mN));
        const int pp = base + lp(k);
        if (d.fx) x = dd_add(x, dd_mul(dd_from_double(d.fx[pp]), i2hd));
        if (d.fy) y = dd_add(y, dd_mul(dd_from_double(d.fy[pp]), i2hd));
        return make_float4(x.hi, x.lo, y.hi, y.lo);
      };
#pragma unroll 1
      for (int u = 0; u < EPT / 2; ++u) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = inside(kA(u)) ? coeff(kA(u)) : z, b = inside(kB(u)) ? coeff(kB(u)) : z;
        qc[tid + kA(u) * NT] = a;
        qc[tid + kB(u) * NT] = b;
      }
    }
    float qx[EPT], qy[EPT];                      // the hi parts, for the Krylov operator
#pragma unroll
    for (int k = 0; k < EPT; ++k) {
      const float4 q = qc[tid + k * NT];
      qx[k] = q.x;
      qy[k] = q.z;
    }

    float w[EPT];                                // r, then w = A v_j
    float bb[NH], sw[NH];                        // this thread's part of ||b||^2, of the warm start's ||r||^2
#pragma unroll
    for (int h = 0; h < NH; ++h) bb[h] = sw[h] = 0.f;
    auto sumsq = [&](float (&s)[NH]) {
#pragma unroll
      for (int h = 0; h < NH; ++h) s[h] = 0.f;
#pragma unroll
      for (int k = 0; k < EPT; ++k) s[chain(k)] = fmaf(w[k], w[k], s[chain(k)]);
    };
    // push this CTA's edge columns of w to the neighbours' halo buffers
    // (visible after the next cluster barrier)
    auto push_edges = [&]() {
      if (CS == 1 || LONG) return;
      float* wl = rank > 0 ? cluster.map_shared_rank(whalo, rank - 1) + hbuf * 2 * p.hmax + H : nullptr;
      float* wr = rank + 1 < CS ? cluster.map_shared_rank(whalo, rank + 1) + hbuf * 2 * p.hmax : nullptr;
#pragma unroll
      for (int k = 0; k < EPT; ++k) {
        const int l = lp(k);
        if (wl && inside(k) && l < H) wl[l] = w[k];
        if (wr && inside(k) && l >= SL - H) wr[l - (SL - H)] = w[k];
      }
    };
    // sums over the system of nv values -> hb[0..nv) of every warp of every
    // CTA, identical bits; part(i0, nv, a) gives this thread's chains of values
    // i0 .. i0 + 3.  Ends with __syncwarp.
    auto reduce = [&](int nv, auto&& part) {
      for (int c0 = 0; c0 < nv; c0 += redv) {
        const int nc = min(redv, nv - c0);
        float* rb = red + buf * redv * P;
#pragma unroll 1
        for (int i0 = 0; i0 < nc; i0 += 4) {
          float a[NH][4];
          part(c0 + i0, nv, a);
          const float s = warp_reduce4f<NH>(a, lane);
          // value v of this lane, one of the 8 / NH lanes that hold it, and
          // where the four adding lanes expect it
          const int v = i0 + (NH == 2 ? (lane >> 2) & 3 : lane >> 3), h = NH == 2 ? lane >> 4 : 0;
          const int r0 = NH == 2 ? lane & 3 : lane & 7;
          const int w = warp + (HALF == 1 ? h * (NT / 32) : 0), vc = HALF == 2 ? 2 * rank + h : rank;
          const int la = VC >= 4 ? vc & 3 : VC == 2 ? vc * 2 + (w & 1) : w & 3;
          const int wl = VC >= 4 ? w : VC == 2 ? w >> 1 : w >> 2;
          const int at = ((v * 4 + la) * VL + (VC >= 4 ? vc >> 2 : 0)) * NWL + wl;
          if (v < nc) {
            if (CS == 1) {
              if (r0 == 0) rb[at] = s;
            } else {
              for (int r = r0; r < CS; r += 8 / NH) cluster.map_shared_rank(rb, r)[at] = s;
            }
          }
        }
        if (CS == 1) __syncthreads();
        else cluster.sync();
#pragma unroll 1
        for (int i0 = 0; i0 < nc; i0 += 8) {
          const int i = i0 + (lane >> 2);
          float s = 0.f, e = 0.f;
          if (i < nc) {
            const float* f = rb + (i * 4 + (lane & 3)) * VL * NWL;
#pragma unroll
            for (int u = 0; u < VL; ++u) {
              float x[NWL];
#pragma unroll
              for (int n = 0; n < NWL; ++n) x[n] = f[u * NWL + n];
#pragma unroll
              for (int n = NWL / 2; n > 0; n /= 2)           // warps of a block: FP32
#pragma unroll
                for (int q = 0; q < n; ++q) x[q] += x[q + n];
              if (u == 0) {
                s = x[0];
              } else {
                const dd t = dd_two_sum(s, x[0]);
                s = t.hi;
                e += t.lo;
              }
            }
          }
          auto blocks = [&](int o) {                         // double-float butterfly
            const float so = __shfl_xor_sync(kFull, s, o), eo = __shfl_xor_sync(kFull, e, o);
            const dd t = dd_two_sum(s, so);
            s = t.hi;
            e = (e + eo) + t.lo;
          };
          if (VC >= 4) {
            blocks(2);
            blocks(1);
          } else if (VC == 2) {
            s += __shfl_xor_sync(kFull, s, 1);
            blocks(2);
          } else {
            s += __shfl_xor_sync(kFull, s, 2);
            s += __shfl_xor_sync(kFull, s, 1);
          }
          if ((lane & 3) == 0 && i < nc) hb[c0 + i] = VC > 1 ? as_f2(dd_fast_two_sum(s, e)) : make_float2(s, 0.f);
        }
        buf ^= 1;
      }
      __syncwarp();
    };

    // ---- initial guess
    const bool judge = p.x0_mode == X0_GUESS_PROJECT;
    unsigned long long proj_flops = 0;
    const int sl = d.slot + parity_base;         // the target's seed basis
    const float* U = p.slotV32 + (size_t)sl * (p.max_a + 1) * p.slot_ld;
    SlotMeta mt;
    mt.a = 0;
    if (judge || p.x0_mode == X0_PROJECT || p.x0_mode == X0_GALERKIN) {
      mt = p.slotMeta[sl];
      if (mt.timestep != tstep || mt.N != N) mt.a = 0;   // no basis: no projection
    }
    // x_init of a given guess: the learned guess m~ + dt rho net, from the
    // network's FP32 output, in double-float, or x as it is
    auto load_guess = [&]() {
      if (p.gdelta) {
        const float sg = (float)(p.grho[sysi] * p.gmul);
        const float* dl = p.gdelta + (size_t)sysi * p.gdelta_ld;
        each_ext([&](int, int pp) -> dd {
          return pp >= 0 ? dd_add_f(dd_from_double(d.mt[pp]), sg * dl[pp]) : dd{0.f, 0.f};
        }, put_x);
      } else {
        load_x(d.x);
      }
    };
    if (p.x0_mode != X0_WARM && !judge) {
      sync_x();                                  // every read of the lagged field in the slots is done
      if (p.x0_mode == X0_READ) load_guess();
      else load_x(nullptr);
    }
    if (CS == 1 && p.x0_mode == X0_GALERKIN && p.gram) {
      // Sec. 3, Phase 2 without the seed-matrix shortcut: G alpha = V_a^T b
      // with G = V_a^T A_i V_a of this target's own operator, assembled from
      // the seed basis part G0 and this target's tensor-core part (kp_gram.cu),
      // x0 = V_a alpha; c = V^T b from the projection GEMM.  G (FP64) takes
      // the space of the Hessenberg matrix and the vector slots.
      const int a = mt.a, A = p.gram_a;
      if (a > 0 && a <= A && a * a <= (m + 1) * m && p.cproj) {
        const float* g0 = p.gram0 + (size_t)sl * A * A;
        const float* gi = p.gram + (size_t)sysi * A * A;
        double* G = reinterpret_cast<double*>(Hr);               // a x a, column-major: G[l + k a] = v_l^T A v_k
        double* cv = reinterpret_cast<double*>(hball);
        __syncthreads();                         // the zeroed slots are written
        for (int e = tid; e < a * a; e += NT) {
          const int l = e % a, k = e / a;
          G[e] = (double)g0[l * A + k] + (double)gi[l * A + k];
        }
        if (tid < a) cv[tid] = (double)p.cproj[(size_t)sysi * p.cproj_ld + tid];
        __syncthreads();
        if (warp == 0) {
          const bool ok = lu_solve_warp(G, a, cv, lane);
          for (int i = lane; i < a; i += 32) yf[i] = ok ? (float)cv[i] : 0.f;
        }
        __syncthreads();
        zero_halo();
        add_basis(U, a, true);
        proj_flops = (unsigned long long)(2 * a) * (unsigned long long)N;
      }
    }

    // ---- refinement.  One loop body serves the judge's two residuals, the
    // projection's right-hand side and the residual of every outer step, so
    // that the unrolled stencil exists once (the kernel is sensitive to the
    // size of its code: instruction fetch was its first stall).
    enum { kWarm, kGuess, kProject, kSolve };
    int phase = judge ? kWarm : p.x0_mode == X0_PROJECT && mt.a > 0 ? kProject : kSolve;
    bool first_norm = true;
    dd bnorm = {0.f, 0.f}, rnorm = {0.f, 0.f};   // ||b||, ||r||
    float tolb = 0.f;
    int steps = 0, status = KP_NOT_CONVERGED, outer = 0;
    // power of two that brings the diagonal of H_A to [1, 2): the squares of
    // the least-squares problem then stay inside the FP32 range for any dt
    const unsigned cde = (__float_as_uint(cdd.hi) >> 23) & 255u;
    const float hsc = (cde > 0 && cde < 254) ? __uint_as_float((254u - cde) << 23) : 1.f;
#pragma unroll 1
    for (;;) {
      sync_x();                                  // x complete for the stencil
      const bool no_x = phase == kProject || (p.x0_mode == X0_ZERO && outer == 0);
      // r = b - A x in double-float: the hi parts of the terms are added by
      // TwoSum and all low parts and errors in FP32; the FP32 value of r,
      // which is all the Krylov process and the norms need, goes through the
      // third vector slot to w (no_x: r = b).  The loop is rolled, two points
      // at a time with the next ones' b and q on their way: unrolled over a
      // thread's points, this and the loops above were 70 KB of straight code
      // and instruction fetch was the kernel's first stall (4.3 of 12 cycles
      // between two instructions of a warp).
      {
        float* rs = V + 2 * vld + hal;
        auto mul = [](float ah, float al, float bh, float bl) -> dd {   // a b, unnormalised
          const float t = __fmul_rn(ah, bh);
          return {t, fmaf(al, bh, fmaf(ah, bl, fmaf(ah, bh, -t)))};
        };
        auto point = [&](int k, double bv, float4 q, float& sum) -> float {
          const dd b = dd_from_double(bv);
          sum = fmaf(b.hi, b.hi, sum);
          if (no_x) return b.hi;
          const int at = hal + lp(k);
          const dd x = {xh[at], xl[at]};
          const dd xE = {nbE(xh, at, k), nbE(xl, at, k)}, xW = {nbW(xh, at, k), nbW(xl, at, k)};
          const dd xN = {nbN(xh, at, k), nbN(xl, at, k)}, xS = {nbS(xh, at, k), nbS(xl, at, k)};
          const dd s1 = dd_two_sum(xE.hi, xW.hi), s2 = dd_two_sum(xN.hi, xS.hi), s = dd_two_sum(s1.hi, s2.hi);
          const float sl_ = ((xE.lo + xW.lo) + (xN.lo + xS.lo)) + ((s1.lo + s2.lo) + s.lo);
          const dd dx = dd_two_sum(xE.hi, -xW.hi), dy = dd_two_sum(xN.hi, -xS.hi);
          const float dxl = dx.lo + (xE.lo - xW.lo), dyl = dy.lo + (xN.lo - xS.lo);
          const dd t1 = mul(cdd.hi, cdd.lo, x.hi, x.lo), t2 = mul(ccd.hi, ccd.lo, s.hi, sl_);
          const dd t3 = mul(q.x, q.y, dx.hi, dxl), t4 = mul(q.z, q.w, dy.hi, dyl);
          const dd a1 = dd_two_sum(b.hi, -t1.hi), a2 = dd_two_sum(a1.hi, t2.hi);
          const dd a3 = dd_two_sum(a2.hi, -t3.hi), a4 = dd_two_sum(a3.hi, -t4.hi);
          return a4.hi + (((b.lo - t1.lo) + (t2.lo - t3.lo)) + ((a1.lo + a2.lo) + (a3.lo + a4.lo)) - t4.lo);
        };
        float sA = 0.f, sB = 0.f;
        double bA = 0.0, bB = 0.0;
        float4 qA, qB;
        auto fetch = [&](int u) {
          if (inside(kA(u))) { bA = d.b[base + lp(kA(u))]; qA = qc[tid + kA(u) * NT]; }
          if (inside(kB(u))) { bB = d.b[base + lp(kB(u))]; qB = qc[tid + kB(u) * NT]; }
        };
        fetch(0);
#pragma unroll 1
        for (int u = 0; u < EPT / 2; ++u) {
          const double cA = bA, cB = bB;
          const float4 eA = qA, eB = qB;
          if (u + 1 < EPT / 2) fetch(u + 1);
          const float r0 = inside(kA(u)) ? point(kA(u), cA, eA, sA) : 0.f;
          const float r1 = inside(kB(u)) ? point(kB(u), cB, eB, HALF ? sB : sA) : 0.f;
          if (full || inside(kA(u))) rs[lp(kA(u))] = r0;
          if (full || inside(kB(u))) rs[lp(kB(u))] = r1;
        }
        bb[0] = sA;
        if (HALF) bb[NH - 1] = sB;
#pragma unroll
        for (int k = 0; k < EPT; ++k) w[k] = full || inside(k) ? rs[lp(k)] : 0.f;
      }
      if (phase == kWarm) {
        sumsq(sw);
        sync_x();                                // every read of the warm start in the slots is done
        load_guess();
        phase = kGuess;
        continue;
      }
      bool project = phase == kProject;
      if (!project) {
        if (claimer && first_norm) tell_claim(next_sys);
        push_edges();
        reduce(first_norm ? 3 : 1, [&](int, int, float (&a)[NH][4]) {
          float s[NH];
          sumsq(s);
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            a[h][0] = s[h];
            a[h][1] = bb[h];
            a[h][2] = sw[h];
            a[h][3] = 0.f;
          }
        });
        if (phase == kGuess) {
          // the judge of a given guess (the learned one): its true residual
          // against the warm start's; a kept guess is projected, the warm
          // start (the fallback) starts unprojected, as in the warm mode
          proj_flops = 26ull * (unsigned long long)N;
          phase = kSolve;
          if (hb[2].x < hb[0].x || (hb[2].x == hb[0].x && hb[2].y < hb[0].y)) {
            load_x(d.mt);
            continue;
          }
          project = mt.a > 0;
        }
      }
      if (project) {
        // Sec. 3, Phase 2 with the seed's FP32 basis: c = V^T w for w = b (the
        // paper) or the residual of the guess (tensor-core GEMM, or FP32
        // products and sums here), alpha = H_a^{-1} c, x0 = x_init + V alpha
        const int a = mt.a;
        const int nv = mt.lsq ? a + 1 : a;
        if (phase == kProject && p.cproj) {
          if (warp == 0) {
            for (int i = lane; i < nv; i += 32) hb[i] = make_float2(p.cproj[(size_t)sysi * p.cproj_ld + i], 0.f);
            __syncwarp();
          }
        } else {
          reduce(nv, [&](int i0, int n, float (&s)[NH][4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
              for (int h = 0; h < NH; ++h) s[h][u] = 0.f;
              if (i0 + u < n) {
                const float* ui = U + (size_t)(i0 + u) * p.slot_ld + base;
#pragma unroll
                for (int k = 0; k < EPT; ++k)
                  if (inside(k)) s[chain(k)][u] = fmaf(ui[lp(k)], w[k], s[chain(k)][u]);
              }
            }
          });
        }
        if (warp == 0) {
          const double* rot = p.slotRot + (size_t)sl * 3 * p.max_a;
          solve_projected_dd(hb, a, mt.nrot, p.slotR + (size_t)sl * (p.max_a + 1) * p.max_a, p.max_a + 1, rot,
                             rot + 2 * p.max_a, yf, lane);
        }
        __syncthreads();
        add_basis(U, a, phase == kProject);
        proj_flops += (unsigned long long)(2 * nv + 2 * a) * (unsigned long long)N;
        phase = kSolve;
        continue;
      }
      rnorm = dd_sqrt(as_dd(hb[0]));
      if (first_norm) {
        first_norm = false;
        bnorm = dd_sqrt(as_dd(hb[1]));
        tolb = __fmul_rd(__double2float_rd(p.tol), bnorm.hi);   // rounded down
        if (bnorm.hi == 0.f) {
          load_x(nullptr);
          rnorm = bnorm;
          status = KP_OK;
          break;
        }
      }
      const float beta = rnorm.hi;
      // (before the tolerance: an infinite ||b|| is above everything)
      if (!isfinite(beta) || !isfinite(bnorm.hi)) { status = KP_BREAKDOWN; break; }
      // ||r|| <= tol ||b||: by the FP32 values, or in double-float where they
      // are too close (with a margin above its rounding), so that the rel_res
      // of a converged system is not above tol
      bool met = beta <= tolb * (1.f - 0x1p-20f);
      if (!met && beta <= tolb * (1.f + 0x1p-20f)) {
        const dd t = dd_mul(dd_from_double(p.tol), bnorm);
        met = (t.hi - rnorm.hi) + (t.lo - rnorm.lo) >= t.hi * 0x1p-40f;
      }
      if (met) { status = KP_OK; break; }
      if (steps >= p.maxit || outer >= 64) break;
      const bool first = (outer == 0);
      // the seed's captured cycle runs to the seed tolerance, so its basis has
      // the dimension the FP64 method would keep (Sec. 3, Phase 1)
      const float target = (capture && first) ? tolb : fmaxf(kEta * beta, (float)kInnerFloor * tolb);

      // ---- inner FP32 GMRES(m) on A d = r, from d = 0.  v_n = w scale, kept
      // as the next Krylov vector (and captured for the seed basis)
      auto next_vector = [&](int n, float scale) {
        float* vn = slot(n);
        const bool keep = capture && first && n <= p.cap_a;
#pragma unroll
        for (int k = 0; k < EPT; ++k) {
          const int l = lp(k);
          const float v = w[k] * scale;
          if (full || inside(k)) vn[hal + l] = v;
          if (LONG && inside(k))
            to_neighbours(l, [&](int r, int o) {
              (n < p.S ? cluster.map_shared_rank(vn, r) : vn + (r - rank) * (long long)p.ws_ld)[o] = v;
            });
          if (keep && inside(k)) {
            capV[(size_t)n * p.cap_ld + base + l] = v;
            if (p.capVb && n < kVbRows)
              p.capVb[((size_t)cidx * kVbRows + n) * p.capVb_ld + base + l] = __float2bfloat16_rn(v);
          }
        }
        if ((LONG || !full) && n >= zeroed) {    // (vectors come in order)
          zero_outside(n);
          zeroed = n + 1;
        }
        if (CS > 1 && !LONG) {
          const float* wh = whalo + hbuf * 2 * p.hmax;
          for (int q = tid; q < 2 * H; q += NT) vn[q < H ? q : SL + q] = wh[q] * scale;
        } else if (REG && n >= p.S) {
          for (int q = tid; q < 2 * H; q += NT) vn[q < H ? q : SL + q] = 0.f;
        }
      };
      next_vector(0, 1.f / beta);
      hbuf ^= 1;
      int kdone = 0, brk = 0;
      dd gcur = rnorm;                           // running right-hand side (warp 0)
#pragma unroll 1
      for (int j = 0; j < m; ++j) {
        // v_j complete (own slice and halo; LONG: by the barrier that ends a step)
        if (!LONG) __syncthreads();
        else if (j == 0) cluster.sync();
        {
          auto apply = [&](const float* v) {
#pragma unroll
            for (int k = 0; k < EPT; ++k) {
              const int at = hal + lp(k);
              float xE = 0.f, xW = 0.f, xN = 0.f, xS = 0.f;
              if (full || inside(k)) {
                xE = nbE(v, at, k);
                xW = nbW(v, at, k);
                xN = nbN(v, at, k);
                xS = nbS(v, at, k);
              }
              w[k] = -ccf * (xE + xW + xN + xS) + qx[k] * (xE - xW) + qy[k] * (xN - xS);
            }
          };
          if (j < p.S) apply(V + (size_t)j * vld);
          else apply(Vg + (size_t)(j - p.S) * vld);
        }
        push_edges();
        ++steps;
        const int nh = j + 1;
        float2* col = Hr + j * (j + 1) / 2;      // column j of the Hessenberg matrix (warp 0)
        float ww0 = 0.f;
        dd hn2 = {0.f, 0.f};                     // ||w||^2 after Gram-Schmidt
        // Gram-Schmidt: pass 0; pass 1 (re-orthogonalisation) always or, with
        // reorth, when the first removed more than half of ||w||^2; pass 2
        // only measures the norm, after a large correction in pass 1
#pragma unroll 1
        for (int pass = 0;; ++pass) {
          reduce(nh + 1, [&](int i0, int n, float (&s)[NH][4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
#pragma unroll
              for (int h = 0; h < NH; ++h) s[h][u] = 0.f;
              const int i = i0 + u;
              if (i < n - 1) {
                auto dot = [&](const float* vi) {
#pragma unroll
                  for (int k = 0; k < EPT; ++k) s[chain(k)][u] = fmaf(vi[lp(k)], w[k], s[chain(k)][u]);   // (w = 0 outside)
                };
                if (i < p.S) dot(V + (size_t)i * vld + hal);
                else dot(Vg + (size_t)(i - p.S) * vld + hal);
              } else if (i == n - 1) {
                float q[NH];
                sumsq(q);
#pragma unroll
                for (int h = 0; h < NH; ++h) s[h][u] = q[h];
              }
            }
          });
          const dd ww = as_dd(hb[nh]);
          if (pass == 2) { hn2 = ww; break; }
          float sqh = 0.f, sql = 0.f;            // sum of the squared coefficients
          for (int i = 0; i < nh; ++i) {
            const float2 h = hb[i];
            const float t = __fmul_rn(h.x, h.x);
            const dd a = dd_two_sum(sqh, t);
            sqh = a.hi;
            sql += a.lo + fmaf(2.f * h.x, h.y, fmaf(h.x, h.x, -t));
          }
          const dd sq = dd_fast_two_sum(sqh, sql);
          hn2 = dd_sub(ww, sq);
          if (warp == 0)
            for (int i = lane; i < nh; i += 32) col[i] = pass ? as_f2(dd_add(as_dd(col[i]), as_dd(hb[i]))) : hb[i];
          // w -= sum h_i v_i on the slice and on the halo.  A thread's first
          // halo point goes along with its points of the slice, the others of
          // long columns several at a time: in a loop of its own each waited a
          // latency per vector (L2 past the window; 128x128, 300 systems, warm:
          // 1126 -> 1097 us, 2048x8 36.6 -> 22.7 ms)
          float* wh = whalo + hbuf * 2 * p.hmax;
          const bool hq = CS > 1 && !LONG && tid < 2 * H;
          float hv = hq ? wh[tid] : 0.f;
#pragma unroll 1
          for (int i = 0; i < nh; ++i) {
            const float hi = hb[i].x;
            auto sub_ = [&](const float* vi) {
#pragma unroll
              for (int k = 0; k < EPT; ++k) w[k] = fmaf(-hi, vi[hal + lp(k)], w[k]);
              if (hq) hv = fmaf(-hi, vi[tid < H ? tid : SL + tid], hv);
            };
            if (i < p.S) sub_(V + (size_t)i * vld);
            else sub_(Vg + (size_t)(i - p.S) * vld);
          }
          if (!full)
#pragma unroll
            for (int k = 0; k < EPT; ++k) w[k] = inside(k) ? w[k] : 0.f;
          if (hq) wh[tid] = hv;
          if (CS > 1 && !LONG) {
            constexpr int B = REG ? 1 : 8;       // (REG: H <= NT)
#pragma unroll 1
            for (int q0 = tid + NT; q0 < 2 * H; q0 += B * NT) {
              float v[B];
#pragma unroll
              for (int u = 0; u < B; ++u) v[u] = q0 + u * NT < 2 * H ? wh[q0 + u * NT] : 0.f;
#pragma unroll 1
              for (int i = 0; i < nh; ++i) {
                const float hi = hb[i].x;
                const float* vi = slot(i);
#pragma unroll
                for (int u = 0; u < B; ++u) {
                  const int q = q0 + u * NT;
                  if (q < 2 * H) v[u] = fmaf(-hi, vi[q < H ? q : SL + q], v[u]);
                }
              }
#pragma unroll
              for (int u = 0; u < B; ++u)
                if (q0 + u * NT < 2 * H) wh[q0 + u * NT] = v[u];
            }
          }
          if (pass == 0) {
            ww0 = ww.hi;
            if (p.reorth != 0 && hn2.hi >= 0.5f * ww0) break;
          } else if (sq.hi <= 0.25f * ww.hi) {
            break;
          }
        }
        const dd ihn = hn2.hi > 0.f ? dd_rsqrt(hn2) : dd{0.f, 0.f};
        brk = !(hn2.hi > 1e-14f * ww0);          // h_{j+1,j} <= 1e-7 ||w_0||: breakdown at FP32 level
        if (!brk) next_vector(j + 1, ihn.hi);
        hbuf ^= 1;
        if (warp == 0) {
          // Givens step of column j (every lane; lane 0 stores): rotations,
          // residual estimate, stop flag
          __syncwarp();
          const dd hn = dd_mul(hn2, ihn);
          auto entry = [&](int i) -> dd { return i == j ? dd_add(as_dd(col[i]), cdd) : as_dd(col[i]); };   // H_A = H + cd I
          if (capture && first && j < p.cap_a && rank == 0)
            for (int i = lane; i <= j + 1; i += 32) capH[i + j * (p.cap_a + 1)] = dd_to_double(i <= j ? entry(i) : hn);
          auto scaled = [&](dd v) -> dd { return {v.hi * hsc, v.lo * hsc}; };
          dd cur = scaled(entry(0));
          for (int i = 0; i < j; ++i) {
            const dd c = as_dd(cs[i]), s = as_dd(sn[i]), nx = scaled(entry(i + 1));
            const dd top = dd_add(dd_mul(c, cur), dd_mul(s, nx));
            cur = dd_sub(dd_mul(c, nx), dd_mul(s, cur));
            __syncwarp();
            if (lane == 0) col[i] = as_f2(top);
          }
          const dd hs = scaled(hn);
          const dd rr = dd_add(dd_mul(cur, cur), dd_mul(hs, hs));
          const dd ir = dd_rsqrt(rr);
          const dd c = dd_mul(cur, ir), s = dd_mul(hs, ir);
          const dd gj = dd_mul(c, gcur);
          gcur = dd_mul(dd{-s.hi, -s.lo}, gcur);
          __syncwarp();
          if (lane == 0) {
            cs[j] = as_f2(c);
            sn[j] = as_f2(s);
            col[j] = as_f2(dd_mul(rr, ir));
            rinv[j] = as_f2(ir);
            gv[j] = as_f2(gj);
            // fixed basis dimension: the seed's captured cycle reaches cap_a
            // steps before the residual test may end it
            const bool short_of_a = p.fixed_a && capture && first && j + 1 < p.cap_a;
            fl[0] = (fabsf(gcur.hi) <= target && !short_of_a) || brk || (steps >= p.maxit) || (j + 1 == m);
          }
          __syncwarp();
        }
        kdone = j + 1;
        sync_x();
        if (fl[0]) break;
      }
      // y = R^{-1} g: column-oriented back substitution on warp 0 (lane l
      // owns rows l and l + 32), reciprocal pivots from the Givens steps
      if (warp == 0) {
        dd g0 = lane < kdone ? as_dd(gv[lane]) : dd{0.f, 0.f};
        dd g1 = lane + 32 < kdone ? as_dd(gv[lane + 32]) : dd{0.f, 0.f};
        for (int i = kdone - 1; i >= 0; --i) {
          const dd s = i < 32 ? g0 : g1;
          const dd gi = {__shfl_sync(kFull, s.hi, i & 31), __shfl_sync(kFull, s.lo, i & 31)};
          const dd yi = dd_mul(gi, as_dd(rinv[i]));
          if (lane == 0) yf[i] = yi.hi * hsc;    // (R was scaled by hsc)
          const float2* col = Hr + i * (i + 1) / 2;
          if (lane < i) g0 = dd_sub(g0, dd_mul(as_dd(col[lane]), yi));
          if (lane + 32 < i) g1 = dd_sub(g1, dd_mul(as_dd(col[lane + 32]), yi));
        }
      }
      if (warp == 0 && rank == 0 && capture && first) {
        const int a = kdone < p.cap_a ? kdone : p.cap_a;
        const int hn = (a < kdone) || !brk;
        double* rot = p.capRot + (size_t)cidx * 3 * p.cap_a;
        const double us = 1.0 / (double)hsc;     // (a power of two: exact)
        int lsq, nrot;
        store_factors(a, hn, capH, p.cap_a + 1, [&](int i, int j) { return dd_to_double(as_dd(Hr[j * (j + 1) / 2 + i])) * us; },
                      [&](int j) { return dd_to_double(as_dd(cs[j])); }, [&](int j) { return dd_to_double(as_dd(sn[j])); },
                      [&](int j) { return dd_to_double(as_dd(rinv[j])) * (double)hsc; },
                      p.capR + (size_t)cidx * (p.cap_a + 1) * p.cap_a, p.cap_a + 1, rot, rot + 2 * p.cap_a, &lsq, &nrot,
                      kDdPivot, lane);
        if (lane == 0) {
          if (p.factor) {
            SlotMeta sm;
            sm.a = a;
            sm.has_next = hn;
            sm.timestep = tstep;
            sm.N = N;
            sm.lsq = lsq;
            sm.nrot = nrot;
            sm.dense = sm.pad_ = 0;
            p.slotMeta[cidx] = sm;
          } else {
            p.capMeta[sysi].a = a;
            p.capMeta[sysi].has_next = hn;
            p.capMeta[sysi].N = N;
            p.capMeta[sysi].valid = 1;
            p.capMeta[sysi].lsq = lsq;
            p.capMeta[sysi].nrot = nrot;
          }
        }
      }
      __syncthreads();
      // d = V y in FP32, x += d in double-float; x goes to the first two slots
      // (each thread has read its own points of every vector by then)
      each_ext([&](int at, int) -> dd {
        const dd x = as_dd(xs[at]);
        float dv = 0.f;
        for (int i = 0; i < kdone; ++i) dv = fmaf(yf[i], slot(i)[at], dv);
        return dd_add_f(x, dv);
      }, put_x);
      ++outer;
    }
    if (capture && outer == 0 && tid == 0 && rank == 0) {
      if (p.factor) {
        SlotMeta sm;
        sm.a = 0; sm.has_next = 0; sm.timestep = tstep; sm.N = N; sm.lsq = 0; sm.nrot = 0;
        sm.dense = sm.pad_ = 0;
        p.slotMeta[cidx] = sm;
      } else {
        p.capMeta[sysi].a = 0;
        p.capMeta[sysi].has_next = 0;
        p.capMeta[sysi].N = N;
        p.capMeta[sysi].valid = 1;
        p.capMeta[sysi].lsq = p.capMeta[sysi].nrot = 0;
      }
    }
    // (the loop ends with x in the first two slots: every exit follows a
    // residual of x, or x0 = 0 put there)
#pragma unroll 4
    for (int k = 0; k < EPT; ++k)
      if (inside(k)) {
        const int at = hal + lp(k), pp = base + lp(k);
        const dd x = {xh[at], xl[at]};
        // (after a breakdown the low part may hold the infinity or NaN)
        const bool bad = status == KP_BREAKDOWN;
        d.x[pp] = bad ? dd_to_double_any(x) : dd_to_double(x);
        if (p.bnext) p.bnext[(size_t)sysi * p.bnext_ld + pp] = __float2bfloat16_rn(bad ? x.hi + x.lo : x.hi);
      }
    if (tid == 0 && rank == 0) {
      const double rel = bnorm.hi > 0.f ? dd_to_double(rnorm) / dd_to_double(bnorm) : 0.0;
      if (p.info) {
        kp_info inf;
        inf.iters = steps;
        inf.status = status;
        inf.rel_res = rel;
        p.info[sysi] = inf;
      }
      if (p.acc) {
        StepAcc* a = p.acc + tstep;
        // high-precision flops of the refinement (residuals, x update: in
        // double-float); FP32 Krylov work is counted separately
        const unsigned long long fl64 = (unsigned long long)(14 + outer * 13) * (unsigned long long)N;
        const unsigned long long fl32 = (gmres_flops(steps, m) - 14ull) * (unsigned long long)N;
        if (p.acc_kind == 0) {
          atomicAdd(&a->seed_iters, (unsigned long long)steps);
          atomicAdd(&a->seed_flops, fl64 + fl32);
        } else {
          atomicAdd(&a->tgt_iters, (unsigned long long)steps);
          atomicAdd(&a->tgt_flops, fl64);
          atomicAdd(&a->tgt_flops32, fl32);
          atomicMax(&a->tgt_max_iters, (unsigned int)steps);
          atomicMax(&a->max_res_bits, (unsigned long long)__double_as_longlong(rel));
          if (proj_flops) atomicAdd(&a->proj_flops, proj_flops);
        }
        if (status != KP_OK) atomicAdd(&a->not_converged, 1u);
      }
    }
    sync_x();                                    // shared memory is reused by the next system
  }
  if (tid == 0 && rank == 0 && atomicAdd(p.claim + 1, 1) == (int)gridDim.x / CS - 1) {
    p.claim[0] = 0;                              // the last to finish: ready for the next launch
    p.claim[1] = 0;
  }
  if (CS > 1) cluster.sync();                    // no CTA leaves while others write its memory
}

template <int EPT, int NT, int CS, int MINB, int HALF, bool REG, bool LONG = false>
cudaError_t launch_mx(const GmresParams& p, size_t smem, cudaStream_t st) {
  auto k = gmres_mixed_kernel<EPT, NT, CS, MINB, HALF, REG, LONG>;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if (smem > (size_t)optin) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess && CS > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.grid);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CS;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CS > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, k, p);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace
}  // namespace kp
