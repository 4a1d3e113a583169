// kp_conv_train.cu -- the 3x3 convolutions of the network's training as GEMMs
// on the tcgen05 tensor cores, with the im2col operand built in shared memory:
//   forward      Z[p][co]  = sum_k Xcol[p][k]  W[co][k]         k = c*9 + tap
//   input grad   dX[p][c]  = sum_k dZcol[p][k] W2[c][k]         k = co*9 + tap
//   weight grad  dW[co][k] = sum_p XcolT[k][p] dZ[co][p]        (split over p)
// Activations and gradients are FP32 planes [B][C][H*W]; operands are rounded
// to BF16 as they are staged, sums are FP32 in TMEM.  The K order of forward
// and input gradient is that of an im2col matrix in memory, so the results
// have its bits.
//
// Why: with the im2col matrices in memory a training step at 128x128, batch 16
// moved 151 MB per layer and direction and spent 2.4 of its 3.7 ms writing
// them (8-byte bursts of a 576-byte row per pixel), 0.7 ms reading them back.
// Staged, the nine taps come out of L1, and bias, ReLU, ReLU mask and bias
// gradient ride along.  What bounds the kernels now is the staging itself:
// loads from L1 and their conversion (72 loads, 36 packs and 9 stores per
// pixel and 8 channels).
#include <algorithm>

#include "kp_internal.cuh"
#include "kp_tc.cuh"

namespace kp {
namespace {

// Whether tap (di, dj) = sign (tap/3 - 1, tap%3 - 1) of pixel (i, j) lies in
// the grid, for all nine taps.
__device__ __forceinline__ unsigned tap_mask(int i, int j, int H, int W, int sign) {
  unsigned m = 0;
#pragma unroll
  for (int t = 0; t < 9; ++t) {
    const int ii = i + sign * (t / 3 - 1), jj = j + sign * (t % 3 - 1);
    m |= ((unsigned)ii < (unsigned)W && (unsigned)jj < (unsigned)H ? 1u : 0u) << t;
  }
  return m;
}

struct TrainConvArgs {
  const float* X;              // [B][C][P]
  const __nv_bfloat16* Wb;     // [N][ldw], K-major (k = channel * 9 + tap)
  int ldw;
  const float* bias;           // forward: [N]; input gradient: null
  const float* gate;           // input gradient: [B][N][P], passes where > 0
  float* Y;                    // [B][N][P]
  int B, C, N, H, W, sign, relu;
  int* err;
};

// One CTA per SM makes a run of consecutive tiles of 128 pixels x N <= 32
// outputs.  Sixteen warps stage a tile's im2col rows (a pixel per thread and a
// quarter of the channels) into one of two buffers while the MMAs of the other
// run, a seventeenth issues the MMAs over the whole K, and the sixteen read the
// earlier tile's TMEM back.
//
// The staging is what bounds this kernel, in instructions: taken tap by tap
// from global memory it was some 16 instructions per value (address,
// predicate, load, conversion; 83 us per 32 -> 32 layer of 2048 tiles).  So the tile's
// window (its pixels and H + 1 before and after) is converted to BF16 in
// shared memory once, a tap is one load at a precomputed offset (an
// immediate away from channel to channel), and the border is masked in pairs
// after packing.  The next tile's window is loaded into registers meanwhile:
// four rounds of load latency were half of the kernel.  Columns too long for the window (H > 191) are staged from
// global memory.
constexpr int kWin = 512;                          // pixels of a channel's window

constexpr int kStageThreads = 512;
constexpr int kTrainThreads = kStageThreads + 32;

__device__ __forceinline__ int k_groups(int C) { return (C + 7) / 8; }           // 72 k values each
__host__ __device__ inline int k_chunks(int C) { return ((C + 7) / 8 * 72 + 63) / 64; }   // 64 k values each

template <bool WIN>
__global__ void __launch_bounds__(kTrainThreads, 1) train_conv_kernel(const TrainConvArgs a) {
  extern __shared__ unsigned char train_smem[];
  unsigned char* base = train_smem + ((1024u - (su32(train_smem) & 1023u)) & 1023u);
  const int nch = k_chunks(a.C);
  unsigned char* Ws = base;                        // [nch][32 rows][128 bytes], swizzled
  unsigned char* As0 = base + (size_t)nch * 4096;  // [2][nch][128 rows][128 bytes], swizzled
  uint16_t* win = reinterpret_cast<uint16_t*>(As0 + (size_t)nch * 2 * 16384);   // [8 ng][kWin] BF16 (WIN)
  __shared__ uint64_t done[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  volatile int* abort = &abort_s;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(kFull, tid >> 5, 0);   // (uniform, and known to be)
  const int P = a.H * a.W, K = 9 * a.C;
  const int total = a.B * P;                       // (at most 2^30)
  const int ntiles = (total + 127) / 128;
  const int t0 = (int)((long long)ntiles * blockIdx.x / gridDim.x), t1 = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
  const int nout = a.N > 16 ? 32 : 16;             // MMA width
  const int ksteps = (K + 15) / 16;
  const int row = tid & 127, part = tid >> 7;      // (staging warps)
  const bool stager = warp < kStageThreads / 32;
  const int ng = k_groups(a.C);

  if (tid == 0) {
    bar_init(&done[0], 1);
    bar_init(&done[1], 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the weights, zero past K and past N (zero operands meet zero operands)
  for (int e = tid; e < nch * 32 * 8; e += kTrainThreads) {
    const int u = e & 7, r = (e >> 3) & 31, c = e >> 8;
    const int k0 = c * 64 + u * 8;
    __nv_bfloat16 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      v[q] = (r < a.N && k0 + q < K) ? a.Wb[(size_t)r * a.ldw + k0 + q] : __float2bfloat16_rn(0.f);
    *reinterpret_cast<uint4*>(Ws + c * 4096 + r * 128 + ((u ^ (r & 7)) << 4)) = *reinterpret_cast<uint4*>(v);
  }
  // an odd number of groups ends half-way through a K step: zeros behind it
  if ((ng & 1) && part < 2)                        // (parts 0 and 1: the two buffers)
    *reinterpret_cast<uint4*>(As0 + ((size_t)part * nch + ((ng * 9) >> 3)) * 16384 + row * 128 +
                              ((((ng * 9) & 7) ^ (row & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();                              // (the MMA warp wrote its share of the weights too)
  if (warp == 0) tmem_alloc(&tmem_slot, 64);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // TMEM of tile t (use number it of the buffers) -> planes: warp w reads
  // lanes 32 (w % 4) .. = pixels, outputs 8 (w / 4) ..
  auto epilogue = [&](int t, int it) {
    if (!bar_wait(&done[it & 1], (uint32_t)(it >> 1) & 1u, abort)) *abort = 1;
    tc_fence_after();
    const int c0 = (warp >> 2) * 8;
    if (c0 < nout) {
      const int pq = t * 128 + (warp & 3) * 32 + lane;
      float v[8];
      tmem_ld_x8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((it & 1) * 32 + c0), v);
      if (pq < total) {
        const int pb = pq / P, pp = pq - pb * P;
        // (all loads before the first store: the compiler has to keep the
        // order of loads and stores that may alias, one memory latency each)
        const size_t at = ((size_t)pb * a.N + c0) * P + pp;
        float g[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
          g[e] = c0 + e < a.N ? (a.gate ? a.gate[at + (size_t)e * P] : a.bias[c0 + e]) : 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (c0 + e < a.N) {
            float z = a.gate ? (g[e] > 0.f ? v[e] : 0.f) : v[e] + g[e];
            if (a.relu) z = fmaxf(z, 0.f);
            a.Y[at + (size_t)e * P] = z;
          }
      }
    }
    tc_fence_before();
  };

  // the window: pixel w of it is pixel t 128 - H - 1 + w of the batch (pixels
  // of another image or outside the batch are only read by masked taps);
  // channels past C are zero
  float wv[32];
  auto load_window = [&](int t) {
    const int wq = t * 128 - a.H - 1 + tid;
    const bool in = wq >= 0 && wq < total && tid < 128 + 2 * a.H + 2;
    const int wb = in ? wq / P : 0;
    const float* xw = a.X + (size_t)wb * a.C * P + (in ? wq - wb * P : 0);
#pragma unroll
    for (int c = 0; c < 32; ++c) wv[c] = (in && c < a.C) ? xw[(size_t)c * P] : 0.f;
  };
  if (WIN && stager && t0 < t1) load_window(t0);

  int it = 0;
  for (int t = t0; t < t1; ++t, ++it) {
    // buffer it & 1 is free: the epilogue of tile it - 2 waited for its MMAs
    unsigned char* As = As0 + (size_t)(it & 1) * nch * 16384;
    if (WIN && stager) {
#pragma unroll
      for (int c = 0; c < 32; ++c)
        if (c < ng * 8) win[c * kWin + tid] = __bfloat16_as_ushort(__float2bfloat16_rn(wv[c]));
    }
    if (WIN) __syncthreads();
    if (stager) {
      const int q = t * 128 + row;
      const int b = q < total ? q / P : 0, p = q < total ? q - b * P : 0;
      const unsigned tm = q < total ? tap_mask(p / a.H, p % a.H, a.H, a.W, a.sign) : 0u;
      if (WIN) {
        if (t + 1 < t1) load_window(t + 1);
        // taps outside the grid read the pixel itself and are masked: pair e of
        // the 72 values of 8 channels holds taps 2e mod 9 and 2e + 1 mod 9
        int wt[9];
        uint32_t keep[9];
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          wt[tap] = row + a.H + 1 + ((tm >> tap & 1u) ? a.sign * ((tap / 3 - 1) * a.H + (tap % 3 - 1)) : 0);
          const int x = (2 * tap) % 9, y = (2 * tap + 1) % 9;
          keep[tap] = ((tm >> x & 1u) ? 0xFFFFu : 0u) | ((tm >> y & 1u) ? 0xFFFF0000u : 0u);
        }
#pragma unroll 1
        for (int g = part; g < ng; g += 4) {
          const uint16_t* wg = win + g * 8 * kWin;
#pragma unroll
          for (int u0 = 0; u0 < 9; u0 += 3) {      // loads in groups, ahead of their stores
            uint32_t pk[3][4];
#pragma unroll
            for (int u = 0; u < 3; ++u)
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int k = (u0 + u) * 8 + 2 * e;  // of the group's 72
                const uint32_t lo = wg[wt[k % 9] + (k / 9) * kWin], hi = wg[wt[(k + 1) % 9] + ((k + 1) / 9) * kWin];
                pk[u][e] = (lo | hi << 16) & keep[(k / 2) % 9];
              }
#pragma unroll
            for (int u = 0; u < 3; ++u) {
              const int uu = g * 9 + u0 + u;
              *reinterpret_cast<uint4*>(As + (uu >> 3) * 16384 + row * 128 + (((uu & 7) ^ (row & 7)) << 4)) =
                  make_uint4(pk[u][0], pk[u][1], pk[u][2], pk[u][3]);
            }
          }
        }
      } else {
        const float* xb = a.X + ((size_t)b * a.C) * P + p;
#pragma unroll 1
        for (int g = part; g < ng; g += 4) {
#pragma unroll
          for (int u = 0; u < 9; ++u) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float v[2];
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const int k = u * 8 + 2 * e + h, c = g * 8 + k / 9, tap = k % 9;
                v[h] = (c < a.C && (tm >> tap & 1u)) ? xb[(size_t)c * P + a.sign * ((tap / 3 - 1) * a.H + (tap % 3 - 1))] : 0.f;
              }
              __nv_bfloat162 h2 = __floats2bfloat162_rn(v[0], v[1]);
              pk[e] = *reinterpret_cast<uint32_t*>(&h2);
            }
            const int uu = g * 9 + u;
            *reinterpret_cast<uint4*>(As + (uu >> 3) * 16384 + row * 128 + (((uu & 7) ^ (row & 7)) << 4)) =
                make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
      }
      fence_async_smem();
    }
    __syncthreads();                               // tile staged; TMEM buffer it & 1 read (epilogue of it - 2)
    if (!stager) {
      if (!*abort) {
        tc_fence_after();
        const bool issue = lane == 0;
        const uint32_t idesc = idesc_f16(128, nout);
        const uint64_t ad0 = desc_sw128(su32(As)), bd0 = desc_sw128(su32(Ws));
        for (int ks = 0; ks < ksteps; ++ks) {
          const int c = ks >> 2, kk = ks & 3;
          mma_f16_one(issue, tmem + (uint32_t)((it & 1) * 32), ad0 + (uint64_t)(c * 1024 + kk * 2),
                  bd0 + (uint64_t)(c * 256 + kk * 2), idesc, ks > 0 ? 1u : 0u);
        }
        if (issue) mma_commit_to(&done[it & 1]);
      }
      __syncwarp();
    } else if (it > 0) {
      epilogue(t - 1, it - 1);
    }
  }
  if (stager && it > 0) epilogue(t1 - 1, it - 1);
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && *abort) atomicOr(a.err, 1);
  if (warp == 0) tmem_free(tmem, 64);
}

struct WgradArgs {
  const float* X;              // [B][C][P]
  const float* dZ;             // [B][N][P]
  float* dW;                   // [N][9 C], added to
  double* db;                  // [N], added to
  int B, C, N, H, W;
  int* err;
};

// Weight and bias gradients: D[k][co] = sum over pixels, M = k in tiles of 128,
// N = outputs, K = pixels in chunks of 64.  CTA (M tile, split): 16 warps stage
// the tile's rows (c, tap) of two chunks -- a channel per warp, two pixels per
// lane and chunk, from a BF16 window in shared memory, the next one already on
// its way, as in the forward kernel
// (868 instructions per warp and two chunks taken from global memory, 158 us
// for 32 -> 32 channels) -- into one of two buffers while the MMAs of the
// other run, and add their sums to dW at the end.  The
// splits of the pixels are as many as two CTAs per SM and 48 values of k give
// (their number fixes the length of the FP32 sums in TMEM, which truncate);
// with M tiles as the other grid axis they fill the SMs once.
constexpr int kWgThreads = kStageThreads + 32;     // sixteen staging warps, one MMA warp
constexpr uint32_t kWgA = 2 * 16384, kWgB = 2 * 4096;   // bytes per buffer

template <bool WIN>
__global__ void __launch_bounds__(kWgThreads, 1) train_wgrad_kernel(const WgradArgs a) {
  extern __shared__ unsigned char train_smem[];
  unsigned char* base = train_smem + ((1024u - (su32(train_smem) & 1023u)) & 1023u);
  __shared__ uint64_t done[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  volatile int* abort = &abort_s;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(kFull, tid >> 5, 0);   // (uniform, and known to be)
  const int P = a.H * a.W, rows = 9 * a.C, mi = blockIdx.y;
  const int r0 = mi * 128, rn = min(128, rows - r0);
  const int total = a.B * P;                       // (at most 2^30)
  const int nchunk = (total + 63) / 64;
  const int ch0 = (int)((long long)nchunk * blockIdx.x / gridDim.x), ch1 = (int)((long long)nchunk * (blockIdx.x + 1) / gridDim.x);
  const int nout = a.N > 16 ? 32 : 16;

  if (tid == 0) {
    bar_init(&done[0], 1);
    bar_init(&done[1], 1);
    abort_s = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_slot, 32);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  const bool stager = warp < kStageThreads / 32;
  // channels of this tile: (r0 + 127) / 9 - r0 / 9 + 1 <= 16 of them, one per warp
  const int c = r0 / 9 + warp;
  const bool has_c = stager && c < a.C && c * 9 < r0 + rn;
  // two pixels of row r: bytes 4 lane .. + 3 of the row, in piece lane / 4
  auto put = [&](unsigned char* tile, int r, uint32_t v) {
    *reinterpret_cast<uint32_t*>(tile + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4) = v;
  };
  auto pack = [](float v, float w) {
    __nv_bfloat162 h2 = __floats2bfloat162_rn(v, w);
    return *reinterpret_cast<uint32_t*>(&h2);
  };
  uint16_t* msk = reinterpret_cast<uint16_t*>(base + 2 * (kWgA + kWgB));        // [2][128] taps inside the grid
  uint16_t* win = msk + 2 * 128 + (stager ? warp : 0) * kWin;                   // this warp's channel (WIN)
  const int wlen = 128 + 2 * a.H + 2;
  auto masks = [&](int ch, uint16_t* out) {        // of the 128 pixels from chunk ch
    if (tid < 128) {
      const int q = ch * 64 + tid;
      const int p = q < total ? q % P : 0;
      out[tid] = (uint16_t)(q < total && ch + (tid >> 6) < ch1 ? tap_mask(p / a.H, p % a.H, a.H, a.W, 1) : 0u);
    }
  };
  // outputs' gradients (two pixels per lane and chunk, outputs warp, warp + 16)
  // and the channel's window of the two chunks from ch
  float z[2][2][2], wv[kWin / 32];
  // image and pixel of this lane's first point of the next load, kept from one
  // to the next (a division by P a point was a third of the instructions)
  const size_t CP = (size_t)a.C * P, NP = (size_t)a.N * P;
  auto place = [&](int q, int* b, int* p) {
    *b = q >= 0 ? q / P : 0;
    *p = q - *b * P;
  };
  int zb, zp, xb, xp;
  place(ch0 * 64 + 2 * lane, &zb, &zp);
  place(ch0 * 64 - a.H - 1, &xb, &xp);
  xp += lane;                                      // (negative before the first image)
  auto load = [&](int ch) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        int b = zb, p = zp + 64 * h + e;
        while (p >= P) { p -= P; ++b; }
        const bool in = stager && b < a.B && ch + h < ch1;
        const float* zc = a.dZ + (in ? b * NP + p : 0);
#pragma unroll
        for (int u = 0; u < 2; ++u) z[h][e][u] = (in && warp + 16 * u < a.N) ? zc[(size_t)(warp + 16 * u) * P] : 0.f;
      }
    zp += 128;
    while (zp >= P) { zp -= P; ++zb; }
    if (WIN && has_c) {
      int b = xb, p = xp;
      while (p >= P) { p -= P; ++b; }
      const float* xc = a.X + b * CP + (size_t)c * P;
#pragma unroll
      for (int e = 0; e < kWin / 32; ++e, p += 32) {
        while (p >= P) { p -= P; ++b; xc += CP; }
        wv[e] = (e * 32 + lane < wlen && p >= 0 && b < a.B) ? xc[p] : 0.f;
      }
      xp += 128;
      while (xp - lane >= P) { xp -= P; ++xb; }
    }
  };
  // this lane's part of db of outputs warp, warp + 16: an FP32 sum and the
  // errors of its additions (TwoSum, Knuth), since the chain is as long as the
  // split; the CTAs' sums are added in FP64 (constant gradients at 128x128, batch
  // 64: 2.2e-6 off with FP32 sums throughout, at most 6e-8 now)
  float bsum[2] = {0.f, 0.f}, berr[2] = {0.f, 0.f};
  auto add_b = [&](int u, float v) {
    const float t = bsum[u] + v, w = t - bsum[u];
    berr[u] += (bsum[u] - (t - w)) + (v - w);
    bsum[u] = t;
  };
  int it = 0;
  if (ch0 < ch1) {
    masks(ch0, msk);
    load(ch0);
  }
  __syncthreads();
  for (int ch = ch0; ch < ch1; ch += 2, ++it) {
    const int s = it & 1;
    unsigned char* As = base + s * (kWgA + kWgB);
    unsigned char* Bs = As + kWgA;
    if (stager) {
      if (WIN && has_c) {
#pragma unroll
        for (int e = 0; e < kWin / 32; ++e) win[e * 32 + lane] = __bfloat16_as_ushort(__float2bfloat16_rn(wv[e]));
        __syncwarp();
      }
      // the buffer's previous MMAs are done
      if (it >= 2 && !bar_wait(&done[s], (uint32_t)((it >> 1) - 1) & 1u, abort)) *abort = 1;
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (warp + 16 * u < a.N) {
            if (h == 0) add_b(u, (z[0][0][u] + z[0][1][u]) + (z[1][0][u] + z[1][1][u]));
            put(Bs + h * 4096, warp + 16 * u, pack(z[h][0][u], z[h][1][u]));
          }
      if (ch + 2 < ch1) load(ch + 2);
      if (has_c) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t mm = *reinterpret_cast<const uint32_t*>(msk + s * 128 + h * 64 + 2 * lane);
          uint32_t v[9];
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int off = (tap / 3 - 1) * a.H + (tap % 3 - 1);
            if (WIN) {
              const uint16_t* x = win + h * 64 + 2 * lane + a.H + 1 + off;
              v[tap] = ((uint32_t)x[0] | (uint32_t)x[1] << 16) & ((mm >> tap & 0x00010001u) * 0xFFFFu);
            } else {
              float f[2];
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const int q = (ch + h) * 64 + 2 * lane + e;
                const bool in = mm >> (16 * e + tap) & 1u;
                const int b = in ? q / P : 0;
                f[e] = in ? a.X[((size_t)b * a.C + c) * P + (q - b * P) + off] : 0.f;
              }
              v[tap] = pack(f[0], f[1]);
            }
          }
#pragma unroll
          for (int tap = 0; tap < 9; ++tap) {
            const int r = c * 9 + tap - r0;
            if (r >= 0 && r < rn) put(As + h * 16384, r, v[tap]);
          }
        }
      }
      if (ch + 2 < ch1) masks(ch + 2, msk + (s ^ 1) * 128);
      fence_async_smem();
    }
    __syncthreads();
    if (!stager) {
      if (!*abort) {
        tc_fence_after();
        const bool issue = lane == 0;
        const uint32_t idesc = idesc_f16(128, nout);
        const uint64_t ad0 = desc_sw128(su32(As)), bd0 = desc_sw128(su32(Bs));
        const int nk = ch + 1 < ch1 ? 8 : 4;       // K steps of 16 pixels
        for (int kk = 0; kk < nk; ++kk)
          mma_f16_one(issue, tmem, ad0 + (uint64_t)((kk >> 2) * 1024 + (kk & 3) * 2), bd0 + (uint64_t)((kk >> 2) * 256 + (kk & 3) * 2),
                  idesc, (it > 0 || kk > 0) ? 1u : 0u);
        if (issue) mma_commit_to(&done[s]);
      }
      __syncwarp();
    }
  }
  // the last commit waits for all MMAs before it
  if (it > 0 && !bar_wait(&done[(it - 1) & 1], (uint32_t)((it - 1) >> 1) & 1u, abort)) *abort = 1;
  tc_fence_after();
  if (mi == 0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float e = __shfl_xor_sync(kFull, berr[u], o);
        add_b(u, __shfl_xor_sync(kFull, bsum[u], o));
        berr[u] += e;
      }
      if (stager && lane == 0 && warp + 16 * u < a.N) atomicAdd(a.db + warp + 16 * u, (double)bsum[u] + (double)berr[u]);
    }
  }
  // warp w: k = lanes 32 (w % 4) .., outputs 8 (w / 4) ..
  const int c0 = (warp >> 2) * 8;
  if (stager && it > 0 && c0 < nout && !*abort) {
    const int k = (warp & 3) * 32 + lane;
    float v[8];
    tmem_ld_x8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
    if (k < rn)
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (c0 + e < a.N) atomicAdd(a.dW + (size_t)(c0 + e) * rows + r0 + k, v[e]);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && *abort) atomicOr(a.err, 1);
  if (warp == 0) tmem_free(tmem, 32);
}

}  // namespace

// Y = act(conv3x3(X, W) + bias) (gate null), or the input gradient through a
// ReLU: Y = (gate > 0) conv3x3 with the taps mirrored (sign -1, W transposed).
cudaError_t launch_train_conv(const float* X, int B, int C, int H, int W, const __nv_bfloat16* Wb, int ldw, int N,
                              const float* bias, int relu, const float* gate, int sign, float* Y, int* err, int sms,
                              cudaStream_t st) {
  if (C < 1 || C > 32 || N < 1 || N > 32) return cudaErrorInvalidValue;
  TrainConvArgs a{X, Wb, ldw, bias, gate, Y, B, C, N, H, W, sign, relu, err};
  const bool win = 128 + 2 * H + 2 <= kWin;
  const size_t smem = (size_t)k_chunks(C) * (2 * 16384 + 4096) + 1024 + (win ? (size_t)((C + 7) / 8 * 8) * kWin * 2 : 0);
  auto k = win ? train_conv_kernel<true> : train_conv_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long ntiles = ((long long)B * H * W + 127) / 128;
  k<<<(unsigned)std::min<long long>(ntiles, sms), kTrainThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_train_wgrad(const float* X, const float* dZ, int B, int C, int N, int H, int W, float* dW, double* db,
                               int* err, int sms, cudaStream_t st) {
  if (C < 1 || C > 32 || N < 1 || N > 32) return cudaErrorInvalidValue;
  WgradArgs a{X, dZ, dW, db, B, C, N, H, W, err};
  const bool win = 128 + 2 * H + 2 <= kWin;
  const size_t smem = 2 * (size_t)(kWgA + kWgB) + 1024 + 2 * 128 * 2 + (win ? (size_t)(kStageThreads / 32) * kWin * 2 : 0);
  auto k = win ? train_wgrad_kernel<true> : train_wgrad_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long nchunk = ((long long)B * H * W + 63) / 64;
  const int tiles48 = (9 * C + 47) / 48;
  const long long splits = std::max<long long>(1, std::min<long long>(nchunk, 2 * sms / tiles48));
  k<<<dim3((unsigned)splits, (9 * C + 127) / 128), kWgThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace kp
