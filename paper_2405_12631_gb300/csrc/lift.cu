// CNN lifting wavelet transform (Section 3.1, Fig. 2), temporal lifting
// (Section 3.3), colour conversion and the scalar quantiser.
//
// One lifting half-step computes v = lin(src) + CNN(src) along a direction
// and writes out = other + sign * v; the inverse transform runs the steps
// of the forward transform backwards, so it reconstructs perfectly for any
// network weights. The CNN residual is conv3x3(1->16), tanh,
// conv3x3(16->16), tanh, conv3x3(16->1) with zero padding, fused in one
// kernel per output tile (halo of 3, all activations in shared memory). Linear parts: LeGall 5/3 (P = (s[n] + s[n+1]) / 2,
// U = (s[n-1] + s[n]) / 4, edges clamped = whole-sample symmetric) for the
// spatial transform; Haar (P = s, U = s / 2) for the temporal one. Integer
// mode (lossless) rounds P with floor(v) and U with floor(v + 1/2), which
// makes the transform the JPEG 2000 reversible 5/3 when the CNN is zero.
//
// An integer lifting step reconstructs exactly only if encoder and decoder
// round the same P and U values, so in integer mode the CNN is evaluated as
// a fixed sequence of FP32 operations that any IEEE implementation
// reproduces bit for bit: every layer starts from its bias and adds, tap by
// tap in raster order (dy, dx) and within a tap input channel by input
// channel in ascending order, the product w * x (product and sum each
// rounded to nearest even, never fused), the activation is tanh32_spec, and
// v = lin + CNN is one rounded addition before the floor. The lossy steps
// keep fused multiply-adds and the CUDA tanh.
#include <cuda_bf16.h>

#include <cstring>
#include <mutex>

#include "pw_internal.cuh"
#include "lift_kernels.cuh"
#include "spec_math.cuh"
#include "f32x2.cuh"
#include "tc_ptx.cuh"

namespace pw {

constexpr int LF = 16;            // CNN channels
// the tensor-core step's tile
constexpr int LT = 16;            // output tile
constexpr int L1 = LT + 4;        // layer-1 region (20)
constexpr int L2 = LT + 2;        // layer-2 region (18)
constexpr int LI = LT + 6;        // input region (22)

// The activation: CUDA's tanhf, or (kExact) tanh32_spec.
template <bool kExact>
__device__ __forceinline__ float act(float v) {
  return kExact ? tanh32_spec(v) : tanhf(v);
}

// Two accumulators at once, acc + w x: per element a fused multiply-add, or
// (kExact) a rounded product and a rounded sum.
template <bool kExact>
__device__ __forceinline__ uint64_t mac2(uint64_t acc, uint64_t w, uint64_t x) {
  return kExact ? add2(acc, mul2(w, x)) : fma2(w, x, acc);
}

__device__ __forceinline__ float acc_get(const PlaneAcc &a, int p, int y, int x) {
  return a.p[(int64_t)p * a.ps + (int64_t)y * a.rs + (int64_t)x * a.cs];
}
__device__ __forceinline__ void acc_set(const PlaneAcc &a, int p, int y, int x, float v) {
  a.p[(int64_t)p * a.ps + (int64_t)y * a.rs + (int64_t)x * a.cs] = v;
}

// The linear part and the output at (y, x) of a plane: c points at the source
// sample in the staged input, whose rows are `stride` apart; r_out is the CNN
// residual.
template <bool kExact>
__device__ __forceinline__ void lift_out(const LiftStepParams &a, int p, int H, int W, int y,
                                         int x, const float *c, int stride, float r_out) {
  const float s0 = c[0];
  float lin;
  if (a.lin == LIN_P53) {
    const float s1 = a.dir == 0 ? (x + 1 < W ? c[1] : s0) : (y + 1 < H ? c[stride] : s0);
    lin = 0.5f * (s0 + s1);
  } else if (a.lin == LIN_U53) {
    const float sm = a.dir == 0 ? (x > 0 ? c[-1] : s0) : (y > 0 ? c[-stride] : s0);
    lin = 0.25f * (sm + s0);
  } else if (a.lin == LIN_ID) {
    lin = s0;
  } else if (a.lin == LIN_HALF) {
    lin = 0.5f * s0;
  } else {  // LIN_ZERO: the CNN alone (post-processing)
    lin = 0.f;
  }
  float v = kExact ? __fadd_rn(lin, r_out) : lin + r_out;
  if (a.round == 1) v = floorf(v);
  else if (a.round == 2) v = floorf(v + 0.5f);
  const float o = acc_get(a.other, p, y, x);
  acc_set(a.out, p, y, x, a.sign > 0 ? o + v : o - v);
  if (a.copy.p) acc_set(a.copy, p, y, x, s0);
}

// One lifting step on FP32 cores, one TW x TH output tile per block.
//
// What bounds it: the FP32 pipe. Layer 2 is 2304 of the 2592 multiply-adds
// of a sample (in the exact mode each is a product and a sum, and the 32
// tanh32_spec of a sample cost a third as much again). So the tile is chosen
// for layer 2: its region, one wider than the tile on every side, is 512
// positions for 30 x 14 (a 22 % surplus, two positions x 16 channels per
// thread, every lane busy) and 128 for 14 x 6 (one position x 8 channels),
// the small tile for planes that do not fill the chip with large ones.
// Activations lie in four planes of 4 channels (16 bytes per position):
// neighbouring lanes read neighbouring 16 bytes, where a 64-byte pixel cost
// four times the shared-memory passes. Layer 2's result overwrites layer
// 1's slab once every thread holds its own, so four blocks share an SM.
// Layer 2's weights are the same for every lane: the large tile reads them
// from the kernel's parameters (constant bank), since broadcast loads from
// shared memory return 16 bytes to each of 32 lanes and had the port busy
// for longer than the arithmetic; the small tile, whose threads split the
// channels, reads shared memory (11 us against 16 us a launch).
// Measured: 2 lossless 3840x2160 12-bit RGB images, all steps, 51.7 ms (16 x
// 16 tile, 64-byte pixels, 162 of 256 threads in layer 2, tanh by branches)
// -> 28.2 -> 23.6 ms with the weights as parameters; forward lifting of 12
// 768x512 RGB images 10.7 -> 6.7 -> 5.1 ms; a 250x333 plane, 24 steps, 0.67
// -> 0.27 ms (small tile).
// Every layer's per-element operation order is the definition's: bias, then
// tap by tap, input channel by input channel (channels or outputs in packed
// FP32 pairs, each element rounded as its scalar operation).
template <int TW, int TH>
struct LiftCfg {
  static constexpr int IW = TW + 6, IH = TH + 6;              // input region
  static constexpr int W1 = TW + 4, H1 = TH + 4, N1 = W1 * H1;   // layer-1 region
  static constexpr int W2 = TW + 2, H2 = TH + 2, N2 = W2 * H2;   // layer-2 region
  static constexpr int NO = TW * TH;
  static constexpr int PP = N2 >= 512 ? N2 / 256 : 1;         // layer-2 positions per thread
  static constexpr int CH = 16 * N2 / (256 * PP);             // and channels
  static_assert(PP * CH * 256 == 16 * N2 && (CH == 16 || CH == 8), "layer-2 work split");
  static_assert(NO <= 512, "outputs per thread");
  struct Smem {
    alignas(16) float act[4 * N1 * 4];   // [channel / 4][position][channel % 4]
    alignas(16) float wt[kLiftSmall + (CH == 16 ? 0 : kLiftW2)];
    alignas(16) float in[IW * IH];
  };
  // layer 2's weights as a kernel parameter (unused by the small tile)
  struct Wt2 {
    alignas(16) float v[CH == 16 ? kLiftW2 : 4];
  };
};

template <bool kExact, int TW, int TH>
__global__ void __launch_bounds__(256, 4) k_lift_step(
    const __grid_constant__ LiftStepParams a,
    const __grid_constant__ typename LiftCfg<TW, TH>::Wt2 w2p) {
  using C = LiftCfg<TW, TH>;
  extern __shared__ __align__(16) uint8_t lift_smem[];
  typename C::Smem &S = *reinterpret_cast<typename C::Smem *>(lift_smem);
  float4 *act4 = reinterpret_cast<float4 *>(S.act);
  const float *w1t = S.wt, *w3t = S.wt + 144, *b1 = S.wt + 288, *b2 = S.wt + 304;
  const int t = threadIdx.x;
  const int p = blockIdx.z;
  const int tiles_x = (a.W + TW - 1) / TW;
  const int y0 = (blockIdx.x / tiles_x) * TH, x0 = (blockIdx.x % tiles_x) * TW;
  const bool cnn = a.net.w1 != nullptr;
  int H, W;
  lift_extent(a, p, H, W);
  if (y0 >= H || x0 >= W) return;  // a tile beyond this plane of a ragged batch

  for (int e = t; e < C::IW * C::IH; e += 256) {
    const int yy = y0 + e / C::IW - 3, xx = x0 + e % C::IW - 3;
    S.in[e] = (yy >= 0 && yy < H && xx >= 0 && xx < W) ? acc_get(a.src, p, yy, xx) : 0.f;
  }
  if (cnn)
    for (int e = t; e < (int)(sizeof(S.wt) / 16); e += 256)
      reinterpret_cast<float4 *>(S.wt)[e] = __ldg(reinterpret_cast<const float4 *>(a.net.wt) + e);
  __syncthreads();
  float res[2] = {0.f, 0.f};   // CNN residual of outputs t and t + 256
  if (cnn) {
    // layer 1: one position and 8 channels per item
    for (int it = t; it < 2 * C::N1; it += 256) {
      const int g = it >= C::N1 ? 1 : 0, pos = it - g * C::N1;
      const int ly = pos / C::W1, lx = pos % C::W1;
      const int yy = y0 + ly - 2, xx = x0 + lx - 2;
      const bool inside = yy >= 0 && yy < H && xx >= 0 && xx < W;
      uint64_t accp[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) accp[k] = f2pack(b1[8 * g + 2 * k], b1[8 * g + 2 * k + 1]);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const float iv = S.in[(ly + tap / 3) * C::IW + lx + tap % 3];
        const uint64_t xv = f2pack(iv, iv);
        const ulonglong2 *wp = reinterpret_cast<const ulonglong2 *>(w1t + tap * LF + 8 * g);
        const ulonglong2 wa = wp[0], wb = wp[1];
        accp[0] = mac2<kExact>(accp[0], wa.x, xv);
        accp[1] = mac2<kExact>(accp[1], wa.y, xv);
        accp[2] = mac2<kExact>(accp[2], wb.x, xv);
        accp[3] = mac2<kExact>(accp[3], wb.y, xv);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        float v[4];
        f2unpack(accp[2 * k], v[0], v[1]);
        f2unpack(accp[2 * k + 1], v[2], v[3]);
        act4[(2 * g + k) * C::N1 + pos] =
            inside ? make_float4(act<kExact>(v[0]), act<kExact>(v[1]), act<kExact>(v[2]),
                                 act<kExact>(v[3]))
                   : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    __syncthreads();
    // layer 2: positions q + 256 i, channels c0 .. c0 + CH - 1
    {
      const int c0 = C::CH == 8 && t >= 128 ? 8 : 0;
      const int q = C::CH == 8 ? (t & 127) : t;
      uint64_t acc[C::PP][C::CH / 2];
      int base[C::PP];
#pragma unroll
      for (int i = 0; i < C::PP; ++i) {
        const int e = q + 256 * i;
        base[i] = (e / C::W2) * C::W1 + e % C::W2;
#pragma unroll
        for (int k = 0; k < C::CH / 2; ++k)
          acc[i][k] = f2pack(b2[c0 + 2 * k], b2[c0 + 2 * k + 1]);
      }
#pragma unroll 1
      for (int tap = 0; tap < 9; ++tap) {
        const int off = (tap / 3) * C::W1 + tap % 3;
        const float *wrow = C::CH == 16 ? w2p.v + tap * LF * LF
                                        : S.wt + kLiftSmall + tap * LF * LF + c0;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          float xv[C::PP][4];
#pragma unroll
          for (int i = 0; i < C::PP; ++i) {
            const float4 f = act4[g * C::N1 + base[i] + off];
            xv[i][0] = f.x; xv[i][1] = f.y; xv[i][2] = f.z; xv[i][3] = f.w;
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const ulonglong2 *wp =
                reinterpret_cast<const ulonglong2 *>(wrow + (4 * g + e) * LF);
#pragma unroll
            for (int k = 0; k < C::CH / 4; ++k) {
              const ulonglong2 w = wp[k];
#pragma unroll
              for (int i = 0; i < C::PP; ++i) {
                const uint64_t xx = f2pack(xv[i][e], xv[i][e]);
                acc[i][2 * k] = mac2<kExact>(acc[i][2 * k], w.x, xx);
                acc[i][2 * k + 1] = mac2<kExact>(acc[i][2 * k + 1], w.y, xx);
              }
            }
          }
        }
      }
      __syncthreads();   // layer 1's slab is consumed: layer 2's goes over it
#pragma unroll
      for (int i = 0; i < C::PP; ++i) {
        const int e = q + 256 * i;
        const int yy = y0 + e / C::W2 - 1, xx = x0 + e % C::W2 - 1;
        const bool inside = yy >= 0 && yy < H && xx >= 0 && xx < W;
#pragma unroll
        for (int k = 0; k < C::CH / 4; ++k) {
          float v[4];
          f2unpack(acc[i][2 * k], v[0], v[1]);
          f2unpack(acc[i][2 * k + 1], v[2], v[3]);
          act4[(c0 / 4 + k) * C::N2 + e] =
              inside ? make_float4(act<kExact>(v[0]), act<kExact>(v[1]), act<kExact>(v[2]),
                                   act<kExact>(v[3]))
                     : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
    }
    __syncthreads();
    // layer 3: outputs t and t + 256 as one packed pair
    {
      const int oa = min(t, C::NO - 1), ob = min(t + 256, C::NO - 1);
      const int pa = (oa / TW) * C::W2 + oa % TW, pb = (ob / TW) * C::W2 + ob % TW;
      const float b3 = S.wt[320];
      uint64_t v = f2pack(b3, b3);
#pragma unroll 1
      for (int tap = 0; tap < 9; ++tap) {
        const int off = (tap / 3) * C::W2 + tap % 3;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const float4 w = *reinterpret_cast<const float4 *>(w3t + tap * LF + 4 * g);
          const float4 xa = act4[g * C::N2 + pa + off];
          const float4 xb = C::NO > 256 ? act4[g * C::N2 + pb + off] : xa;
          v = mac2<kExact>(v, f2pack(w.x, w.x), f2pack(xa.x, xb.x));
          v = mac2<kExact>(v, f2pack(w.y, w.y), f2pack(xa.y, xb.y));
          v = mac2<kExact>(v, f2pack(w.z, w.z), f2pack(xa.z, xb.z));
          v = mac2<kExact>(v, f2pack(w.w, w.w), f2pack(xa.w, xb.w));
        }
      }
      f2unpack(v, res[0], res[1]);
    }
  }
#pragma unroll
  for (int i = 0; i < (C::NO > 256 ? 2 : 1); ++i) {
    const int o = t + 256 * i;
    if (o >= C::NO) break;
    const int ly = o / TW, lx = o % TW;
    const int y = y0 + ly, x = x0 + lx;
    if (y < H && x < W)
      lift_out<kExact>(a, p, H, W, y, x, S.in + (ly + 3) * C::IW + lx + 3, C::IW, res[i]);
  }
}

// ---------------------------------------------------------------------------
// Lifting step with the CNN's second and third layers (conv3x3 16 -> 16 and
// 16 -> 1, 95 % of its FLOPs) on the tensor cores: BF16 operands, FP32
// accumulation in tensor memory. Layer 1, the linear part and the output
// stay FP32.
//
// Rows of every GEMM are positions of a region laid out with a row stride of
// RS = 24 positions: row m = r * RS + c. Layer 1 (20 x 20 region) and layer 2
// (18 x 18) are stored as BF16 slabs with that stride, so tap (dy, dx) of row
// m reads position m + dy * RS + dx of the layer below: each tap is one MMA
// per 128-row block whose A operand is the slab shifted by a constant
// (columns c >= 18, resp. 16, are padding whose results are never used).
// Slabs: [2 channel groups][positions][8] BF16 (K-major core matrices, no
// swizzle); B: [tap][2][16 outputs][8] (layer 3: output 0 only, rest zero).
constexpr int kRS = 24;                   // row stride of the regions
constexpr int kMT = 4;                    // layer-2 blocks (18 * 24 = 432 rows)
constexpr int kMT3 = 3;                   // layer-3 blocks (16 * 24 = 384 rows)
constexpr int kA = 576;                   // layer-1 positions kept (> 511 + 2 * 24 + 2)
constexpr int kA2 = 448;                  // layer-2 positions kept (> 383 + 2 * 24 + 2)

struct LiftTcSmem {
  // layer-1 slab; once the layer-2 MMAs have completed, the layer-2 slab
  // (2 * kA2 * 8 elements) is written over it
  alignas(128) __nv_bfloat16 a1[2 * kA * 8];
  alignas(128) __nv_bfloat16 w2[9 * 2 * LF * 8];
  alignas(128) __nv_bfloat16 w3[9 * 2 * LF * 8];
  alignas(16) float in[LI * LI];
  alignas(16) float rout[LT * LT];
  alignas(8) uint64_t bar;
  uint32_t tmem;
};
// The FP32 weights of a step as a kernel parameter: w1 [tap][c], the biases.
struct LiftTcWt {
  alignas(16) float w1[9 * LF];
  float b1[LF], b2[LF], b3;
};

// Bounded wait of every thread for completion phase `parity` of the MMA
// barrier (lane 0 polls, the rest follow); false on expiry.
__device__ __forceinline__ bool lift_mma_wait(uint64_t *bar, uint32_t parity) {
  const int lane = threadIdx.x & 31;
  int ok = 1;
  if (lane == 0) {
    // suspended try_wait: the waiting warps leave the issue slots to the
    // other CTAs' warps on the SM instead of spinning
    const long long t0 = clock64();
    while (!mbar_try_sleep(bar, parity, 2000u))
      if (clock64() - t0 > kWaitCycles) { ok = 0; break; }
  }
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (ok && lane != 0) while (!mbar_try(bar, parity)) {}
  __syncwarp();
  fence_after();
  return ok != 0;
}

// (six resident CTAs per SM: 40 registers instead of 48, which allowed five;
// lifting class 4.50 -> 4.45 ms per batch of 24. Layer 1 from the parameter
// bank and on its 400 positions only: 4.36 -> 3.51 ms, with 4 bytes spilled;
// what bounds it now is issue (58 % of the slots with 2304 blocks) and the
// waits between the phases of a tile.)
__global__ void __launch_bounds__(256, 6) k_lift_tc(const __grid_constant__ LiftStepParams a,
                                                    const __grid_constant__ LiftTcWt wt) {
  extern __shared__ __align__(1024) uint8_t lsm_raw[];
  LiftTcSmem &S = *reinterpret_cast<LiftTcSmem *>(lsm_raw);
  __nv_bfloat16 *const a2 = S.a1;   // layer-2 slab over the consumed layer-1 slab
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int p = blockIdx.z;
  const int tiles_x = (a.W + LT - 1) / LT;
  const int y0 = (blockIdx.x / tiles_x) * LT, x0 = (blockIdx.x % tiles_x) * LT;
  int H, W;
  lift_extent(a, p, H, W);
  if (y0 >= H || x0 >= W) return;  // a tile beyond this plane of a ragged batch (uniform)
  // TMEM columns: layer 2 in [0, 64) (4 blocks x 16), then layer 3 in
  // [0, 48) once the layer-2 epilogue has read them
  constexpr uint32_t kCols = 64;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&S.tmem)),
                 "r"(kCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (t == 32) {
    mbar_init(&S.bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = t; e < LI * LI; e += 256) {
    const int yy = y0 + e / LI - 3, xx = x0 + e % LI - 3;
    S.in[e] = (yy >= 0 && yy < H && xx >= 0 && xx < W) ? acc_get(a.src, p, yy, xx) : 0.f;
  }
  {
    // the packed B operands of layers 2 and 3 (9 x 2 x 16 x 8 BF16 each)
    constexpr int kB16 = 9 * 2 * LF * 8 * 2 / 16;
    const uint4 *src2 = reinterpret_cast<const uint4 *>(a.net.w2b);
    const uint4 *src3 = reinterpret_cast<const uint4 *>(a.net.w3b);
    for (int i = t; i < kB16; i += 256) {
      reinterpret_cast<uint4 *>(S.w2)[i] = __ldg(src2 + i);
      reinterpret_cast<uint4 *>(S.w3)[i] = __ldg(src3 + i);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tbase = S.tmem;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(LF >> 3) << 17) |
                         ((uint32_t)(128 >> 4) << 24);

  // layer 1 on the 20 x 20 region (origin y0 - 2, x0 - 2), one position per
  // item. (The slab's padding stays as it is: an MMA row reads the rows of
  // its own taps only, and rows that read padding are not used.) The weights
  // come from the parameter bank: as broadcast loads from shared memory they
  // had its port at 86 %, the bound of this kernel.
  for (int it = t; it < L1 * L1; it += 256) {
    const int r = it / L1, c = it % L1, pos = r * kRS + c;
    const int yy = y0 - 2 + r, xx = x0 - 2 + c;
    const bool inside = yy >= 0 && yy < H && xx >= 0 && xx < W;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      // channel pairs in packed FP32 FMAs (the same rounding as fmaf)
      uint64_t acc[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[k] = f2pack(wt.b1[8 * g + 2 * k], wt.b1[8 * g + 2 * k + 1]);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const float iv = S.in[(r + tap / 3) * LI + c + tap % 3];
        const uint64_t iv2 = f2pack(iv, iv);
        const uint64_t *w = reinterpret_cast<const uint64_t *>(wt.w1 + tap * LF + 8 * g);
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] = fma2(w[k], iv2, acc[k]);
      }
      __align__(16) __nv_bfloat16 hb[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float lo, hi;
        f2unpack(acc[k], lo, hi);
        hb[2 * k] = __float2bfloat16_rn(inside ? tanh_fast(lo) : 0.f);
        hb[2 * k + 1] = __float2bfloat16_rn(inside ? tanh_fast(hi) : 0.f);
      }
      *reinterpret_cast<uint4 *>(S.a1 + ((size_t)g * kA + pos) * 8) =
          *reinterpret_cast<const uint4 *>(hb);
    }
  }
  fence_proxy_async();
  __syncthreads();

  // layer 2: 4 blocks x 9 taps MMAs (M = 128, N = 16, K = 16), one thread
  if (t == 0) {
    fence_after();
    const uint32_t abase = smem_u32(S.a1), bbase = smem_u32(S.w2);
#pragma unroll
    for (int i = 0; i < kMT; ++i) {
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const uint32_t arow = (uint32_t)(i * 128 + (tap / 3) * kRS + tap % 3);
        const uint64_t ad = sdesc(abase + arow * 16u, kA * 16u, 128u);
        const uint64_t bd = sdesc(bbase + (uint32_t)tap * (2 * LF * 16), LF * 16u, 128u);
        mma_bf16(tbase + (uint32_t)(i * LF), ad, bd, idesc, tap > 0 ? 1u : 0u);
      }
    }
    mma_commit(&S.bar);
  }
  bool ok = lift_mma_wait(&S.bar, 0);
  // layer-2 epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 of blocks
  // w / 4 and w / 4 + 2 -> tanh(acc + b2) (0 outside the image and in the
  // padding rows / columns) into the layer-2 slab
  if (ok) {
    const int q = warp & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = (warp >> 2) + 2 * h;
      float v[LF];
      tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(i * LF), v);
      const int m = i * 128 + 32 * q + lane;
      if (m < kA2) {
        const int r2 = m / kRS, c2 = m % kRS;
        const int yy = y0 - 1 + r2, xx = x0 - 1 + c2;
        const bool live = r2 < L2 && c2 < L2 && yy >= 0 && yy < H && xx >= 0 && xx < W;
        __align__(16) __nv_bfloat16 hb[LF];
#pragma unroll
        for (int k = 0; k < LF; ++k)
          hb[k] = __float2bfloat16_rn(live ? tanh_fast(v[k] + wt.b2[k]) : 0.f);
        *reinterpret_cast<uint4 *>(a2 + (size_t)m * 8) = *reinterpret_cast<const uint4 *>(hb);
        *reinterpret_cast<uint4 *>(a2 + ((size_t)kA2 + m) * 8) =
            *reinterpret_cast<const uint4 *>(hb + 8);
      }
    }
  }
  fence_proxy_async();
  fence_before();
  __syncthreads();
  fence_after();

  // layer 3: 3 blocks x 9 taps MMAs into TMEM columns 64 + 16 i
  if (t == 0 && ok) {
    const uint32_t abase = smem_u32(a2), bbase = smem_u32(S.w3);
#pragma unroll
    for (int i = 0; i < kMT3; ++i) {
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const uint32_t arow = (uint32_t)(i * 128 + (tap / 3) * kRS + tap % 3);
        const uint64_t ad = sdesc(abase + arow * 16u, kA2 * 16u, 128u);
        const uint64_t bd = sdesc(bbase + (uint32_t)tap * (2 * LF * 16), LF * 16u, 128u);
        mma_bf16(tbase + (uint32_t)(i * LF), ad, bd, idesc, tap > 0 ? 1u : 0u);
      }
    }
    mma_commit(&S.bar);
  }
  if (ok) ok = lift_mma_wait(&S.bar, 1);
  if (!ok && lane == 0) atomicOr(a.status, kStTimeout);
  // layer-3 epilogue: column 0 of each block -> residual of output (r, c)
  if (ok) {
    const int q = warp & 3;
    for (int i = warp >> 2; i < kMT3; i += 2) {
      float v[LF];
      tmem_ld16(tbase + ((uint32_t)(32 * q) << 16) + (uint32_t)(i * LF), v);
      const int m = i * 128 + 32 * q + lane;
      const int r = m / kRS, c = m % kRS;
      if (r < LT && c < LT) S.rout[r * LT + c] = v[0] + wt.b3;
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(kCols));
  }
  const int oy = y0 + t / LT, ox = x0 + t % LT;
  if (ok && oy < H && ox < W)
    lift_out<false>(a, p, H, W, oy, ox, S.in + (t / LT + 3) * LI + t % LT + 3, LI, S.rout[t]);
}

// Component planes [B][nc][Hp][Wp] -> interleaved samples (crop, inverse
// colour transform, floor(v + 1/2), clip).
__global__ void k_colour_out(const float *__restrict__ planes, int B, int nc, int Hp, int Wp,
                             int H, int W, int colour, int bitdepth, void *out,
                             int64_t img_stride, int64_t row_stride, int out16) {
  const int64_t n = (int64_t)B * H * W;
  const float off = (float)(1 << (bitdepth - 1));
  const float maxv = (float)((1 << bitdepth) - 1);
  const float kr = 0.299f, kb = 0.114f, kg = 1.f - 0.299f - 0.114f;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(e % W);
    const int y = (int)((e / W) % H);
    const int b = (int)(e / ((int64_t)W * H));
    const float *pl = planes + (int64_t)b * nc * Hp * Wp + (int64_t)y * Wp + x;
    float v[3];
    if (nc == 1) {
      v[0] = pl[0] + off;
    } else {
      const float Y = pl[0] + off, Cb = pl[(int64_t)Hp * Wp], Cr = pl[2 * (int64_t)Hp * Wp];
      if (colour == 2) {
        const float G = Y - floorf((Cb + Cr) * 0.25f);
        v[0] = Cr + G; v[1] = G; v[2] = Cb + G;
      } else {
        const float R = Y + 2.f * (1.f - kr) * Cr;
        const float Bv = Y + 2.f * (1.f - kb) * Cb;
        v[0] = R; v[2] = Bv; v[1] = (Y - kr * R - kb * Bv) / kg;
      }
    }
    for (int c = 0; c < nc; ++c) {
      float s = fminf(fmaxf(floorf(v[c] + 0.5f), 0.f), maxv);
      const int64_t o = (int64_t)b * img_stride + (int64_t)y * row_stride;
      if (out16) reinterpret_cast<uint16_t *>((uint8_t *)out + o)[(int64_t)x * nc + c] = (uint16_t)s;
      else ((uint8_t *)out + o)[(int64_t)x * nc + c] = (uint8_t)s;
    }
  }
}

// Interleaved samples -> component planes [B][nc][Hp][Wp] (colour
// transform, level shift, whole-sample mirror padding).
__global__ void k_colour_in(const void *in, int64_t img_stride, int64_t row_stride, int in16,
                            int B, int nc, int H, int W, int Hp, int Wp, int lossless,
                            int bitdepth, float *__restrict__ planes) {
  const int64_t n = (int64_t)B * Hp * Wp;
  const float off = (float)(1 << (bitdepth - 1));
  const float kr = 0.299f, kb = 0.114f, kg = 1.f - 0.299f - 0.114f;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(e % Wp);
    const int y = (int)((e / Wp) % Hp);
    const int b = (int)(e / ((int64_t)Wp * Hp));
    int sy = y < H ? y : 2 * (H - 1) - y;
    int sx = x < W ? x : 2 * (W - 1) - x;
    sy = min(max(sy, 0), H - 1);
    sx = min(max(sx, 0), W - 1);
    const int64_t o = (int64_t)b * img_stride + (int64_t)sy * row_stride;
    float s[3];
    for (int c = 0; c < nc; ++c)
      s[c] = in16 ? (float)reinterpret_cast<const uint16_t *>((const uint8_t *)in + o)[(int64_t)sx * nc + c]
                  : (float)((const uint8_t *)in + o)[(int64_t)sx * nc + c];
    float *pl = planes + (int64_t)b * nc * Hp * Wp + (int64_t)y * Wp + x;
    const int64_t ps = (int64_t)Hp * Wp;
    if (nc == 1) {
      pl[0] = s[0] - off;
    } else if (lossless) {
      pl[0] = floorf((s[0] + 2.f * s[1] + s[2]) * 0.25f) - off;
      pl[ps] = s[2] - s[1];
      pl[2 * ps] = s[0] - s[1];
    } else {
      const float Y = kr * s[0] + kg * s[1] + kb * s[2];
      pl[0] = Y - off;
      pl[ps] = (s[2] - Y) / (2.f * (1.f - kb));
      pl[2 * ps] = (s[0] - Y) / (2.f * (1.f - kr));
    }
  }
}

__global__ void k_quantise(const float *__restrict__ y, int64_t n, float delta,
                           int32_t *__restrict__ q) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    q[e] = (int32_t)rintf(__fmul_rn(y[e], delta));
}

__global__ void k_dequantise(const int32_t *__restrict__ q, int64_t n, float delta,
                             float *__restrict__ y) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    y[e] = __fdiv_rn((float)q[e], delta);
}

static int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g > 152 * 32 ? 152 * 32 : (g < 1 ? 1 : g));
}

template <bool kExact, int TW, int TH>
static void launch_lift_tile(const LiftStepParams &a, cudaStream_t st) {
  constexpr int smem = (int)sizeof(typename LiftCfg<TW, TH>::Smem);
  static std::atomic<uint64_t> attr{0};
  once_per_device(attr, [] {
    cudaFuncSetAttribute(k_lift_step<kExact, TW, TH>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  });
  dim3 grid(((a.H + TH - 1) / TH) * ((a.W + TW - 1) / TW), 1, a.P);
  typename LiftCfg<TW, TH>::Wt2 w2;
  if (LiftCfg<TW, TH>::CH == 16 && a.net.wt_host)
    std::memcpy(w2.v, a.net.wt_host + kLiftSmall, sizeof(w2.v));
  k_lift_step<kExact, TW, TH><<<grid, 256, smem, st>>>(a, w2);
}

void launch_lift_step(const LiftStepParams &a, cudaStream_t st) {
  if (a.tc && a.net.w1 && a.round == 0) {
    static std::atomic<uint64_t> attr_tc{0};
    once_per_device(attr_tc, [] {
      cudaFuncSetAttribute(k_lift_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)sizeof(LiftTcSmem) + 1024);
    });
    const int tiles = ((a.H + LT - 1) / LT) * ((a.W + LT - 1) / LT);
    dim3 grid(tiles, 1, a.P);
    LiftTcWt wt;
    std::memcpy(wt.w1, a.net.wt_host, sizeof(wt.w1));
    std::memcpy(wt.b1, a.net.wt_host + 288, sizeof(wt.b1));
    std::memcpy(wt.b2, a.net.wt_host + 304, sizeof(wt.b2));
    wt.b3 = a.net.wt_host[320];
    k_lift_tc<<<grid, 256, sizeof(LiftTcSmem) + 1024, st>>>(a, wt);
    return;
  }
  // large tiles where they fill the chip, small ones (a quarter of the work
  // per thread, half as much surplus again) where latency counts
  const int64_t big = (int64_t)((a.H + 13) / 14) * ((a.W + 29) / 30) * a.P;
  // integer (lossless) steps take the exact operation sequence
  if (big > sm_count()) {
    if (a.round != 0) launch_lift_tile<true, 30, 14>(a, st);
    else launch_lift_tile<false, 30, 14>(a, st);
  } else {
    if (a.round != 0) launch_lift_tile<true, 14, 6>(a, st);
    else launch_lift_tile<false, 14, 6>(a, st);
  }
}
void launch_colour_out(const float *planes, int B, int nc, int Hp, int Wp, int H, int W,
                       int colour, int bitdepth, void *out, int64_t img_stride,
                       int64_t row_stride, cudaStream_t st) {
  int64_t n = (int64_t)B * H * W;
  k_colour_out<<<grid_for(n), 256, 0, st>>>(planes, B, nc, Hp, Wp, H, W, colour, bitdepth,
                                             out, img_stride, row_stride, bitdepth > 8);
}
void launch_colour_in(const void *in, int64_t img_stride, int64_t row_stride, int B, int nc,
                      int H, int W, int Hp, int Wp, int lossless, int bitdepth, float *planes,
                      cudaStream_t st) {
  int64_t n = (int64_t)B * Hp * Wp;
  k_colour_in<<<grid_for(n), 256, 0, st>>>(in, img_stride, row_stride, bitdepth > 8, B, nc,
                                            H, W, Hp, Wp, lossless, bitdepth, planes);
}
void launch_quantise(const float *y, int64_t n, float delta, int32_t *q, cudaStream_t st) {
  k_quantise<<<grid_for(n), 256, 0, st>>>(y, n, delta, q);
}
void launch_dequantise(const int32_t *q, int64_t n, float delta, float *y, cudaStream_t st) {
  k_dequantise<<<grid_for(n), 256, 0, st>>>(q, n, delta, y);
}

}  // namespace pw
