// Context model of pWave++ (Section 3.2, Figs. 3-5) on FP32 SIMT cores: the
// plain FP32 path. Activations are NHWC float tensors [P, H, W, C] (P =
// planes: images x colour components). Every kernel here computes each
// output from a fixed sequence of FP32 operations, so results do not depend
// on batch composition or launch order (encoder and decoder agree bit for bit).
//
// Layers (a reading of the text; the paper's figures are not available):
//  ConvLSTM: e = conv3x3(1->C)(up(s_prev)), [i f o g] = conv3x3(2C->4C)([e, up(h)]),
//            c = sig(f) up(c) + sig(i) tanh(g), h = sig(o) tanh(c), l = h.
//  step 1:   z = 1x1(l); z += 1x1(dw3x3(lrelu(1x1 z))); z += 1x1(lrelu(1x1(2C) z));
//            (mu, rho) = 1x1(C->2) z.
//  steps 2-4: a = conv3x3(1->C)(m_<k s); z = 1x1(2C->C)[a, l];
//            z += conv3x3(lrelu(conv3x3 z)); (mu, rho) = 1x1(C->2) z.
// The integer-network class runs the same kernels on integers held exactly
// in floats, with integer epilogues (requantisation, clamps, LeakyReLU
// slope 1/128, hard sigmoid / tanh cell, log-scale head): see rq_ll below.
#include "pw_internal.cuh"
#include "ctx_kernels.cuh"
#include "f32x2.cuh"

#include <algorithm>
#include <atomic>

namespace pw {

__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + expf(-x)); }
__device__ __forceinline__ float lrelu(float x) { return x >= 0.f ? x : 0.01f * x; }

// Integer-network class. Every sum is of integers below 2^24 in magnitude
// (at most 2304 products of weights |w| <= 56 and activations |a| <= 127,
// plus a bias |b| <= 2^18), so FP32 FMAs compute it exactly in any order;
// these helpers then work on the exact integer: requantisation by n bits
// (round half up: floor((x + 2^(n-1)) / 2^n); n <= 0 shifts left),
// clamping, LeakyReLU with slope 1/128 (floor division), hard sigmoid
// clamp(2x + 64, 0, 128) and hard tanh clamp(8x, -128, 128) (7 fractional
// bits).
__device__ __forceinline__ long long rq_ll(long long x, int n) {
  return n > 0 ? ((x + (1LL << (n - 1))) >> n) : (x << (-n));
}
__device__ __forceinline__ long long clamp_ll(long long x, long long lim) {
  return x > lim ? lim : (x < -lim ? -lim : x);
}
__device__ __forceinline__ float rq_f(float v, int n, long long lim) {
  return (float)clamp_ll(rq_ll((long long)v, n), lim);
}
__device__ __forceinline__ float lrelu_i(float v) {
  const long long x = (long long)v;
  return (float)(x >= 0 ? x : (x >> 7));
}
__device__ __forceinline__ long long hsig_i(long long x) {
  return x * 2 + 64 < 0 ? 0 : (x * 2 + 64 > 128 ? 128 : x * 2 + 64);
}
__device__ __forceinline__ long long htanh_i(long long x) { return clamp_ll(8 * x, 128); }

// 16 bytes from global to shared memory, asynchronously; zeros when !valid.
__device__ __forceinline__ void cp16(void *dst, const void *src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}

// Generic NHWC convolution, KS x KS (KS = 1 or 3, zero padding). A block
// computes a tile of 32 PX positions of one plane (blockIdx.z) x WG NC output
// channels from blockIdx.y WG NC on: warp w has channels w NC .. + NC - 1, a
// lane PX positions. Weights are [KS*KS][cin][cout_total].
//
// EPI_HEAD computes the step's own positions only (a quarter of the plane;
// nothing else is used): TH rows x TW positions of a row, x = phase + 4 j,
// the phase by the row's parity.
//
// What bounds it: on large planes the loads from shared memory (a thread
// reads PX + NC values for PX NC multiply-adds, and the port returns one
// register of a warp per cycle), on small ones the latency of a block. So the
// input tile and the weights stream through a ring of kStages stages of CK
// input channels by 16-byte asynchronous copies (one barrier per stage, no
// load is waited for while another could run); the input lies in planes of 4
// channels, 16 bytes per position, which lanes read side by side (for the
// head columns are split by x mod 4, so that a step's positions are
// neighbours too); and a plane with few tiles is split into more and smaller
// blocks (see the launcher). Measured with C = 32, 3x3 32 -> 32 / gates / head
// / 1x1: 24 x 32 plane 23 / 58 / 24 / 10..18 us -> 8 / 13 / 8 / 4 us; 192 x 256
// plane 39 / 240 / 41 / 22 us -> 34 / 181 / 18 / 14..20 us (against four chunks
// of synchronous 4-byte loads, and the head at every position).
//
// Every output is one chain in a fixed order: chunks of 8 input channels (4
// for the head of 128), within a chunk tap by tap, channel by channel.
template <int KS, int WG, int NC, int PX, int EPI>
struct SimtCfg {
  static constexpr int CO = WG * NC;
  static constexpr int TW = PX == 4 ? 16 : 8, TH = 32 * PX / TW;
  static constexpr bool kStep = EPI == EPI_HEAD;
  static constexpr int HH = TH + KS - 1;                       // rows staged
  static constexpr int HW = kStep ? 4 * (TW + 1) : TW + KS - 1;   // slots per row
  static constexpr int HP = HH * HW;
  // input channels per stage
  static constexpr int CK = KS == 1 ? (kStep ? 16 : 32) : (NC == 16 ? 4 : 8);
  static constexpr int kStages = 3;
  static constexpr int kInF = CK * HP, kWF = KS * KS * CK * CO;   // floats of a stage
  static constexpr int kHead = kStep ? 8 * TH * TW * 2 : 0;
  static constexpr int kSmem = (kStages * (kInF + kWF) + kHead) * 4;
};
template <int KS, int WG, int NC, int PX, int EPI>
__global__ void __launch_bounds__(32 * WG) k_conv_simt(const __grid_constant__ ConvParams a) {
  using G = SimtCfg<KS, WG, NC, PX, EPI>;
  constexpr int R = KS / 2, NT = 32 * WG, CK = G::CK;
  extern __shared__ __align__(16) float sm_conv[];
  const int t = threadIdx.x;
  const int lane = t & 31, cg = t >> 5;
  const int p = blockIdx.z;
  // tile origin: row y0, column x0 (head: position j0 of a row)
  const int npos = G::kStep ? max(row_count(a.W, step_phase(a.step, 0)),
                                  row_count(a.W, step_phase(a.step, 1)))
                            : a.W;
  const int tiles_x = (npos + G::TW - 1) / G::TW;
  const int y0 = (blockIdx.x / tiles_x) * G::TH, x0 = (blockIdx.x % tiles_x) * G::TW;
  const int co0 = blockIdx.y * G::CO;
  const float *inp = a.in + (int64_t)p * a.H * a.W * a.in_cs + a.in_co;

  const int nchunk = a.cin / CK;
  auto stage_in = [&](int k) { return sm_conv + (k % G::kStages) * (G::kInF + G::kWF); };
  auto load = [&](int k) {
    float *si = stage_in(k), *sw = si + G::kInF;
    const int c0 = k * CK;
    for (int e = t; e < (CK / 4) * G::HP; e += NT) {
      const int g = e % (CK / 4), q = e / (CK / 4);
      const int r = q / G::HW, u = q % G::HW;
      // head: columns 4 x0 - 1 + u, stored as (u mod 4, u / 4)
      const int yy = y0 + r - R, xx = G::kStep ? 4 * x0 - 1 + u : x0 + u - R;
      const bool in = yy >= 0 && yy < a.H && xx >= 0 && xx < a.W;
      const int slot = G::kStep ? (u & 3) * (G::TW + 1) + (u >> 2) : u;
      cp16(si + (g * G::HP + r * G::HW + slot) * 4,
           inp + (in ? ((int64_t)yy * a.W + xx) * a.in_cs + c0 + 4 * g : 0), in);
    }
    for (int e = t; e < KS * KS * CK * (G::CO / 4); e += NT) {
      const int j = e % (G::CO / 4), row = e / (G::CO / 4);   // row = tap * CK + c
      const int tap = row / CK, c = row % CK;
      cp16(sw + row * G::CO + 4 * j,
           a.w + ((int64_t)tap * a.cin + c0 + c) * a.cout_total + co0 + 4 * j, true);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  // positions of this lane: (ty[i], tx[i]) in the tile, slot of tap column dx
  int base[PX], dxo[PX][KS];
#pragma unroll
  for (int i = 0; i < PX; ++i) {
    const int q = lane + 32 * i, ty = q / G::TW, tx = q % G::TW;
    base[i] = ty * G::HW + tx;
#pragma unroll
    for (int dx = 0; dx < KS; ++dx) {
      if (G::kStep) {
        const int v = step_phase(a.step, (y0 + ty) & 1) + dx + (KS == 1 ? 1 : 0);
        dxo[i][dx] = (v & 3) * (G::TW + 1) + (v >> 2);
      } else {
        dxo[i][dx] = dx;
      }
    }
  }
  // accumulators of output channels (2k, 2k + 1) of a position in one packed
  // FP32 pair: each element takes the same fused multiply-adds in the same
  // order as a scalar accumulator
  uint64_t accp[PX][NC / 2];
#pragma unroll
  for (int i = 0; i < PX; ++i)
#pragma unroll
    for (int k = 0; k < NC / 2; ++k) accp[i][k] = 0ull;

#pragma unroll
  for (int k = 0; k < G::kStages - 1; ++k) {
    if (k < nchunk) load(k);
    else asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = 0; k < nchunk; ++k) {
    asm volatile("cp.async.wait_group %0;" ::"n"(G::kStages - 2) : "memory");
    __syncthreads();   // chunk k landed; chunk k - 1 is consumed
    if (k + G::kStages - 1 < nchunk) load(k + G::kStages - 1);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    const float4 *si = reinterpret_cast<const float4 *>(stage_in(k));
    const float *sw = stage_in(k) + G::kInF + cg * NC;
#pragma unroll
    for (int tap = 0; tap < KS * KS; ++tap) {
      const int dy = tap / KS, dx = tap % KS;
#pragma unroll
      for (int g = 0; g < CK / 4; ++g) {
        float xv[PX][4];
#pragma unroll
        for (int i = 0; i < PX; ++i) {
          const float4 f = si[g * G::HP + base[i] + dy * G::HW + dxo[i][dx]];
          xv[i][0] = f.x; xv[i][1] = f.y; xv[i][2] = f.z; xv[i][3] = f.w;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const ulonglong2 *wrow =
              reinterpret_cast<const ulonglong2 *>(sw + (tap * CK + 4 * g + e) * G::CO);
#pragma unroll
          for (int k2 = 0; k2 < NC / 4; ++k2) {
            const ulonglong2 w2 = wrow[k2];
#pragma unroll
            for (int i = 0; i < PX; ++i) {
              const uint64_t xx = f2pack(xv[i][e], xv[i][e]);
              accp[i][2 * k2] = fma2(w2.x, xx, accp[i][2 * k2]);
              accp[i][2 * k2 + 1] = fma2(w2.y, xx, accp[i][2 * k2 + 1]);
            }
          }
        }
      }
    }
  }
  float acc[PX][NC];
#pragma unroll
  for (int i = 0; i < PX; ++i)
#pragma unroll
    for (int k = 0; k < NC / 2; ++k) f2unpack(accp[i][k], acc[i][2 * k], acc[i][2 * k + 1]);

  // plane position of this lane's i-th position
  auto pos = [&](int q, int &y, int &x) {
    const int ty = q / G::TW, tx = q % G::TW;
    y = y0 + ty;
    x = G::kStep ? step_phase(a.step, y & 1) + 4 * (x0 + tx) : x0 + tx;
  };
  if constexpr (EPI == EPI_STORE) {
    // four channels per 16-byte access (channel counts are multiples of
    // 32, channel offsets and row strides multiples of 4 floats)
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      int y, x;
      pos(lane + 32 * i, y, x);
      if (y >= a.H || x >= a.W) continue;
      const int64_t pix = ((int64_t)p * a.H + y) * a.W + x;
#pragma unroll
      for (int j = 0; j < NC; j += 4) {
        const int co = co0 + cg * NC + j;
        const float4 bb = *reinterpret_cast<const float4 *>(a.b + co);
        float v[4] = {acc[i][j] + bb.x, acc[i][j + 1] + bb.y, acc[i][j + 2] + bb.z,
                      acc[i][j + 3] + bb.w};
        float r[4] = {0.f, 0.f, 0.f, 0.f};
        if (a.res) {
          const float4 rr = *reinterpret_cast<const float4 *>(a.res + pix * a.res_cs + a.res_co + co);
          r[0] = rr.x; r[1] = rr.y; r[2] = rr.z; r[3] = rr.w;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (a.iq) {
            // integer class: act on the accumulator, requantise, then the
            // residual (an activation at the same binary point)
            if (a.act) v[k] = lrelu_i(v[k]);
            v[k] = rq_f(v[k], a.rq, 127);
            if (a.res) v[k] = (float)clamp_ll((long long)v[k] + (long long)r[k], 127);
          } else {
            if (a.res) v[k] += r[k];
            if (a.act) v[k] = lrelu(v[k]);
          }
        }
        *reinterpret_cast<float4 *>(a.out + pix * a.out_cs + a.out_co + co) =
            make_float4(v[0], v[1], v[2], v[3]);
      }
    }
  } else if constexpr (EPI == EPI_LSTM) {
    // output channel o = 4 * ch + gate (gate order i, f, o, g)
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      int y, x;
      pos(lane + 32 * i, y, x);
      if (y >= a.H || x >= a.W) continue;
      const int64_t pix = ((int64_t)p * a.H + y) * a.W + x;
      const int Hp = a.H >> a.up, Wp = a.W >> a.up;
      const int64_t ppix = ((int64_t)p * Hp + (y >> a.up)) * Wp + (x >> a.up);
#pragma unroll
      for (int j = 0; j < NC; j += 4) {
        const int o = co0 + cg * NC + j;
        const int ch = o >> 2;
        float gi = acc[i][j] + a.b[o], gf = acc[i][j + 1] + a.b[o + 1];
        float go = acc[i][j + 2] + a.b[o + 2], gg = acc[i][j + 3] + a.b[o + 3];
        float cp = a.first ? 0.f : a.c_prev[ppix * a.C + ch];
        if (a.iq) {
          // integer cell: gates requantised to 4 fractional bits, hard
          // sigmoid / tanh, c and h with 7
          const long long si = hsig_i((long long)rq_f(gi, a.rq, 127));
          const long long sf = hsig_i((long long)rq_f(gf, a.rq, 127));
          const long long so = hsig_i((long long)rq_f(go, a.rq, 127));
          const long long tg = htanh_i((long long)rq_f(gg, a.rq, 127));
          const long long c = clamp_ll(rq_ll(sf * (long long)cp + si * tg, 7), 32767);
          const long long hq = clamp_ll(rq_ll(so * clamp_ll(c, 128), 7), 127);
          a.c_new[pix * a.C + ch] = (float)c;
          a.out[pix * a.out_cs + a.out_co + ch] = (float)hq;
          continue;
        }
        float cn = sigm(gf) * cp + sigm(gi) * tanhf(gg);
        float hn = sigm(go) * tanhf(cn);
        a.c_new[pix * a.C + ch] = cn;
        a.out[pix * a.out_cs + a.out_co + ch] = hn;
      }
    }
  } else {  // EPI_HEAD: z' = res + acc + b over all C channels, then 1x1(C->2)
    static_assert(WG == 8, "the head's partial sums are those of 8 channel groups");
    float(*s_head)[G::TH * G::TW][2] = reinterpret_cast<float(*)[G::TH * G::TW][2]>(
        sm_conv + G::kStages * (G::kInF + G::kWF));
#pragma unroll
    for (int i = 0; i < PX; ++i) {
      int y, x;
      pos(lane + 32 * i, y, x);
      const bool in = y < a.H && x < a.W;
      const int64_t pix = ((int64_t)p * a.H + min(y, a.H - 1)) * a.W + min(x, a.W - 1);
      float rv[NC], pm = 0.f, pr = 0.f;
#pragma unroll
      for (int j = 0; j < NC; j += 4) {  // the residual, 16 bytes at a time
        float4 r4 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in) r4 = *reinterpret_cast<const float4 *>(a.res + pix * a.res_cs + a.res_co + cg * NC + j);
        rv[j] = r4.x; rv[j + 1] = r4.y; rv[j + 2] = r4.z; rv[j + 3] = r4.w;
      }
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        const int co = cg * NC + j;
        float v = acc[i][j] + a.b[co];
        if (a.iq) {
          v = rq_f(v, a.rq, 127);
          if (in) v = (float)clamp_ll((long long)v + (long long)rv[j], 127);
        } else if (in) {
          v += rv[j];
        }
        pm = fmaf(a.wh[co], v, pm);
        pr = fmaf(a.wh[a.cout_total + co], v, pr);
      }
      s_head[cg][lane + 32 * i][0] = pm;
      s_head[cg][lane + 32 * i][1] = pr;
    }
    __syncthreads();
    if (t < G::TH * G::TW) {
      int yy, xx;
      pos(t, yy, xx);
      if (yy < a.H && xx < a.W) {
        float mu = a.bh[0], rho = a.bh[1];
#pragma unroll
        for (int g = 0; g < 8; ++g) { mu += s_head[g][t][0]; rho += s_head[g][t][1]; }
        const int q = step_index(a.W, a.step, yy, xx);
        if (a.iq) {
          // integer head: t = 16 mu and the scale bin j directly
          const long long ti = clamp_ll(rq_ll((long long)mu, a.rq_mu), 1LL << 23);
          long long j = rq_ll((long long)rho, a.rq_rho) + 24;
          j = j < 0 ? 0 : (j > kNJ - 1 ? kNJ - 1 : j);
          a.idx[(int64_t)p * a.idx_stride + q] =
              ((uint32_t)(ti + (1 << 23)) << 7) | (uint32_t)j;
          if (a.mu_out) {
            const int64_t o = (int64_t)p * a.H * a.W + (int64_t)yy * a.W + xx;
            a.mu_out[o] = (float)ti * 0.0625f;
            a.sg_out[o] = __int_as_float(0x3E000000 + ((int)j << 20) + (1 << 19));
          }
        } else {
          a.idx[(int64_t)p * a.idx_stride + q] = pack_index(mu, rho);
          if (a.mu_out) {
            const int64_t o = (int64_t)p * a.H * a.W + (int64_t)yy * a.W + xx;
            a.mu_out[o] = mu;
            a.sg_out[o] = rho > 20.f ? rho : log1pf(expf(rho));
          }
        }
      }
    }
  }
}

// The SIMT producers below: one block per row (plane p, row y), a thread has
// 4 fixed channels (their 9 taps in registers) and walks the row; per output
// the bias, then the taps in raster order.
struct Taps4 {
  float w[4][9], b[4];
  __device__ __forceinline__ Taps4(const float *wt, const float *bias, int c) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
      for (int t = 0; t < 9; ++t) w[k][t] = __ldg(wt + (c + k) * 9 + t);
      b[k] = __ldg(bias + c + k);
    }
  }
};
__device__ __forceinline__ float4 rq4(const float *v, int rqn) {
  if (rqn == kRqFloat) return make_float4(v[0], v[1], v[2], v[3]);
  return make_float4(rq_f(v[0], rqn, 127), rq_f(v[1], rqn, 127), rq_f(v[2], rqn, 127),
                     rq_f(v[3], rqn, 127));
}

// ConvLSTM input: X[..., 0:C] = conv3x3(1->C)(up(s_prev)) + be,
// X[..., C:2C] = up(h_prev) (zero for the first LSTM step).
__global__ void __launch_bounds__(256) k_lstm_in(
    const int32_t *__restrict__ s_prev, const float *__restrict__ h_prev, int h_cs, int h_co,
    const float *__restrict__ we, const float *__restrict__ be, float *__restrict__ X, int H,
    int W, int C, int up, int first, int rqn) {
  const int y = blockIdx.x % H;
  const int64_t p = blockIdx.x / H;
  const int c = 4 * (threadIdx.x % (C / 4)), nx = blockDim.x / (C / 4);
  const Taps4 k(we, be, c);
  const int Hp = H >> up, Wp = W >> up;
  const int32_t *sp = s_prev + p * Hp * Wp;
  for (int x = threadIdx.x / (C / 4); x < W; x += nx) {
    float v[4] = {k.b[0], k.b[1], k.b[2], k.b[3]};
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int yy = y + tap / 3 - 1, xx = x + tap % 3 - 1;
      if (yy < 0 || yy >= H || xx < 0 || xx >= W) continue;
      int32_t sv = __ldg(sp + (int64_t)(yy >> up) * Wp + (xx >> up));
      if (rqn != kRqFloat) sv = min(max(sv, -127), 127);   // integer class input
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = fmaf(k.w[q][tap], (float)sv, v[q]);
    }
    float *o = X + ((p * H + y) * W + x) * 2 * C + c;
    *reinterpret_cast<float4 *>(o) = rq4(v, rqn);
    float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!first)
      h = *reinterpret_cast<const float4 *>(
          h_prev + ((p * Hp + (y >> up)) * Wp + (x >> up)) * h_cs + h_co + c);
    *reinterpret_cast<float4 *>(o + C) = h;
  }
}

// Masked spatial input of steps 2-4: out[..., 0:C] = conv3x3(1->C)(m_<k s) + b.
__global__ void __launch_bounds__(256) k_masked_in(const int32_t *__restrict__ s,
                                                   const float *__restrict__ wa,
                                                   const float *__restrict__ ba,
                                                   float *__restrict__ out, int out_cs, int H,
                                                   int W, int C, int step, int rqn) {
  const int y = blockIdx.x % H;
  const int64_t p = blockIdx.x / H;
  // taps of an earlier step, by x mod 4 (the pattern's period)
  __shared__ uint32_t smask[4];
  if (threadIdx.x < 4) {
    uint32_t m = 0;
    for (int tap = 0; tap < 9; ++tap)
      if (step_of(y + 2 + tap / 3 - 1, threadIdx.x + 4 + tap % 3 - 1) < step) m |= 1u << tap;
    smask[threadIdx.x] = m;
  }
  const int c = 4 * (threadIdx.x % (C / 4)), nx = blockDim.x / (C / 4);
  const Taps4 k(wa, ba, c);
  __syncthreads();
  const int32_t *sp = s + p * H * W;
  for (int x = threadIdx.x / (C / 4); x < W; x += nx) {
    const uint32_t m = smask[x & 3];
    float v[4] = {k.b[0], k.b[1], k.b[2], k.b[3]};
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int yy = y + tap / 3 - 1, xx = x + tap % 3 - 1;
      if (!((m >> tap) & 1u) || yy < 0 || yy >= H || xx < 0 || xx >= W) continue;
      int32_t sv = __ldg(sp + (int64_t)yy * W + xx);
      if (rqn != kRqFloat) sv = min(max(sv, -127), 127);   // integer class input
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = fmaf(k.w[q][tap], (float)sv, v[q]);
    }
    *reinterpret_cast<float4 *>(out + ((p * H + y) * W + x) * out_cs + c) = rq4(v, rqn);
  }
}

// Depthwise 3x3 (zero padding): out = dw(in) + b, NHWC with C channels.
__global__ void __launch_bounds__(256) k_dw3x3(const float *__restrict__ in,
                                               const float *__restrict__ w,
                                               const float *__restrict__ b,
                                               float *__restrict__ out, int H, int W, int C,
                                               int rqn) {
  const int y = blockIdx.x % H;
  const int64_t p = blockIdx.x / H;
  const int c = 4 * (threadIdx.x % (C / 4)), nx = blockDim.x / (C / 4);
  const Taps4 k(w, b, c);
  const float *ip = in + p * H * W * C + c;
  for (int x = threadIdx.x / (C / 4); x < W; x += nx) {
    float v[4] = {k.b[0], k.b[1], k.b[2], k.b[3]};
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int yy = y + tap / 3 - 1, xx = x + tap % 3 - 1;
      if (yy < 0 || yy >= H || xx < 0 || xx >= W) continue;
      const float4 f = __ldg(reinterpret_cast<const float4 *>(ip + ((int64_t)yy * W + xx) * C));
      v[0] = fmaf(k.w[0][tap], f.x, v[0]);
      v[1] = fmaf(k.w[1][tap], f.y, v[1]);
      v[2] = fmaf(k.w[2][tap], f.z, v[2]);
      v[3] = fmaf(k.w[3][tap], f.w, v[3]);
    }
    *reinterpret_cast<float4 *>(out + ((p * H + y) * W + x) * C + c) = rq4(v, rqn);
  }
}

bool &launch_failed() {
  static thread_local bool f = false;
  return f;
}

template <int KS, int WG, int NC, int PX, int EPI>
static void launch_simt_cfg(const ConvParams &a, cudaStream_t st) {
  using G = SimtCfg<KS, WG, NC, PX, EPI>;
  static std::atomic<uint64_t> attr{0};
  once_per_device(attr, [] {
    cudaFuncSetAttribute(k_conv_simt<KS, WG, NC, PX, EPI>,
                         cudaFuncAttributeMaxDynamicSharedMemorySize, G::kSmem);
  });
  const int npos = G::kStep ? std::max(row_count(a.W, step_phase(a.step, 0)),
                                       row_count(a.W, step_phase(a.step, 1)))
                            : a.W;
  const int tiles = ((a.H + G::TH - 1) / G::TH) * ((npos + G::TW - 1) / G::TW);
  if (tiles == 0) return;   // a head of a step without positions
  k_conv_simt<KS, WG, NC, PX, EPI>
      <<<dim3(tiles, a.cout_total / G::CO, a.P), 32 * WG, G::kSmem, st>>>(a);
}

void launch_conv_simt(int ks, const ConvParams &a, int epi, cudaStream_t st) {
  // Large blocks (128 positions x 32 or 64 channels, 8 warps) where they give
  // every SM at least two; else small ones, 64 positions x 8 channels in 2
  // warps (the shared-memory port of an SM then serves few warps, and a tiny
  // plane spreads over the SMs). The head has all channels in a block: 128 or
  // 32 positions.
  const int64_t px = (int64_t)((a.H + 7) / 8) * ((a.W + 15) / 16) * a.P;
  const int co = a.cout_total;
  const bool c64 = co >= 64;
  const bool large = epi == EPI_HEAD ? px / 4 >= 2 * sm_count()
                                     : px * (co / (c64 ? 64 : 32)) >= 2 * sm_count();
  const bool fits = co % 32 == 0 && (!c64 || co % 64 == 0) && a.cin % 32 == 0;
#define PW_CONV_CASE(KS_, EPI_)                                                      \
  if (fits && ks == KS_ && epi == EPI_) {                                            \
    if (!large) launch_simt_cfg<KS_, 2, 4, 2, EPI_>(a, st);                          \
    else if (c64) launch_simt_cfg<KS_, 8, 8, 4, EPI_>(a, st);                        \
    else launch_simt_cfg<KS_, 8, 4, 4, EPI_>(a, st);                                 \
    return;                                                                          \
  }
#define PW_HEAD_CASE(KS_, C_)                                                        \
  if (fits && ks == KS_ && epi == EPI_HEAD && co == C_) {                            \
    if (!large) launch_simt_cfg<KS_, 8, C_ / 8, 1, EPI_HEAD>(a, st);                 \
    else launch_simt_cfg<KS_, 8, C_ / 8, 4, EPI_HEAD>(a, st);                        \
    return;                                                                          \
  }
  PW_CONV_CASE(1, EPI_STORE) PW_CONV_CASE(3, EPI_STORE) PW_CONV_CASE(3, EPI_LSTM)
  PW_HEAD_CASE(1, 32) PW_HEAD_CASE(1, 64) PW_HEAD_CASE(1, 128)
  PW_HEAD_CASE(3, 32) PW_HEAD_CASE(3, 64) PW_HEAD_CASE(3, 128)
#undef PW_CONV_CASE
#undef PW_HEAD_CASE
  set_last_error("no convolution kernel for this shape");
  launch_failed() = true;
}

void launch_lstm_in(const int32_t *s_prev, const float *h_prev, int h_cs, int h_co,
                    const float *we, const float *be, float *X, int P, int H, int W, int C,
                    int up, int first, cudaStream_t st, int rqn) {
  k_lstm_in<<<P * H, 256, 0, st>>>(s_prev, h_prev, h_cs, h_co, we, be, X, H, W, C, up, first,
                                   rqn);
}
void launch_masked_in(const int32_t *s, const float *wa, const float *ba, float *out,
                      int out_cs, int P, int H, int W, int C, int step, cudaStream_t st,
                      int rqn) {
  k_masked_in<<<P * H, 256, 0, st>>>(s, wa, ba, out, out_cs, H, W, C, step, rqn);
}
void launch_dw3x3(const float *in, const float *w, const float *b, float *out, int P, int H,
                  int W, int C, cudaStream_t st, int rqn) {
  k_dw3x3<<<P * H, 256, 0, st>>>(in, w, b, out, H, W, C, rqn);
}

}  // namespace pw
