// Integer entropy-coding kernels: the Laplace CDF table bank and the
// warp-interleaved rANS decoder / encoder.
//
// The paper codes every quantised coefficient with a Laplace distribution
// whose mean and scale come from the context model, using adaptive
// arithmetic coding (Section 3.1). Encoder and decoder must agree bit for
// bit on every frequency table, so the tables are defined by a fixed
// sequence of FP32 operations:
//   table (phi, j), phi in [-8, 7], j in [0, 127]: mean phi / 16, scale
//   b_j = float with bits 0x3E000000 + (j << 20) + (1 << 19);
//   F(u) = exp(u / b) / 2 (u < 0), 1 - exp(-u / b) / 2 (u >= 0) at the 126
//   symbol edges u = k - 62.5 - phi / 16; p = differences of F with the two
//   tails as escape symbols; f = 1 + floor(max(p, 0) * (M - 127)); the
//   signed remainder M - sum f goes to the first largest f.
// exp() here is the library's own routine (Cody-Waite reduction by ln 2 and a
// degree-6 Taylor polynomial in Horner order) written with explicitly
// rounded intrinsics, so no contraction or library-specific rounding enters.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <type_traits>

#include "pw_internal.cuh"
#include "ctx_kernels.cuh"
#include "spec_math.cuh"
#include "cdf_warp.cuh"
#include "tc_ptx.cuh"

namespace pw {

// One warp per table. Lane l owns symbols 4l .. 4l+3 (127 symbols) and the
// CDF entries 4l .. 4l+3 (128 entries: cdf[0] = 0 .. cdf[127] = M).
// coarse (optional): every 8th CDF entry of each table, [table][16], the
// first level of the decoder's symbol search.
__global__ void k_cdf_bank(uint16_t *__restrict__ bank, uint16_t *__restrict__ coarse) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= kNTables) return;
  const int phi = warp / kNJ - 8;
  const int j = warp % kNJ;
  const float mup = __fdiv_rn((float)phi, 16.f);
  const float b = __int_as_float(0x3E000000 + (j << 20) + (1 << 19));
  const float inv_b = __fdiv_rn(1.f, b);
  // F at edges e = 0..125 (edge e separates symbol e and e+1)
  float F[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int e = 4 * lane + i;
    float u = __fsub_rn(__fsub_rn((float)e, 62.5f), mup);
    float z = __fmul_rn(u, inv_b);
    float v;
    if (u < 0.f) v = __fmul_rn(0.5f, exp32_spec(z));
    else v = __fsub_rn(1.f, __fmul_rn(0.5f, exp32_spec(-z)));
    F[i] = (e < kNSym - 1) ? v : 1.f;
  }
  int f[4];
  int run = warp_cdf(F, lane, f);
  uint16_t *row = bank + (size_t)warp * (kNSym + 1);
  if (coarse && (lane & 1) == 0) coarse[(size_t)warp * kCoarse + (lane >> 1)] = (uint16_t)run;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int s = 4 * lane + i;  // cdf index s = sum of f[0..s-1]
    if (s <= kNSym) row[s] = (uint16_t)(s == kNSym ? kM : run);
    run += f[i];
  }
}

// ---------------------------------------------------------------------------
// rANS decoding. One warp decodes a chunk; lane l < nl owns symbols l, l+nl, ...
// Round 0 of every iteration decodes each active lane's main symbol; escape
// symbols are followed by bypass rounds (frequency M/2 per bit). After each
// round the lanes whose state fell below 2^16 read one 16-bit word each, in
// ascending lane order (ballot + popc). All loops are bounded by the chunk
// size and the escape-length limit; overruns set kStCorrupt.

// DecChunk (ctx_kernels.cuh): data = nl u32 states then u16 words; count
// symbols; first = index of its first symbol in the output list.

// SWAR compare of the two u16 entries of w against slot (< 2^15): with
// s2 = (slot | 0x8000) in both halves, each half of s2 - w is
// 0x8000 + slot - e, which lies in [0, 0xFFFF] for every entry e <= 2^15,
// so no borrow crosses the halves and bit 15 of a half is set exactly when
// e <= slot. le2 returns those two bits at positions 0 and 16.
__device__ __forceinline__ uint32_t le2(uint32_t s2, uint32_t w) {
  return ((s2 - w) >> 15) & 0x10001u;
}
// Two consecutive 16-bit words k, k + 1 of a chunk's word stream (0 past the
// end), byte loads so that no alignment is assumed.
__device__ __forceinline__ uint32_t ld_words2(const uint8_t *wp, uint32_t k, uint32_t nwords) {
  uint32_t v = 0;
  if (k < nwords) v = (uint32_t)__ldg(wp + 2 * k) | ((uint32_t)__ldg(wp + 2 * k + 1) << 8);
  if (k + 1 < nwords)
    v |= ((uint32_t)__ldg(wp + 2 * k + 2) << 16) | ((uint32_t)__ldg(wp + 2 * k + 3) << 24);
  return v;
}
// The lanes' initial states of a chunk (lane l < nl: its l-th u32).
__device__ __forceinline__ uint32_t ld_state(const uint8_t *base, int lane, int nl) {
  if (lane >= nl) return kRansL;
  const uint8_t *sp = base + 4 * lane;
  return (uint32_t)sp[0] | ((uint32_t)sp[1] << 8) | ((uint32_t)sp[2] << 16) |
         ((uint32_t)sp[3] << 24);
}
__device__ __forceinline__ bool chunk_ok(const DecChunk &ch) {
  const int nl = ch.lanes;
  return nl >= 1 && nl <= 32 && ch.nbytes >= 4u * nl && !((ch.nbytes - 4u * nl) & 1u);
}

// SIMD min / max of signed 16-bit halves.
__device__ __forceinline__ uint32_t min16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// The sign bits of the halves of a and b as four bytes 0xFF / 0x00 (-1 / 0).
__device__ __forceinline__ int sign4(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("prmt.b32 %0, %1, %2, 0xFDB9;" : "=r"(r) : "r"(a), "r"(b));
  return (int)r;
}
// 16 bytes from global to shared memory, asynchronously.
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}
__device__ __forceinline__ void trio_sync(int id) {
  asm volatile("bar.sync %0, 96;" ::"r"(id) : "memory");
}

// Laplace decoder: K chunks per block (host: as few as keep every SM at one
// block), each served by three warps. Warp w < K decodes chunk w; warp K + w
// turns its packed indices into table rows, eight rounds at a time and ahead
// of it; warp 2 K + w turns decoded residuals into values at their positions
// behind it. The chunk's serial chain then holds nothing but the coder
// itself. (With both helper jobs in one warp, the helper was the slower one:
// 88 us instead of 66 us for the 384-round chunk below.)
//
// What bounds it: one dependent chain per chunk (state -> symbol -> state ->
// shared word stream), a few hundred rounds long, one warp wide; the SMs are
// otherwise idle. A round is laid out for the shortest chain (it takes 0.16
// us, about 330 cycles; of them about 35 are the shared-memory load, 45 the
// shuffle and the ballot, 25 the population count):
//  * The block first copies the table rows its symbols use (all indices of
//    the pass are known) into shared memory, fine level and coarse level;
//    rows beyond the shared memory's capacity, the ones whose scale is
//    furthest from the chunk's mean, are read through L1, where the helper
//    warp prefetches them (a second loop, compiled apart).
//  * Level 1 (16 coarse entries, in registers a round ahead): T = 0x8000 +
//    slot - e for the entries e, two per word; the signs of T counted by
//    prmt + dp4a give the address of the 8-entry block directly.
//  * Level 2 needs no index: with lo / hi the largest entry <= slot and the
//    smallest > slot, min T (signed) = 0x8000 + slot - lo and max T =
//    0x8000 + slot - hi, so the frequency is min T - max T and the new state
//    f (x >> 15) + (min T - 0x8000). hi may be the next block's first entry,
//    which is a coarse entry, so the max runs over level 1 too. The symbol's
//    index (for the output) is counted off the chain.
//  * Lanes without a symbol in a round get a dummy row whose only symbol
//    fills the interval (the state stays), so the round has no predicates.
//    Such a lane reads no word as long as its state is at least 2^16, which
//    every state of an encoder is and stays. A chunk with an initial state
//    below that is decoded round by round, where only lanes with a symbol
//    may read.
//  * Renormalisation: lane l holds word ptr + l of the stream; a lane's word
//    is one shuffle by its rank among the lanes that need one. Words come
//    from a ring in shared memory, refilled 64 at a time from a register
//    that was loaded one refill earlier.
//  * Escapes and refills are looked for once per four rounds (a branch costs
//    about 70 cycles of a round); see the loop.
//  * A corrupt chunk (words run out, an escape beyond the limit) ends where
//    that branch finds it: the decoding warp passes the barriers left, and no
//    further value is written. (Asked for at the head of every batch it cost
//    the cases 1.5 %, by a variable loop bound 0.7 %; so, nothing.)
// Measured, decoder launches alone, GB300: 3 chunks of 12,288 symbols on 32
// lanes (384 rounds) 207 -> 68 us, of 4,096 (128 rounds) 72 -> 27 us, 192
// chunks of 16,200 273 -> 98 us, 1,200 chunks of 16,384 453 -> 202 us, against
// one warp per chunk with the tables read through L1.
//
// Output: positions of a four-step subband plane (step >= 0), or a linear
// array (step < 0, out[first + i]).
// kRag (ragged batches, step >= 0): planes of different sizes on one canvas
// of width w. A chunk's symbols are the step positions of its own plane,
// whose subband width is ext[plane].y >> esh; their packed indices sit at
// the canvas's step positions (the context model runs on the canvas) and
// their values go to canvas rows of stride w.
constexpr int kRound = 8;                        // rounds per batch
constexpr int kGroup = 4;                        // rounds decoded between two checks
constexpr uint32_t kRowBytes = 2 * (kNSym + 1) + 2 * kCoarse;   // 288
constexpr uint32_t kMapBytes = 2 * kNTables;     // table id -> shared row
constexpr uint32_t kRowBufBytes = 3 * kRound * 32 * 4;   // row of each symbol, 3 batches
constexpr uint32_t kResBytes = 2 * kRound * 32 * 4;      // residuals, 2 batches
constexpr uint32_t kRing = 512, kFill = 384;     // words of the ring, of them loaded ahead
constexpr uint32_t kRingBytes = 2 * (kRing + 32);   // (the first 32 words again at the end)
constexpr uint32_t kStopOff = kRowBufBytes + kResBytes + kRingBytes;   // first batch not written
constexpr uint32_t kPairBytes = kStopOff + 16;
constexpr int kMaxEscPasses = 2 * kMaxEscBits + 2;   // one bit each from states below 2^16
constexpr uint32_t kRowGlobal = 0x80000000u;     // row entry: table id in global memory
static_assert(2 * kNTables + 256 <= (int)kPairBytes, "row list and partial sums fit a pair area");

// Positions of a chunk's symbols, walked with a constant stride.
struct StepCursor {
  int y2, r, dq, dr, pair;
  __device__ __forceinline__ StepCursor(int q0, int stride, int pair_) : pair(pair_) {
    y2 = q0 / pair; r = q0 - y2 * pair;
    dq = stride / pair; dr = stride - dq * pair;
  }
  __device__ __forceinline__ void next() {
    y2 += dq; r += dr;
    if (r >= pair) { r -= pair; ++y2; }
  }
};

template <bool kRag>
__global__ void __launch_bounds__(768) k_rans_decode(
    const DecChunk *__restrict__ chunks, int nchunks, int K, int cap,
    const uint16_t *__restrict__ bank, const uint16_t *__restrict__ coarse,
    const uint32_t *__restrict__ idx, int64_t idx_stride, int32_t *__restrict__ out,
    int64_t out_stride, int w, int step, uint32_t *status, const int2 *__restrict__ ext,
    int esh) {
  extern __shared__ __align__(16) uint8_t sm[];
  const int t = threadIdx.x, nt = blockDim.x, warp = t >> 5, lane = t & 31;
  const int c0 = blockIdx.x * K, nc = min(K, nchunks - c0);
  uint16_t *map = reinterpret_cast<uint16_t *>(sm);
  const uint32_t rows0 = kMapBytes + (uint32_t)K * kPairBytes;   // row 0: the dummy
  const uint4 *bank4 = reinterpret_cast<const uint4 *>(bank);
  const uint4 *coarse4 = reinterpret_cast<const uint4 *>(coarse);
  const int ae = step >= 0 ? step_phase(step, 0) : 0, ao = step >= 0 ? step_phase(step, 1) : 0;
  const int neC = row_count(w, ae), pairC = neC + row_count(w, ao);

  // ---- the block's table rows -------------------------------------------
  {
    uint8_t *flag = sm;                                           // [kNTables]
    uint16_t *list = reinterpret_cast<uint16_t *>(sm + kMapBytes);   // table of each row
    uint32_t *part = reinterpret_cast<uint32_t *>(sm + kMapBytes + 2 * kNTables);
    for (int i = t; i < kNTables / 4; i += nt) reinterpret_cast<uint32_t *>(flag)[i] = 0u;
    if (t < 10) part[t] = 0u;
    __syncthreads();
    uint32_t sj = 0, sn = 0;
    for (int c = 0; c < nc; ++c) {
      const DecChunk ch = chunks[c0 + c];
      if (!chunk_ok(ch)) continue;
      const uint32_t *ip = idx + (int64_t)ch.plane * idx_stride;
      const int count = (int)ch.count;
      if constexpr (kRag) {
        const int wq = ext[ch.plane].y >> esh, ne = row_count(wq, ae), pair = ne + row_count(wq, ao);
        if (pair == 0 || wq > w) continue;
        StepCursor cu((int)ch.first + t, nt, pair);
        for (int i = t; i < count; i += nt, cu.next()) {
          const uint32_t v = __ldg(ip + (int64_t)cu.y2 * pairC +
                                   (cu.r < ne ? cu.r : neC + (cu.r - ne)));
          flag[(v + 1024u) & (kNTables - 1)] = 1;
          sj += v & (kNJ - 1);
          ++sn;
        }
      } else {
        // 16-byte loads from the aligned address below the first index on
        // (every group loaded holds one of the chunk's indices, so it lies in
        // the allocation, whose granularity is larger)
        const uint32_t *cp = ip + ch.first;
        const int off = (int)((reinterpret_cast<uintptr_t>(cp) >> 2) & 3);
        const uint4 *cp4 = reinterpret_cast<const uint4 *>(cp - off);
        const int lo = off, hi = off + count, n4 = (hi + 3) >> 2;
        for (int g0 = t; g0 < n4; g0 += 4 * nt) {
          uint4 v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (g0 + u * nt < n4) v[u] = __ldg(cp4 + g0 + u * nt);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int i = 4 * (g0 + u * nt) + k;
              if (i >= lo && i < hi) {
                flag[(e[k] + 1024u) & (kNTables - 1)] = 1;
                sj += e[k] & (kNJ - 1);
                ++sn;
              }
            }
          }
        }
      }
    }
    sj = __reduce_add_sync(0xffffffffu, sj);
    sn = __reduce_add_sync(0xffffffffu, sn);
    if (lane == 0) { atomicAdd(&part[8], sj); atomicAdd(&part[9], sn); }
    __syncthreads();
    // rows in order of |scale bin - mean bin|: threads 0..255 take 8 tables
    // (half a scale bin) each
    const int j0 = min(kNJ - 1, (int)(part[8] / max(part[9], 1u)));
    const int d = min(j0, kNJ - 1 - j0);
    const int jp = t >> 1;
    const int j = jp <= 2 * d ? j0 + ((jp & 1) ? (jp + 1) / 2 : -(jp / 2))
                              : (j0 < kNJ - 1 - j0 ? jp : kNJ - 1 - jp);
    uint32_t used = 0;
    if (t < 256)
#pragma unroll
      for (int k = 0; k < 8; ++k)
        used |= (flag[(((t & 1) * 8 + k) * kNJ) + j] ? 1u : 0u) << k;
    uint32_t incl = __popc(used);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (warp < 8 && lane == 31) part[warp] = incl;
    __syncthreads();   // every flag read: the map may be written over them
    uint32_t rank = incl - __popc(used), total = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const uint32_t v = part[k];
      if (k < warp) rank += v;
      total += v;
    }
    if (t < 256)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int tid = ((t & 1) * 8 + k) * kNJ + j;
        if ((used >> k) & 1u) {
          map[tid] = rank < (uint32_t)cap ? (uint16_t)(rank + 1) : (uint16_t)0xFFFFu;
          if (rank < (uint32_t)cap) list[rank] = (uint16_t)tid;
          ++rank;
        }
      }
    // the dummy row: entries 0..7 zero, the rest M
    uint4 *rows = reinterpret_cast<uint4 *>(sm + rows0);
    if (t < 18) {
      const uint32_t m2 = kM | (kM << 16);
      rows[t] = t == 0 ? make_uint4(0u, 0u, 0u, 0u)
                       : make_uint4(t == 16 ? kM << 16 : m2, m2, m2, m2);
    }
    if (t == 0) part[10] = total;
    __syncthreads();
    const int n18 = (int)min(total, (uint32_t)cap) * 18;
    for (int e = t; e < n18; e += nt) {
      const int r = e / 18, k = e - 18 * r;
      const uint32_t tid = list[r];
      cp_async16(rows + 18 + e, k < 16 ? bank4 + tid * 16 + k : coarse4 + tid * 2 + (k - 16));
    }
    cp_async_wait();
  }
  const bool over = reinterpret_cast<uint32_t *>(sm + kMapBytes + 2 * kNTables)[10] > (uint32_t)cap;
  __syncthreads();

  // ---- three warps per chunk ------------------------------------------------
  const int role = warp / K, pr = warp - role * K;
  if (role > 2 || pr >= nc) return;
  const DecChunk ch = chunks[c0 + pr];
  const int nl = ch.lanes, count = (int)ch.count;
  int wq = w, ne = neC, pair = pairC;
  if constexpr (kRag) {
    wq = ext[ch.plane].y >> esh;
    ne = row_count(wq, ae);
    pair = ne + row_count(wq, ao);
  }
  // (a step without positions has no chunks)
  if (!chunk_ok(ch) || (step >= 0 && (pair == 0 || wq > w))) {
    if (role == 0 && lane == 0) atomicOr(status, kStCorrupt);
    return;
  }
  const uint32_t pbase = kMapBytes + (uint32_t)pr * kPairBytes;
  const int niter = (count + nl - 1) / nl;
  const int nbatch = (niter + kRound - 1) / kRound;
  const int bar = 1 + pr;
  // first batch that is not written (batch b sets it to b or leaves it, which
  // the third warp sees after barrier b + 1)
  volatile int *const stop = reinterpret_cast<volatile int *>(sm + pbase + kStopOff);

  if (role > 0) {
    // ---- helper warps: 1 prepares table rows, 2 writes values -----------------
    const uint32_t *ip = idx + (int64_t)ch.plane * idx_stride + (kRag ? 0 : ch.first);
    const bool live = lane < nl;
    StepCursor cl((int)ch.first + lane, nl, step >= 0 ? pair : 1), co = cl;   // loads, output
    // packed indices of batch b, loaded a batch before their use
    uint32_t v[kRound];
    auto load = [&](int b) {
#pragma unroll
      for (int u = 0; u < kRound; ++u) {
        const int i = (b * kRound + u) * nl + lane;
        const int64_t q = kRag ? (int64_t)cl.y2 * pairC + (cl.r < ne ? cl.r : neC + (cl.r - ne))
                               : (int64_t)i;
        v[u] = live && i < count ? __ldg(ip + q) : 0u;
        if (kRag) cl.next();
      }
    };
    if (role == 1) {
      auto prepare = [&](int b) {
        uint32_t *rb = reinterpret_cast<uint32_t *>(sm + pbase) + (b % 3) * kRound * 32 + lane;
#pragma unroll
        for (int u = 0; u < kRound; ++u) {
          const int i = (b * kRound + u) * nl + lane;
          uint32_t e = rows0;
          if (live && i < count) {
            const uint32_t tid = (v[u] + 1024u) & (kNTables - 1);
            const uint32_t m = map[tid];
            e = rows0 + m * kRowBytes;
            if (m == 0xFFFFu) {
              e = kRowGlobal | tid;
              const uint16_t *fr = bank + (size_t)tid * (kNSym + 1);
              asm volatile("prefetch.global.L1 [%0];" ::"l"(fr));
              asm volatile("prefetch.global.L1 [%0];" ::"l"(fr + 64));
              asm volatile("prefetch.global.L1 [%0];" ::"l"(coarse + (size_t)tid * kCoarse));
            }
          }
          rb[u * 32] = e;
        }
        load(b + 1);
      };
      load(0);
      prepare(0);
      prepare(1);
      for (int b = 0; b < nbatch; ++b) {
        trio_sync(bar);
        prepare(b + 2);
      }
      trio_sync(bar);
      return;
    }
    int32_t *outp = out + (int64_t)ch.plane * out_stride + (step >= 0 ? 0 : ch.first);
    auto finish = [&](int b) {
      const int32_t *rs = reinterpret_cast<const int32_t *>(sm + pbase + kRowBufBytes) +
                          (b & 1) * kRound * 32 + lane;
#pragma unroll
      for (int u = 0; u < kRound; ++u) {
        const int i = (b * kRound + u) * nl + lane;
        int o = i;
        if (step >= 0) {   // a plane has less than 2^31 samples
          o = (co.r < ne ? 2 * co.y2 * w + ae + 4 * co.r
                         : (2 * co.y2 + 1) * w + ao + 4 * (co.r - ne));
          co.next();
        }
        if (live && i < count) {
          int ctr, tid;
          unpack_index(v[u], ctr, tid);
          outp[o] = ctr + rs[u * 32];
        }
      }
      load(b + 1);
    };
    load(0);
    for (int b = 0; b < nbatch; ++b) {
      trio_sync(bar);
      if (b > 0 && *stop >= b) finish(b - 1);
    }
    trio_sync(bar);
    if (nbatch > 0 && *stop >= nbatch) finish(nbatch - 1);
    return;
  }

  // ---- decoding warp ---------------------------------------------------------
  const uint32_t nwords = (ch.nbytes - 4u * nl) >> 1;
  const uint8_t *wp = ch.data + 4 * nl;
  uint32_t x = ld_state(ch.data, lane, nl);
  // (a round and its word leave a state below 2^16 only if it was there)
  const bool low = __any_sync(0xffffffffu, x < kRansL);
  uint16_t *ring = reinterpret_cast<uint16_t *>(sm + pbase + kRowBufBytes + kResBytes);
  // words k, k + 1 (k = base + 2 lane) into the ring
  auto put = [&](uint32_t k, uint32_t v) {
    const uint32_t o = k & (kRing - 1);
    *reinterpret_cast<uint32_t *>(ring + o) = v;
    if (o < 32u) *reinterpret_cast<uint32_t *>(ring + kRing + o) = v;
  };
  {
    uint32_t wi[kFill / 64];
#pragma unroll
    for (uint32_t k = 0; k < kFill / 64; ++k) wi[k] = ld_words2(wp, 64 * k + 2 * lane, nwords);
#pragma unroll
    for (uint32_t k = 0; k < kFill / 64; ++k) put(64 * k + 2 * lane, wi[k]);
  }
  uint32_t wnxt = ld_words2(wp, kFill + 2 * lane, nwords);
  uint32_t wb = 0, ptr = 0;   // next word; the ring holds words [wb, wb + kFill)
  __syncwarp();
  uint32_t took = 0;   // words of the round before, added to ptr a round late
  const uint32_t lt = (1u << lane) - 1u;
  auto refill = [&]() {
    put(wb + kFill + 2 * lane, wnxt);
    wb += 64;
    wnxt = ld_words2(wp, wb + kFill + 2 * lane, nwords);
    __syncwarp();
  };
  bool bad = false;
  if (lane == 0) *stop = 0x7FFFFFFF;

  auto loop = [&](auto gen) {
    constexpr bool kGen = decltype(gen)::value;
    auto ldrow = [&](uint32_t e, uint32_t byte) -> uint4 {
      if (kGen && (e & kRowGlobal)) {
        const uint32_t tid = e & (kNTables - 1);
        return byte >= 256u ? __ldg(coarse4 + tid * 2 + ((byte - 256u) >> 4))
                            : __ldg(bank4 + tid * 16 + (byte >> 4));
      }
      return *reinterpret_cast<const uint4 *>(sm + e + byte);
    };
    auto lds = [&](uint32_t a) { return *reinterpret_cast<const uint32_t *>(sm + a); };
    // One round up to the shuffle: from the state and the coarse level (ca,
    // cb) of row rw, the lanes that need a word (m) and the symbol's residual;
    // shadow() runs while the fine level's load is in flight.
    auto round = [&](uint32_t rw, const uint4 ca, const uint4 cb, uint32_t &m, int &r,
                     auto shadow) {
      // level 1
      uint32_t s2;
      asm("prmt.b32 %0, %1, %1, 0x1010;" : "=r"(s2) : "r"(x));
      s2 |= 0x80008000u;
      const uint32_t t0 = s2 - ca.x, t1 = s2 - ca.y, t2 = s2 - ca.z, t3 = s2 - ca.w;
      const uint32_t t4 = s2 - cb.x, t5 = s2 - cb.y, t6 = s2 - cb.z, t7 = s2 - cb.w;
      constexpr int km16 = (int)0xF0F0F0F0u, km1 = (int)0xFFFFFFFFu;   // -16, -1 per byte
      const int na = __dp4a(sign4(t2, t3), km16, __dp4a(sign4(t0, t1), km16, -16));
      const int nb = __dp4a(sign4(t6, t7), km16, __dp4a(sign4(t4, t5), km16, 0));
      const uint32_t blk = (uint32_t)(na + nb);   // 16 x block, byte offset in the row
      const uint4 f = ldrow(rw, blk);
      shadow();
      const uint32_t mxc = max16x2(max16x2(max16x2(t0, t1), max16x2(t2, t3)),
                                   max16x2(max16x2(t4, t5), max16x2(t6, t7)));
      // level 2
      const uint32_t u0 = s2 - f.x, u1 = s2 - f.y, u2 = s2 - f.z, u3 = s2 - f.w;
      uint32_t mn = min16x2(min16x2(u0, u1), min16x2(u2, u3));
      uint32_t mx = max16x2(max16x2(max16x2(u0, u1), max16x2(u2, u3)), mxc);
      mn = min16x2(mn, mn >> 16);   // low half: the minimum of both (the high half is unused)
      mx = max16x2(mx, mx >> 16);
      x = ((mn - mx) & 0xFFFFu) * (x >> kLogM) + (mn & 0x7FFFu);
      m = __ballot_sync(0xffffffffu, x < kRansL);
      r = __dp4a(sign4(u2, u3), km1, __dp4a(sign4(u0, u1), km1, (int)(blk >> 1) - 2 - kT));
    };
    auto is_esc = [](int r) { return (uint32_t)(r + kT) > 2u * kT; };   // first or last symbol
    const uint32_t rb0 = pbase + 4 * lane, rs0 = rb0 + kRowBufBytes;
    auto row_at = [&](uint32_t it) {   // table row of round it
      return lds(rb0 + (it % (3 * kRound)) * 128u);
    };
    uint32_t row = 0, rown = 0;   // rows of the next round and the one after
    uint4 ca, cb;                 // coarse level of the next round
    uint32_t rb = rb0;            // row buffer of the batch
    for (int b = 0; b < nbatch; ++b) {
      trio_sync(bar);   // batches b and b + 1 prepared, the residuals of b - 2 consumed
      if (b == 0) {
        row = lds(rb);
        rown = lds(rb + 128);
        ca = ldrow(row, 256u);
        cb = ldrow(row, 272u);
      }
      const uint32_t rbn = rb == rb0 + 2 * kRound * 128 ? rb0 : rb + kRound * 128;
      // always kRound rounds: past the chunk's end every lane has the dummy row
#pragma unroll 1
      for (int g = 0; g < kRound; g += kGroup) {
        // A group of rounds without a branch. Escapes are rare: they are
        // looked for once per group, and a group that has one is done again
        // from its start, round by round.
        const uint32_t x0 = x;
        const uint32_t p0 = ptr + took;
        const uint32_t rsg = rs0 + ((b & 1) * kRound + g) * 128u;
        bool esc = low;
#pragma unroll
        for (int u = 0; u < kGroup; ++u) {
          const uint32_t rw = row;
          const uint4 c0v = ca, c1v = cb;
          uint32_t m, wcur;
          int r;
          round(rw, c0v, c1v, m, r, [&]() {
            // the words from ptr on (one per lane), the next round's rows
            ptr += took;
            wcur = ring[(ptr & (kRing - 1)) + lane];
            row = rown;
            ca = ldrow(row, 256u);
            cb = ldrow(row, 272u);
            rown = lds(g + u + 2 < kRound ? rb + (g + u + 2) * 128u
                                          : rbn + (g + u + 2 - kRound) * 128u);
          });
          const uint32_t wv = __shfl_sync(0xffffffffu, wcur, __popc(m & lt));
          x = x < kRansL ? (x << 16) | wv : x;
          took = __popc(m);
          *reinterpret_cast<int32_t *>(sm + rsg + u * 128) = r;
          esc = esc || is_esc(r);
        }
        // (refills may be a round late: ptr - wb < 64 + 32 at a group's start)
        if (__builtin_expect(__any_sync(0xffffffffu, esc || ptr - wb >= 64u), 0)) {
          if (__any_sync(0xffffffffu, esc)) {
            x = x0;
            ptr = p0;
            took = 0;
#pragma unroll 1
            for (int u = 0; u < kGroup; ++u) {
              const uint32_t it = (uint32_t)(b * kRound + g + u);
              const uint32_t rw = row_at(it);
              uint32_t m;
              int r;
              round(rw, ldrow(rw, 256u), ldrow(rw, 272u), m, r, [] {});
              // lanes with a symbol in this round
              const int nsym = min(nl, max(0, count - (int)it * nl));
              m &= (uint32_t)((1ull << nsym) - 1);
              while (ptr - wb >= 64u) refill();
              if ((m >> lane) & 1u)
                x = (x << 16) | ring[(ptr & (kRing - 1)) + __popc(m & lt)];
              ptr += __popc(m);
              // Escapes: ones up to a zero, then as many bits, one bypass bit
              // a round, the lanes whose state fell below 2^16 taking a word
              // after each, in lane order. A bypass bit is bit 14 of the
              // state, and is deleted from it; so a state of n + 16 bits gives
              // its next n bits at once (bit 14 first) and takes a word after
              // the n-th, later one every 16 bits. Hence passes of up to n
              // bits per lane: within a pass a lane's word comes in the order
              // (rounds to its first word, lane).
              bool pend = is_esc(r);
              int kcnt = 0, e = 0;
              bool tail = false;   // in the bits after the zero
              uint32_t v = 0;
              for (int pass = 0; pass < kMaxEscPasses; ++pass) {
                if (!__any_sync(0xffffffffu, pend)) break;
                bool nd = false;
                if (pend) {
                  const int n = max(1, 16 - __clz(x));
                  uint32_t bits = x >> 14;
                  int left = n;
                  if (!tail) {
                    const int c = min(__ffs(~bits) - 1, n);
                    kcnt += c;
                    if (kcnt > kMaxEscBits) bad = true;   // also when the zero follows
                    left -= c;
                    if (left > 0) {
                      tail = true;
                      v = 1;
                      --left;
                      bits >>= c + 1;
                    }
                  }
                  if (tail) {
                    const int q = min(kcnt, left);
                    v = (v << q) | ((__brev(bits) >> 1) >> (31 - q));
                    kcnt -= q;
                    left -= q;
                  }
                  x = ((x >> (14 + n - left)) << 14) | (x & 0x3FFFu);
                  nd = left == 0;
                  if (pass == 0) e = n - 1;
                  if (bad || (tail && kcnt == 0)) pend = false;
                }
                uint32_t eq = __ballot_sync(0xffffffffu, nd), less = 0;
                const uint32_t all = eq;
                if (all) {
#pragma unroll
                  for (int k = 3; k >= 0; --k) {
                    const uint32_t one = __ballot_sync(0xffffffffu, (e >> k) & 1);
                    if ((e >> k) & 1) { less |= eq & ~one; eq &= one; }
                    else eq &= ~one;
                  }
                  while (ptr - wb >= 64u) refill();
                  if (nd)
                    x = (x << 16) |
                        ring[(ptr & (kRing - 1)) + __popc(less) + __popc(eq & lt)];
                  ptr += __popc(all);
                }
              }
              if (pend) bad = true;
              if (is_esc(r)) r = r < 0 ? -(int)(v - 1) - kT - 1 : (int)(v - 1) + kT + 1;
              *reinterpret_cast<int32_t *>(sm + rsg + u * 128) = r;
            }
          }
          while (ptr + took - wb >= 64u) refill();
          if (__builtin_expect(__any_sync(0xffffffffu, bad || ptr + took > nwords), 0)) {
            if (lane == 0) *stop = b;
            bad = true;
            __syncwarp();
            for (; b < nbatch; ++b) trio_sync(bar);
            return;
          }
        }
      }
      rb = rbn;
    }
    ptr += took;
    trio_sync(bar);
  };
  if (over) loop(std::integral_constant<bool, true>());
  else loop(std::integral_constant<bool, false>());
  // words past the end read as zeros, so an overrun shows in ptr
  if (lane < nl && x != kRansL) bad = true;
  if (ptr != nwords) bad = true;
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kStCorrupt);
}

// Symbol search: the largest s in [0, 126] with t[s] <= slot, in two levels:
// the table's 16 coarse entries (every 8th, shared memory) give the block
// b = s / 8, one 16-byte load gives its 8 entries. The entries are strictly
// increasing with t[0] = 0, t[127] = M = 2^15 > slot, and all are <= 2^15,
// so the SWAR counts below are exactly that s. Returns s; lo = t[s],
// hi = t[s + 1].
// The table's coarse entries come in registers (c0 = entries 0..7, c1 =
// 8..15, two per word, low half first), loaded one round ahead; the entry
// after block b also comes from them.
__device__ __forceinline__ int cdf_search_r(const uint16_t *__restrict__ row, const uint4 c0,
                                            const uint4 c1, uint32_t slot, uint32_t &lo,
                                            uint32_t &hi) {
  const uint32_t s2 = (slot | 0x8000u) * 0x10001u;
  uint32_t a = le2(s2, c0.x) + le2(s2, c0.y) + le2(s2, c0.z) + le2(s2, c0.w) + le2(s2, c1.x) +
               le2(s2, c1.y) + le2(s2, c1.z) + le2(s2, c1.w);
  const int b = (int)((a & 0xFFFFu) + (a >> 16)) - 1;
  const uint4 f = __ldg(reinterpret_cast<const uint4 *>(row + 8 * b));
  a = le2(s2, f.x) + le2(s2, f.y) + le2(s2, f.z) + le2(s2, f.w);
  const int i = (int)((a & 0xFFFFu) + (a >> 16)) - 1;
  // coarse entry b + 1 (clamped; its low 16 bits are what is used)
  const int bn = min(b + 1, kCoarse - 1), wn = bn >> 1;
  const uint32_t q0 = (wn & 1) ? c0.y : c0.x, q1 = (wn & 1) ? c0.w : c0.z;
  const uint32_t q2 = (wn & 1) ? c1.y : c1.x, q3 = (wn & 1) ? c1.w : c1.z;
  const uint32_t r0 = (wn & 2) ? q1 : q0, r1 = (wn & 2) ? q3 : q2;
  const uint32_t wsel = (wn & 4) ? r1 : r0;
  const uint32_t nxt = (bn & 1) ? (wsel >> 16) : wsel;
  const int wi = i >> 1;
  const uint32_t w0 = (wi & 2) ? ((wi & 1) ? f.w : f.z) : ((wi & 1) ? f.y : f.x);
  const uint32_t w1 = (wi & 2) ? ((wi & 1) ? nxt : f.w) : ((wi & 1) ? f.z : f.y);
  const uint32_t pair = (i & 1) ? __funnelshift_r(w0, w1, 16) : w0;
  lo = pair & 0xFFFFu;
  hi = pair >> 16;
  return 8 * b + i;
}

// Decoder of logistic-mixture chunks: one warp per chunk, up to 8 per block.
// Every symbol has its own table row in global memory (rows = the step's,
// kMixRow entries each, the coarse level in the row's last 16), written just
// before by the mixture head; idx holds the centres. The coarse entries of a
// lane's symbol are loaded two rounds ahead, its fine row prefetched into L1
// two rounds ahead. The renormalisation words come from a 128-word window
// that the warp keeps in registers (lane l holds words wb + 2l, wb + 2l + 1
// in cur and the same 64 words later in nxt) and reads with shuffles; the
// window moves by 64 words once 64 are consumed, loading the next 64 one
// shift ahead. Output: the step's positions of a plane of width w.
__global__ void __launch_bounds__(256) k_rans_decode_mix(
    const DecChunk *__restrict__ chunks, int nchunks, const uint16_t *__restrict__ rows,
    const uint32_t *__restrict__ idx, int64_t idx_stride, int32_t *__restrict__ out,
    int64_t out_stride, int w, int step, uint32_t *status) {
  const int cw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (cw >= nchunks) return;
  const DecChunk ch = chunks[cw];
  const int nl = ch.lanes;
  const int count = (int)ch.count;
  const int ae = step_phase(step, 0), ao = step_phase(step, 1);
  const int ne = row_count(w, ae), pair = ne + row_count(w, ao);
  // chunk layouts hold no empty chunks, and none of a step without positions
  if (!chunk_ok(ch) || count == 0 || pair == 0) {
    if (lane == 0) atomicOr(status, kStCorrupt);
    return;
  }
  const uint32_t nwords = (ch.nbytes - 4u * nl) >> 1;
  uint32_t x = ld_state(ch.data, lane, nl);
  const uint8_t *wp = ch.data + 4 * nl;
  uint32_t wb = 0;
  uint32_t wcur = ld_words2(wp, 2 * lane, nwords), wnxt = ld_words2(wp, 64 + 2 * lane, nwords);
  uint32_t ptr = 0;
  bool bad = false;
  const uint32_t lt = (1u << lane) - 1u;
  // word k of the stream (k - wb in [0, 128) for every calling lane)
  auto word = [&](uint32_t k) -> uint32_t {
    const uint32_t r = k - wb;
    const int src = (int)((r & 63u) >> 1);
    const uint32_t a = __shfl_sync(0xffffffffu, wcur, src);
    const uint32_t b = __shfl_sync(0xffffffffu, wnxt, src);
    const uint32_t v = r < 64u ? a : b;
    return (r & 1u) ? (v >> 16) : (v & 0xFFFFu);
  };
  auto advance = [&](uint32_t n) {
    ptr += n;
    if (ptr - wb >= 64u) {
      wcur = wnxt;
      wnxt = ld_words2(wp, wb + 128 + 2 * lane, nwords);
      wb += 64;
    }
  };
  const uint32_t *idxp = idx + (int64_t)ch.plane * idx_stride + ch.first;
  int32_t *outp = out + (int64_t)ch.plane * out_stride;
  const int niter = (count + nl - 1) / nl;
  StepCursor pos((int)ch.first + lane, nl, pair);   // output position of the lane's symbol
  // centres of this lane's next two symbols, the coarse rows likewise
  uint32_t ctr_a = (lane < nl && lane < count) ? __ldg(idxp + lane) : 0u;
  uint32_t ctr_b = (lane < nl && lane + nl < count) ? __ldg(idxp + lane + nl) : 0u;
  // row of the chunk's symbol i (inactive lanes use the first one)
  const uint16_t *mrows = rows + ((int64_t)ch.plane * idx_stride + ch.first) * kMixRow;
  auto mix_row = [&](int i) { return mrows + (int64_t)(i < count ? i : 0) * kMixRow; };
  const uint4 *ra = reinterpret_cast<const uint4 *>(mix_row(lane) + kNSym + 1);
  const uint4 *rb = reinterpret_cast<const uint4 *>(mix_row(lane + nl) + kNSym + 1);
  uint4 ca0 = __ldg(ra), ca1 = __ldg(ra + 1), cb0 = __ldg(rb), cb1 = __ldg(rb + 1);
  for (int it = 0; it < niter; ++it) {
    const int p = it * nl + lane;
    const bool active = lane < nl && p < count;
    const int ctr = (int)ctr_a;
    const uint4 c0 = ca0, c1 = ca1;
    ca0 = cb0; ca1 = cb1;
    const uint16_t *frow = mix_row(p + 2 * nl);
    const uint4 *cr = reinterpret_cast<const uint4 *>(frow + kNSym + 1);
    cb0 = __ldg(cr); cb1 = __ldg(cr + 1);
    asm volatile("prefetch.global.L1 [%0];" ::"l"(frow));
    asm volatile("prefetch.global.L1 [%0];" ::"l"(frow + 64));
    ctr_a = ctr_b;
    ctr_b = (active && p + 2 * nl < count) ? __ldg(idxp + p + 2 * nl) : 0u;
    // every lane runs the search (inactive lanes on a valid table, their
    // state kept), so the round has no branch around it
    const uint16_t *trow = mix_row(active ? p : 0);
    const uint32_t slot = x & (kM - 1);
    uint32_t lo, hi;
    const int s = cdf_search_r(trow, c0, c1, slot, lo, hi);
    {
      const uint32_t xn = (hi - lo) * (x >> kLogM) + slot - lo;
      x = active ? xn : x;
      const bool need = active && x < kRansL;
      const uint32_t m = __ballot_sync(0xffffffffu, need);
      const uint32_t k = ptr + __popc(m & lt);
      const uint32_t wv = word(need ? k : ptr);
      bad = bad || (need && k >= nwords);
      x = need ? ((x << 16) | (k < nwords ? wv : 0u)) : x;
      advance(__popc(m));
    }
    // escapes: phase 0 counts ones up to a zero, phase 1 reads k bits
    bool pend = active && (s == 0 || s == kNSym - 1);
    int phase = 0, kcnt = 0;
    uint32_t v = 0;
    if (__builtin_expect(__any_sync(0xffffffffu, pend), 0))
    for (int rnd = 0; rnd < 2 * kMaxEscBits + 2; ++rnd) {
      if (!__any_sync(0xffffffffu, pend)) break;
      if (pend) {
        const uint32_t slot = x & (kM - 1);
        const uint32_t bit = slot >> (kLogM - 1);
        x = (kM >> 1) * (x >> kLogM) + (slot & ((kM >> 1) - 1));
        if (phase == 0) {
          if (bit) { if (++kcnt > kMaxEscBits) { bad = true; } }
          else { phase = 1; v = 1; }
        } else {
          v = (v << 1) | bit;
          --kcnt;
        }
      }
      const bool need = pend && x < kRansL;
      const uint32_t m = __ballot_sync(0xffffffffu, need);
      if (m) {
        const uint32_t k = ptr + __popc(m & lt);
        const uint32_t wv = word(need ? k : ptr);
        if (need) {
          if (k >= nwords) bad = true;
          x = (x << 16) | (k < nwords ? wv : 0u);
        }
        advance(__popc(m));
      }
      if (pend && ((phase == 1 && kcnt == 0) || bad)) pend = false;
    }
    if (pend) bad = true;
    if (active) {
      int r;
      if (s == 0) r = -(int)(v - 1) - kT - 1;
      else if (s == kNSym - 1) r = (int)(v - 1) + kT + 1;
      else r = s - kT - 1;
      const int yy = 2 * pos.y2 + (pos.r < ne ? 0 : 1);
      const int xx = pos.r < ne ? ae + 4 * pos.r : ao + 4 * (pos.r - ne);
      outp[(int64_t)yy * w + xx] = ctr + r;
    }
    pos.next();
    // every loop is bounded, so a corrupt chunk only has to stop early
    // eventually: vote every 32 iterations
    if ((it & 31) == 31 && __any_sync(0xffffffffu, bad)) break;
  }
  if (lane < nl && x != kRansL) bad = true;
  if (lane == 0 && ptr != nwords) bad = true;
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kStCorrupt);
}

// ---------------------------------------------------------------------------
// rANS encoding (reverse of the decoder). One warp per chunk; iterations,
// rounds and lanes run in descending order; each emitted word is written at
// a decreasing address of the chunk's scratch region, so the words read
// forward from the lowest written address are in decoder order.

// EncChunk (ctx_kernels.cuh): the chunk's symbols are idx[sym_base + i] /
// vals[sym_base + i]; scratch_end = word index one past its scratch region.

__device__ __forceinline__ void esc_code(int r, int &s, uint32_t &v, int &k) {
  if (r >= -kT && r <= kT) { s = r + kT + 1; v = 0; k = -1; return; }
  uint32_t e = (r < -kT) ? (uint32_t)(-r - kT - 1) : (uint32_t)(r - kT - 1);
  s = (r < -kT) ? 0 : kNSym - 1;
  v = e + 1;
  k = 31 - __clz(v);
}

// ops of a symbol: 1 main + (2k + 1) bypass bits for an escape
// (mix: idx holds the centres)
__global__ void k_rans_count_ops(const EncChunk *__restrict__ chunks, int nchunks,
                                 const uint32_t *__restrict__ idx,
                                 const int32_t *__restrict__ vals,
                                 uint32_t *__restrict__ ops, int mix) {
  const int cw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (cw >= nchunks) return;
  EncChunk ch = chunks[cw];
  uint32_t tot = 0;
  for (uint32_t i = lane; i < ch.count; i += 32) {
    const int64_t q = (int64_t)ch.sym_base + i;
    int ctr, tid;
    if (mix) ctr = (int)idx[q];
    else unpack_index(idx[q], ctr, tid);
    int s, k;
    uint32_t v;
    esc_code(vals[q] - ctr, s, v, k);
    tot += 1 + (k >= 0 ? 2 * k + 1 : 0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if (lane == 0) ops[cw] = tot;
}

__global__ void k_rans_encode(const EncChunk *__restrict__ chunks, int nchunks,
                              const uint16_t *__restrict__ bank,
                              const uint32_t *__restrict__ idx,
                              const int32_t *__restrict__ vals,
                              uint16_t *__restrict__ scratch,
                              uint32_t *__restrict__ states_out,  // 32 per chunk
                              uint32_t *__restrict__ nwords_out, uint32_t *status,
                              const uint32_t *__restrict__ cf) {
  const int cw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (cw >= nchunks) return;
  const EncChunk ch = chunks[cw];
  const int nl = ch.lanes;
  uint32_t x = kRansL;
  uint64_t wpos = ch.scratch_end;
  const uint32_t gt = ~((2u << lane) - 1u);  // lanes above me
  const int niter = (ch.count + nl - 1) / nl;
  bool bad = false;
  for (int it = niter - 1; it >= 0; --it) {
    const int p = it * nl + lane;
    const bool active = lane < nl && p < (int)ch.count;
    int s = 0, k = -1;
    uint32_t v = 0, c0 = 0, f0 = 1;
    if (active) {
      const int64_t q = (int64_t)ch.sym_base + p;
      int ctr, tid;
      if (cf) {
        // logistic mixture: the symbol's own (cdf, frequency), centre in idx
        ctr = (int)idx[q];
        esc_code(vals[q] - ctr, s, v, k);
        c0 = cf[q] & 0xFFFFu;
        f0 = cf[q] >> 16;
      } else {
        unpack_index(idx[q], ctr, tid);
        esc_code(vals[q] - ctr, s, v, k);
        const uint16_t *t = bank + (size_t)tid * (kNSym + 1);
        c0 = t[s];
        f0 = (uint32_t)t[s + 1] - c0;
      }
      if (k > kMaxEscBits) bad = true;
    }
    const int nops = active ? 1 + (k >= 0 ? 2 * k + 1 : 0) : 0;
    int rounds = nops;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rounds = max(rounds, __shfl_xor_sync(0xffffffffu, rounds, o));
    for (int rnd = rounds - 1; rnd >= 0; --rnd) {
      const bool has = rnd < nops;
      uint32_t c = c0, f = f0;
      if (has && rnd > 0) {
        int b = rnd - 1;          // bypass bit index in decode order
        uint32_t bit;
        if (b < k) bit = 1;
        else if (b == k) bit = 0;
        else bit = (v >> (2 * k - b)) & 1u;
        c = bit * (kM >> 1);
        f = kM >> 1;
      }
      const bool emit = has && x >= (f << 17);
      const uint32_t m = __ballot_sync(0xffffffffu, emit);
      if (emit) {
        uint64_t pos = wpos - 1 - __popc(m & gt);
        scratch[pos] = (uint16_t)(x & 0xFFFFu);
        x >>= 16;
      }
      wpos -= __popc(m);
      if (has) x = (x / f) * kM + (x % f) + c;
    }
  }
  if (lane < nl) states_out[(size_t)cw * 32 + lane] = x;
  if (lane == 0) nwords_out[cw] = (uint32_t)(ch.scratch_end - wpos);
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kStRange);
}

// Copy encoded chunks (states + words) into the packed payload.
__global__ void k_rans_pack(const EncChunk *__restrict__ chunks, int nchunks,
                            const uint16_t *__restrict__ scratch,
                            const uint32_t *__restrict__ states,
                            const uint32_t *__restrict__ nwords,
                            const uint64_t *__restrict__ out_off,
                            uint8_t *__restrict__ payload) {
  const int cw = blockIdx.x;
  if (cw >= nchunks) return;
  const EncChunk ch = chunks[cw];
  const int nl = ch.lanes;
  uint8_t *dst = payload + out_off[cw];
  for (int i = threadIdx.x; i < 4 * nl; i += blockDim.x) {
    uint32_t st = states[(size_t)cw * 32 + i / 4];
    dst[i] = (uint8_t)(st >> (8 * (i & 3)));
  }
  const uint32_t nw = nwords[cw];
  const uint16_t *src = scratch + (ch.scratch_end - nw);
  uint8_t *dw = dst + 4 * nl;
  for (uint32_t i = threadIdx.x; i < nw; i += blockDim.x) {
    uint16_t v = src[i];
    dw[2 * i] = (uint8_t)(v & 0xFF);
    dw[2 * i + 1] = (uint8_t)(v >> 8);
  }
}

// Entropy-parameter index decision over arrays (stage API).
__global__ void k_pack_index(const float *__restrict__ mu, const float *__restrict__ rho_or_sigma,
                             int64_t n, int is_sigma, uint32_t *__restrict__ idx) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float m = mu[i], s = rho_or_sigma[i];
  if (is_sigma) {
    // sigma given directly: bypass the softplus by mapping through rho = s
    // only for the bin computation
    float t = rintf(__fmul_rn(m, 16.f));
    t = fminf(fmaxf(t, -8388608.f), 8388608.f);
    int j = (__float_as_int(s) - 0x3E000000) >> 20;
    j = min(max(j, 0), kNJ - 1);
    idx[i] = ((uint32_t)((int)t + (1 << 23)) << 7) | (uint32_t)j;
  } else {
    idx[i] = pack_index(m, s);
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
void launch_cdf_bank(uint16_t *bank, uint16_t *coarse, cudaStream_t st) {
  k_cdf_bank<<<kNTables * 32 / 256, 256, 0, st>>>(bank, coarse);
}
void launch_rans_decode(const DecChunk *chunks, int nchunks, const uint16_t *bank,
                        const uint16_t *coarse, const uint32_t *idx, int64_t idx_stride,
                        int32_t *out, int64_t out_stride, int h, int w, int step,
                        uint32_t *status, cudaStream_t st, bool mix, const int2 *ext,
                        int esh) {
  if (nchunks <= 0) return;
  const int nsm = sm_count();
  if (mix) {
    // one warp per chunk; with few chunks, fewer warps per block so that the
    // chunks spread over the SMs (one warp per scheduler)
    int wpb = 8;
    while (wpb > 1 && (nchunks + wpb - 1) / wpb < nsm) wpb >>= 1;
    k_rans_decode_mix<<<(nchunks + wpb - 1) / wpb, 32 * wpb, 0, st>>>(
        chunks, nchunks, bank, idx, idx_stride, out, out_stride, w, step, status);
    return;
  }
  constexpr uint32_t maxsm = 227 * 1024;
  static std::atomic<uint64_t> attr{0};
  once_per_device(attr, [] {
    cudaFuncSetAttribute(k_rans_decode<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)maxsm);
    cudaFuncSetAttribute(k_rans_decode<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)maxsm);
  });
  // chunks per block: one while every chunk finds an SM of its own, then as
  // many as that takes, up to 8 (24 warps; past that the shared-memory port is
  // near its limit: 0.16 us a round for one chunk, 0.31 us for eight)
  const int K = std::min(8, (nchunks + nsm - 1) / nsm);
  // table rows in shared memory: no more than the block has symbols (idx_stride
  // symbols a plane, 0 when unknown), so that small passes take little of it
  int64_t cap = (maxsm - kMapBytes - K * kPairBytes) / kRowBytes - 1;
  cap = std::min<int64_t>(cap, kNTables - 1);
  if (idx_stride > 0) cap = std::min<int64_t>(cap, idx_stride * K);
  const size_t smem = kMapBytes + (size_t)K * kPairBytes + (size_t)(cap + 1) * kRowBytes;
  const int grid = (nchunks + K - 1) / K, threads = std::max(256, 96 * K);
  if (ext && step >= 0)
    k_rans_decode<true><<<grid, threads, smem, st>>>(chunks, nchunks, K, (int)cap, bank, coarse,
                                                     idx, idx_stride, out, out_stride, w, step,
                                                     status, ext, esh);
  else
    k_rans_decode<false><<<grid, threads, smem, st>>>(chunks, nchunks, K, (int)cap, bank, coarse,
                                                      idx, idx_stride, out, out_stride, w, step,
                                                      status, nullptr, 0);
}
void launch_rans_count_ops(const EncChunk *chunks, int nchunks, const uint32_t *idx,
                           const int32_t *vals, uint32_t *ops, cudaStream_t st, bool mix) {
  if (nchunks <= 0) return;
  k_rans_count_ops<<<(nchunks + 3) / 4, 128, 0, st>>>(chunks, nchunks, idx, vals, ops,
                                                      mix ? 1 : 0);
}
void launch_rans_encode(const EncChunk *chunks, int nchunks, const uint16_t *bank,
                        const uint32_t *idx, const int32_t *vals, uint16_t *scratch,
                        uint32_t *states, uint32_t *nwords, uint32_t *status,
                        cudaStream_t st, const uint32_t *cf) {
  if (nchunks <= 0) return;
  k_rans_encode<<<(nchunks + 3) / 4, 128, 0, st>>>(chunks, nchunks, bank, idx, vals, scratch,
                                                   states, nwords, status, cf);
}
void launch_rans_pack(const EncChunk *chunks, int nchunks, const uint16_t *scratch,
                      const uint32_t *states, const uint32_t *nwords,
                      const uint64_t *out_off, uint8_t *payload, cudaStream_t st) {
  if (nchunks <= 0) return;
  k_rans_pack<<<nchunks, 256, 0, st>>>(chunks, nchunks, scratch, states, nwords, out_off,
                                       payload);
}
void launch_pack_index(const float *mu, const float *s, int64_t n, int is_sigma,
                       uint32_t *idx, cudaStream_t st) {
  if (n <= 0) return;
  k_pack_index<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mu, s, n, is_sigma, idx);
}

}  // namespace pw
