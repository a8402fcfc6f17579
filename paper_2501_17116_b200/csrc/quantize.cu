// Quantiser kernels: exact quantile selection, clamp, vector-wise absmax, E2M1 encoding in both
// packed layouts, and extraction of the sparse residual (Eq. 1, Appendix A, Section 3.2).
//
// Passes over a [rows x cols] BF16 tensor:
//   with outlier clamping (activations)
//     1. tail_select      one read: exact counts of the BF16 bit patterns in the two tails (shared
//                         memory) + signed max / min of every row; the block that finishes last
//     2.                  turns the cumulative counts into the two order statistics lo, hi
//     3. encode           one read: clamp, per-row scale from the clamped row extremes, Q, both
//                         nibble layouts, a 1-bit-per-element mask of the clamped entries, and
//                         the number of clamped entries per row and per (64-row strip, column)
//     4. mask -> CSR/CSC  prefix sums of those counts and ordered fills driven by the mask (1/16
//                         of the tensor); values are gathered from the few marked entries
//   without clamping (weights, output gradients)
//     1. absmax           one read: max |x| per row and / or per column (after the prescale)
//     2. encode           one read
// The "dual" mode serves the backward pass: one read of dY yields the token-wise codes of
// dY (.) d_W[n] and the channel-wise codes of dY (.) d_A[m].
#include <cmath>
#include <mutex>

#include "common.cuh"

namespace {

constexpr int ENC_TM = 64;                        // tile rows of the encoder (= one strip)
constexpr int ENC_TK = 256;                       // tile columns
constexpr int ENC_THREADS = 256;
constexpr int SUPER = 16;                         // strips whose column counts are also kept as one sum

enum Mode { MODE_ROWS = 0, MODE_COLS = 1, MODE_DUAL = 2 };

__device__ __forceinline__ int float_to_ordered(float f) {
  const int b = __float_as_int(f);
  return b ^ ((b >> 31) & 0x7FFFFFFF);            // signed integer order == float order
}
__device__ __forceinline__ float ordered_to_float(int k) {
  return __int_as_float(k ^ ((k >> 31) & 0x7FFFFFFF));
}
// Two fp32 numbers in a register pair: one instruction multiplies or fuses both (each rounded as usual).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2_rm(f32x2 a, f32x2 b) {      // toward -infinity
  f32x2 r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// max(|m|, |a|, |b|); a NaN wins
__device__ __forceinline__ float absmax3(float m, float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(a)), "f"(fabsf(b)));
  return r;
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// ------------------------------------------------------------------------------------------
// 1. + 2. row extremes, histogram of the tails, order statistics -- one kernel
// ------------------------------------------------------------------------------------------
// The two thresholds are order statistics far out in the tails, so only the tails are counted value by
// value.  Every block draws the same SEL_SAMPLES elements (SEL_GROUPS groups of neighbours, stratified over
// the tensor, jittered by a hash of the stratum) and takes from them a bracket Q < P that leaves more than
// n_tail elements on either side: the k-th smallest / largest sample.  Elements strictly between Q and P are
// the bulk: a vector of eight costs the packed maxima and minima that the row extremes need anyway and two
// packed comparisons.  The others are counted by pattern.  The number of bulk
// elements B is n minus what was counted, so the rank r of the whole tensor is rank r of the counters
// below the bulk and rank r - B above it.  The result is exact whatever the sample was: a rank that does
// not fall into its tail makes the last block count the whole tensor by itself, which takes a hundred times
// as long.  k is chosen for that to happen to one tensor in 10^8 at most, also where the tail consists of
// whole tokens, so that neighbours lie in it together: the groups, not the elements, are the independent
// draws then.  (A margin for 2048 independent ones is half as wide: 8192 x 4096, clamped and encoded, 76.4
// us instead of 78 at 0.1 % per tail, 105 instead of 109 at 3 %.  But it misses one layout of outlier
// tokens in 3000, and on every call where they stay in place, because the positions depend on the size alone.)
//
// What bounds it: a fixed chain of about 8 us (sample -> bracket, and flush -> ticket -> selection), then
// HBM for light clamps and the counting loop for heavy ones.  A histogram of every element needed 180 KB
// of shared memory (one block per SM) and 12 instructions per element; 8192 x 4096 at 0.1 % per tail
// went from 28.8 to 24.5 us, 8192 x 5120 at 0.01 % from 34.7 to 27.6, 16384 x 13824 at 1 % from 130 to
// 117 (L2 flushed by reads before each).  Samples are taken four adjacent elements at a time: one load
// per thread; every block reading 2048 separate sectors cost 2 us more.
//
// Counters: 32-bit in shared memory over a window of SEL_EXPS binary exponents (both signs, all 128
// mantissas), SEL_HEADROOM binades above the largest magnitude of the sample.  Counted elements outside
// the window (tiny values of a bracket around zero, later giants) go to the global counters with
// atomics and exact zeros are counted in registers, so every element is counted exactly once.
//
// A block owns whole rows (a contiguous range of them), so the signed max / min of a row are
// reduced in shared memory and written with plain stores, as is the zero that starts the row's
// count of clamped entries: nothing the kernel writes per row needs initialising.
//
// Every count also goes into one of 32 coarse counters (2048 consecutive positions of the
// ascending real order each).  The block that finishes last (a ticket, no waiting) finds the
// coarse range of each of the two ranks and reads only those 2048 fine counters: lo and hi.
// The context keeps two sets of counters and a device-side parity: a call counts into set p,
// clears set 1 - p at its start (every block a slice, plain stores) and flips the parity at its
// end, so the set a call counts into is always zero and no separate clearing pass exists.  With
// `parity` null (the allocation-free entry point, which clears its one set itself) set 0 is used.
constexpr int SEL_THREADS = 512;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_BLOCKS_PER_SM = 2;
constexpr int SEL_GROUP = 4, SEL_GROUPS = SEL_THREADS;        // one 8-byte load per thread
constexpr int SEL_SAMPLES = SEL_GROUP * SEL_GROUPS;
constexpr int SEL_EXPS = 24;
constexpr int SEL_WINDOW = SEL_EXPS * 128;         // 3072 magnitudes in the window, per sign
constexpr int SEL_ALL = 8192;                       // elements per SM below which everything is counted
constexpr int SEL_HEADROOM = 2;                    // binades between the sample's maximum and the window's top
constexpr int SEL_FLY = 4;                         // vectors a lane loads per unit
constexpr int SEL_DYN_SMEM = 2 * SEL_FLY * SEL_THREADS * 16;   // two units of every warp
constexpr int SEL_ROW_SLOTS = 128;                 // rows whose extremes a block reduces at a time
constexpr int SEL_BIN_SHIFT = 4;                   // sample histogram: 16 positions per bin
constexpr int SEL_BINS = 65536 >> SEL_BIN_SHIFT;
constexpr int HIST_COARSE = 32;                    // coarse counters: 2048 positions each
constexpr int HIST_SET_WORDS = 65536 + HIST_COARSE; // one set: fine counters, then coarse counters

// Position p in ascending real order: p < 32768 are the negative patterns from 0xFFFF down to
// 0x8000 (-0), p >= 32768 the non-negative patterns from 0x0000 up.
__device__ __forceinline__ uint32_t pos_to_bits(int p) { return p < 32768 ? uint32_t(0xFFFF - p) : uint32_t(p - 32768); }
__device__ __forceinline__ int bits_to_pos(uint32_t bits) { return (bits & 0x8000u) ? int(0xFFFFu - bits) : int(bits) + 32768; }

// Stratum i of SEL_THREADS over n elements -> the first of its four sampled elements (n is a multiple of 4).
__device__ __forceinline__ long long sample_index(int i, long long n) {
  const long long q = n >> 2, b = q * i / SEL_THREADS, e = q * (i + 1) / SEL_THREADS;
  uint32_t h = uint32_t(i) * 2654435761u + 0x9E3779B9u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 13;
  return 4 * (b + (long long)(h % uint32_t(e - b)));
}

__device__ __forceinline__ __nv_bfloat162 bf162_of(uint32_t bits) {
  const __nv_bfloat16 v = __ushort_as_bfloat16((unsigned short)bits);
  return __halves2bfloat162(v, v);
}

struct SelectArgs {
  const uint4* x;
  int rows, vec_per_row;
  uint32_t* sets;               // global counters (two sets with `parity`, else one)
  unsigned* parity;
  unsigned* ticket;
  int* row_max;
  int* row_min;
  int* row_cnt;                 // zeroed (or null)
  int* clear;                   // `clear_words` ints that a later kernel adds to: zeroed (or null)
  int clear_words;
  long long n, n_tail;
  int sample_rank;              // k: the bracket is the k-th smallest / largest sample (0-based); -1: none, count all
  float* thresholds;
  int32_t* status;
  int abs_mode;
};

struct SelectShared {
  union {
    uint32_t window[2 * SEL_WINDOW];                // positive, then negative magnitudes
    uint32_t bins[SEL_BINS];                        // histogram of the sample
  };
  int rmax[SEL_ROW_SLOTS], rmin[SEL_ROW_SLOTS];
  uint32_t coarse[HIST_COARSE];
  int warp_tot[SEL_WARPS];
  uint32_t top;
  int p_pos, q_pos;
  int last, fail;
  uint32_t step[2][8];
};

// Inclusive scan of one value per lane over the warp.
template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const T up = __shfl_up_sync(0xFFFFFFFFu, v, off);
    if (lane >= off) v += up;
  }
  return v;
}

// One counted element: into the window, or past it (rare) into the global counters.
__device__ __forceinline__ void select_count(SelectShared& s, uint32_t bits, uint32_t base, uint32_t* ghist, uint32_t& zeros_pos,
                                             uint32_t& zeros_neg, bool& nonfinite) {
  const uint32_t m15 = bits & 0x7FFFu, off = m15 - base;
  if (off < uint32_t(SEL_WINDOW)) {
    atomicAdd(&s.window[off + (bits >> 15) * SEL_WINDOW], 1u);
  } else if (m15 == 0) {
    if (bits) ++zeros_neg; else ++zeros_pos;
  } else {
    atomicAdd(&ghist[bits], 1u);
    atomicAdd(&s.coarse[bits_to_pos(bits) >> 11], 1u);
    if (m15 >= 0x7F80u) nonfinite = true;             // infinity or NaN: always outside the window
  }
}

// A unit is a stretch of consecutive vectors of one row, FLY per lane (vectors lane, lane + 32, ... of the
// stretch); warp w takes units w, w + 16, ...  Units travel to shared memory (cp.async), two of a warp's in
// flight; every lane reads only what it copied itself, so waiting for its own copies is all the
// synchronisation there is.
extern __shared__ __align__(16) unsigned char s_vec[];        // [2][SEL_FLY][SEL_THREADS] vectors
template <int FLY>
__device__ __forceinline__ void select_request(const SelectArgs& a, int u, int units, int r0, int stage) {
  if (u < units) {
    const int chunks_per_row = (a.vec_per_row + 32 * FLY - 1) / (32 * FLY), lane = threadIdx.x & 31;
    const int row = u / chunks_per_row, v0 = (u - row * chunks_per_row) * 32 * FLY;
    const uint4* px = a.x + ((long long)(r0 + row) * a.vec_per_row + v0 + lane);
    const int mine = min(32 * FLY, a.vec_per_row - v0) - lane;             // vectors lane, lane + 32, ... below this
    const uint32_t slot = uint32_t(__cvta_generic_to_shared(s_vec + (stage * SEL_FLY * SEL_THREADS + threadIdx.x) * 16));
#pragma unroll
    for (int k = 0; k < FLY; ++k)
      if (32 * k < mine)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot + uint32_t(k * SEL_THREADS * 16)), "l"(px + 32 * k)
                     : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// Rows [r_begin, r_end): extremes of every row, and the counts of the elements outside (Q, P), or of all.
// `requested`: the warp's first two units are on their way.
template <bool ALL>
__device__ __forceinline__ void select_count_rows(const SelectArgs& a, SelectShared& s, int r_begin, int r_end,
                                                  uint32_t p_bits, uint32_t q_bits, uint32_t base, uint32_t* ghist,
                                                  bool requested) {
  const int tid = threadIdx.x, lane = tid & 31;
  const __nv_bfloat162 p2 = bf162_of(p_bits), q2 = bf162_of(q_bits);
  // with everything counted a vector is work enough per lane
  constexpr int FLY = ALL ? 1 : SEL_FLY, CHUNK = 32 * FLY;
  const int chunks_per_row = (a.vec_per_row + CHUNK - 1) / CHUNK;
  uint32_t zeros_pos = 0, zeros_neg = 0;
  bool nonfinite = false;
  for (int r0 = r_begin; r0 < r_end; r0 += SEL_ROW_SLOTS) {
    const int r1 = min(r_end, r0 + SEL_ROW_SLOTS);
    for (int r = tid; r < r1 - r0; r += SEL_THREADS) {
      s.rmax[r] = INT_MIN;
      s.rmin[r] = INT_MAX;
    }
    __syncthreads();
    const int units = (r1 - r0) * chunks_per_row;
    int u = tid >> 5, stage = 0;
    if (r0 != r_begin || !requested) {
      select_request<FLY>(a, u, units, r0, 0);
      select_request<FLY>(a, u + SEL_WARPS, units, r0, 1);
    }
    for (; u < units; u += SEL_WARPS, stage ^= 1) {
      const int row = u / chunks_per_row, v0 = (u - row * chunks_per_row) * CHUNK;
      const int mine = min(CHUNK, a.vec_per_row - v0) - lane;
      const unsigned char* slot = s_vec + (stage * SEL_FLY * SEL_THREADS + tid) * 16;
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      // Extremes of the unit, packed (a NaN loses here: it is seen below), and one bit per element that
      // is not strictly inside the bracket (a NaN never is): bit 4 k + q for the lower, 16 + 4 k + q for
      // the upper half of word q of vector k.
      __nv_bfloat162 umax = __float2bfloat162_rn(-INFINITY), umin = __float2bfloat162_rn(INFINITY);
      uint32_t tail = 0;
#pragma unroll
      for (int k = 0; k < FLY; ++k) {
        if (32 * k >= mine) break;
        const uint4 vv = *reinterpret_cast<const uint4*>(slot + k * SEL_THREADS * 16);
        const uint32_t w[4] = {vv.x, vv.y, vv.z, vv.w};
        const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(w);
        umax = __hmax2(umax, __hmax2(__hmax2(p[0], p[1]), __hmax2(p[2], p[3])));
        umin = __hmin2(umin, __hmin2(__hmin2(p[0], p[1]), __hmin2(p[2], p[3])));
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (ALL) {
            select_count(s, w[q] & 0xFFFFu, base, ghist, zeros_pos, zeros_neg, nonfinite);
            select_count(s, w[q] >> 16, base, ghist, zeros_pos, zeros_neg, nonfinite);
          } else {
            tail |= ~(__hlt2_mask(p[q], p2) & __hgt2_mask(p[q], q2)) & (0x00010001u << (4 * k + q));
          }
        }
      }
      if (!ALL) {
        // Counted elements are picked out of shared memory rather than out of the registers by a chain of
        // selections: the lanes hold few of them, and a lane's four vectors share one loop.
        while (tail) {
          const uint32_t b = 31u - __clz(tail);
          tail ^= 1u << b;
          const uint32_t at = ((b >> 2) & 3u) * (SEL_THREADS * 16) | ((b & 3u) << 2) | ((b >> 3) & 2u);
          select_count(s, *reinterpret_cast<const unsigned short*>(slot + at), base, ghist, zeros_pos, zeros_neg, nonfinite);
        }
      }
      select_request<FLY>(a, u + 2 * SEL_WARPS, units, r0, stage);
      int kmax = float_to_ordered(fmaxf(__low2float(umax), __high2float(umax)));
      int kmin = float_to_ordered(fminf(__low2float(umin), __high2float(umin)));
      kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
      kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
      if (lane == 0) {
        atomicMax(&s.rmax[row], kmax);
        atomicMin(&s.rmin[row], kmin);
      }
    }
    __syncthreads();
    for (int r = tid; r < r1 - r0; r += SEL_THREADS) {
      a.row_max[r0 + r] = s.rmax[r];
      a.row_min[r0 + r] = s.rmin[r];
      if (a.row_cnt) a.row_cnt[r0 + r] = 0;
    }
    __syncthreads();
  }
  if (__any_sync(0xFFFFFFFFu, nonfinite) && lane == 0 && a.status) atomicOr(a.status, FP4_DEV_NONFINITE);
  zeros_pos = __reduce_add_sync(0xFFFFFFFFu, zeros_pos);
  zeros_neg = __reduce_add_sync(0xFFFFFFFFu, zeros_neg);
  if (lane == 0) {
    if (zeros_pos) { atomicAdd(&ghist[0x0000], zeros_pos); atomicAdd(&s.coarse[bits_to_pos(0x0000u) >> 11], zeros_pos); }
    if (zeros_neg) { atomicAdd(&ghist[0x8000], zeros_neg); atomicAdd(&s.coarse[bits_to_pos(0x8000u) >> 11], zeros_neg); }
  }
}

// The block's counters (of the magnitudes from base + `from` up, `from` a multiple of 64) into the global
// ones.  Two neighbouring counters (an even pattern and the next one: same sign, same coarse range) leave
// with one 64-bit add; no 32-bit half can overflow into the other (n < 2^31).  A warp's 32 pairs lie in one
// coarse range, whose counter gets one add per warp.
__device__ __forceinline__ void select_flush(SelectShared& s, uint32_t base, uint32_t* ghist, int from) {
  const int pairs = (SEL_WINDOW - from) / 2;         // per sign; a multiple of 32
  for (int idx = threadIdx.x; idx < 2 * pairs; idx += SEL_THREADS) {
    const int neg = idx >= pairs, off = from + 2 * (idx - neg * pairs);
    const uint2 c = *reinterpret_cast<const uint2*>(&s.window[neg * SEL_WINDOW + off]);
    const uint32_t bits = (uint32_t(neg) << 15) | (base + uint32_t(off));
    if (c.x | c.y)
      atomicAdd(reinterpret_cast<unsigned long long*>(&ghist[bits]), (unsigned long long)c.x | ((unsigned long long)c.y << 32));
    const uint32_t t = __reduce_add_sync(0xFFFFFFFFu, c.x + c.y);
    if ((threadIdx.x & 31) == 0 && t) atomicAdd(&s.coarse[bits_to_pos(bits) >> 11], t);
  }
}

// The order statistics from the global counters, by all threads of one block.  `bulk` elements lie
// between the tails and were not counted; a rank that falls inside them sets s.fail.
__device__ __forceinline__ void select_ranks(const SelectArgs& a, SelectShared& s, const uint32_t* ghist,
                                             const uint32_t* gcoarse, bool whole) {
  // Rank q (0: lower, 1: upper) is served by warps 8 q .. 8 q + 7.  Every warp finds the rank's coarse
  // range (one coarse counter per lane), then warp st of the 8 reads step st of the range's 2048 fine
  // counters: 256 consecutive positions, 8 per lane.  The step totals meet in shared memory; the warp
  // whose step holds the rank writes the threshold.
  static_assert(SEL_WARPS == 16, "two ranks x eight steps, one warp each");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp >> 3, st = warp & 7;
  // abs_mode: one rank in the order of the magnitudes (both warp groups find it, the first writes
  // -t and t): magnitude range c holds the positive range 16 + c and the negative range 15 - c.
  // (counts and ranks fit 32 bits: n < 2^31)
  const uint32_t raw = __ldcg(&gcoarse[lane]);
  const uint32_t raw_mag = a.abs_mode && lane < 16 ? __ldcg(&gcoarse[16 + lane]) + __ldcg(&gcoarse[15 - lane]) : 0u;
  const uint32_t n = uint32_t(a.n), n_tail = uint32_t(a.n_tail), bulk = n - __reduce_add_sync(0xFFFFFFFFu, raw);
  const bool upper = a.abs_mode || q == 1;
  const uint32_t rank = a.abs_mode ? n - 1 - 2 * n_tail - bulk : (q == 0 ? n_tail : n - 1 - n_tail - bulk);
  const uint32_t cc = a.abs_mode ? raw_mag : raw;
  const uint32_t sc = warp_inclusive_scan(cc);
  const unsigned holds = __ballot_sync(0xFFFFFFFFu, rank >= sc - cc && rank < sc);   // at most one lane
  const int region = holds ? __ffs(holds) - 1 : 0;
  uint32_t run = __shfl_sync(0xFFFFFFFFu, sc - cc, region);                           // counts before the range
  if (!holds && lane == 0) s.fail = 1;
  // positions of the range in ascending order; in memory they ascend (region >= 16) or descend
  const bool desc = !a.abs_mode && region < 16;
  const uint32_t* first = a.abs_mode ? ghist + 2048 * region
                                     : ghist + (desc ? (0xFFFF - 2048 * region - 2047) : 2048 * (region - 16));
  const int word = desc ? (2048 - 256 * st - 8 * lane - 8) : (256 * st + 8 * lane);
  uint32_t c[8];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint4 t = __ldcg(reinterpret_cast<const uint4*>(first + word) + h);
    if (a.abs_mode) {                                 // the same magnitudes with the sign bit set
      const uint4 tn = __ldcg(reinterpret_cast<const uint4*>(first + 0x8000 + word) + h);
      t = make_uint4(t.x + tn.x, t.y + tn.y, t.z + tn.z, t.w + tn.w);
    }
    const uint32_t tt[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {                     // in ascending position order
      if (desc) c[7 - 4 * h - i] = tt[i]; else c[4 * h + i] = tt[i];
    }
  }
  uint32_t mine = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) mine += c[i];
  const uint32_t incl = warp_inclusive_scan(mine);
  if (lane == 31) s.step[q][st] = incl;
  __syncthreads();
  for (int j = 0; j < st; ++j) run += s.step[q][j];
  uint32_t before = run + incl - mine;
  if (holds && rank >= before && rank < before + mine) {
    int k = 0;
#pragma unroll
    for (int i = 0; i < 7; ++i) {
      if (k == i && rank >= before + c[i]) { before += c[i]; k = i + 1; }
    }
    const int at = 2048 * region + 256 * st + 8 * lane + k;
    if (a.abs_mode) {
      const uint32_t m15 = uint32_t(at);              // `at` counts magnitudes here
      if (!whole && at + 32768 < s.p_pos) s.fail = 1;
      if (q == 0) {
        a.thresholds[1] = __uint_as_float(m15 << 16);
        a.thresholds[0] = __uint_as_float(m15 ? (m15 | 0x8000u) << 16 : 0u);
      }
    } else {
      if (!whole && (upper ? at < s.p_pos : at > s.q_pos)) s.fail = 1;
      const uint32_t bits = pos_to_bits(at);
      a.thresholds[q] = __uint_as_float((bits == 0x8000u ? 0u : bits) << 16);   // thresholds are real numbers: -0 is +0
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(SEL_THREADS, SEL_BLOCKS_PER_SM)
tail_select_kernel(const __grid_constant__ SelectArgs a) {
  __shared__ SelectShared s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r_begin = int((long long)a.rows * blockIdx.x / gridDim.x);
  const int r_end = int((long long)a.rows * (blockIdx.x + 1) / gridDim.x);
  // loads issued first, so that their latency runs under the clearing below; the parity is not looked at before the
  // sample has been (the clearing of the global counters, which needs it, waited a microsecond for it alone)
  const unsigned par = a.parity ? (*reinterpret_cast<volatile unsigned*>(a.parity) & 1u) : 0u;
  const bool sampled = a.sample_rank >= 0;
  uint2 sample = make_uint2(0, 0);
  uint4 first = make_uint4(0, 0, 0, 0);
  if (sampled) {
    sample = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const unsigned short*>(a.x) + sample_index(tid, a.n)));
  } else if (tid < (long long)(r_end - r_begin) * a.vec_per_row) {
    first = __ldg(&a.x[(long long)r_begin * a.vec_per_row + tid]);
  }
  {
    const int rows0 = min(r_end - r_begin, SEL_ROW_SLOTS), v = a.vec_per_row;
    if (sampled) {
      const int units = rows0 * ((v + 32 * SEL_FLY - 1) / (32 * SEL_FLY));
      select_request<SEL_FLY>(a, warp, units, r_begin, 0);
      select_request<SEL_FLY>(a, warp + SEL_WARPS, units, r_begin, 1);
    } else {
      const int units = rows0 * ((v + 31) / 32);
      select_request<1>(a, warp, units, r_begin, 0);
      select_request<1>(a, warp + SEL_WARPS, units, r_begin, 1);
    }
  }
  for (int i = tid; i < 2 * SEL_WINDOW / 4; i += SEL_THREADS) reinterpret_cast<uint4*>(s.window)[i] = make_uint4(0, 0, 0, 0);
  if (tid < HIST_COARSE) s.coarse[tid] = 0;
  if (tid == 0) { s.top = 0; s.fail = 0; }
  __syncthreads();
  // Everything is counted (no sample), or what lies outside the sample's bracket.
  uint32_t p_bits = 0, q_bits = 0;
  int p_pos = 0, q_pos = 65535;
  if (!sampled) {
    // the window's top: from the block's first vectors
    const uint32_t w[4] = {first.x, first.y, first.z, first.w};
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) m = max(m, max(w[q] & 0x7FFFu, (w[q] >> 16) & 0x7FFFu));
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0 && m) atomicMax(&s.top, m);
  } else {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w = i & 2 ? sample.y : sample.x, bits = i & 1 ? w >> 16 : w & 0xFFFFu;
      atomicAdd(&s.bins[bits_to_pos(a.abs_mode ? bits & 0x7FFFu : bits) >> SEL_BIN_SHIFT], 1u);
      m = max(m, bits & 0x7FFFu);
    }
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0 && m) atomicMax(&s.top, m);
    __syncthreads();
    // bins 8 tid .. 8 tid + 7 of this thread; the thread whose bins hold a rank notes the bin
    static_assert(SEL_BINS == 8 * SEL_THREADS, "eight bins per thread");
    uint4* bins4 = reinterpret_cast<uint4*>(s.bins) + 2 * tid;
    const uint4 b0 = bins4[0], b1 = bins4[1];
    bins4[0] = bins4[1] = make_uint4(0, 0, 0, 0);      // the same words are the window's counters from here on
    const int c[8] = {int(b0.x), int(b0.y), int(b0.z), int(b0.w), int(b1.x), int(b1.y), int(b1.z), int(b1.w)};
    const int mine = c[0] + c[1] + c[2] + c[3] + c[4] + c[5] + c[6] + c[7];
    const int incl = warp_inclusive_scan(mine);
    if (lane == 31) s.warp_tot[warp] = incl;
    __syncthreads();
    int before = incl - mine;
    for (int w = 0; w < warp; ++w) before += s.warp_tot[w];
    const int k_lo = min(a.sample_rank, SEL_SAMPLES - 1), k_hi = SEL_SAMPLES - 1 - k_lo;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (k_lo >= before && k_lo < before + c[i]) s.q_pos = ((8 * tid + i) << SEL_BIN_SHIFT) + (1 << SEL_BIN_SHIFT) - 1;
      if (k_hi >= before && k_hi < before + c[i]) s.p_pos = (8 * tid + i) << SEL_BIN_SHIFT;
      before += c[i];
    }
    __syncthreads();
    // The bracket as numbers.  Comparisons do not tell -0 from +0, so a bound at a zero takes in both; a
    // bound among the NaN patterns (only with non-finite inputs) leaves no bulk.
    p_pos = s.p_pos;
    q_pos = a.abs_mode ? 65535 - p_pos : s.q_pos;
    if (p_pos == bits_to_pos(0x0000u)) p_pos = bits_to_pos(0x8000u);
    if (q_pos == bits_to_pos(0x8000u)) q_pos = bits_to_pos(0x0000u);
    p_bits = pos_to_bits(p_pos);
    q_bits = pos_to_bits(q_pos);
  }
  __syncthreads();
  uint32_t* ghist = a.sets + size_t(par) * HIST_SET_WORDS;
  uint32_t* gcoarse = ghist + 65536;
  if (a.parity) {
    // this block's slice of the other set, for the next call
    uint32_t* other = a.sets + size_t(par ^ 1u) * HIST_SET_WORDS;
    const int per = (HIST_SET_WORDS + gridDim.x - 1) / gridDim.x;
    const int w0 = blockIdx.x * per, w1 = min(HIST_SET_WORDS, w0 + per);
    for (int i = w0 + tid; i < w1; i += SEL_THREADS) other[i] = 0;
  }
  for (int i = blockIdx.x * SEL_THREADS + tid; i < a.clear_words; i += gridDim.x * SEL_THREADS) a.clear[i] = 0;
  if (tid == 0) { s.p_pos = p_pos; s.q_pos = q_pos; }
  const int e_top = min(254, int(s.top >> 7) + SEL_HEADROOM);
  const uint32_t base = uint32_t(max(0, e_top - SEL_EXPS + 1)) << 7;
  if (sampled)
    select_count_rows<false>(a, s, r_begin, r_end, p_bits, q_bits, base, ghist, true);
  else
    select_count_rows<true>(a, s, r_begin, r_end, p_bits, q_bits, base, ghist, true);
  __syncthreads();
  // counted magnitudes start at the smaller bound where the bracket holds zero (else anywhere)
  const uint32_t lowest = sampled && !(p_bits & 0x8000u) && (q_bits & 0x8000u) ? min(p_bits, q_bits & 0x7FFFu) : 0u;
  select_flush(s, base, ghist, lowest > base ? int(lowest - base) & ~63 : 0);
  __syncthreads();
  if (tid < HIST_COARSE && s.coarse[tid]) atomicAdd(&gcoarse[tid], s.coarse[tid]);
  // ---- the last block to get here selects -------------------------------------------------
  // (one thread's fences, behind and ahead of a barrier, order the whole block's counters)
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    s.last = atomicAdd(a.ticket, 1u) == gridDim.x - 1;
    __threadfence();
  }
  __syncthreads();
  if (!s.last) return;
  select_ranks(a, s, ghist, gcoarse, false);
  if (s.fail) {
    // The bracket missed: count the whole tensor into the cleared set, nothing left out.
    for (int i = tid; i < HIST_SET_WORDS; i += SEL_THREADS) ghist[i] = 0;
    for (int i = tid; i < 2 * SEL_WINDOW; i += SEL_THREADS) s.window[i] = 0;
    if (tid < HIST_COARSE) s.coarse[tid] = 0;
    __threadfence();
    __syncthreads();
    select_count_rows<true>(a, s, 0, a.rows, 0, 0, base, ghist, false);
    __syncthreads();
    select_flush(s, base, ghist, 0);
    __syncthreads();
    if (tid < HIST_COARSE) gcoarse[tid] = s.coarse[tid];
    __threadfence();
    __syncthreads();
    select_ranks(a, s, ghist, gcoarse, true);
  }
  if (tid == 0) {
    if (a.parity) *a.parity = par ^ 1u;
    *a.ticket = 0;
  }
}

// Sample rank of the bracket (see above): four times the number of groups that a tail of whole groups is hit by with a
// probability of 1e-8 at most, by Chernoff's bound for a binomial (Poisson) variable of mean m:
// P(X >= g) <= exp(-(g ln(g / m) - g + m)).
int select_sample_rank(long long n, long long n_tail) {
  const double m = double(n_tail) / double(n) * SEL_GROUPS;
  int g = int(m) + 1;
  while (m > 0.0 && g * std::log(g / m) - g + m < 18.42) ++g;
  return (g - 1) * SEL_GROUP;
}

// ------------------------------------------------------------------------------------------
// 1c. thresholds per token (a variant outside the paper, which clamps at tensor-wide quantiles)
// ------------------------------------------------------------------------------------------
// One block per row: exact order statistics of the row's 16-bit patterns by a two-pass radix
// select in shared memory (high byte of the position in ascending real order, then the low byte
// inside the bin that holds the rank), both ranks at once; also the row's extremes, the zero that
// starts its count of clamped entries, and the non-finite flag, like the tensor-wide kernel.
// thresholds[2 m] = lo of row m, thresholds[2 m + 1] = hi (a -0 threshold is written as +0).
__global__ void __launch_bounds__(256)
row_select_kernel(const uint4* __restrict__ x, int vec_per_row, int n_tail, int* __restrict__ row_max,
                  int* __restrict__ row_min, int* __restrict__ row_cnt, float* __restrict__ thresholds,
                  int32_t* status) {
  __shared__ uint32_t hist[3][256];          // pass 1; pass 2 for the lower rank; pass 2 for the upper rank
  __shared__ int s_bin[2], s_rank[2], s_max[8], s_min[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = blockIdx.x;
  const uint4* row = x + (long long)m * vec_per_row;
  const int cols = 8 * vec_per_row;
  for (int i = tid; i < 3 * 256; i += 256) (&hist[0][0])[i] = 0;
  __syncthreads();
  int kmax = INT_MIN, kmin = INT_MAX;
  bool nonfinite = false;
  for (int v = tid; v < vec_per_row; v += 256) {
    const uint4 q = __ldg(&row[v]);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t bits = (e & 1) ? (w[e >> 1] >> 16) : (w[e >> 1] & 0xFFFFu);
      atomicAdd(&hist[0][bits_to_pos(bits) >> 8], 1u);
      if ((bits & 0x7FFFu) >= 0x7F80u) nonfinite = true;
      const int key = float_to_ordered(__uint_as_float(bits << 16));
      kmax = max(kmax, key);
      kmin = min(kmin, key);
    }
  }
  kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
  kmin = __reduce_min_sync(0xFFFFFFFFu, kmin);
  if (lane == 0) { s_max[warp] = kmax; s_min[warp] = kmin; }
  if (__any_sync(0xFFFFFFFFu, nonfinite) && lane == 0 && status) atomicOr(status, FP4_DEV_NONFINITE);
  __syncthreads();
  if (tid == 0) {
    int a = s_max[0], b = s_min[0];
    for (int i = 1; i < 8; ++i) { a = max(a, s_max[i]); b = min(b, s_min[i]); }
    row_max[m] = a;
    row_min[m] = b;
    if (row_cnt) row_cnt[m] = 0;
  }
  // the bin of each rank: warp q scans the 256 counts for rank q (8 per lane)
  if (warp < 2) {
    const int rank = warp == 0 ? n_tail : cols - 1 - n_tail;
    int c[8], mine = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { c[i] = int(hist[0][8 * lane + i]); mine += c[i]; }
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += up;
    }
    int before = incl - mine;
    if (rank >= before && rank < incl) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (rank >= before && rank < before + c[i]) { s_bin[warp] = 8 * lane + i; s_rank[warp] = rank - before; }
        before += c[i];
      }
    }
  }
  __syncthreads();
  const int bin_lo = s_bin[0], bin_hi = s_bin[1];
  for (int v = tid; v < vec_per_row; v += 256) {      // second pass: the row is in L1 / L2 now
    const uint4 q = __ldg(&row[v]);
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const uint32_t bits = (e & 1) ? (w[e >> 1] >> 16) : (w[e >> 1] & 0xFFFFu);
      const int pos = bits_to_pos(bits);
      if ((pos >> 8) == bin_lo) atomicAdd(&hist[1][pos & 255], 1u);
      if ((pos >> 8) == bin_hi) atomicAdd(&hist[2][pos & 255], 1u);
    }
  }
  __syncthreads();
  if (warp < 2) {
    const int rank = s_rank[warp];
    int c[8], mine = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) { c[i] = int(hist[1 + warp][8 * lane + i]); mine += c[i]; }
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int up = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += up;
    }
    int before = incl - mine;
    if (rank >= before && rank < incl) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (rank >= before && rank < before + c[i]) {
          const uint32_t bits = pos_to_bits(256 * s_bin[warp] + 8 * lane + i);
          thresholds[2 * m + warp] = __uint_as_float((bits == 0x8000u ? 0u : bits) << 16);
        }
        before += c[i];
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// absmax without clamping
// ------------------------------------------------------------------------------------------
// d[i] = amax[i] / MAX rounded once (MAX = 6 for E2M1, 448 for E4M3): the de-scale vector of a
// quantised operand, used as a prescale
__global__ void descale_kernel(const float* __restrict__ amax, int n, float div, float* __restrict__ d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = __fdiv_rn(amax[i], div);
}

struct AbsmaxArgs {
  const uint4* x;
  int rows, cols;
  const float* pre_col;         // PRE: multiplies along columns before the row-wise maximum
  const float* pre_row;         // PRE: multiplies along rows before the column-wise maximum
  float pre_col_div, pre_row_div;   // > 0: the vector holds amax values: use amax / div (6 or 448) and store it
  float* d_col_out;             // dual mode: the de-scale vectors actually used, for the encoder
  float* d_row_out;
  uint32_t* amax_rows;          // float bits, zero-initialised (non-negative floats order as integers)
  uint32_t* amax_cols;
  int32_t* status;              // FP4_DEV_NONFINITE is raised when a maximum is infinite or NaN
};

// Without a prescale: maxima of packed BF16 magnitudes (a NaN wins and is seen).  Tile of 64 rows x 256 columns per
// block, same thread mapping as the encoder: warp w owns rows 8w..8w+7, lane l the 8 columns 8l..8l+7.  It needs no
// scales and few registers, and many short blocks keep HBM busy (13824 x 13824, columns: 53 us, 7.1 TB/s).
template <int MODE>
__global__ void __launch_bounds__(ENC_THREADS)
absmax_tile_kernel(const AbsmaxArgs a) {
  __shared__ uint32_t s_cmax[8][ENC_TK];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row0 = blockIdx.y * ENC_TM + 8 * warp, col = blockIdx.x * ENC_TK + 8 * lane;
  const int vec_per_row = a.cols >> 3;
  constexpr bool want_rows = MODE != MODE_COLS, want_cols = MODE != MODE_ROWS;
  uint4 v[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    v[r] = make_uint4(0, 0, 0, 0);
    if (col < a.cols) v[r] = __ldg(&a.x[(long long)(row0 + r) * vec_per_row + (col >> 3)]);
  }
  __nv_bfloat162 cmax[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) cmax[q] = __float2bfloat162_rn(0.0f);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    __nv_bfloat162 m[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) m[q] = __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w[q]));
    if (want_cols) {
#pragma unroll
      for (int q = 0; q < 4; ++q) cmax[q] = __hmax2_nan(cmax[q], m[q]);
    }
    if (want_rows) {
      const __nv_bfloat162 t = __hmax2_nan(__hmax2_nan(m[0], m[1]), __hmax2_nan(m[2], m[3]));
      const uint32_t bits = *reinterpret_cast<const uint32_t*>(&t);
      const uint32_t g = __reduce_max_sync(0xFFFFFFFFu, max(bits << 16, bits & 0x7FFF0000u));
      if (lane == 0) {
        atomicMax(&a.amax_rows[row0 + r], g);
        if (g >= 0x7F800000u && a.status) atomicOr(a.status, FP4_DEV_NONFINITE);
      }
    }
  }
  if (want_cols) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t bits = *reinterpret_cast<const uint32_t*>(&cmax[q]);
      s_cmax[warp][8 * lane + 2 * q] = bits << 16;
      s_cmax[warp][8 * lane + 2 * q + 1] = bits & 0xFFFF0000u;
    }
    __syncthreads();
    uint32_t m = 0;
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) m = max(m, s_cmax[w8][tid]);
    const int c = blockIdx.x * ENC_TK + tid;
    if (c < a.cols) {
      atomicMax(&a.amax_cols[c], m);
      if (m >= 0x7F800000u && a.status) atomicOr(a.status, FP4_DEV_NONFINITE);
    }
  }
}

// With a prescale: a block walks down a strip of 256 columns, 32 rows per step: warp w owns rows 4w..4w+3 of a step, lane l the 8
// columns 8l..8l+7.  Steps travel to shared memory (cp.async), two in flight while one is looked at; every lane reads
// only what it copied itself.  The grid is one wave of blocks, four per SM.  (Blocks that loaded one tile each, scales
// first, spent two thirds of their time waiting for it: dY of 8192 x 5120, both axes, 25 us, 18 now; 13824 x 5120
// 45 -> 30.)  Maxima of three, products two at a time; a NaN wins and is seen.
constexpr int AB_ROWS = 32, AB_STAGES = 3;
template <int MODE>
__global__ void __launch_bounds__(ENC_THREADS, 4)
absmax_strip_kernel(const AbsmaxArgs a) {
  __shared__ __align__(16) uint4 s_buf[AB_STAGES][4][ENC_THREADS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int col = blockIdx.x * ENC_TK + 8 * lane;
  const bool in_cols = col < a.cols;
  const int vec_per_row = a.cols >> 3;
  constexpr bool want_rows = MODE != MODE_COLS, want_cols = MODE != MODE_ROWS;
  const int steps = a.rows / AB_ROWS;
  const int st0 = blockIdx.y, stride = gridDim.y;     // all blocks go down the tensor together
  auto request = [&](int st, int stage) {
    if (in_cols && st < steps) {
      const uint4* px = a.x + (long long)(AB_ROWS * st + 4 * warp) * vec_per_row + (col >> 3);
      const uint32_t slot = uint32_t(__cvta_generic_to_shared(&s_buf[stage][0][tid]));
#pragma unroll
      for (int r = 0; r < 4; ++r)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(slot + uint32_t(r * ENC_THREADS * 16)),
                     "l"(px + (long long)r * vec_per_row)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  request(st0, 0);
  request(st0 + stride, 1);
  f32x2 pc[4];
  if (want_rows) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float p[2] = {0.0f, 0.0f};
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (in_cols) {
          const float v = __ldg(&a.pre_col[col + 2 * q + h]);
          p[h] = a.pre_col_div > 0.0f ? __fdiv_rn(v, a.pre_col_div) : v;
          if (a.d_col_out && blockIdx.y == 0 && warp == 0) a.d_col_out[col + 2 * q + h] = p[h];
        }
      pc[q] = pack2(p[0], p[1]);
    }
  }
  float cmax[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  float prow = 0.0f;                                  // lane r: prescale of the step's row r (r = lane mod 4)
  auto fetch_prow = [&](int st) {
    if (want_cols && st < steps) prow = __ldg(&a.pre_row[AB_ROWS * st + 4 * warp + (lane & 3)]);
  };
  fetch_prow(st0);
  int stage = 0;
  for (int st = st0; st < steps; st += stride) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    const int row = AB_ROWS * st + 4 * warp;
    const uint4* slot = &s_buf[stage][0][tid];
    uint4 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = in_cols ? slot[r * ENC_THREADS] : make_uint4(0, 0, 0, 0);
    request(st + 2 * stride, stage == 0 ? 2 : stage - 1);       // the stage before this one
    stage = stage == AB_STAGES - 1 ? 0 : stage + 1;
    float pr = prow;
    if (want_cols) {
      if (a.pre_row_div > 0.0f) pr = __fdiv_rn(pr, a.pre_row_div);
      if (a.d_row_out && blockIdx.x == 0 && lane < 4) a.d_row_out[row + lane] = pr;
      fetch_prow(st + stride);
    }
    uint32_t rm[4];                                   // bits of the maxima: they order like the numbers
#pragma unroll
    for (int r = 0; r < 4; r += 2) {                // two rows at a time
      const uint32_t w[2][4] = {{v[r].x, v[r].y, v[r].z, v[r].w}, {v[r + 1].x, v[r + 1].y, v[r + 1].z, v[r + 1].w}};
      float rmax[2] = {0.0f, 0.0f};
      f32x2 p[2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (want_cols) {
          const float t = __shfl_sync(0xFFFFFFFFu, pr, r + i);
          p[i] = pack2(t, t);
        }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        float lo[2], hi[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const f32x2 x = pack2(bf16_lo(w[i][q]), bf16_hi(w[i][q]));
          if (want_rows) {
            float f, g;
            unpack2(mul2(x, pc[q]), f, g);
            rmax[i] = absmax3(rmax[i], f, g);
          }
          if (want_cols) unpack2(mul2(x, p[i]), lo[i], hi[i]);
        }
        if (want_cols) {
          cmax[2 * q] = absmax3(cmax[2 * q], lo[0], lo[1]);
          cmax[2 * q + 1] = absmax3(cmax[2 * q + 1], hi[0], hi[1]);
        }
      }
      rm[r] = __float_as_uint(rmax[0]);
      rm[r + 1] = __float_as_uint(rmax[1]);
    }
    if (want_rows) {
      // four reductions over the warp; lane r keeps row r's
      uint32_t g = 0;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint32_t t = __reduce_max_sync(0xFFFFFFFFu, rm[r]);
        if (lane == r) g = t;
      }
      if (lane < 4) {
        atomicMax(&a.amax_rows[row + lane], g);
        if (g >= 0x7F800000u && a.status) atomicOr(a.status, FP4_DEV_NONFINITE);
      }
    }
  }
  if (want_cols) {
    uint32_t* s_cmax = reinterpret_cast<uint32_t*>(&s_buf[0][0][0]);      // [8][ENC_TK]
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 8; ++c) s_cmax[warp * ENC_TK + 8 * lane + c] = __float_as_uint(cmax[c]);
    __syncthreads();
    uint32_t m = 0;
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) m = max(m, s_cmax[w8 * ENC_TK + tid]);
    const int c = blockIdx.x * ENC_TK + tid;
    if (c < a.cols) {
      atomicMax(&a.amax_cols[c], m);
      if (m >= 0x7F800000u && a.status) atomicOr(a.status, FP4_DEV_NONFINITE);
    }
  }
}

// ------------------------------------------------------------------------------------------
// 3. encoder
// ------------------------------------------------------------------------------------------
// Q of Appendix A for eight float32 values -> eight nibbles (element 0 in bits 3:0).
// The chain sends a value that equals a threshold to the larger neighbour, i.e. it rounds to the
// nearest grid value with ties toward +infinity.  The hardware conversion rounds ties to even, so
// each input is first moved off the tie, to the inside of its cell of width 1/8: thresholds are multiples of 1/4, and a
// value belongs to the cell it is the lower end of.  Added to TIE_C with rounding toward -infinity it becomes the cell's
// lower end w (units of 1/8 are the last place there); w + TIE_C times 1 - 2^-24, minus TIE_C - 1/8, is w + 1/32 less
// w 2^-24.  Two instructions for two values, where nudging the bit patterns took four on the unit that bounds the
// encoders (8192 x 5120 clamped and encoded 78.8 -> 76.7 us, 8192 x 4096 71.4 -> 69.8; backward of 4096 x 2048 x 5504
// 111.0 -> 109.1).  The conversion's "-0" nibble is cleared: a nibble's magnitude + 7 reaches bit 3 where it is not zero,
// and never the next nibble.
constexpr float TIE_C = 1572864.0f;                    // 1.5 * 2^20
__device__ __forceinline__ uint32_t encode8(const f32x2 (&v)[4]) {
  const f32x2 up = pack2(TIE_C, TIE_C), scale = pack2(0x0.FFFFFFp0f, 0x0.FFFFFFp0f), down = pack2(0.125f - TIE_C, 0.125f - TIE_C);
  float f[8];
#pragma unroll
  for (int q = 0; q < 4; ++q) unpack2(fma2(add2_rm(v[q], up), scale, down), f[2 * q], f[2 * q + 1]);
  uint32_t w;
  asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t}"
      : "=r"(w)
      : "f"(f[0]), "f"(f[1]), "f"(f[2]), "f"(f[3]), "f"(f[4]), "f"(f[5]), "f"(f[6]), "f"(f[7]));
  return w & (((w & 0x77777777u) + 0x77777777u) | 0x77777777u);
}

// 8 x 8 nibble transpose: in[r] nibble c  ->  out[c] nibble r
__device__ __forceinline__ void transpose8x8_nibbles(uint32_t (&r)[8]) {
  uint32_t t[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {                       // swap the off-diagonal 4x4 blocks
    t[i] = __byte_perm(r[i], r[i + 4], 0x5410);
    t[i + 4] = __byte_perm(r[i], r[i + 4], 0x7632);
  }
#pragma unroll
  for (int g = 0; g < 8; g += 4) {                    // 2x2 blocks inside each 4x4 block
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      r[g + i] = __byte_perm(t[g + i], t[g + i + 2], 0x6240);
      r[g + i + 2] = __byte_perm(t[g + i], t[g + i + 2], 0x7351);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; i += 2) {                    // single nibbles inside each 2x2 block
    const uint32_t a = r[i], b = r[i + 1];
    r[i] = (a & 0x0F0F0F0Fu) | ((b << 4) & 0xF0F0F0F0u);
    r[i + 1] = ((a >> 4) & 0x0F0F0F0Fu) | (b & 0xF0F0F0F0u);
  }
}

// A load that stays where it is written.
__device__ __forceinline__ uint4 load_now(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

struct EncodeArgs {
  const uint4* x;
  int rows, cols;
  const float* pre_col;         // prescale along columns (row-scaled output) or null
  const float* pre_row;         // prescale along rows (column-scaled output) or null
  const uint32_t* amax_rows;    // no clamp: max |x| per row (float bits)
  const uint32_t* amax_cols;    // max |x| per column
  const int* row_max;           // clamp: ordered-int row extremes
  const int* row_min;
  const float* thresholds;      // clamp: lo, hi
  uint32_t* codes;              // [rows x cols/8] words or null   (row-scaled in dual mode)
  uint32_t* codes_t;            // [cols x rows/8] words or null   (column-scaled in dual mode)
  float* amax_out_rows;
  float* amax_out_cols;
  uint8_t* mask;                // clamp: [rows x cols/8] bytes
  int* row_cnt;                 // clamp: clamped entries per row (zero-initialised)
  uint8_t* strip_cnt;           // clamp: [rows/64 x cols] clamped entries per (strip, column)
  int* col_cnt;                 // clamp: clamped entries per column (zero-initialised)
  int* super_cnt;               // clamp: [groups of SUPER strips x cols] clamped entries (zero-initialised)
  float fmax;                   // FP8 encoder: the format's largest value (448 or 57344)
  int e5m2;                     // FP8 encoder: E5M2 bytes instead of E4M3 bytes
};

// MODE_ROWS: one scale per row -> codes and / or codes_t.  MODE_COLS: one scale per column.
// MODE_DUAL: codes hold the row-scaled tensor x (.) pre_col, codes_t the column-scaled tensor
// x (.) pre_row.  OCC (clamping) implies MODE_ROWS without prescale.
template <int MODE, bool OCC, bool PRESCALE, bool PER_TOKEN = false>
__global__ void __launch_bounds__(ENC_THREADS, 4)
encode_kernel(const EncodeArgs a) {
  __shared__ __align__(16) float s_gcol[ENC_TK];
  __shared__ float s_grow[ENC_TM];
  __shared__ float s_prow[ENC_TM];
  __shared__ uint32_t tile_t[8 * 8 * 32];
  __shared__ int s_colcnt[OCC ? ENC_TK : 1];
  __shared__ float s_thr[PER_TOKEN ? 2 * ENC_TM : 1];      // per-token clamp: lo, hi of the tile's rows
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int strip = gridDim.y - 1 - blockIdx.y;       // from the end: what the pass before read last is still in L2
  const int row0 = strip * ENC_TM;
  const int col0 = blockIdx.x * ENC_TK;
  const int vec_per_row = a.cols >> 3;
  constexpr bool ROW_SCALED = MODE != MODE_COLS;      // a row-scaled output exists
  constexpr bool COL_SCALED = MODE != MODE_ROWS;
  uint4 v[8];
  // The tile is requested ahead of the scales, so that one latency runs under the other: by columns (5120 x 13824, absmax and
  // codes, 65.8 -> 63.9 us) and with the clamp, whose scales come out of three reads and two minima (quantising 16384 x 13824
  // 300 -> 294, smaller tensors as before).  Rows without the clamp wait for one read only and run slower (4096 x 512 x 5504
  // forward 29.3 -> 29.8); both axes have more scales to hold beside the tile (145 -> 149).
  constexpr bool TILE_FIRST = MODE == MODE_COLS || OCC;
  if (TILE_FIRST) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = make_uint4(0, 0, 0, 0);
      if (col0 + 8 * lane < a.cols) v[r] = load_now(&a.x[(long long)(row0 + 8 * warp + r) * vec_per_row + (col0 >> 3) + lane]);
    }
  }
  float lo = 0.f, hi = 0.f;
  if (OCC) {
    if constexpr (!PER_TOKEN) {
      lo = a.thresholds[0];
      hi = a.thresholds[1];
    }
    s_colcnt[tid] = 0;
  }

  if (ROW_SCALED && tid < ENC_TM) {
    const int r = row0 + tid;
    float amax;
    if (OCC) {
      if constexpr (PER_TOKEN) {
        lo = s_thr[2 * tid] = a.thresholds[2 * r];
        hi = s_thr[2 * tid + 1] = a.thresholds[2 * r + 1];
      }
      const float mx = fminf(fmaxf(ordered_to_float(a.row_max[r]), lo), hi);
      const float mn = fminf(fmaxf(ordered_to_float(a.row_min[r]), lo), hi);
      amax = fmaxf(fabsf(mx), fabsf(mn));
    } else {
      amax = __uint_as_float(a.amax_rows[r]);
    }
    s_grow[tid] = amax > 0.0f ? __fdiv_rn(6.0f, amax) : 0.0f;
    if (blockIdx.x == 0) a.amax_out_rows[r] = amax;
  }
  if (COL_SCALED) {
    const int c = col0 + tid;
    if (c < a.cols) {
      const float amax = __uint_as_float(a.amax_cols[c]);
      s_gcol[tid] = amax > 0.0f ? __fdiv_rn(6.0f, amax) : 0.0f;
      if (blockIdx.y == 0) a.amax_out_cols[c] = amax;
    }
    if (PRESCALE && tid < ENC_TM) s_prow[tid] = __ldg(&a.pre_row[row0 + tid]);
  }
  __syncthreads();

  const int col = col0 + 8 * lane;                   // first of this thread's 8 columns
  const bool in_cols = col < a.cols;                 // ragged last tile in the column direction
  if (!TILE_FIRST) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = make_uint4(0, 0, 0, 0);
      if (in_cols) v[r] = __ldg(&a.x[(long long)(row0 + 8 * warp + r) * vec_per_row + (col >> 3)]);
    }
  }
  f32x2 gc[4], pc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (COL_SCALED) gc[q] = in_cols ? *reinterpret_cast<const f32x2*>(&s_gcol[8 * lane + 2 * q]) : 0ull;
    if (ROW_SCALED && PRESCALE) {
      const int c = in_cols ? col + 2 * q : 0;
      const float2 p = make_float2(__ldg(&a.pre_col[c]), __ldg(&a.pre_col[c + 1]));
      pc[q] = in_cols ? pack2(p.x, p.y) : 0ull;
    }
  }

  uint32_t word[8];                                   // codes of the row-major output
  uint32_t word_t[MODE == MODE_DUAL ? 8 : 1];         // dual: codes of the column-scaled tensor
  uint32_t any_bits = 0, lo4 = 0, hi4 = 0;            // clamp: mask bytes of rows 0..3 / 4..7
  __nv_bfloat162 lo2, hi2;                            // the thresholds are BF16 numbers: the clamp needs no unpacking
  if (OCC && !PER_TOKEN) { lo2 = __float2bfloat162_rn(lo); hi2 = __float2bfloat162_rn(hi); }
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    f32x2 f[4], f2[4];
    uint32_t obits = 0;
    const float grow1 = ROW_SCALED ? s_grow[8 * warp + r] : 0.0f;
    const float prow1 = (COL_SCALED && PRESCALE) ? s_prow[8 * warp + r] : 1.0f;
    const f32x2 grow = pack2(grow1, grow1), prow = pack2(prow1, prow1);
    if constexpr (PER_TOKEN) {
      lo2 = __float2bfloat162_rn(s_thr[2 * (8 * warp + r)]);
      hi2 = __float2bfloat162_rn(s_thr[2 * (8 * warp + r) + 1]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t x = w[q];
      if (OCC) {
        const __nv_bfloat162 xb = *reinterpret_cast<const __nv_bfloat162*>(&w[q]);
        const __nv_bfloat162 xc = __hmin2(__hmax2(xb, lo2), hi2);
        // bit 2 q for the lower element, 17 + 2 q for the upper one
        obits |= __hne2_mask(xc, xb) & (0x00020001u << (2 * q));
        x = *reinterpret_cast<const uint32_t*>(&xc);
      }
      const f32x2 xv = pack2(bf16_lo(x), bf16_hi(x));
      if constexpr (MODE == MODE_ROWS) {
        f[q] = mul2(PRESCALE ? mul2(xv, pc[q]) : xv, grow);
      } else if constexpr (MODE == MODE_COLS) {
        f[q] = mul2(PRESCALE ? mul2(xv, prow) : xv, gc[q]);
      } else {
        f[q] = mul2(mul2(xv, pc[q]), grow);
        f2[q] = mul2(mul2(xv, prow), gc[q]);
      }
    }
    if (OCC) obits = in_cols ? (obits | (obits >> 16)) & 0xFFu : 0u;   // beyond the tensor: its zeros may lie outside [lo, hi]
    word[r] = encode8(f);
    if constexpr (MODE == MODE_DUAL) word_t[r] = encode8(f2);
    if (in_cols) {
      const long long o = (long long)(row0 + 8 * warp + r) * vec_per_row + (col >> 3);
      if (a.codes) a.codes[o] = word[r];
      if (OCC) a.mask[o] = uint8_t(obits);
    }
    if (OCC) {
      any_bits |= obits;
      if (r < 4) lo4 |= obits << (8 * r); else hi4 |= obits << (8 * (r - 4));
      const int cnt = __reduce_add_sync(0xFFFFFFFFu, __popc(obits));
      if (lane == 0 && cnt) atomicAdd(&a.row_cnt[row0 + 8 * warp + r], cnt);
    }
  }
  if (OCC) {
    // per-column counts of this 64-row strip: only threads that saw a clamped entry take part
    while (any_bits) {
      const int c = __ffs(any_bits) - 1;
      any_bits &= any_bits - 1;
      const uint32_t sel = 0x01010101u << c;
      atomicAdd(&s_colcnt[8 * lane + c], __popc(lo4 & sel) + __popc(hi4 & sel));
    }
  }

  if (a.codes_t) {
    if constexpr (MODE == MODE_DUAL) {
#pragma unroll
      for (int r = 0; r < 8; ++r) word[r] = word_t[r];
    }
    transpose8x8_nibbles(word);
#pragma unroll
    for (int c = 0; c < 8; ++c) tile_t[(c * 8 + warp) * 32 + lane] = word[c];
  }
  __syncthreads();
  if (OCC && col0 + tid < a.cols) {
    a.strip_cnt[(long long)strip * a.cols + col0 + tid] = uint8_t(s_colcnt[tid]);
    if (s_colcnt[tid]) {                              // integer sums: order-independent
      atomicAdd(&a.col_cnt[col0 + tid], s_colcnt[tid]);
      atomicAdd(&a.super_cnt[(long long)(strip / SUPER) * a.cols + col0 + tid], s_colcnt[tid]);
    }
  }
  if (a.codes_t) {
    // thread (c = warp, j = lane) owns column col0 + 8 j + c: 64 rows = 8 words = 32 bytes
    const int k = col0 + 8 * lane + warp;
    if (k < a.cols) {
      uint32_t o[8];
#pragma unroll
      for (int w8 = 0; w8 < 8; ++w8) o[w8] = tile_t[(warp * 8 + w8) * 32 + lane];
      uint4* dst = reinterpret_cast<uint4*>(a.codes_t + (long long)k * (a.rows >> 3) + (row0 >> 3));
      dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
      dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
  }
}

// ------------------------------------------------------------------------------------------
// 3b. FP8 encoder (FP8 operands of the W4A8 / W8A4 settings and of the FP8 reading of dY)
// ------------------------------------------------------------------------------------------
// Two floats -> two FP8 bytes (first value in the low byte), E4M3 or E5M2: nearest even, saturating
// at the format's largest finite value (448 / 57344), the sign kept also on zero.
template <bool E5M2>
__device__ __forceinline__ uint32_t fp8x2(f32x2 v) {
  float lo, hi;
  unpack2(v, lo, hi);
  uint16_t r;
  if (E5M2)
    asm("cvt.rn.satfinite.e5m2x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  else
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
// eight values -> eight bytes
template <bool E5M2>
__device__ __forceinline__ uint2 fp8x8(const f32x2 (&v)[4]) {
  return make_uint2(fp8x2<E5M2>(v[0]) | (fp8x2<E5M2>(v[1]) << 16), fp8x2<E5M2>(v[2]) | (fp8x2<E5M2>(v[3]) << 16));
}
// 4 x 4 byte transpose: in[r] byte c -> out[c] byte r
__device__ __forceinline__ void transpose4x4_bytes(uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t (&c)[4]) {
  const uint32_t t0 = __byte_perm(a0, a1, 0x5140), t1 = __byte_perm(a2, a3, 0x5140);
  const uint32_t t2 = __byte_perm(a0, a1, 0x7362), t3 = __byte_perm(a2, a3, 0x7362);
  c[0] = __byte_perm(t0, t1, 0x5410);
  c[1] = __byte_perm(t0, t1, 0x7632);
  c[2] = __byte_perm(t2, t3, 0x5410);
  c[3] = __byte_perm(t2, t3, 0x7632);
}

// Same tile and thread mapping as encode_kernel, one byte per element: `codes` [rows x cols] bytes
// (row-scaled in dual mode), `codes_t` [cols x rows] bytes (column-scaled in dual mode).  No
// clamping: outlier clamping belongs to 4-bit activations.
// (Values in pairs and the format known when compiled: backward of 4096 x 2048 x 2048 with dY in E5M2 51.5 -> 49.5 us.  Columns'
// tiles ahead of their scales: 5120 x 13824, absmax and codes, 88 -> 84.  Rows keep five blocks per SM: with four 8192 x 13824
// took 131 us instead of 128.)
template <int MODE, bool PRESCALE, bool E5M2>
__global__ void __launch_bounds__(ENC_THREADS, MODE == MODE_DUAL ? 3 : MODE == MODE_ROWS && !PRESCALE ? 5 : 4)
encode_fp8_kernel(const EncodeArgs a) {
  __shared__ __align__(16) float s_gcol[ENC_TK];
  __shared__ float s_grow[ENC_TM];
  __shared__ float s_prow[ENC_TM];
  __shared__ uint2 tile_t[8 * 8 * 32];
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int strip = gridDim.y - 1 - blockIdx.y;       // from the end: what the pass before read last is still in L2
  const int row0 = strip * ENC_TM;
  const int col0 = blockIdx.x * ENC_TK;
  const int vec_per_row = a.cols >> 3;
  constexpr bool ROW_SCALED = MODE != MODE_COLS;
  constexpr bool COL_SCALED = MODE != MODE_ROWS;
  uint4 v[8];
  if (MODE == MODE_COLS) {                            // the tile is requested ahead of the scales (see the encoder)
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = make_uint4(0, 0, 0, 0);
      if (col0 + 8 * lane < a.cols) v[r] = load_now(&a.x[(long long)(row0 + 8 * warp + r) * vec_per_row + (col0 >> 3) + lane]);
    }
  }
  if (ROW_SCALED && tid < ENC_TM) {
    const int r = row0 + tid;
    const float amax = __uint_as_float(a.amax_rows[r]);
    s_grow[tid] = amax > 0.0f ? __fdiv_rn(a.fmax, amax) : 0.0f;
    if (blockIdx.x == 0) a.amax_out_rows[r] = amax;
  }
  if (COL_SCALED) {
    const int c = col0 + tid;
    if (c < a.cols) {
      const float amax = __uint_as_float(a.amax_cols[c]);
      s_gcol[tid] = amax > 0.0f ? __fdiv_rn(a.fmax, amax) : 0.0f;
      if (blockIdx.y == 0) a.amax_out_cols[c] = amax;
    }
    if (PRESCALE && tid < ENC_TM) s_prow[tid] = __ldg(&a.pre_row[row0 + tid]);
  }
  __syncthreads();

  const int col = col0 + 8 * lane;
  const bool in_cols = col < a.cols;
  if (MODE != MODE_COLS) {
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      v[r] = make_uint4(0, 0, 0, 0);
      if (in_cols) v[r] = __ldg(&a.x[(long long)(row0 + 8 * warp + r) * vec_per_row + (col >> 3)]);
    }
  }
  f32x2 gc[4], pc[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (COL_SCALED) gc[q] = in_cols ? *reinterpret_cast<const f32x2*>(&s_gcol[8 * lane + 2 * q]) : 0ull;
    if (ROW_SCALED && PRESCALE) {
      const int c = in_cols ? col + 2 * q : 0;
      const float2 p = make_float2(__ldg(&a.pre_col[c]), __ldg(&a.pre_col[c + 1]));
      pc[q] = in_cols ? pack2(p.x, p.y) : 0ull;
    }
  }
  uint32_t lo4[8], hi4[8];                            // bytes of columns 0..3 / 4..7 of each row (output for codes_t)
  uint8_t* codes8 = reinterpret_cast<uint8_t*>(a.codes);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const uint32_t w[4] = {v[r].x, v[r].y, v[r].z, v[r].w};
    f32x2 f[4], f2[4];
    const float grow1 = ROW_SCALED ? s_grow[8 * warp + r] : 0.0f;
    const float prow1 = (COL_SCALED && PRESCALE) ? s_prow[8 * warp + r] : 1.0f;
    const f32x2 grow = pack2(grow1, grow1), prow = pack2(prow1, prow1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const f32x2 xv = pack2(bf16_lo(w[q]), bf16_hi(w[q]));
      if constexpr (MODE == MODE_ROWS) {
        f[q] = mul2(PRESCALE ? mul2(xv, pc[q]) : xv, grow);
      } else if constexpr (MODE == MODE_COLS) {
        f[q] = mul2(PRESCALE ? mul2(xv, prow) : xv, gc[q]);
      } else {
        f[q] = mul2(mul2(xv, pc[q]), grow);
        f2[q] = mul2(mul2(xv, prow), gc[q]);
      }
    }
    const uint2 bytes = fp8x8<E5M2>(f);
    if (in_cols && codes8) *reinterpret_cast<uint2*>(codes8 + (long long)(row0 + 8 * warp + r) * a.cols + col) = bytes;
    const uint2 bytes_t = MODE == MODE_DUAL ? fp8x8<E5M2>(f2) : bytes;
    lo4[r] = bytes_t.x;
    hi4[r] = bytes_t.y;
  }
  if (a.codes_t) {
    // 8 x 8 byte transpose in registers: column c of this thread's block as the bytes of rows 0..7
    uint32_t q00[4], q01[4], q10[4], q11[4];
    transpose4x4_bytes(lo4[0], lo4[1], lo4[2], lo4[3], q00);     // columns 0..3, rows 0..3
    transpose4x4_bytes(lo4[4], lo4[5], lo4[6], lo4[7], q01);     // columns 0..3, rows 4..7
    transpose4x4_bytes(hi4[0], hi4[1], hi4[2], hi4[3], q10);     // columns 4..7, rows 0..3
    transpose4x4_bytes(hi4[4], hi4[5], hi4[6], hi4[7], q11);     // columns 4..7, rows 4..7
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      tile_t[(c * 8 + warp) * 32 + lane] = make_uint2(q00[c], q01[c]);
      tile_t[((c + 4) * 8 + warp) * 32 + lane] = make_uint2(q10[c], q11[c]);
    }
  }
  __syncthreads();
  if (a.codes_t) {
    // thread (c = warp, j = lane) owns column col0 + 8 j + c: 64 rows = 64 bytes
    const int k = col0 + 8 * lane + warp;
    if (k < a.cols) {
      uint2 o[8];
#pragma unroll
      for (int w8 = 0; w8 < 8; ++w8) o[w8] = tile_t[(warp * 8 + w8) * 32 + lane];
      uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<uint8_t*>(a.codes_t) + (long long)k * a.rows + row0);
#pragma unroll
      for (int h = 0; h < 4; ++h) dst[h] = make_uint4(o[2 * h].x, o[2 * h].y, o[2 * h + 1].x, o[2 * h + 1].y);
    }
  }
}

template <int MODE, bool PRESCALE>
void launch_encode_fp8(dim3 grid, cudaStream_t stream, const EncodeArgs& a) {
  if (a.e5m2)
    encode_fp8_kernel<MODE, PRESCALE, true><<<grid, ENC_THREADS, 0, stream>>>(a);
  else
    encode_fp8_kernel<MODE, PRESCALE, false><<<grid, ENC_THREADS, 0, stream>>>(a);
}

// ------------------------------------------------------------------------------------------
// 4. mask -> CSR / CSC
// ------------------------------------------------------------------------------------------
// The CSR and the CSC of the residual are built from the encoder's mask and counts in three launches: the
// two pointer arrays, then the two fills.
//
// Launch 1, sparse_prefix_kernel: block 0 turns the row counts into csr_rowptr (and nnz); every
// other block owns 1024 columns and their column pointers -- the counts of all earlier columns are
// summed by the block itself, so no block waits for another.  (Where a strip's entries start inside a
// column is worked out by the fill from the counts per strip and per SUPER strips.  A running sum over
// the strips here was a serial loop on a handful of SMs: 14 us of 8192 x 4096.)
// (A total cannot exceed the caller's capacity: the host refuses capacities below 2 n_tail, and at
// most n_tail entries lie beyond either threshold.  The fill kernels still guard every write.)

// Inclusive scan of one value per thread over a block of 1024 threads; the total is left in warp_tot[31].
__device__ __forceinline__ int block_scan_1024(int v, int* warp_tot /*[32] shared*/) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  v = warp_inclusive_scan(v);
  if (lane == 31) warp_tot[warp] = v;
  __syncthreads();
  if (warp == 0) warp_tot[lane] = warp_inclusive_scan(warp_tot[lane]);
  __syncthreads();
  if (warp > 0) v += warp_tot[warp - 1];
  return v;
}

__global__ void __launch_bounds__(1024, 1)
sparse_prefix_kernel(const int* __restrict__ row_cnt, int rows, int* __restrict__ rowptr, int* __restrict__ nnz_out,
                     const int* __restrict__ col_cnt, int cols, int* __restrict__ colptr) {
  __shared__ int warp_tot[32];
  const int t = threadIdx.x;
  if (blockIdx.x == 0) {
    // four rows per thread and round
    int base = 0;
    for (int r0 = 0; r0 < rows; r0 += 4096) {
      const int r = r0 + 4 * t;
      int4 c = make_int4(0, 0, 0, 0);
      if (r < rows) c = *reinterpret_cast<const int4*>(row_cnt + r);
      const int mine = c.x + c.y + c.z + c.w;
      const int incl = block_scan_1024(mine, warp_tot);
      const int at = base + incl - mine;
      if (r < rows) {                                 // (the caller's pointer array is aligned to 4 bytes only)
        rowptr[r] = at;
        rowptr[r + 1] = at + c.x;
        rowptr[r + 2] = at + c.x + c.y;
        rowptr[r + 3] = at + c.x + c.y + c.z;
      }
      base += warp_tot[31];
      __syncthreads();                                // warp_tot is written again in the next round
    }
    if (t == 0) {
      rowptr[rows] = base;
      if (nnz_out) *nnz_out = base;
    }
    return;
  }
  const int c0 = (int(blockIdx.x) - 1) * 1024;
  // entries of all earlier columns
  int before = 0;
  for (int i = 4 * t; i < c0; i += 4096) {
    const int4 c = *reinterpret_cast<const int4*>(col_cnt + i);
    before += c.x + c.y + c.z + c.w;
  }
  const int k = c0 + t;
  const int mine = k < cols ? col_cnt[k] : 0;
  block_scan_1024(before, warp_tot);
  const int base = warp_tot[31];
  __syncthreads();
  const int incl = block_scan_1024(mine, warp_tot);
  if (k < cols) colptr[k] = base + incl - mine;
  if (k == cols - 1) colptr[cols] = base + incl;
}

// Both fills hand the marked entries of a warp's piece of the mask out to the lanes, 32 at a time and in
// output order: lane i finds the word that holds entry i by a binary search over the scanned bit counts,
// and its bit by halving.  So all lanes fetch a value at once, and the entries leave in order.  (Fetching
// every value by the lane that holds the word made the reads of a lane wait for one another: csr 12, csc 26
// us of 1920 x 5504 at 3 % per tail, 8 and 10 now.)  No shared memory: a GEMM that runs beside the fills
// leaves none on its SM, and blocks that need some would wait for its end.
constexpr int FILL_WARPS = 8;
// Entries among 1024 columns from which a row's columns are taken one after another instead, all 32 words of them in
// four rounds of loads: what ten rounds of the search take (from 256 on the two were equal at 128 x 65536).  Every
// hundredth token beyond the thresholds as a whole, alpha 0.99: 2048 x 11008 186 -> 115 us, 128 x 65536 631 -> 261.
constexpr int FILL_DENSE = 320;

// Position of set bit number r (from 0, r < popc(m)) of m.
__device__ __forceinline__ int nth_set_bit(uint32_t m, int r) {
  int pos = 0;
#pragma unroll
  for (int s = 16; s; s >>= 1) {
    const int c = __popc(m & ((1u << s) - 1u));
    if (r >= c) { r -= c; m >>= s; pos += s; }
  }
  return pos;
}

// Lane that holds entry i, given every lane's inclusive count: the first lane whose count exceeds i.
__device__ __forceinline__ int lane_of_entry(int i, int incl) {
  int lane = 0;
#pragma unroll
  for (int s = 16; s; s >>= 1) {
    const int c = __shfl_sync(0xFFFFFFFFu, incl, lane + s - 1);
    if (i >= c) lane += s;
  }
  return lane;
}

// CSR: one warp per row, 32 mask words (1024 columns) at a time.  A round's values are stored in the next
// round, so that their latency runs under its search.
__global__ void __launch_bounds__(32 * FILL_WARPS)
csr_fill_kernel(const uint32_t* __restrict__ mask, const __nv_bfloat16* __restrict__ x, int rows, int cols,
                const float* __restrict__ thresholds, int thr_per_row, const int* __restrict__ rowptr, long long cap,
                int* __restrict__ csr_col, float* __restrict__ csr_val) {
  const int row = blockIdx.x * FILL_WARPS + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  int base = rowptr[row];
  if (rowptr[row + 1] == base) return;                // nothing clamped in this row
  const int words = cols >> 5;
  const uint32_t* mrow = mask + (long long)row * words;
  const __nv_bfloat16* xrow = x + (long long)row * cols;
  const float lo = thresholds[thr_per_row ? 2 * row : 0], hi = thresholds[thr_per_row ? 2 * row + 1 : 1];
  int held_at = -1, held_col = 0;                     // the previous round's entry of this lane
  __nv_bfloat16 held = __float2bfloat16(0.0f);
  auto put = [&]() {
    if (held_at >= 0 && held_at < cap) {
      const float v = __bfloat162float(held);
      csr_col[held_at] = held_col;
      csr_val[held_at] = __fsub_rn(v, v > hi ? hi : lo);
    }
  };
  uint32_t next = lane < words ? mrow[lane] : 0u;
  for (int w0 = 0; w0 < words; w0 += 32) {
    const uint32_t m = next;
    next = w0 + 32 + lane < words ? mrow[w0 + 32 + lane] : 0u;
    const int c = __popc(m);
    const int incl = warp_inclusive_scan(c), total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    if (total >= FILL_DENSE) {
      // word by word, a lane per column: the row's own order, eight coalesced loads in flight
#pragma unroll 1
      for (int j0 = 0; j0 < 32 && w0 + j0 < words; j0 += 8) {
        __nv_bfloat16 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = xrow[32 * min(w0 + j0 + u, words - 1) + lane];
#pragma unroll
        for (int u = 0; u < 8; ++u) {                   // (words beyond the row are zero)
          const uint32_t word = __shfl_sync(0xFFFFFFFFu, m, j0 + u);
          const int at = base + __shfl_sync(0xFFFFFFFFu, incl - c, j0 + u) + __popc(word & ((1u << lane) - 1u));
          if (((word >> lane) & 1u) && at < cap) {
            const float f = __bfloat162float(v[u]);
            csr_col[at] = 32 * (w0 + j0 + u) + lane;
            csr_val[at] = __fsub_rn(f, f > hi ? hi : lo);
          }
        }
      }
      base += total;
      continue;
    }
    for (int i0 = 0; i0 < total; i0 += 32) {
      const int i = min(i0 + lane, total - 1);
      const int src = lane_of_entry(i, incl);
      const uint32_t word = __shfl_sync(0xFFFFFFFFu, m, src);
      const int first = __shfl_sync(0xFFFFFFFFu, incl - c, src);
      const int col = 32 * (w0 + src) + nth_set_bit(word, i - first);
      put();
      held_at = i0 + lane < total ? base + i : -1;
      held_col = col;
      held = xrow[col];
    }
    base += total;
  }
  put();
}

// 32 x 32 bit transpose over a warp: bit c of lane r -> bit r of lane c.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t v) {
  const int lane = threadIdx.x & 31;
  uint32_t keep = 0x0000FFFFu;
#pragma unroll
  for (int j = 16; j; j >>= 1) {
    const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, v, j);
    v = lane & j ? (v & ~keep) | ((o >> j) & keep) : (v & keep) | ((o << j) & ~keep);
    keep ^= keep << (j >> 1);
  }
  return v;
}

// CSC: one warp per (64-row strip, 32-column word of the mask).  The word's two 32 x 32 blocks are
// transposed: lane c holds the marked rows of column c.
__global__ void __launch_bounds__(32 * FILL_WARPS)
csc_fill_kernel(const uint32_t* __restrict__ mask, const __nv_bfloat16* __restrict__ x, int rows, int cols,
                const float* __restrict__ thresholds, int thr_per_row, const int* __restrict__ colptr,
                const uint8_t* __restrict__ strip_cnt, const int* __restrict__ super_cnt, long long cap,
                int* __restrict__ csc_row, float* __restrict__ csc_val) {
  const int lane = threadIdx.x & 31;
  const int q = blockIdx.x * FILL_WARPS + (threadIdx.x >> 5), strip = blockIdx.y;
  const int words_per_row = cols >> 5;
  if (q >= words_per_row) return;
  const int r0 = strip * ENC_TM;
  const uint32_t w0 = mask[(long long)(r0 + lane) * words_per_row + q];
  const uint32_t w1 = mask[(long long)(r0 + 32 + lane) * words_per_row + q];
  if (!__any_sync(0xFFFFFFFFu, w0 | w1)) return;
  // where this strip's entries of column 32 q + lane start: the column's pointer, whole groups of SUPER
  // strips, then the strips of the own group
  const int k = 32 * q + lane;
  int at = colptr[k];
  const int sup = strip / SUPER;
  for (int g = 0; g < sup; ++g) at += super_cnt[(long long)g * cols + k];
#pragma unroll
  for (int g = 0; g < SUPER - 1; ++g)
    if (sup * SUPER + g < strip) at += strip_cnt[(long long)(sup * SUPER + g) * cols + k];
  const uint32_t t0 = transpose_bits(w0), t1 = transpose_bits(w1);       // rows 0..31 / 32..63 of column `lane`
  const int c0 = __popc(t0), c = c0 + __popc(t1);
  const int incl = warp_inclusive_scan(c), total = __shfl_sync(0xFFFFFFFFu, incl, 31);
  const float lo = thresholds[0], hi = thresholds[1];
  int held_at = -1, held_row = 0;                     // the previous round's entry of this lane
  __nv_bfloat16 held = __float2bfloat16(0.0f);
  auto put = [&]() {
    if (held_at >= 0 && held_at < cap) {
      float l = lo, h = hi;
      if (thr_per_row) { l = thresholds[2 * held_row]; h = thresholds[2 * held_row + 1]; }
      const float v = __bfloat162float(held);
      csc_row[held_at] = held_row;
      csc_val[held_at] = __fsub_rn(v, v > h ? h : l);
    }
  };
  for (int i0 = 0; i0 < total; i0 += 32) {
    const int i = min(i0 + lane, total - 1);
    const int src = lane_of_entry(i, incl);
    const uint32_t m0 = __shfl_sync(0xFFFFFFFFu, t0, src), m1 = __shfl_sync(0xFFFFFFFFu, t1, src);
    const int n0 = __shfl_sync(0xFFFFFFFFu, c0, src), first = __shfl_sync(0xFFFFFFFFu, incl - c, src);
    const int to = __shfl_sync(0xFFFFFFFFu, at, src);
    const int j = i - first;                          // number of the entry inside its column
    const int r = r0 + (j < n0 ? nth_set_bit(m0, j) : 32 + nth_set_bit(m1, j - n0));
    put();
    held_at = i0 + lane < total ? to + j : -1;
    held_row = r;
    held = x[(long long)r * cols + 32 * q + src];
  }
  put();
}

// At most two blocks per SM, and as few as give no block more rows than that.  Small tensors (a block
// holds a few thousand elements) are counted whole: the sample's chain would cost more than it saves.
void launch_select(SelectArgs& a, int num_sms, cudaStream_t stream) {
  const int most = SEL_BLOCKS_PER_SM * num_sms, per = (a.rows + most - 1) / most;
  // abs mode has one bracket on the magnitudes, with both tails in it
  const int k = select_sample_rank(a.n, a.abs_mode ? 2 * a.n_tail : a.n_tail);
  a.sample_rank = a.n < (long long)SEL_ALL * num_sms ? -1 : k;
  tail_select_kernel<<<(a.rows + per - 1) / per, SEL_THREADS, SEL_DYN_SMEM, stream>>>(a);
}

// One wave of blocks, four per SM, each with at least one step of rows.
dim3 absmax_grid(int rows, int cols, int num_sms) {
  const int strips = (cols + ENC_TK - 1) / ENC_TK, steps = rows / AB_ROWS;
  int groups = 4 * num_sms / strips;
  groups = groups < 1 ? 1 : groups > steps ? steps : groups;
  return dim3(strips, groups);
}

size_t r256(size_t b) { return (b + 255) & ~size_t(255); }

struct Scratch {
  int* row_max;
  int* row_min;
  uint32_t* amax_rows;
  uint32_t* amax_cols;
  uint8_t* mask;
  int* row_cnt;
  int* col_cnt;
  uint8_t* strip_cnt;
  int* super_cnt;               // directly behind col_cnt: cleared together
  int count_words;              // of both
  float* pre_rows;
  float* pre_cols;
  bool ok;
};

int supers_of(int rows) { return (rows / ENC_TM + SUPER - 1) / SUPER; }

Scratch carve(Arena& arena, int rows, int cols, bool occ) {
  Scratch s = {};
  s.row_max = arena.take<int>(rows);
  s.row_min = arena.take<int>(rows);
  s.amax_rows = arena.take<uint32_t>(rows);
  s.amax_cols = arena.take<uint32_t>(cols);
  s.row_cnt = arena.take<int>(rows);
  s.pre_rows = arena.take<float>(rows);
  s.pre_cols = arena.take<float>(cols);
  if (occ) {
    s.mask = arena.take<uint8_t>(size_t(rows) * cols / 8);
    s.strip_cnt = arena.take<uint8_t>(size_t(rows / ENC_TM) * cols);
    s.count_words = cols * (1 + supers_of(rows));
    s.col_cnt = arena.take<int>(size_t(s.count_words));
    s.super_cnt = s.col_cnt + cols;
  }
  s.ok = arena.ok;
  return s;
}

}  // namespace

// Once per device, before the first launch there.
int quantize_setup() {
  FP4_CUDA_TRY(cudaFuncSetAttribute(tail_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SEL_DYN_SMEM));
  return FP4_OK;
}

// Counters of the quantile selection that live as long as the context: two sets, parity, ticket.
size_t quantize_persistent_bytes() { return (2 * size_t(HIST_SET_WORDS) + 64) * 4; }

size_t quantize_scratch_bytes(int64_t rows, int64_t cols) {
  size_t b = 0;
  b += 5 * r256(size_t(rows) * 4) + 2 * r256(size_t(cols) * 4);   // per-row / per-column vectors
  b += r256(size_t(rows) * size_t(cols) / 8);                    // outlier mask
  b += r256(size_t(rows / ENC_TM) * size_t(cols));               // per-strip column counts (bytes)
  b += r256(size_t(cols) * size_t(1 + supers_of(int(rows))) * 4);   // column counts, whole and per SUPER strips
  return b;
}

int launch_csc_fill(fp4_ctx* ctx, cudaStream_t stream, const CscFill& f) {
  KernelScope scope(ctx, stream, KC_SPARSE, 1);
  const dim3 grid((f.cols / 32 + FILL_WARPS - 1) / FILL_WARPS, f.rows / ENC_TM);
  csc_fill_kernel<<<grid, 32 * FILL_WARPS, 0, stream>>>(f.mask, static_cast<const __nv_bfloat16*>(f.x_bf16), f.rows, f.cols,
                                                       f.thresholds, f.thr_per_row, f.colptr, f.strip_cnt, f.super_cnt, f.cap,
                                                       f.csc_row, f.csc_val);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

int launch_quantize(fp4_ctx* ctx, cudaStream_t stream, Arena& arena, const void* x_bf16, int64_t rows64,
                    int64_t cols64, int scale_axis, double alpha, const float* prescale, float prescale_div,
                    fp4_qtensor* out, int32_t* status, const SparseOverlap* overlap) {
  const int rows = int(rows64), cols = int(cols64);
  const long long n = (long long)rows * cols;
  const bool occ = alpha < 1.0;
  const bool e4m3 = out->format == FP4_FORMAT_E4M3 || out->format == FP4_FORMAT_E5M2;   // an FP8 format
  if (out->format != FP4_FORMAT_E2M1 && !e4m3) return FP4_ERR_ARG;
  if (e4m3 && occ) return FP4_ERR_ARG;               // outlier clamping belongs to 4-bit activations
  const uint4* x = static_cast<const uint4*>(x_bf16);
  Scratch sc = carve(arena, rows, cols, occ);
  if (!sc.ok) return FP4_ERR_WORKSPACE;

  EncodeArgs ea = {};
  ea.x = x;
  ea.rows = rows;
  ea.cols = cols;
  ea.amax_rows = sc.amax_rows;
  ea.amax_cols = sc.amax_cols;
  ea.row_max = sc.row_max;
  ea.row_min = sc.row_min;
  ea.thresholds = out->thresholds;
  ea.codes = reinterpret_cast<uint32_t*>(out->codes);
  ea.codes_t = reinterpret_cast<uint32_t*>(out->codes_t);
  ea.amax_out_rows = out->amax;
  ea.amax_out_cols = out->amax;
  ea.mask = sc.mask;
  ea.row_cnt = sc.row_cnt;
  ea.strip_cnt = sc.strip_cnt;
  ea.col_cnt = sc.col_cnt;
  ea.super_cnt = sc.super_cnt;
  ea.e5m2 = out->format == FP4_FORMAT_E5M2;
  ea.fmax = fp8_max(out->format);
  const dim3 tile_grid((cols + ENC_TK - 1) / ENC_TK, rows / ENC_TM);

  const int per_token = occ && ctx->quantile_mode == FP4_QUANTILE_TOKEN;
  if (occ) {
    const long long n_tail = llround((1.0 - alpha) * double(n));
    if (per_token) {
      KernelScope scope(ctx, stream, KC_SELECT, 1);
      const int n_tail_row = int(llround((1.0 - alpha) * double(cols)));
      FP4_CUDA_TRY(cudaMemsetAsync(sc.col_cnt, 0, size_t(sc.count_words) * 4, stream));     // the encoder adds to these
      row_select_kernel<<<rows, 256, 0, stream>>>(x, cols / 8, n_tail_row, sc.row_max, sc.row_min, sc.row_cnt,
                                                  out->thresholds, status);
    } else {
      // The two sets of global counters, their parity and the ticket belong to the context: the
      // kernel keeps the set it is about to use zero (see there), so nothing is cleared here.
      KernelScope scope(ctx, stream, KC_SELECT, 1);
      SelectArgs sa = {};
      sa.x = x;
      sa.rows = rows;
      sa.vec_per_row = cols / 8;
      sa.sets = ctx->occ_hist;
      sa.parity = reinterpret_cast<unsigned*>(ctx->occ_hist + 2 * HIST_SET_WORDS);
      sa.ticket = sa.parity + 1;
      sa.row_max = sc.row_max;
      sa.row_min = sc.row_min;
      sa.row_cnt = sc.row_cnt;
      sa.n = n;
      sa.n_tail = n_tail;
      sa.thresholds = out->thresholds;
      sa.status = status;
      sa.abs_mode = ctx->quantile_mode == FP4_QUANTILE_ABS;
      sa.clear = sc.col_cnt;                          // the encoder adds to these
      sa.clear_words = sc.count_words;
      launch_select(sa, ctx->num_sms, stream);
    }
    {
      KernelScope scope(ctx, stream, KC_ENCODE, 1);
      if (per_token)
        encode_kernel<MODE_ROWS, true, false, true><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
      else
        encode_kernel<MODE_ROWS, true, false><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
    }
    cudaStream_t sp = stream;
    if (overlap && overlap->stream) {
      sp = overlap->stream;
      FP4_CUDA_TRY(cudaEventRecord(overlap->encoded, stream));
      FP4_CUDA_TRY(cudaStreamWaitEvent(sp, overlap->encoded, 0));
    }
    const uint32_t* mask32 = reinterpret_cast<const uint32_t*>(sc.mask);
    const __nv_bfloat16* xb = static_cast<const __nv_bfloat16*>(x_bf16);
    // The CSC's fill takes a stream of its own where the caller offers one: either fill is bound by the latency of its
    // chain (mask -> bits -> value), which the other's warps cover (8192 x 4096 at 0.1 %
    // per tail, clamped and encoded: 77.8 us one after the other, 72.0 now; as one launch of both 74).
    cudaStream_t sc2 = sp;
    {
      KernelScope scope(ctx, sp, KC_SPARSE, 2);
      sparse_prefix_kernel<<<1 + (cols + 1023) / 1024, 1024, 0, sp>>>(sc.row_cnt, rows, out->csr_rowptr, out->nnz,
                                                                    sc.col_cnt, cols, out->csc_colptr);
      if (overlap && overlap->colptr_done) FP4_CUDA_TRY(cudaEventRecord(overlap->colptr_done, sp));
      if (overlap && overlap->stream_csc && overlap->colptr_done) {
        sc2 = overlap->stream_csc;
        FP4_CUDA_TRY(cudaStreamWaitEvent(sc2, overlap->colptr_done, 0));
      }
      csr_fill_kernel<<<(rows + FILL_WARPS - 1) / FILL_WARPS, 32 * FILL_WARPS, 0, sp>>>(mask32, xb, rows, cols, out->thresholds, per_token, out->csr_rowptr,
                                                      out->sparse_cap, out->csr_col, out->csr_val);
    }
    if (sp != stream) FP4_CUDA_TRY(cudaEventRecord(overlap->csr_done, sp));
    const CscFill fill = {mask32, x_bf16, rows, cols, out->thresholds, per_token, out->csc_colptr,
                          sc.strip_cnt, sc.super_cnt, out->sparse_cap, out->csc_row, out->csc_val};
    if (sp != stream && overlap->later) {
      *overlap->later = fill;
      return FP4_OK;
    }
    const int rc = launch_csc_fill(ctx, sc2, fill);
    if (rc != FP4_OK) return rc;
    if (sc2 != stream && overlap->csc_done) {
      FP4_CUDA_TRY(cudaEventRecord(overlap->csc_done, sc2));
      if (sp == stream) FP4_CUDA_TRY(cudaStreamWaitEvent(stream, overlap->csc_done, 0));   // nobody else waits for it
    }
  } else {
    if (prescale && prescale_div > 0.0f) {
      float* d = scale_axis == 0 ? sc.pre_cols : sc.pre_rows;
      const int np = scale_axis == 0 ? cols : rows;
      KernelScope scope(ctx, stream, KC_ABSMAX, 1);
      descale_kernel<<<(np + 255) / 256, 256, 0, stream>>>(prescale, np, prescale_div, d);
      prescale = d;
    }
    AbsmaxArgs aa = {};
    aa.x = x;
    aa.rows = rows;
    aa.cols = cols;
    aa.amax_rows = sc.amax_rows;
    aa.amax_cols = sc.amax_cols;
    aa.status = status;
    if (scale_axis == 0) {
      aa.pre_col = prescale;
      ea.pre_col = prescale;
      FP4_CUDA_TRY(cudaMemsetAsync(sc.amax_rows, 0, size_t(rows) * 4, stream));
      {
        KernelScope scope(ctx, stream, KC_ABSMAX, 1);
        if (prescale)
          absmax_strip_kernel<MODE_ROWS><<<absmax_grid(rows, cols, ctx->num_sms), ENC_THREADS, 0, stream>>>(aa);
        else
          absmax_tile_kernel<MODE_ROWS><<<tile_grid, ENC_THREADS, 0, stream>>>(aa);
      }
      KernelScope scope(ctx, stream, KC_ENCODE, 1);
      if (e4m3 && prescale)
        launch_encode_fp8<MODE_ROWS, true>(tile_grid, stream, ea);
      else if (e4m3)
        launch_encode_fp8<MODE_ROWS, false>(tile_grid, stream, ea);
      else if (prescale)
        encode_kernel<MODE_ROWS, false, true><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
      else
        encode_kernel<MODE_ROWS, false, false><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
    } else {
      aa.pre_row = prescale;
      ea.pre_row = prescale;
      FP4_CUDA_TRY(cudaMemsetAsync(sc.amax_cols, 0, size_t(cols) * 4, stream));
      {
        KernelScope scope(ctx, stream, KC_ABSMAX, 1);
        if (prescale)
          absmax_strip_kernel<MODE_COLS><<<absmax_grid(rows, cols, ctx->num_sms), ENC_THREADS, 0, stream>>>(aa);
        else
          absmax_tile_kernel<MODE_COLS><<<tile_grid, ENC_THREADS, 0, stream>>>(aa);
      }
      KernelScope scope(ctx, stream, KC_ENCODE, 1);
      if (e4m3 && prescale)
        launch_encode_fp8<MODE_COLS, true>(tile_grid, stream, ea);
      else if (e4m3)
        launch_encode_fp8<MODE_COLS, false>(tile_grid, stream, ea);
      else if (prescale)
        encode_kernel<MODE_COLS, false, true><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
      else
        encode_kernel<MODE_COLS, false, false><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
    }
  }
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

// One read of dY for both backward GEMMs: row-scaled codes of dY (.) (amax_col_pre / 6) and
// column-scaled transposed codes of dY (.) (amax_row_pre / 6).
int launch_quantize_dual(fp4_ctx* ctx, cudaStream_t stream, Arena& arena, const void* x_bf16, int64_t rows64,
                         int64_t cols64, const float* amax_col_pre, const float* amax_row_pre, uint8_t* codes_rows,
                         float* amax_rows_out, uint8_t* codes_t_cols, float* amax_cols_out, int32_t* status,
                         int format, float col_pre_div, float row_pre_div) {
  const bool e4m3 = format != FP4_FORMAT_E2M1;       // an FP8 format
  const int rows = int(rows64), cols = int(cols64);
  Scratch sc = carve(arena, rows, cols, false);
  if (!sc.ok) return FP4_ERR_WORKSPACE;
  const dim3 tile_grid((cols + ENC_TK - 1) / ENC_TK, rows / ENC_TM);
  AbsmaxArgs aa = {};
  aa.x = static_cast<const uint4*>(x_bf16);
  aa.rows = rows;
  aa.cols = cols;
  aa.pre_col = amax_col_pre;
  aa.pre_row = amax_row_pre;
  aa.pre_col_div = col_pre_div;
  aa.pre_row_div = row_pre_div;
  aa.d_col_out = sc.pre_cols;
  aa.d_row_out = sc.pre_rows;
  aa.amax_rows = sc.amax_rows;
  aa.amax_cols = sc.amax_cols;
  aa.status = status;
  // amax_rows and amax_cols are carved one behind the other: one clearing covers both
  FP4_CUDA_TRY(cudaMemsetAsync(sc.amax_rows, 0,
                               size_t(reinterpret_cast<char*>(sc.amax_cols + cols) - reinterpret_cast<char*>(sc.amax_rows)),
                               stream));
  {
    KernelScope scope(ctx, stream, KC_ABSMAX, 1);
    absmax_strip_kernel<MODE_DUAL><<<absmax_grid(rows, cols, ctx->num_sms), ENC_THREADS, 0, stream>>>(aa);
  }
  EncodeArgs ea = {};
  ea.x = aa.x;
  ea.rows = rows;
  ea.cols = cols;
  ea.pre_col = sc.pre_cols;
  ea.pre_row = sc.pre_rows;
  ea.amax_rows = sc.amax_rows;
  ea.amax_cols = sc.amax_cols;
  ea.codes = reinterpret_cast<uint32_t*>(codes_rows);
  ea.codes_t = reinterpret_cast<uint32_t*>(codes_t_cols);
  ea.amax_out_rows = amax_rows_out;
  ea.amax_out_cols = amax_cols_out;
  ea.e5m2 = format == FP4_FORMAT_E5M2;
  ea.fmax = fp8_max(format);
  KernelScope scope(ctx, stream, KC_ENCODE, 1);
  if (e4m3)
    launch_encode_fp8<MODE_DUAL, true>(tile_grid, stream, ea);
  else
    encode_kernel<MODE_DUAL, false, true><<<tile_grid, ENC_THREADS, 0, stream>>>(ea);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

// ------------------------------------------------------------------------------------------
// Quantile thresholds without any allocation
// ------------------------------------------------------------------------------------------
// Scratch of fp4_quantile_thresholds_static: the 65536-bin histogram, the select kernel's segment
// sums and ticket, and the row extremes of up to FP4_STATIC_MAX_ROWS rows.  It lives in the
// library image: every GPU that loads the library holds these 769 KB until the process exits.
namespace {
constexpr size_t STATIC_HIST_BYTES = 65536 * sizeof(uint32_t);
constexpr size_t STATIC_SELECT_BYTES = 1024;      // 32 coarse counters, then (at 512) the ticket
constexpr size_t STATIC_SCRATCH_BYTES =
    STATIC_HIST_BYTES + STATIC_SELECT_BYTES + 2 * size_t(FP4_STATIC_MAX_ROWS) * sizeof(int);
constexpr int STATIC_MAX_DEVICES = 64;
}  // namespace
static __device__ __align__(256) unsigned char g_static_scratch[STATIC_SCRATCH_BYTES];

extern "C" int fp4_quantile_thresholds_static(void* stream, const void* x_bf16, int64_t rows, int64_t cols,
                                              double alpha, float* thresholds) {
  // In host code `g_static_scratch` is only a handle; the device address of this device's copy
  // is looked up once per device and cached (under a lock: host threads may race to the first call).
  static void* scratch_of_device[STATIC_MAX_DEVICES] = {};
  static int sms_of_device[STATIC_MAX_DEVICES] = {};
  static std::mutex setup_lock;
  if (!x_bf16 || !thresholds) return FP4_ERR_NULL;
  if (rows <= 0 || cols <= 0 || (rows % 128) || (cols % 128) || rows * cols >= (int64_t(1) << 31))
    return FP4_ERR_SHAPE;
  if (rows > FP4_STATIC_MAX_ROWS) return FP4_ERR_STATIC_LIMIT;
  if (!(alpha > 0.5 && alpha < 1.0)) return FP4_ERR_ALPHA;
  if (reinterpret_cast<uintptr_t>(x_bf16) & 15) return FP4_ERR_ALIGN;
  const long long n = (long long)rows * cols;
  const long long n_tail = llround((1.0 - alpha) * double(n));
  if (2 * n_tail >= n) return FP4_ERR_ALPHA;

  int device = -1;
  FP4_CUDA_TRY(cudaGetDevice(&device));
  if (device < 0 || device >= STATIC_MAX_DEVICES) return FP4_ERR_ARG;
  std::unique_lock<std::mutex> guard(setup_lock);
  if (!scratch_of_device[device]) {
    void* ptr = nullptr;
    FP4_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_static_scratch));
    int sms = 0;
    FP4_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    const int rc = quantize_setup();
    if (rc != FP4_OK) return rc;
    sms_of_device[device] = sms;
    scratch_of_device[device] = ptr;
  }
  const int num_sms = sms_of_device[device];
  unsigned char* base = static_cast<unsigned char*>(scratch_of_device[device]);
  guard.unlock();
  uint32_t* hist = reinterpret_cast<uint32_t*>(base);
  unsigned* ticket = reinterpret_cast<unsigned*>(base + STATIC_HIST_BYTES + 512);   // behind the coarse counters
  int* row_max = reinterpret_cast<int*>(base + STATIC_HIST_BYTES + STATIC_SELECT_BYTES);
  int* row_min = row_max + FP4_STATIC_MAX_ROWS;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // The array keeps what the previous call left (a call that was cut short may have left counts
  // behind): the histogram and the ticket are cleared; the row extremes are written before read.
  FP4_CUDA_TRY(cudaMemsetAsync(base, 0, STATIC_HIST_BYTES + STATIC_SELECT_BYTES, st));
  SelectArgs sa = {};
  sa.x = static_cast<const uint4*>(x_bf16);
  sa.rows = int(rows);
  sa.vec_per_row = int(cols / 8);
  sa.sets = hist;
  sa.ticket = ticket;
  sa.row_max = row_max;
  sa.row_min = row_min;
  sa.n = n;
  sa.n_tail = n_tail;
  sa.thresholds = thresholds;
  launch_select(sa, num_sms, st);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}
