// Outlier compensation (Section 3.2: the sparse residual times a dense high-precision matrix):
// forward fused with the final store, weight gradient (Eq. 6) as rows for the GEMM's epilogue.
//
//   forward   Y[m, :]  = store( Y1[m, :] + sum_{(m,k) in dA} dA[m,k] * W[k, :] )
//   wgrad     C[k, :] = sum_{(m,k) in dA} dA[m,k] * dY[m, :]   for the columns k that hold entries;
//             the weight-gradient GEMM adds C and applies the DGE factor in its epilogue
//
// Both are "sparse row times dense BF16 matrix" with fp32 accumulation on the plain ALUs: a warp
// owns one output row and 256 of its columns (8 per lane); the sparse entries of that row (CSR
// for the forward, CSC for the weight gradient) are walked in order, so the result is
// deterministic.  The FP4 branch and the compensation meet in fp32 and are rounded once.
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "gather.cuh"

namespace {

constexpr int COMP_THREADS = 256;          // 8 warps = 8 output rows per block
constexpr int COMP_COLS = 256;             // columns per block (8 per lane)

template <int n>
__device__ __forceinline__ void add_kept(float (&acc)[8], const uint2* __restrict__ kept, const uint4* __restrict__ dense,
                                         int vec_per_row, int vcol) {
  uint2 t[n];
  uint4 d[n];
#pragma unroll
  for (int u = 0; u < n; ++u) t[u] = __ldg(&kept[u]);
#pragma unroll
  for (int u = 0; u < n; ++u) d[u] = __ldg(&dense[(long long)t[u].x * vec_per_row + vcol]);
#pragma unroll
  for (int u = 0; u < n; ++u) fma8(acc, __uint_as_float(t[u].y), d[u]);
}

// Y1 is read for the last time and Y leaves with streaming stores, so that neither pushes the rest of Y1 and the slab
// of weight rows out of L2; two or three last entries of a token travel together.  One token per
// warp and few registers: the chain row pointer -> entry -> weight row is hidden by the other warps (walking tokens with the next
// Y1 in flight took 17 us of 4096 x 2048 x 2048 instead of 11).  8192 x 5120 x 5120 at 0.01 %: 65 -> 52.5 us, 4096 x
// 2048 x 5504 at 0.1 %: 37 -> 28, with the walk from the end below.  Blocks of four warps: with eight, a block's
// slots waited for its slowest warp (51 % of the warps active; 51.8 -> 49.6, 28.1 -> 26.9; blocks of two are slower;
// comp_fwd_kept, 2048 x 512 x 2048 at 1 %: 9.4 -> 8.9).
// Long rows, 32 entries at a time: forward 128 x 4096 x 4096 with every hundredth token beyond the thresholds 682 -> 450
// us.  Ten blocks of 48 registers per SM instead of twelve of 40 cost light residuals 1 to 3 % of their forward; 52
// registers without a bound gain the long rows little (618).
constexpr int FWD_THREADS = 128;
__device__ __forceinline__ float4 load_y1(const float* p) {
  float4 v;
  asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}
__global__ void __launch_bounds__(FWD_THREADS, 10)
comp_fwd_kernel(const float* __restrict__ y1, const int* __restrict__ rowptr, const int* __restrict__ col,
                const float* __restrict__ val, const uint4* __restrict__ w, int M, int N, void* y, int out_f32) {
  // blocks that follow one another share the 256 output columns, i.e. the same slab of the weight
  // rows (K x 512 bytes): it stays in L2 while the tokens stream past
  // (from the end: what the GEMM wrote last is still in L2)
  const int m = (gridDim.x - 1 - blockIdx.x) * (FWD_THREADS / 32) + (threadIdx.x >> 5);
  const int n0 = (gridDim.y - 1 - blockIdx.y) * COMP_COLS + 8 * (threadIdx.x & 31);
  if (m >= M) return;
  const bool live = n0 < N;                           // (every lane takes part in the walk over a long row)
  // Y1 is requested first: its latency runs under the dependent chain row pointer -> entry -> weight row
  const long long off = (long long)m * N + (live ? n0 : 0);
  float4 a = load_y1(y1 + off), b = load_y1(y1 + off + 4);
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const int vcol = live ? n0 >> 3 : 0, e1 = __ldg(&rowptr[m + 1]);
  int e = __ldg(&rowptr[m]);
  if (e + 32 <= e1) {
    add_groups_of_32(acc, col, val, e, e1, w, N >> 3, vcol);
    e += (e1 - e) & ~31;
    a = load_y1(y1 + off);                            // (not kept over the walk: registers)
    b = load_y1(y1 + off + 4);
  }
  sparse_row_times_dense(acc, col, val, e, e1, w, N >> 3, vcol);
  if (!live) return;
  const float y8[8] = {a.x + acc[0], a.y + acc[1], a.z + acc[2], a.w + acc[3],
                       b.x + acc[4], b.y + acc[5], b.z + acc[6], b.w + acc[7]};
  store8(y, out_f32, off, y8);
}

// The forward compensation when the dense tail is in use: tail_a has listed, per token, the entries
// the tail does not cover (`kept`: column and value bits, at the token's own range of the CSR, ending
// at kept_end[m]), so this kernel walks a plain list: one 8-byte broadcast load per entry, eight
// weight-row gathers in flight per lane at 32 warps per SM (measured on the 13B layer: four in flight 9.3 ms per
// step, eight 7.7 ms, twelve at 24 warps 8.0 ms, sixteen at 16 warps 10.2 ms).  If the tail was switched off on the
// device (*tail_count == 0: a value FP16 cannot hold) the list is not valid and the whole CSR row is added instead.
constexpr int FWD_FLY = 8;                 // weight-row gathers a lane keeps in flight
__global__ void __launch_bounds__(FWD_THREADS, 8)
comp_fwd_kept_kernel(const float* __restrict__ y1, const int* __restrict__ rowptr, const int* __restrict__ col,
                     const float* __restrict__ val, const uint2* __restrict__ kept, const int* __restrict__ kept_end,
                     const uint4* __restrict__ w, int M, int N, void* y, int out_f32,
                     const int* __restrict__ tail_count) {
  const int m = (gridDim.x - 1 - blockIdx.x) * (FWD_THREADS / 32) + (threadIdx.x >> 5);
  const int n0 = (gridDim.y - 1 - blockIdx.y) * COMP_COLS + 8 * (threadIdx.x & 31);
  if (m >= M || n0 >= N) return;
  const long long off = (long long)m * N + n0;
  const float4 a = __ldcs(reinterpret_cast<const float4*>(y1 + off));
  const float4 b = __ldcs(reinterpret_cast<const float4*>(y1 + off + 4));
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const int vec_per_row = N >> 3, vcol = n0 >> 3;
  if (__ldg(tail_count) > 0) {
    int e = __ldg(&rowptr[m]);
    const int e1 = __ldg(&kept_end[m]);
    for (; e + FWD_FLY <= e1; e += FWD_FLY) add_kept<FWD_FLY>(acc, kept + e, w, vec_per_row, vcol);
    // the last one to seven: four, two, one
    if (e + 4 <= e1) {
      add_kept<4>(acc, kept + e, w, vec_per_row, vcol);
      e += 4;
    }
    if (e + 2 <= e1) {
      add_kept<2>(acc, kept + e, w, vec_per_row, vcol);
      e += 2;
    }
    if (e < e1) add_kept<1>(acc, kept + e, w, vec_per_row, vcol);
  } else {
    sparse_row_times_dense(acc, col, val, __ldg(&rowptr[m]), __ldg(&rowptr[m + 1]), w, vec_per_row, vcol);
  }
  const float y8[8] = {a.x + acc[0], a.y + acc[1], a.z + acc[2], a.w + acc[3],
                       b.x + acc[4], b.y + acc[5], b.z + acc[6], b.w + acc[7]};
  store8(y, out_f32, off, y8);
}

// Columns of the residual by how many entries they hold.  LONG_COLUMN (and M / 4) entries make a column a
// candidate for the dense class: an outlier channel that most tokens hit (Appendix D).
constexpr int LONG_COLUMN = 512;
// From how many entries a column's gathers are spread over a whole cluster of blocks instead of one warp:
// LONG_FEW entries as long as those columns keep a cluster per SM busy for LONG_FEW_ROUNDS items at most, else
// LONG_COLUMN.  A warp walks eight entries per round trip to L2, so the few outlier channels of a small batch (256
// entries: 32 round trips) are what everything waits for (256 x 4096 x 4096 with 40 of them, four rounds: backward 91
// us by clusters, 99 by warps).  An item of a cluster takes about 4 us however short its column is: a hundred channels
// with 400 entries each (512 x 11008 x 4096, 16 items a channel: 150 us by warps, 176 by clusters) or a few hundred
// columns with 64 (2048 x 512 x 2048 at 4 %: 72 and 92) stay with the warps.
constexpr int LONG_FEW = 64, LONG_FEW_ROUNDS = 5;

struct ColumnClasses {
  int* list_dense;             // [DENSE_TC_MAX] dense columns, ascending
  int* list_long;              // [K]
  int4* list_short;            // [K] column, its entries' range
  int* counts;                 // numbers of dense, long and short columns
  int* slot_of_col;            // [K] position among the dense columns; DENSE_TC_MAX for a long or short one; -1: empty
};

// Exclusive counts of a flag over a block of 1024 threads: how many threads before this one have it set.  Two flags travel
// together (low and high half of a word).
__device__ __forceinline__ int block_rank_1024(bool f, bool g, int* warp_tot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned mf = __ballot_sync(0xFFFFFFFFu, f), mg = __ballot_sync(0xFFFFFFFFu, g), below = (1u << lane) - 1u;
  if (lane == 0) warp_tot[warp] = __popc(mf) | (__popc(mg) << 16);
  __syncthreads();
  const int before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? warp_tot[lane] : 0);     // (at most 1024 each)
  return before + (__popc(mf & below) | (__popc(mg & below) << 16));
}

// Dense columns: the first DENSE_TC_MAX, in ascending order, that hold at least `dense_from` entries (INT_MAX:
// none).  With ALL the others are listed too, long and short ones, in ascending order.
// A block owns 1024 columns and counts all earlier ones itself (coalesced reads of a few KB from L2), so no
// block waits for another: one block walking all columns in stretches took 4.5 us of 2048 and 17.5 of 11008.  The
// sums meet behind one barrier and the ranks come from ballots (a barrier or two for every sum and scan: backward of 128 x 4096 x 11008 112.6 us, 111.1 now).
template <bool ALL>
__global__ void __launch_bounds__(1024, 1)
classify_columns_kernel(const int* __restrict__ colptr, int K, int dense_from, int few_max, const ColumnClasses out) {
  constexpr int SUMS = ALL ? 8 : 2;
  __shared__ int part[SUMS][32], rank_tot[2][32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, c0 = blockIdx.x * 1024, k = c0 + t;
  const int e0 = k < K ? __ldg(&colptr[k]) : 0, n = k < K ? __ldg(&colptr[k + 1]) - e0 : 0;
  // candidates, columns with LONG_FEW entries and more, with LONG_COLUMN and more (both without candidates), with any:
  // in all, and before c0
  int sum[SUMS] = {};
  for (int j = t; j < K; j += 1024) {
    const int m = __ldg(&colptr[j + 1]) - __ldg(&colptr[j]);
    const bool b = j < c0, c = m >= dense_from;
    sum[0] += c;
    sum[1] += c && b;
    if constexpr (ALL) {
      sum[2] += m >= LONG_FEW && !c;
      sum[3] += m >= LONG_FEW && !c && b;
      sum[4] += m >= LONG_COLUMN && !c;
      sum[5] += m >= LONG_COLUMN && !c && b;
      sum[6] += m > 0;
      sum[7] += m > 0 && b;
    }
  }
#pragma unroll
  for (int i = 0; i < SUMS; ++i) {
    const int v = __reduce_add_sync(0xFFFFFFFFu, sum[i]);
    if (lane == 0) part[i][warp] = v;
  }
  const bool is_cand = n >= dense_from;
  const int cand_rank = block_rank_1024(is_cand, false, rank_tot[0]);       // (its barrier is the sums' too)
#pragma unroll
  for (int i = 0; i < SUMS; ++i) sum[i] = __reduce_add_sync(0xFFFFFFFFu, part[i][lane]);
  const int cand = sum[0], cand_b = sum[1], n_dense = min(cand, DENSE_TC_MAX), rank = cand_b + cand_rank;
  const bool dense = is_cand && rank < DENSE_TC_MAX;
  if (dense) out.list_dense[rank] = k;
  if constexpr (!ALL) {
    if (k < K) out.slot_of_col[k] = dense ? rank : -1;
    if (k == 0) out.counts[0] = n_dense;
  } else {
    const bool use_few = sum[2] <= few_max;
    const int long_from = use_few ? LONG_FEW : LONG_COLUMN;
    // (candidates beyond DENSE_TC_MAX hold LONG_COLUMN entries or more: they are long)
    const int large = (use_few ? sum[2] : sum[4]) + cand - n_dense;
    const int large_b = (use_few ? sum[3] : sum[5]) + max(0, cand_b - DENSE_TC_MAX);
    const int any = sum[6], any_b = sum[7];
    const bool is_long = !dense && n >= long_from, is_short = !dense && !is_long && n > 0;
    const int ranks = block_rank_1024(is_long, is_short, rank_tot[1]);
    if (is_long) out.list_long[large_b + (ranks & 0xFFFF)] = k;
    if (is_short) out.list_short[any_b - large_b - min(cand_b, DENSE_TC_MAX) + (ranks >> 16)] = make_int4(k, e0, e0 + n, 0);
    if (k < K) out.slot_of_col[k] = dense ? rank : n > 0 ? DENSE_TC_MAX : -1;
    if (k == 0) {
      out.counts[0] = n_dense;
      out.counts[1] = large;
      out.counts[2] = any - n_dense - large;
    }
  }
}

// Two-term FP16 split of x: hi = RN16(x), lo = RN16(x - hi), stored for the cross products as
// hi_small = hi / TAIL_BALANCE and lo_big = TAIL_BALANCE * lo (exact powers of two: see GemmTail).
__device__ __forceinline__ void split_half(float x, __half& hi, __half& hi_small, __half& lo_big) {
  hi = __float2half_rn(x);
  const float h = __half2float(hi);
  hi_small = __float2half_rn(h * (1.0f / TAIL_BALANCE));
  lo_big = __float2half_rn((x - h) * TAIL_BALANCE);
}

// A operand of the dense tail: row m holds, for hot column s = 64 j + c, the value
// x = residual[m, k_s] / (d_A[m] * TAIL_SCALE) as x_hi at column 192 j + c, x_hi / TAIL_BALANCE at
// 192 j + 64 + c and TAIL_BALANCE x_lo at 192 j + 128 + c; zero elsewhere.  One warp per token walks the token's CSR row.  A value
// that FP16 cannot hold (or a token whose de-scale is zero, or a list that is too short) switches the tail off for this call:
// *count becomes 0 and the per-entry kernel keeps every entry.
__global__ void __launch_bounds__(COMP_THREADS)
tail_a_kernel(const int* __restrict__ rowptr, const int* __restrict__ col, const float* __restrict__ val,
              const int* __restrict__ slot_of_col, int* __restrict__ count, const float* __restrict__ amax_row,
              float row_div, __half* __restrict__ ta, int M, uint2* __restrict__ kept, int kept_cap, int* __restrict__ kept_end) {
  const int hot = *count;
  if (hot == 0) return;
  const int lane = threadIdx.x & 31;
  const int m = blockIdx.x * (COMP_THREADS / 32) + (threadIdx.x >> 5);
  if (m >= M) return;
  uint32_t* row32 = reinterpret_cast<uint32_t*>(ta + size_t(m) * TAIL_WIDTH);
  for (int i = lane; i < TAIL_WIDTH / 2; i += 32) row32[i] = 0u;
  __syncwarp();
  const float scale = __fdiv_rn(__ldg(&amax_row[m]), row_div) * TAIL_SCALE;
  __half* row = ta + size_t(m) * TAIL_WIDTH;
  bool bad = false;
  const int e0 = rowptr[m], e1 = rowptr[m + 1];
  int n_kept = e0;                                       // the kept entries go to this token's own range
  for (int base = e0; base < e1; base += 32) {
    const int e = base + lane;
    int k = 0, slot = -1;
    float v = 0.0f;
    if (e < e1) {
      k = col[e];
      v = val[e];
      slot = slot_of_col[k];
    }
    const bool is_hot = e < e1 && unsigned(slot) < unsigned(hot);
    const bool keep = e < e1 && !is_hot;
    {                                                    // entries the tail does not cover, in column order
      const unsigned km = __ballot_sync(0xFFFFFFFFu, keep);
      const int at = n_kept + __popc(km & ((1u << lane) - 1u));
      if (keep && at < kept_cap) kept[at] = make_uint2(uint32_t(k), __float_as_uint(v));
      bad |= keep && at >= kept_cap;                     // (more entries than were noted beside the operand)
      n_kept += __popc(km);
    }
    if (!is_hot) continue;
    const float x = __fdiv_rn(v, scale);
    if (!(fabsf(x) <= 65504.0f)) { bad = true; continue; }         // also catches NaN (0 / 0)
    __half hi, hi_small, lo_big;
    split_half(x, hi, hi_small, lo_big);
    const int at = 192 * (slot >> 6) + (slot & 63);
    row[at] = hi;
    row[at + 64] = hi_small;
    row[at + 128] = lo_big;
  }
  if (lane == 0) kept_end[m] = n_kept;
  if (bad) atomicExch(count, 0);
}

// B operand of the dense tail: row n holds, for hot column s = 64 j + c, the value
// x = TAIL_SCALE * W[k_s, n] / d_W[n] as x_hi at 192 j + c, TAIL_BALANCE x_lo at 192 j + 64 + c and
// x_hi / TAIL_BALANCE at 192 j + 128 + c (|x| <= 6 * 4, or 448 * 4 for an E4M3 weight; no tail with E5M2, 57344 * 4: the weight is at
// most amax in magnitude), zero beyond the last hot column of a block of 64; blocks without one are not read.
// A block of threads makes 64 rows of such a block: whole lines of W in, a shared tile, whole lines out.  (A thread per
// row and column wrote three halfwords into lines of 768 bytes each: 2048 x 11008 x 1024 at alpha 0.995 forward 117.5 us, 109 now.)
constexpr int TAIL_B_ROWS = 64, TAIL_B_PITCH = 192 + 2;      // (halves; an odd number of words: no bank conflicts)
__global__ void __launch_bounds__(256)
tail_b_kernel(const __nv_bfloat16* __restrict__ w, const int* __restrict__ list_hot, const int* __restrict__ count,
              const float* __restrict__ amax_col, float col_div, __half* __restrict__ tb, int N) {
  __shared__ __align__(16) __half tile[TAIL_B_ROWS * TAIL_B_PITCH];           // (read by words)
  const int hot = *count, s0 = 64 * blockIdx.y, n0 = TAIL_B_ROWS * blockIdx.x;
  if (s0 >= hot) return;
  const int warp = threadIdx.x >> 5, n = 2 * (threadIdx.x & 31);             // rows n0 + n and the next one
  float d[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) d[i] = __fdiv_rn(__ldg(&amax_col[n0 + n + i]), col_div);
  __nv_bfloat162 v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int s = s0 + 8 * u + warp;
    v[u] = s < hot ? *reinterpret_cast<const __nv_bfloat162*>(w + size_t(__ldg(&list_hot[s])) * N + n0 + n)
                   : __float2bfloat162_rn(0.0f);
  }
#pragma unroll
  for (int u = 0; u < 8; ++u)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float wv = i ? __high2float(v[u]) : __low2float(v[u]);
      const float x = d[i] > 0.0f ? __fdiv_rn(wv * TAIL_SCALE, d[i]) : 0.0f;
      __half hi, hi_small, lo_big;
      split_half(x, hi, hi_small, lo_big);
      __half* at = tile + (n + i) * TAIL_B_PITCH + 8 * u + warp;
      at[0] = hi;
      at[64] = lo_big;
      at[128] = hi_small;
    }
  __syncthreads();
  constexpr int WORDS = 192 / 2;
  for (int i = threadIdx.x; i < TAIL_B_ROWS * WORDS; i += 256) {
    const int r = i / WORDS, c = i - r * WORDS;
    reinterpret_cast<uint32_t*>(tb + size_t(n0 + r) * TAIL_WIDTH + 192 * blockIdx.y)[c] =
        *reinterpret_cast<const uint32_t*>(tile + r * TAIL_B_PITCH + 2 * c);
  }
}

// Dense columns (their partial sums come from the tensor-core kernel, one set per range of tokens):
// C[column of slot s, n] = sum over the ranges, in order.
__global__ void __launch_bounds__(256)
dense_reduce_kernel(float* __restrict__ comp, const float* __restrict__ partial, const int* __restrict__ list_dense,
                    const int* __restrict__ counts, int N, int chunks, long long chunk_stride) {
  const int n4 = N >> 2;
  const int total = counts[0] * n4;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int s = i / n4;
    float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int c0 = 0; c0 < chunks; c0 += 4) {            // four loads in flight, added in chunk order
      float4 p[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        p[u] = c0 + u < chunks ? __ldg(reinterpret_cast<const float4*>(partial + (long long)(c0 + u) * chunk_stride) + i)
                               : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int u = 0; u < 4; ++u) { t.x += p[u].x; t.y += p[u].y; t.z += p[u].z; t.w += p[u].w; }
    }
    reinterpret_cast<float4*>(comp + (long long)list_dense[s] * N)[i - s * n4] = t;
  }
}

// acc[0..7] += sum of val[e] * dense[idx[e], vcol] over e = first, first + step, ... < e1, eight
// gathers in flight and the indices of the next round fetched under them.
__device__ __forceinline__ void strided_entries_times_dense(float (&acc)[8], const int* __restrict__ idx,
                                                            const float* __restrict__ val, int first, int e1,
                                                            int step, const uint4* __restrict__ dense,
                                                            int vec_per_row, int vcol) {
  int r[8];
  float v[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const bool live = first + step * u < e1;          // past the end: value 0 times row 0
    r[u] = live ? __ldg(&idx[first + step * u]) : 0;
    v[u] = live ? __ldg(&val[first + step * u]) : 0.0f;
  }
  for (int e = first; e < e1; e += 8 * step) {
    uint4 d[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) d[u] = __ldg(&dense[(long long)r[u] * vec_per_row + vcol]);
    int rn[8];
    float vn[8];
    const int nxt = e + 8 * step;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool live = nxt + step * u < e1;
      rn[u] = live ? __ldg(&idx[nxt + step * u]) : 0;
      vn[u] = live ? __ldg(&val[nxt + step * u]) : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) fma8(acc, v[u], d[u]);
#pragma unroll
    for (int u = 0; u < 8; ++u) { r[u] = rn[u]; v[u] = vn[u]; }
  }
}

// Weight-gradient compensation of the columns that are not dense:
//   comp[k, :] = sum over the entries of column k of dA[m,k] * dY[m, :].
// Long columns: a cluster of four blocks per (column, 256 outputs).  Its 32 warps take the entries
// round-robin; every block adds a quarter of the outputs, all 32 partial sums of each in warp order
// (distributed shared memory), so the result does not depend on scheduling nor on the cluster's size.
// (One block of 32 warps per item left ten outlier channels x 8 blocks of outputs with 80 blocks for 148 SMs.)
constexpr int LONG_CLUSTER = 4, LONG_WARPS = 8;
__global__ void __cluster_dims__(LONG_CLUSTER, 1, 1) __launch_bounds__(32 * LONG_WARPS, 4)
comp_wgrad_long_kernel(float* __restrict__ comp, const int* __restrict__ colptr, const int* __restrict__ row,
                       const float* __restrict__ val, const uint4* __restrict__ dy, const int* __restrict__ list,
                       const int* __restrict__ counts, int N) {
  __shared__ float part[LONG_WARPS][32][9];         // [warp][lane][8 (+1 pad)]
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_long = counts[1], n_blocks = (N + COMP_COLS - 1) / COMP_COLS;
  const int clusters = gridDim.x / LONG_CLUSTER, rank = int(cluster.block_rank());
  bool read = true;                                 // the sums of the item before have been read by all four blocks
  for (int it = blockIdx.x / LONG_CLUSTER; it < n_long * n_blocks; it += clusters) {
    const int nb = it / n_long, k = list[it - nb * n_long];
    const int n0 = nb * COMP_COLS + 8 * lane;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (n0 < N)
      strided_entries_times_dense(acc, row, val, colptr[k] + rank * LONG_WARPS + warp, colptr[k + 1], LONG_CLUSTER * LONG_WARPS,
                                  dy, N >> 3, n0 >> 3);
    if (!read) cluster.barrier_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) part[warp][lane][c] = acc[c];
    cluster.sync();
    constexpr int OWN = COMP_COLS / LONG_CLUSTER;   // outputs that this block adds, one per thread
    const int o = rank * OWN + tid;
    if (tid < OWN && nb * COMP_COLS + o < N) {
      float p[LONG_CLUSTER][LONG_WARPS];
#pragma unroll
      for (int r = 0; r < LONG_CLUSTER; ++r) {
        const float* from = cluster.map_shared_rank(&part[0][o >> 3][o & 7], r);
#pragma unroll
        for (int w = 0; w < LONG_WARPS; ++w) p[r][w] = from[w * 32 * 9];
      }
      float t = 0.0f;
#pragma unroll
      for (int r = 0; r < LONG_CLUSTER; ++r)
#pragma unroll
        for (int w = 0; w < LONG_WARPS; ++w) t += p[r][w];
      comp[(long long)k * N + nb * COMP_COLS + o] = t;
    }
    cluster.barrier_arrive();                       // (waited for behind the next item's gathers: backward of 512 x 4096 x 4096 107.2 -> 106.0 us)
    read = false;
  }
  if (!read) cluster.barrier_wait();
}

// Short columns: one warp per (column, 256 outputs), entries in order.  The work items (block of 256
// outputs, group of 8 columns) are numbered with the block of outputs as the slow index and taken
// in that order, so that the blocks in flight at any time read one or two 512-byte-wide slabs of dY
// (tokens x 512 bytes: a few MB, which stay in L2) instead of all of it: every token's piece of a
// slab is gathered by about 1 % of the columns, and those re-reads then hit L2.
// Heavy residuals are bound by L2; light ones (one or two entries per column) by the chain of loads per kilobyte of
// output: the list holds the column's range of entries, the next item's is fetched beside this one, and the last one
// to seven entries travel four, two and one at a time.  8192 x 5120 x 5120 at 0.01 %: 51 -> 43 us.
__global__ void __launch_bounds__(COMP_THREADS, 4)
comp_wgrad_short_kernel(float* __restrict__ comp, const int* __restrict__ row, const float* __restrict__ val,
                        const uint4* __restrict__ dy, const int4* __restrict__ list, const int* __restrict__ counts, int N) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_cols = counts[2];
  const unsigned groups = unsigned(n_cols + 7) >> 3;
  const unsigned items = groups * unsigned((N + COMP_COLS - 1) / COMP_COLS);
  int4 next = make_int4(-1, 0, 0, 0);                 // the warp's column of the item after this one
  int next_n0 = 0;
  auto fetch = [&](unsigned it) {
    const unsigned nb = it / groups;
    const int slot = int(it - nb * groups) * 8 + warp;
    next_n0 = int(nb) * COMP_COLS + 8 * lane;
    next.x = -1;
    if (slot < n_cols && next_n0 < N) next = __ldg(&list[slot]);
  };
  if (blockIdx.x < items) fetch(blockIdx.x);
  for (unsigned it = blockIdx.x; it < items; it += gridDim.x) {
    const int4 c = next;
    const int k = c.x, n0 = next_n0;
    if (it + gridDim.x < items) fetch(it + gridDim.x);
    if (k < 0) continue;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    {
      const int vec_per_row = N >> 3, vcol = n0 >> 3;
      int e = c.y;
      const int e1 = c.z;
      for (; e + 8 <= e1; e += 8)                   // eight gathers in flight, entries in order
        add_entries<8>(acc, row + e, val + e, dy, vec_per_row, vcol);
      // the last one to seven: four, two, one
      if (e + 4 <= e1) {
        add_entries<4>(acc, row + e, val + e, dy, vec_per_row, vcol);
        e += 4;
      }
      if (e + 2 <= e1) {
        add_entries<2>(acc, row + e, val + e, dy, vec_per_row, vcol);
        e += 2;
      }
      if (e < e1) add_entries<1>(acc, row + e, val + e, dy, vec_per_row, vcol);
    }
    float4* dst = reinterpret_cast<float4*>(comp + (long long)k * N + n0);   // streaming: dY stays in L2
    __stcs(dst, make_float4(acc[0], acc[1], acc[2], acc[3]));
    __stcs(dst + 1, make_float4(acc[4], acc[5], acc[6], acc[7]));
  }
}

// Measurement support: every block reads the whole buffer once per repeat with 16-byte loads that
// bypass L1, starting at its own offset, so that a buffer smaller than L2 is served by L2 alone.
__global__ void __launch_bounds__(256)
l2_read_probe_kernel(const uint4* __restrict__ buf, long long n_vec, int repeats, unsigned* __restrict__ sink) {
  unsigned acc = 0;
  const long long start = ((long long)blockIdx.x * 9973 * 256) % n_vec;
  for (int r = 0; r < repeats; ++r) {
    for (long long i0 = 0; i0 < n_vec; i0 += 8 * 256) {
      uint4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        long long i = start + i0 + u * 256 + threadIdx.x;
        if (i >= n_vec) i -= n_vec;
        if (i >= n_vec) i -= n_vec;
        asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w)
                     : "l"(buf + i));
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) acc ^= v[u].x ^ v[u].y ^ v[u].z ^ v[u].w;
    }
  }
  if (acc == 0x9E3779B9u) *sink = acc;               // keeps the loads alive
}

}  // namespace

extern "C" int fp4_l2_read_probe(void* stream, const void* buf, size_t bytes, int repeats, int blocks, unsigned* sink) {
  if (!buf || !sink) return FP4_ERR_NULL;
  if (bytes < 4096 * 16 || (bytes % (8 * 256 * 16)) || repeats <= 0 || blocks <= 0 ||
      (reinterpret_cast<uintptr_t>(buf) & 15))
    return FP4_ERR_ARG;
  l2_read_probe_kernel<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint4*>(buf), (long long)(bytes / 16), repeats, sink);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

int launch_comp_fwd(fp4_ctx* ctx, cudaStream_t stream, const float* y1, const int32_t* rowptr, const int32_t* col,
                    const float* val, const void* w_bf16, int64_t M, int64_t, int64_t N, void* y, int out_f32,
                    const int* tail_count, const void* kept, const int* kept_end) {
  const unsigned rows = FWD_THREADS / 32;             // a warp each
  const dim3 grid(unsigned((M + rows - 1) / rows), unsigned((N + COMP_COLS - 1) / COMP_COLS));
  KernelScope scope(ctx, stream, KC_COMP_FWD, 1);
  if (kept && kept_end && tail_count)
    comp_fwd_kept_kernel<<<grid, FWD_THREADS, 0, stream>>>(y1, rowptr, col, val, static_cast<const uint2*>(kept),
                                                            kept_end, static_cast<const uint4*>(w_bf16), int(M), int(N),
                                                            y, out_f32, tail_count);
  else
    comp_fwd_kernel<<<grid, FWD_THREADS, 0, stream>>>(y1, rowptr, col, val, static_cast<const uint4*>(w_bf16), int(M),
                                                       int(N), y, out_f32);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

size_t comp_wgrad_scratch_bytes(int64_t M, int64_t K, int64_t N) {
  auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
  size_t b = r256((size_t(K) + DENSE_TC_MAX + 4) * 4) + r256(size_t(K) * 16) + r256(size_t(K) * 4);      // lists + counters, slots
  b += dense_tc_scratch_bytes(M, N);                                                  // BF16 terms, partial sums
  return b;
}

// Residual entries the forward with a dense tail may have to list (heavier residuals take no tail).
static int64_t kept_list_capacity(int64_t M, int64_t K) { return M * K / RESIDUAL_FULL_SHARE; }

size_t fwd_tail_scratch_bytes(int64_t M, int64_t K, int64_t N) {
  auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
  return r256(size_t(M) * TAIL_WIDTH * 2) + r256(size_t(N) * TAIL_WIDTH * 2) + r256(size_t(K) * 4) +
         r256(TAIL_MAX_COLS * 4) + 256 + r256(size_t(kept_list_capacity(M, K)) * 8) + r256(size_t(M) * 4);
}

// Prepares the dense tail of the forward GEMM from the saved activation `a` (CSR, CSC column
// pointers, row amax) and the weights; fills `tail` and hands back the list
// for the per-entry kernel.  Buffers come from `scratch` (fwd_tail_scratch_bytes).
// The hot columns and W's operand hang on the column pointers alone: they are made before the stream waits for the CSR
// (`csr_done`, may be null), beside its fill on another stream.
int launch_fwd_tail(fp4_ctx* ctx, cudaStream_t stream, cudaEvent_t csr_done, const fp4_qtensor* a, const void* w_bf16,
                    const float* w_amax, float w_div, Arena& scratch, int64_t M, int64_t K, int64_t N, GemmTail* tail,
                    const void** kept_out, const int** kept_end_out) {
  __half* ta = scratch.take<__half>(size_t(M) * TAIL_WIDTH);
  __half* tb = scratch.take<__half>(size_t(N) * TAIL_WIDTH);
  int* slot_of_col = scratch.take<int>(size_t(K));
  int* list_hot = scratch.take<int>(TAIL_MAX_COLS);
  int* count = scratch.take<int>(1);
  uint2* kept = scratch.take<uint2>(size_t(kept_list_capacity(M, K)));
  int* kept_end = scratch.take<int>(size_t(M));
  if (!scratch.ok) return FP4_ERR_WORKSPACE;
  *kept_out = kept;
  *kept_end_out = kept_end;
  const int hot_from = int(M / 4 > LONG_COLUMN ? M / 4 : LONG_COLUMN);
  const ColumnClasses classes = {list_hot, nullptr, nullptr, count, slot_of_col};
  KernelScope scope(ctx, stream, KC_COMP_FWD, 3);
  classify_columns_kernel<false><<<unsigned((K + 1023) / 1024), 1024, 0, stream>>>(a->csc_colptr, int(K), hot_from, 0, classes);
  tail_b_kernel<<<dim3(unsigned(N / TAIL_B_ROWS), TAIL_MAX_COLS / 64), 256, 0, stream>>>(
      static_cast<const __nv_bfloat16*>(w_bf16), list_hot, count, w_amax, w_div, tb, int(N));
  if (csr_done) FP4_CUDA_TRY(cudaStreamWaitEvent(stream, csr_done, 0));
  tail_a_kernel<<<unsigned((M + 7) / 8), COMP_THREADS, 0, stream>>>(a->csr_rowptr, a->csr_col, a->csr_val, slot_of_col,
                                                                   count, a->amax, 6.0f, ta, int(M), kept,
                                                                   int(kept_list_capacity(M, K)), kept_end);
  FP4_CUDA_TRY(cudaGetLastError());
  tail->a = ta;
  tail->b = tb;
  tail->count = count;
  return FP4_OK;
}

int launch_comp_wgrad(fp4_ctx* ctx, cudaStream_t stream, const fp4_qtensor* a, const void* dy_bf16, Arena& scratch,
                      const int** slot_of_col_out, float* comp, int64_t M, int64_t K, int64_t N, int32_t* status,
                      const CompOverlap* overlap) {
  // lists: [K] long columns, the dense columns, three counters
  int* lists = scratch.take<int>(size_t(K) + DENSE_TC_MAX + 4);
  int4* list_short = scratch.take<int4>(size_t(K));
  int* slot_of_col = scratch.take<int>(size_t(K));
  const int splits = dense_tc_splits(ctx, M, N);
  void* vt = scratch.take<uint16_t>(size_t(3) * DENSE_TC_MAX * size_t(M));
  float* partial = scratch.take<float>(size_t(splits) * DENSE_TC_MAX * size_t(N));
  if (!scratch.ok) return FP4_ERR_WORKSPACE;
  *slot_of_col_out = slot_of_col;
  const ColumnClasses classes = {lists + K, lists, list_short, lists + K + DENSE_TC_MAX, slot_of_col};
  // Columns that at least a quarter of the tokens hit (the outlier channels) form the dense class,
  // whose product runs on the tensor cores.  It costs three launches, which pay
  // when the residual is heavy: when it may hold at least 1 % of the activation (alpha <= 0.995).
  // (No column can reach LONG_COLUMN entries with fewer tokens than that.)
  const bool dense = a->csr_rowptr != nullptr && residual_entries(a) * 100 >= M * K && M >= LONG_COLUMN;
  const int dense_from = dense ? int(M / 4 > LONG_COLUMN ? M / 4 : LONG_COLUMN) : INT_MAX;
  KernelScope scope(ctx, stream, KC_COMP_WGRAD, 3 + (dense ? 3 : 0));
  const unsigned n_blocks = unsigned((N + COMP_COLS - 1) / COMP_COLS);
  const int few_max = int(LONG_FEW_ROUNDS * unsigned(ctx->num_sms) / n_blocks);
  classify_columns_kernel<true><<<unsigned((K + 1023) / 1024), 1024, 0, stream>>>(a->csc_colptr, int(K), dense_from, few_max, classes);
  const uint4* dy = static_cast<const uint4*>(dy_bf16);
  // The long columns (a few blocks, latency) run beside the others, and beside the dense columns' chain of three launches the
  // short ones: at a thousand tokens each of these is a few microseconds of latency (backward with hot columns 1024 x 2048 x
  // 2048 at alpha 0.995 47.3 -> 41.0 us, 2048 x 11008 x 1024 111 -> 99, 4096^3 at 0.99 260 -> 255).  The host knows that dense
  // columns are allowed, not whether there are any; without one, where the chain is idle, the fork is worth -1.3 to 1.5 % (the same
  // sizes with Laplace activations 37.7 -> 38.2, 102.8 -> 101.3, 272 -> 269).  At LONG_COLUMN tokens no column is dense unless
  // every token hits it: the hot ones are long, and the short ones beside them cost more (512 x 4096 x 4096 107 -> 111).
  cudaStream_t sl = stream, ss = stream;
  if (overlap) {
    sl = overlap->stream;
    FP4_CUDA_TRY(cudaEventRecord(overlap->classified, stream));
    FP4_CUDA_TRY(cudaStreamWaitEvent(sl, overlap->classified, 0));
    if (dense && M > LONG_COLUMN && overlap->stream_short) {
      ss = overlap->stream_short;
      FP4_CUDA_TRY(cudaStreamWaitEvent(ss, overlap->classified, 0));
    }
  }
  if (dense) {
    const int rc = launch_comp_wgrad_dense_tc(ctx, stream, a, classes.list_dense, classes.counts, dy_bf16, vt, partial, splits,
                                              M, N, status);
    if (rc != FP4_OK) return rc;
    dense_reduce_kernel<<<unsigned(2 * ctx->num_sms), 256, 0, stream>>>(comp, partial, classes.list_dense, classes.counts,
                                                                       int(N), splits, (long long)DENSE_TC_MAX * N);
  }
  // long columns: up to four blocks per SM
  const unsigned clusters = unsigned(4 * ctx->num_sms / LONG_CLUSTER);
  comp_wgrad_long_kernel<<<clusters * LONG_CLUSTER, 32 * LONG_WARPS, 0, sl>>>(comp, a->csc_colptr, a->csc_row, a->csc_val, dy,
                                                                             classes.list_long, classes.counts, int(N));
  {
    // short columns: 8 per block; about 32 blocks per SM in all, each taking work items in order
    const long long max_items = (long long)((K + 7) / 8) * n_blocks;
    long long g = 32LL * ctx->num_sms;
    g = g > max_items ? max_items : g;
    comp_wgrad_short_kernel<<<unsigned(g), COMP_THREADS, 0, ss>>>(comp, a->csc_row, a->csc_val, dy, classes.list_short,
                                                                     classes.counts, int(N));
  }
  if (ss != stream) {
    FP4_CUDA_TRY(cudaEventRecord(overlap->short_done, ss));
    FP4_CUDA_TRY(cudaStreamWaitEvent(stream, overlap->short_done, 0));
  }
  if (sl != stream) {
    FP4_CUDA_TRY(cudaEventRecord(overlap->long_done, sl));
    FP4_CUDA_TRY(cudaStreamWaitEvent(stream, overlap->long_done, 0));
  }
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}
