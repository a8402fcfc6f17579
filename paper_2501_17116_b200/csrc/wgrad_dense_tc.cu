// Weight-gradient compensation of the residual's channel-dense columns on the tensor cores.
//
// Section 3.2 adds the product of the sparse residual dA = A - A_c with a dense high-precision
// matrix; in the weight gradient (Eq. 6) that product is dA^T dY.  The outlier channels of
// Appendix D make a handful of columns of dA dense (most tokens exceed the threshold there), so
// for those columns the product is a skinny dense contraction over the tokens,
//     C[s, n] = sum_m V[m, s] * dY[m, n],        s < h <= 128 dense columns,
// and it runs on tcgen05.mma instead of gathering one dY row per entry:
//   * dY is the M-side operand, read by TMA straight from the caller's BF16 tensor ([tokens x N],
//     N contiguous: an MN-major operand whose contraction runs over the box's rows);
//   * V is the N-side operand.  Its fp32 values are split exactly into three BF16 terms
//     (v = b1 + b2 + b3, each 8 significant bits), stored K-major as Vt[term][s][m]; BF16 products
//     are exact in fp32, so the tensor cores add exactly the products the fp32 kernel would form;
//   * the tensor cores accumulate one chunk of 128 tokens at a time in tensor memory (24
//     instructions, whose fp32 additions are not round-to-nearest); the epilogue warps drain each
//     chunk into registers and add the chunks in token order with ordinary fp32 additions, so the
//     number of tensor-core additions behind any output stays at 24 however many tokens there are;
//   * a CTA owns 256 output columns and a contiguous range of chunks; the ranges' partial sums go to
//     global memory and are added in range order by dense_reduce (compensate.cu): the result does
//     not depend on scheduling.
// Roles per CTA: warp 0 TMA producer, warp 1 tensor-memory allocation + MMA issue, warps 2..9
// epilogue.  Every wait is bounded (FP4_DEV_TIMEOUT).
#include <cuda.h>

#include "common.cuh"
#include "gather.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int DT_TOK = 64;                       // tokens per stage
constexpr int DT_CHUNK = 2 * DT_TOK;             // tokens accumulated in tensor memory before a drain
constexpr int DT_NT = 256;                       // output columns per CTA
constexpr int DT_BOX = 64 * 64 * 2;              // one 64 x 64 BF16 box: 8 KB
constexpr int DT_DY_BYTES = (DT_NT / 64) * DT_BOX;      // 32 KB of dY per stage
constexpr int DT_THREADS = 64 + 8 * 32;
constexpr int DT_RING = 3 * (DT_DY_BYTES + 4 * DT_BOX);      // 3 stages of up to four V boxes or 2 of six
constexpr int DT_SMEM = 1024 + DT_RING + 256;

// Shared-memory matrix descriptor of an MN-major operand tile made of 64 x 64 BF16 boxes (128-byte
// rows = 64 consecutive MN elements of one contraction index, 128-byte swizzle): groups of 8
// contraction rows are 1024 bytes apart (stride offset), blocks of 64 MN elements one box apart
// (leading offset).
__device__ __forceinline__ uint64_t make_smem_desc_mn(uint32_t smem_addr, uint32_t box_bytes) {
  uint64_t d = 0;
  d |= uint64_t((smem_addr & 0x3FFFFu) >> 4);
  d |= uint64_t(box_bytes >> 4) << 16;
  d |= uint64_t(1024 >> 4) << 32;
  d |= uint64_t(1) << 46;
  d |= uint64_t(2) << 61;
  return d;
}

// kind::f16, BF16 x BF16 -> fp32, A MN-major (dY), B K-major (Vt), M = 128, N = n
__device__ __forceinline__ uint32_t idesc_dense(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (uint32_t(n >> 3) << 17) | (uint32_t(128 >> 4) << 24);
}

// The same product with the operands in the other places, for whole residuals: A = Vt (K-major, M = 128 rows of the
// result), B = the dense matrix (MN-major, N = 256).  An instruction of 128 x 256 x 16 reads 12 KB of shared memory in
// the 131 cycles it takes, one of 128 x 128 x 16 8 KB in 65: more than the port gives beside the copies.
__device__ __forceinline__ uint32_t idesc_full() {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | (uint32_t(DT_NT >> 3) << 17) | (uint32_t(128 >> 4) << 24);
}

// Vt[term][s][m]: the three BF16 terms of the dense columns' residual values, zero where a token has
// no entry.  A block owns SPLIT_TOK tokens of one column: it finds their entries in the column's list (one
// sample per thread brackets the first one), scatters them into a shared tile and writes that out as whole
// lines.  Only rows of boxes the GEMM will load (64 per box) are written.  (Walking the tokens' rows instead, one
// dependent look-up per entry, took 46 us of 16384 x 5120 and 69 of 8192 x 11008; 6 and 5 now.)
constexpr int SPLIT_TOK = 2048;
__global__ void __launch_bounds__(256)
dense_split_kernel(const int* __restrict__ colptr, const int* __restrict__ row, const float* __restrict__ val,
                   const int* __restrict__ list_dense, const int* __restrict__ counts, __nv_bfloat16* __restrict__ vt,
                   int M) {
  __shared__ __align__(16) __nv_bfloat16 tile[3][SPLIT_TOK];
  const int n_dense = min(counts[0], DENSE_TC_MAX), s = blockIdx.y, t = threadIdx.x;
  if (s >= ((n_dense + 63) / 64) * 64) return;
  const int m0 = blockIdx.x * SPLIT_TOK, m1 = min(M, m0 + SPLIT_TOK);
  uint4* t4 = reinterpret_cast<uint4*>(&tile[0][0]);
  for (int i = t; i < 3 * SPLIT_TOK / 8; i += 256) t4[i] = make_uint4(0, 0, 0, 0);
  if (s < n_dense) {
    const int e0 = colptr[list_dense[s]], n = colptr[list_dense[s] + 1] - e0;
    // entries before the sample of the last thread whose sample lies before m0 are before m0 as well
    const int before = __syncthreads_count(n > 0 && row[e0 + int((long long)n * t / 256)] < m0);
    const int first = before ? int((long long)n * (before - 1) / 256) : 0;
    for (int e = first + t; e < n; e += 256) {
      const int m = row[e0 + e];
      if (m >= m1) break;
      if (m < m0) continue;
      const float v = val[e0 + e];
      const __nv_bfloat16 b1 = __float2bfloat16_rn(v);
      const float r1 = v - __bfloat162float(b1);                 // exact
      const __nv_bfloat16 b2 = __float2bfloat16_rn(r1);
      const float r2 = r1 - __bfloat162float(b2);                // exact
      tile[0][m - m0] = b1;
      tile[1][m - m0] = b2;
      tile[2][m - m0] = __float2bfloat16_rn(r2);                 // exact: 24 bits in three terms of 8
    }
  }
  __syncthreads();
  for (int i = t; i < 3 * (SPLIT_TOK / 8); i += 256) {
    const int term = i / (SPLIT_TOK / 8), c = i - term * (SPLIT_TOK / 8);
    if (m0 + 8 * c < m1)
      *reinterpret_cast<uint4*>(vt + size_t(term * DENSE_TC_MAX + s) * size_t(M) + size_t(m0) + 8 * c) = t4[i];
  }
}

// The whole residual (or its transpose) as a dense operand, for residuals so heavy that gathering costs more:
// row r of Vt[term][r][c] holds the terms of the residual's row r, zeros elsewhere.  Terms 1 and 2 are written always;
// term 3 is zero unless a value spans more than 16 bits (500 times the threshold): *third says so, and a second launch
// then writes it.
//
// dense_act_kernel writes it from the activation itself, eight elements per thread: it needs the thresholds and the number
// of entries, so it runs beside the FP4 GEMM and the CSR's fill (1920 x 5504 at alpha 0.97: both were ahead of it on the one
// path).  Where the entries are too few for the product it does nothing.
struct DenseActArgs {
  const uint4* x;              // rows row0 .. of the activation
  long long n_vec;             // of the slab
  int vec_per_row, row0;
  const float* thresholds;
  int thr_per_row;
  uint4* vt;                   // [term][rows][C]
  int* third;
  const int* entries;          // number of entries (device); fewer than dense_from: nothing to do
  int dense_from;
};
template <bool THIRD>
__global__ void __launch_bounds__(256)
dense_act_kernel(const __grid_constant__ DenseActArgs a) {
  if (*a.entries < a.dense_from || (THIRD && *a.third == 0)) return;
  constexpr int FLY = 4;
  const long long i0 = (long long)blockIdx.x * (256 * FLY) + threadIdx.x;
  uint4 v[FLY];
#pragma unroll
  for (int u = 0; u < FLY; ++u)
    if (i0 + 256 * u < a.n_vec) v[u] = __ldg(&a.x[i0 + 256 * u]);
  float lo = a.thresholds[0], hi = a.thresholds[1];
  bool any = false;
#pragma unroll
  for (int u = 0; u < FLY; ++u) {
    const long long i = i0 + 256 * u;
    if (i >= a.n_vec) break;
    if (a.thr_per_row) {
      const int row = a.row0 + int(i / a.vec_per_row);
      lo = a.thresholds[2 * row];
      hi = a.thresholds[2 * row + 1];
    }
    const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
    uint32_t o1[4], o2[4], o3[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float r[2], b1[2], b2[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float x = __uint_as_float(h ? w[q] & 0xFFFF0000u : w[q] << 16);
        r[h] = x > hi ? __fsub_rn(x, hi) : x < lo ? __fsub_rn(x, lo) : 0.0f;
      }
      const __nv_bfloat162 t1 = __floats2bfloat162_rn(r[0], r[1]);
      b1[0] = __low2float(t1); b1[1] = __high2float(t1);
      const float s0 = r[0] - b1[0], s1 = r[1] - b1[1];            // exact
      const __nv_bfloat162 t2 = __floats2bfloat162_rn(s0, s1);
      b2[0] = __low2float(t2); b2[1] = __high2float(t2);
      any |= s0 != b2[0] || s1 != b2[1];
      const __nv_bfloat162 t3 = __floats2bfloat162_rn(s0 - b2[0], s1 - b2[1]);          // exact
      o3[q] = *reinterpret_cast<const uint32_t*>(&t3);
      o1[q] = *reinterpret_cast<const uint32_t*>(&t1);
      o2[q] = *reinterpret_cast<const uint32_t*>(&t2);
    }
    if (THIRD) {
      a.vt[2 * a.n_vec + i] = make_uint4(o3[0], o3[1], o3[2], o3[3]);
    } else {
      a.vt[i] = make_uint4(o1[0], o1[1], o1[2], o1[3]);
      a.vt[a.n_vec + i] = make_uint4(o2[0], o2[1], o2[2], o2[3]);
    }
  }
  if (!THIRD && any) *a.third = 1;                             // (any number of threads writes the same)
}

// The same from the sparse form (the transpose, or an activation that was quantised by an earlier call): a block
// writes one row, in segments of ROW_SEG contraction indices.
// How many entries there are is known on the device only (ties at the thresholds leave fewer than alpha allows,
// an activation of three values none): below `dense_from` of them the product is left out, and
// dense_rows_kernel<true> adds the entries one by one instead, a warp per row and 256 outputs.  Its other task is the
// third term (write_third).
constexpr int ROW_SEG = 8192;
struct DenseRowsArgs {
  const int* ptr;              // the whole matrix: R rows
  const int* idx;
  const float* val;
  int R, C, row0, rows;        // the slab: rows row0 ..
  int dense_from;
  bool write_third;
  __nv_bfloat16* vt;
  int* third;
  const uint4* dense;          // [C x N]
  int N;
  ResidualOut out;
};
template <bool SECOND>
__global__ void __launch_bounds__(256, SECOND ? 5 : 6)
dense_rows_kernel(const __grid_constant__ DenseRowsArgs a) {
  __shared__ __align__(16) __nv_bfloat16 tile[SECOND ? 1 : 2][ROW_SEG];
  const int* __restrict__ ptr = a.ptr;
  const int* __restrict__ idx = a.idx;
  const float* __restrict__ val = a.val;
  const int t = threadIdx.x;
  if (__ldg(&ptr[a.R]) < a.dense_from) {
    if (!SECOND) return;
    // (outputs the slow index: the rows of the dense matrix that are in use at a time stay in L2)
    const int groups = a.rows >> 3, items = groups * ((a.N + 255) >> 8);
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
      const int nb = it / groups, row = a.row0 + (it - nb * groups) * 8 + (t >> 5), n0 = 256 * nb + 8 * (t & 31);
      const int vcol = n0 < a.N ? n0 >> 3 : 0, e1 = __ldg(&ptr[row + 1]);      // (every lane takes part in the walk)
      int e = __ldg(&ptr[row]);
      float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      add_groups_of_32(acc, idx, val, e, e1, a.dense, a.N >> 3, vcol);
      e += max(e1 - e, 0) & ~31;
      sparse_row_times_dense(acc, idx, val, e, e1, a.dense, a.N >> 3, vcol);
      if (n0 >= a.N) continue;
      const long long off = (long long)row * a.N + n0;
      if (a.out.y1) {
        const float4 p = *reinterpret_cast<const float4*>(a.out.y1 + off), q = *reinterpret_cast<const float4*>(a.out.y1 + off + 4);
        const float y1[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = y1[c] + acc[c];
      }
      store8(a.out.y, a.out.f32, off, acc);
    }
    return;
  }
  if (SECOND && (!a.write_third || *a.third == 0)) return;
  for (int r = blockIdx.x; r < a.rows; r += gridDim.x) {
    const int e0 = __ldg(&ptr[a.row0 + r]), e1 = __ldg(&ptr[a.row0 + r + 1]);
    uint4* t4 = reinterpret_cast<uint4*>(&tile[0][0]);
    bool any = false;
    for (int c0 = 0; c0 < a.C; c0 += ROW_SEG) {
      const int c1 = min(a.C, c0 + ROW_SEG);
      for (int i = t; i < (SECOND ? 1 : 2) * ROW_SEG / 8; i += 256) t4[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
      for (int e = e0 + t; e < e1; e += 256) {
        const int c = __ldg(&idx[e]);
        if (c < c0 || c >= c1) continue;
        const float v = __ldg(&val[e]);
        const __nv_bfloat16 b1 = __float2bfloat16_rn(v);
        const float r1 = v - __bfloat162float(b1);                 // exact
        const __nv_bfloat16 b2 = __float2bfloat16_rn(r1);
        const float r2 = r1 - __bfloat162float(b2);                // exact
        if (SECOND) {
          tile[0][c - c0] = __float2bfloat16_rn(r2);               // exact
        } else {
          tile[0][c - c0] = b1;
          tile[1 - SECOND][c - c0] = b2;
          any |= r2 != 0.0f;
        }
      }
      __syncthreads();
#pragma unroll
      for (int term = 0; term < 2 - SECOND; ++term)
        for (int i = t; i < (c1 - c0) / 8; i += 256)
          *reinterpret_cast<uint4*>(a.vt + (size_t(SECOND ? 2 : term) * a.rows + r) * size_t(a.C) + c0 + 8 * i) =
              *reinterpret_cast<const uint4*>(&tile[term][8 * i]);
      __syncthreads();
    }
    if (!SECOND && any) *a.third = 1;                // (any number of threads writes the same)
  }
}

struct DenseTcArgs {
  int M, N;                  // length of the contraction, output columns
  int tiles;                 // blocks of DT_NT output columns
  int splits;                // ranges of chunks per tile; FULL: blocks of 128 rows
  int vt_rows;               // rows of a term of Vt
  const int* counts;         // counts[0] = number of dense columns (device); FULL: whether the third term is needed
  float* partial;            // [splits][DENSE_TC_MAX][N]
  ResidualOut out;           // FULL: rows of the slab
  const int* entries;        // FULL: number of entries (device); fewer than dense_from: nothing to do
  int dense_from;
  int32_t* status;
};

// FULL: every row of the result, in blocks of 128; else the dense columns' rows, in ranges of the contraction.
// FULL drains tensor memory every 64 contraction indices: of the 8 or 12 truncating additions behind a drained sum four
// bring its leading term.  (Chunks of 128, terms interleaved: 7 % further from the exact sum than the gathers' fused
// multiply-adds at a contraction of 512 without hot columns, now 3 % nearer; and slower, 1920 x 5504 x 2048 at alpha
// 0.97 forward 167 us, 158 now: a stage is freed and a drain begins twice as often.)
template <bool FULL>
__global__ void __launch_bounds__(DT_THREADS, 1)
comp_wgrad_dense_tc_kernel(const __grid_constant__ CUtensorMap map_dy, const __grid_constant__ CUtensorMap map_vt,
                           const __grid_constant__ DenseTcArgs args) {
  extern __shared__ uint8_t smem_raw[];
  const int n_dense = FULL ? DENSE_TC_MAX : min(__ldg(args.counts), DENSE_TC_MAX);
  if (n_dense == 0 || (FULL && __ldg(args.entries) < args.dense_from)) return;      // uniform: nothing allocated yet
  const int terms = FULL && *args.counts == 0 ? 2 : 3;
  const int nb = (n_dense + 63) / 64;                     // 64-row boxes of V per term
  const int stages = nb == 1 || terms == 2 ? 3 : 2;
  const uint32_t v_bytes = uint32_t(terms * nb * DT_BOX);
  const uint32_t stage_bytes = uint32_t(DT_DY_BYTES) + v_bytes;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_misc = smem + DT_RING;
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem_misc);
  uint64_t* empty_bar = full_bar + 3;
  uint64_t* acc_full = empty_bar + 3;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* final_bar = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(final_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xFFFFFFFFu, int(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int tile = blockIdx.x % args.tiles, split = blockIdx.x / args.tiles;
  constexpr int HALVES = FULL ? 1 : 2, CHUNK = HALVES * DT_TOK;      // stages and contraction indices per chunk
  const int chunks_total = (args.M + CHUNK - 1) / CHUNK;
  const int c_begin = FULL ? 0 : int((long long)chunks_total * split / args.splits);
  const int c_end = FULL ? chunks_total : int((long long)chunks_total * (split + 1) / args.splits);
  const int s0 = FULL ? split * DENSE_TC_MAX : 0;         // first row of Vt
  const int n_chunks = c_end - c_begin;
  const int n0 = tile * DT_NT;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 3; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 8);
    }
    mbar_init(final_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_dy) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_vt) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer -------
    if (elect_one()) {                            // (see the FP4 GEMM)
      int stage = 0;
      uint32_t phase = 0, fills = 0;
      bool ok = true;
      for (int c = 0; c < HALVES * n_chunks && ok; ++c) {       // one stage = 64 tokens
        const int m0 = c_begin * CHUNK + c * DT_TOK;
        ok = mbar_wait(&empty_bar[stage], phase ^ 1u, abort_flag, args.status);
        if (!ok) break;
        uint8_t* dst = smem + stage * stage_bytes;
        mbar_arrive_expect_tx(&full_bar[stage], stage_bytes);
        for (int j = 0; j < DT_NT / 64; ++j)                    // dY: box j = columns n0 + 64 j .. + 63, 64 tokens
          tma_load_2d(dst + j * DT_BOX, &map_dy, &full_bar[stage], n0 + 64 * j, m0);
        for (int t = 0; t < terms; ++t)                         // V terms: 64 tokens x 64 rows per box
          for (int b = 0; b < nb; ++b)
            tma_load_2d(dst + DT_DY_BYTES + (t * nb + b) * DT_BOX, &map_vt, &full_bar[stage], m0,
                        t * args.vt_rows + s0 + 64 * b);
        ++fills;
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
      if (!ok) {
        // gave up: let the copies already in flight land before shared memory is released
        const uint32_t last = fills < uint32_t(stages) ? fills : uint32_t(stages);
        for (uint32_t back = 1; back <= last; ++back) {
          const uint32_t f = fills - back;
          const uint64_t t0 = global_timer_ns();
          while (!mbar_try_wait(&full_bar[f % stages], (f / stages) & 1u)) {
            if (global_timer_ns() - t0 > 1000000ull) break;
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer ---------
    if (elect_one()) {                            // (see the FP4 GEMM)
      int stage = 0;
      uint32_t phase = 0;
      int acc = 0;
      uint32_t acc_phase = 0;
      bool ok = true;
      const uint32_t idesc = FULL ? idesc_full() : idesc_dense(64 * nb);
      for (int c = 0; c < n_chunks && ok; ++c) {
        ok = mbar_wait(&acc_empty[acc], acc_phase ^ 1u, abort_flag, args.status);
        if (!ok) break;
        tc_fence_after();
        for (int half = 0; half < HALVES && ok; ++half) {       // the stages of this chunk
          ok = mbar_wait(&full_bar[stage], phase, abort_flag, args.status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t dy_addr = smem_u32(smem + stage * stage_bytes);
          const uint32_t v_addr = dy_addr + DT_DY_BYTES;
          if (FULL) {
            // The small terms first: what an addition loses grows with the running sum, which the last term brings.
            const uint32_t d_tmem = tmem_base + uint32_t(acc * 256);
            uint32_t accumulate = 0u;
#pragma unroll
            for (int t = 2; t >= 0; --t)
              if (t < terms) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {                   // 16 contraction indices per instruction
                  mma_f16(d_tmem, make_smem_desc(v_addr + uint32_t(t * 2 * DT_BOX + k * 32)),
                          make_smem_desc_mn(dy_addr + uint32_t(k * 2048), DT_BOX), idesc, accumulate);
                  accumulate = 1u;
                }
              }
          } else
#pragma unroll
          for (int h = 0; h < 2; ++h) {                         // output columns n0 + 128 h .. + 127
            const uint32_t d_tmem = tmem_base + uint32_t(acc * 256 + h * 128);
#pragma unroll
            for (int k = 0; k < 4; ++k) {                       // 16 tokens per instruction
              const uint64_t a_desc = make_smem_desc_mn(dy_addr + uint32_t(2 * h * DT_BOX + k * 2048), DT_BOX);
#pragma unroll
              for (int t = 0; t < 3; ++t) {
                const uint64_t b_desc = make_smem_desc(v_addr + uint32_t(t * nb * DT_BOX + k * 32));
                mma_f16(d_tmem, a_desc, b_desc, idesc, (half | k | t) != 0 ? 1u : 0u);
              }
            }
          }
          tc_commit(&empty_bar[stage]);
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        tc_commit(&acc_full[acc]);
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
      tc_commit(final_bar);
      const uint64_t t0 = global_timer_ns();
      while (!mbar_try_wait(final_bar, 0)) {
        if (global_timer_ns() - t0 > WAIT_LIMIT_NS) {
          atomicOr(args.status, FP4_DEV_TIMEOUT);
          break;
        }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue -----------
    // Warp (h, q) owns output columns n0 + 128 h + 32 q .. + 31 (one per lane) and all dense rows; FULL: rows
    // s0 + 32 q .. + 31 (one per lane) and output columns n0 + 128 h .. + 127.
    const int quarter = warp & 3;
    const int h = (warp - 2) >> 2;
    float run[DENSE_TC_MAX];
#pragma unroll
    for (int i = 0; i < DENSE_TC_MAX; ++i) run[i] = 0.0f;
    int acc = 0;
    uint32_t acc_phase = 0;
    bool gave_up = false;
    // The stage goes back as soon as its last columns are in registers, ahead of their additions.  (The warps stay together
    // from chunk to chunk: left to drift apart they take longer, 1920 x 5504 x 2048 at alpha 0.97 142 us, 146 then.)
    for (int c = 0; c < n_chunks; ++c) {
      const bool ok = mbar_wait(&acc_full[acc], acc_phase, abort_flag, args.status);
      if (epilogue_bar_any(!ok, 8 * 32)) { gave_up = true; break; }
      tc_fence_after();
      const uint32_t t_base = tmem_base + (uint32_t(quarter * 32) << 16) + uint32_t(acc * 256 + h * 128);
#pragma unroll
      for (int c0 = 0; c0 < DENSE_TC_MAX; c0 += 32) {
        if (c0 < 64 * nb) {
          uint32_t v[32];
          tmem_ld_32x32(t_base + uint32_t(c0), v);
          tmem_ld_wait(v);
          if (c0 + 32 == DENSE_TC_MAX || c0 + 32 == 64 * nb) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[acc]);
          }
#pragma unroll
          for (int i = 0; i < 32; ++i) run[c0 + i] += __uint_as_float(v[i]);
        }
      }
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    const int n = FULL ? n0 + 128 * h : n0 + 128 * h + 32 * quarter + lane;
    if (FULL) {
      // Every MMA has retired, so the ring is free: a warp's 32 x 128 sums go through it, a row at a time to the
      // output (a lane's own row piece by piece touched 32 lines with every store).
      if (!gave_up && n < args.N) {         // (N is a multiple of 128)
        constexpr int PITCH = 128 + 4;
        float* mine = reinterpret_cast<float*>(smem) + (warp - 2) * 32 * PITCH;
#pragma unroll
        for (int j = 0; j < DENSE_TC_MAX / 4; ++j)
          *reinterpret_cast<float4*>(mine + lane * PITCH + 4 * j) =
              make_float4(run[4 * j], run[4 * j + 1], run[4 * j + 2], run[4 * j + 3]);
        __syncwarp();
        const long long off = (long long)(s0 + 32 * quarter) * args.N + n + 4 * lane;
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += 8) {
          float4 y1[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            y1[u] = args.out.y1 ? __ldcs(reinterpret_cast<const float4*>(args.out.y1 + off + (long long)(r0 + u) * args.N))
                                : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const float4 v = *reinterpret_cast<const float4*>(mine + (r0 + u) * PITCH + 4 * lane);
            const float4 y = args.out.y1 ? make_float4(y1[u].x + v.x, y1[u].y + v.y, y1[u].z + v.z, y1[u].w + v.w) : v;
            const long long o = off + (long long)(r0 + u) * args.N;
            if (args.out.f32) {
              *reinterpret_cast<float4*>(static_cast<float*>(args.out.y) + o) = y;
            } else {
              const __nv_bfloat162 p = __floats2bfloat162_rn(y.x, y.y), q = __floats2bfloat162_rn(y.z, y.w);
              *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(args.out.y) + o) =
                  make_uint2(*reinterpret_cast<const uint32_t*>(&p), *reinterpret_cast<const uint32_t*>(&q));
            }
          }
        }
      }
    } else if (!gave_up && n < args.N) {
      float* dst = args.partial + size_t(split) * DENSE_TC_MAX * size_t(args.N) + n;
#pragma unroll
      for (int s = 0; s < DENSE_TC_MAX; ++s)
        if (s < n_dense) dst[size_t(s) * size_t(args.N)] = run[s];
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512) : "memory");
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// BF16 [rows x cols] row-major, boxes of 64 columns (128 bytes) x 64 rows, 128-byte swizzle.
int make_bf16_map(fp4_ctx* ctx, CUtensorMap* map, const void* base, int64_t rows, int64_t cols) {
  EncodeTiledFn encode = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled);
  if (!encode) return FP4_ERR_CUDA;
  if (reinterpret_cast<uintptr_t>(base) & 15) return FP4_ERR_ALIGN;
  const cuuint64_t dims[2] = {cuuint64_t(cols), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(cols) * 2};
  const cuuint32_t box[2] = {64, 64};
  const cuuint32_t elem_strides[2] = {1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                            elem_strides, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? FP4_OK : FP4_ERR_CUDA;
}

}  // namespace

// Ranges of chunks per block of output columns: the split (at most 16 ranges) whose CTAs, taken
// in rounds of one per SM, finish soonest -- rounds x chunks per CTA, plus about one chunk's time per
// round for filling the pipeline.
static int splits_for(int sms, int64_t M, int64_t N) {
  const int tiles = int((N + DT_NT - 1) / DT_NT);
  const int chunks = int((M + DT_CHUNK - 1) / DT_CHUNK);
  if (sms > 148) sms = 148;
  int best = 1;
  long long best_cost = -1;
  for (int s = 1; s <= 16 && s <= chunks; ++s) {
    const long long rounds = (tiles * s + sms - 1) / sms;
    const long long cost = rounds * ((chunks + s - 1) / s + 1);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = s; }
  }
  return best;
}

int dense_tc_splits(const fp4_ctx* ctx, int64_t M, int64_t N) { return splits_for(ctx->num_sms, M, N); }

size_t dense_tc_scratch_bytes(int64_t M, int64_t N) {
  auto r256 = [](size_t b) { return (b + 255) & ~size_t(255); };
  return r256(size_t(3) * DENSE_TC_MAX * size_t(M) * 2) + r256(size_t(splits_for(148, M, N)) * DENSE_TC_MAX * size_t(N) * 4);
}

// C[s, :] for the dense columns s < counts[0] into `partial` ([splits][DENSE_TC_MAX][N]); the caller
// adds the splits in order.  M must be a multiple of 128.
int launch_comp_wgrad_dense_tc(fp4_ctx* ctx, cudaStream_t stream, const fp4_qtensor* a, const int* list_dense,
                               const int* counts, const void* dy_bf16, void* vt, float* partial, int splits,
                               int64_t M, int64_t N, int32_t* status) {
  CUtensorMap map_dy, map_vt;
  int rc = make_bf16_map(ctx, &map_dy, dy_bf16, M, N);
  if (rc != FP4_OK) return rc;
  rc = make_bf16_map(ctx, &map_vt, vt, 3 * DENSE_TC_MAX, M);
  if (rc != FP4_OK) return rc;
  dense_split_kernel<<<dim3(unsigned((M + SPLIT_TOK - 1) / SPLIT_TOK), DENSE_TC_MAX), 256, 0, stream>>>(
      a->csc_colptr, a->csc_row, a->csc_val, list_dense, counts, static_cast<__nv_bfloat16*>(vt), int(M));
  DenseTcArgs args;
  args.M = int(M);
  args.N = int(N);
  args.tiles = int((N + DT_NT - 1) / DT_NT);
  args.splits = splits;
  args.vt_rows = DENSE_TC_MAX;
  args.counts = counts;
  args.partial = partial;
  args.out = ResidualOut{nullptr, nullptr, 1};
  args.status = status;
  args.entries = nullptr;
  args.dense_from = 0;
  FP4_CUDA_TRY(cudaFuncSetAttribute(comp_wgrad_dense_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, DT_SMEM));
  comp_wgrad_dense_tc_kernel<false><<<unsigned(args.tiles * splits), DT_THREADS, DT_SMEM, stream>>>(map_dy, map_vt, args);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

// Rows of the result that one slab of Vt holds (a multiple of 128).
static int64_t full_slab_rows(int64_t R, int64_t C) {
  const int64_t fit = FULL_SLAB_BYTES / (6 * C) / 128 * 128;
  return fit >= R ? R : fit;
}

size_t residual_full_scratch_bytes(int64_t R, int64_t C) {
  const int64_t rows = full_slab_rows(R, C);
  return rows < 128 ? 0 : ((size_t(6) * size_t(rows) * size_t(C) + 255) & ~size_t(255)) + 256;
}

// In ns: 15 TB/s of gathered rows (2 N bytes an entry) against 1.9 us per 128 contraction indices of a 128 x 256 tile,
// one tile per SM at a time, slab after slab (4096 x 11008 x 512: three slabs of 30 tiles, 480 us; the gathers 220),
// and the operand's 4 bytes per element.  The backward pays all of that.  In the forward the first slab's operand is made
// beside the GEMM, so that the rule asks for up to a tenth more entries there than the product would need (1920 x 5504 x
// 2048: 3.3 % of the activation, 3.0 % without the operand's time): one rule for both directions, on the safe side.
int64_t residual_full_from(const fp4_ctx* ctx, int64_t R, int64_t C, int64_t N) {
  const int64_t slab = full_slab_rows(R, C);
  if (slab < 128) return INT64_MAX;
  int64_t ns = 0;
  for (int64_t r0 = 0; r0 < R; r0 += slab) {
    const int64_t rows = R - r0 < slab ? R - r0 : slab;
    const int64_t tiles = rows / 128 * ((N + DT_NT - 1) / DT_NT), rounds = (tiles + ctx->num_sms - 1) / ctx->num_sms;
    ns += rounds * (C / 128 * 1900 + 4000) + 6000 + rows * C / 1200;
  }
  return (ns > 5000 ? ns - 5000 : 0) * 7500 / N + 1;
}

int residual_full_begin(const fp4_ctx* ctx, ResidualFull& f, Arena& scratch) {
  f.slab = full_slab_rows(f.R, f.C);
  f.vt = scratch.take<__nv_bfloat16>(size_t(3) * size_t(f.slab) * size_t(f.C));
  f.third = scratch.take<int>(1);
  f.dense_from = int(residual_full_from(ctx, f.R, f.C, f.N));     // (the caller has compared it with a bound below 2^31)
  return scratch.ok ? FP4_OK : FP4_ERR_WORKSPACE;
}

// The slab's rows of the result, or of what is to be stored.
static ResidualOut slab_out(const ResidualFull& f, int64_t r0) {
  const size_t at = size_t(r0) * size_t(f.N);
  return {f.out.y1 ? f.out.y1 + at : nullptr, static_cast<char*>(f.out.y) + at * (f.out.f32 ? 4 : 2), f.out.f32};
}
static DenseRowsArgs dense_rows_args(const ResidualFull& f, int64_t r0, int64_t rows) {
  DenseRowsArgs ra;
  ra.ptr = f.ptr;
  ra.idx = f.idx;
  ra.val = f.val;
  ra.R = int(f.R);
  ra.C = int(f.C);
  ra.row0 = int(r0);
  ra.rows = int(rows);
  ra.dense_from = f.dense_from;
  ra.write_third = !f.act_bf16;
  ra.vt = static_cast<__nv_bfloat16*>(f.vt);
  ra.third = f.third;
  ra.dense = static_cast<const uint4*>(f.dense_bf16);
  ra.N = int(f.N);
  ra.out = f.out;
  return ra;
}

// Idle as a rule: at most four waves of blocks, which calls whose product runs do not show (1920 x 5504 x 2048 at alpha 0.97
// 149.5 us with one wave, 146 with four, runs 18 apart).  With one wave the gathers' last round was half empty: 3 % of entries
// there 110 us, 92 with a block per item.
static void launch_dense_rows_second(const fp4_ctx* ctx, cudaStream_t stream, const DenseRowsArgs& a) {
  const int64_t items = int64_t(a.rows / 8) * ((a.N + 255) / 256), some = 4 * 5 * ctx->num_sms;
  const int64_t blocks = items > a.rows ? items : a.rows;
  dense_rows_kernel<true><<<unsigned(blocks < some ? blocks : some), 256, 0, stream>>>(a);
}

int launch_residual_operand(fp4_ctx* ctx, cudaStream_t stream, const ResidualFull& f, int64_t r0) {
  const int64_t rows = f.R - r0 < f.slab ? f.R - r0 : f.slab;
  if (r0 == 0) FP4_CUDA_TRY(cudaMemsetAsync(f.third, 0, 4, stream));
  KernelScope scope(ctx, stream, f.kernel_class, f.act_bf16 ? 2 : 1);
  if (f.act_bf16) {
    DenseActArgs a;
    a.x = static_cast<const uint4*>(f.act_bf16) + r0 * f.C / 8;
    a.n_vec = rows * f.C / 8;
    a.vec_per_row = int(f.C / 8);
    a.row0 = int(r0);
    a.thresholds = f.thresholds;
    a.thr_per_row = f.thr_per_row;
    a.vt = static_cast<uint4*>(f.vt);
    a.third = f.third;
    a.entries = f.ptr + f.R;
    a.dense_from = f.dense_from;
    const unsigned blocks = unsigned((a.n_vec + 1023) / 1024);
    dense_act_kernel<false><<<blocks, 256, 0, stream>>>(a);
    dense_act_kernel<true><<<blocks, 256, 0, stream>>>(a);
  } else {
    dense_rows_kernel<false><<<unsigned(rows), 256, 0, stream>>>(dense_rows_args(f, r0, rows));
  }
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

int launch_residual_product(fp4_ctx* ctx, cudaStream_t stream, const ResidualFull& f, int64_t r0) {
  const int64_t rows = f.R - r0 < f.slab ? f.R - r0 : f.slab;
  CUtensorMap map_dense, map_vt;
  int rc = make_bf16_map(ctx, &map_dense, f.dense_bf16, f.C, f.N);
  if (rc != FP4_OK) return rc;
  rc = make_bf16_map(ctx, &map_vt, f.vt, 3 * rows, f.C);
  if (rc != FP4_OK) return rc;
  KernelScope scope(ctx, stream, f.kernel_class, 1);
  DenseTcArgs args;
  args.M = int(f.C);
  args.N = int(f.N);
  args.tiles = int((f.N + DT_NT - 1) / DT_NT);
  args.splits = int(rows / DENSE_TC_MAX);
  args.vt_rows = int(rows);
  args.counts = f.third;
  args.partial = nullptr;
  args.out = slab_out(f, r0);
  args.status = f.status;
  args.entries = f.ptr + f.R;
  args.dense_from = f.dense_from;
  FP4_CUDA_TRY(cudaFuncSetAttribute(comp_wgrad_dense_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, DT_SMEM));
  comp_wgrad_dense_tc_kernel<true><<<unsigned(args.tiles * args.splits), DT_THREADS, DT_SMEM, stream>>>(map_dense, map_vt, args);
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}

int launch_residual_full(fp4_ctx* ctx, cudaStream_t stream, const ResidualFull& f, bool first_operand_ready, cudaEvent_t entries_ready) {
  for (int64_t r0 = 0; r0 < f.R; r0 += f.slab) {
    int rc = r0 == 0 && first_operand_ready ? FP4_OK : launch_residual_operand(ctx, stream, f, r0);
    if (rc != FP4_OK) return rc;
    if (!f.act_bf16) {
      // The third term, or where the entries are too few for the product their sums: these read Y1 and store Y, so
      // this launch stands behind whatever makes Y1, not with the first slab's operand.
      KernelScope scope(ctx, stream, f.kernel_class, 1);
      launch_dense_rows_second(ctx, stream, dense_rows_args(f, r0, f.R - r0 < f.slab ? f.R - r0 : f.slab));
    }
    rc = launch_residual_product(ctx, stream, f, r0);
    if (rc != FP4_OK) return rc;
  }
  if (!f.act_bf16) return FP4_OK;
  // The operand was made without the entries: where they are too few for the product they are added now.
  if (entries_ready) FP4_CUDA_TRY(cudaStreamWaitEvent(stream, entries_ready, 0));
  KernelScope scope(ctx, stream, f.kernel_class, 1);
  launch_dense_rows_second(ctx, stream, dense_rows_args(f, 0, f.R));
  FP4_CUDA_TRY(cudaGetLastError());
  return FP4_OK;
}
