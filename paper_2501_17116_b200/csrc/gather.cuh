// Gathers shared by the compensation kernels: sparse entries times rows of a dense BF16 matrix, fp32 sums of eight
// consecutive columns per lane, entries in order.  Internal.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace {

__device__ __forceinline__ void fma8(float (&acc)[8], float v, const uint4& d) {
  const uint32_t w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    acc[2 * q] = fmaf(v, __uint_as_float(w[q] << 16), acc[2 * q]);
    acc[2 * q + 1] = fmaf(v, __uint_as_float(w[q] & 0xFFFF0000u), acc[2 * q + 1]);
  }
}

// eight consecutive outputs, in fp32 or rounded to BF16 once; streaming
__device__ __forceinline__ void store8(void* out, int out_f32, long long off, const float (&y)[8]) {
  if (out_f32) {
    float4* dst = reinterpret_cast<float4*>(static_cast<float*>(out) + off);
    __stcs(dst, make_float4(y[0], y[1], y[2], y[3]));
    __stcs(dst + 1, make_float4(y[4], y[5], y[6], y[7]));
  } else {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      __nv_bfloat162 h = __floats2bfloat162_rn(y[2 * q], y[2 * q + 1]);
      w[q] = *reinterpret_cast<uint32_t*>(&h);
    }
    __stcs(reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(out) + off), make_uint4(w[0], w[1], w[2], w[3]));
  }
}

// acc += n entries, gathered together
template <int n>
__device__ __forceinline__ void add_entries(float (&acc)[8], const int* __restrict__ idx, const float* __restrict__ val,
                                            const uint4* __restrict__ dense, int vec_per_row, int vcol) {
  int r[n];
  float v[n];
  uint4 d[n];
#pragma unroll
  for (int u = 0; u < n; ++u) {
    r[u] = __ldg(&idx[u]);
    v[u] = __ldg(&val[u]);
  }
#pragma unroll
  for (int u = 0; u < n; ++u) d[u] = __ldg(&dense[(long long)r[u] * vec_per_row + vcol]);
#pragma unroll
  for (int u = 0; u < n; ++u) fma8(acc, v[u], d[u]);
}
// The entries of a row in whole groups of 32 (those behind them are the caller's), by all lanes of the warp together.
// A row that holds many (a token that lies beyond the thresholds as a whole) is one chain that nothing hides: the
// lanes fetch 32 entries at once and hand them round, which leaves one round trip to L2 per four entries, not two.
__device__ __forceinline__ void add_groups_of_32(float (&acc)[8], const int* __restrict__ idx, const float* __restrict__ val,
                                                 int e, int e1, const uint4* __restrict__ dense, int vec_per_row, int vcol) {
#pragma unroll 1
  for (; e + 32 <= e1; e += 32) {
    const int r = __ldg(&idx[e + (threadIdx.x & 31)]);
    const float v = __ldg(&val[e + (threadIdx.x & 31)]);
#pragma unroll 1
    for (int u0 = 0; u0 < 32; u0 += 4) {
      uint4 d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        d[u] = __ldg(&dense[(long long)__shfl_sync(0xFFFFFFFFu, r, u0 + u) * vec_per_row + vcol]);
#pragma unroll
      for (int u = 0; u < 4; ++u) fma8(acc, __shfl_sync(0xFFFFFFFFu, v, u0 + u), d[u]);
    }
  }
}

// acc[0..7] += sum over the entries [e0, e1) of val[e] * dense[idx[e], col .. col+7]
__device__ __forceinline__ void sparse_row_times_dense(float (&acc)[8], const int* __restrict__ idx,
                                                       const float* __restrict__ val, int e0, int e1,
                                                       const uint4* __restrict__ dense, int vec_per_row, int vcol) {
  int e = e0;
  for (; e + 4 <= e1; e += 4) add_entries<4>(acc, idx + e, val + e, dense, vec_per_row, vcol);   // four loads in flight
  if (e + 2 <= e1) {
    add_entries<2>(acc, idx + e, val + e, dense, vec_per_row, vcol);
    e += 2;
  }
  if (e < e1) add_entries<1>(acc, idx + e, val + e, dense, vec_per_row, vcol);
}

}  // namespace
