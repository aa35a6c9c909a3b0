// Statistics of the columns of a matrix in one pass over it, shared by k_ozaki.cu and k_batched.cu: a block of
// 32 x 8 threads holds 256 rows of 32 columns in registers and leaves every column's largest magnitude there and the sum
// of squares scaled by its exponent; a second kernel folds the blocks of a column.  (A pass for the maxima with
// atomics and another for the sums read the matrix twice.)
#pragma once
#include "common.cuh"

namespace zf {

constexpr int kColRows = 256;  // rows of a block
inline int col_blocks(int n) { return (n + kColRows - 1) / kColRows; }

// NaN or Inf, or a largest entry that is subnormal (its scaled values would read as zero)
__device__ __forceinline__ bool col_no_bound(unsigned long long m) {
  return m >= 0x7FF0000000000000ull || (m != 0ull && m < (1ull << 52));
}

// Column j = 32 blockIdx.x + threadIdx.x over the rows from r0: maximum (abs_bits) to *pm, scaled sum to *ps.
__device__ __forceinline__ void col_block(const double* __restrict__ X, int n, int ld, int r0, unsigned long long* pm,
                                          float* ps) {
  __shared__ unsigned long long redm[8][33];
  __shared__ float reds[8][33];
  const int tx = threadIdx.x, ty = threadIdx.y, j = blockIdx.x * 32 + tx;
  unsigned long long v[kColRows / 8], m = 0ull;
#pragma unroll
  for (int k = 0; k < kColRows / 8; ++k) {
    const int r = r0 + ty + 8 * k;
    v[k] = j < n && r < n ? abs_bits(X[(size_t)r * ld + j]) : 0ull;
  }
#pragma unroll
  for (int k = 0; k < kColRows / 8; ++k) m = max_bits(m, v[k]);
  redm[ty][tx] = m;
  __syncthreads();
#pragma unroll
  for (int y = 0; y < 8; ++y) m = max_bits(m, redm[y][tx]);
  float acc = 0.0f;
  if (m != 0ull && !col_no_bound(m)) {
    const int e = exp_of_bits(m);
#pragma unroll
    for (int k = 0; k < kColRows / 8; ++k) {
      const float f = scaled_mag_f32(v[k], e);
      acc = fmaf(f, f, acc);
    }
  }
  reds[ty][tx] = acc;
  __syncthreads();
  if (ty == 0 && j < n) {
#pragma unroll
    for (int y = 1; y < 8; ++y) acc += reds[y][tx];
    *pm = m;
    *ps = acc;
  }
}

// The column's maximum (returned) and its rho^2 (FP32 bits; +Inf without a bound) from nb blocks `stride` apart.
__device__ __forceinline__ unsigned long long col_fold(const unsigned long long* pm, const float* ps, size_t stride,
                                                       int nb, unsigned int* rho2) {
  unsigned long long m = 0ull;
#pragma unroll 8
  for (int b = 0; b < nb; ++b) m = max_bits(m, pm[b * stride]);
  *rho2 = 0u;
  if (col_no_bound(m)) {
    *rho2 = 0x7F800000u;
  } else if (m) {
    const int e = exp_of_bits(m);
    float s = 0.0f;
#pragma unroll 8
    for (int b = 0; b < nb; ++b) {
      const unsigned long long mb = pm[b * stride];
      const int d = mb ? 2 * (exp_of_bits(mb) - e) : -200;
      if (d > -126) s = fmaf(ps[b * stride], __uint_as_float((unsigned)(127 + d) << 23), s);
    }
    *rho2 = __float_as_uint(s);
  }
  return m;
}

}  // namespace zf
