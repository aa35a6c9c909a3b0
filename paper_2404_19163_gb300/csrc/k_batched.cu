// Element-wise kernels of the batched (grouped) mode: every instance's matrices are
// stacked along the rows of packed buffers (instance i at row offset row0[i], common
// leading dimension), so that one tensor map and one persistent launch cover all of them.
#include <math.h>

#include "batched.h"
#include "colstats.cuh"

namespace zf {
namespace {

__device__ __forceinline__ uint16_t r16b(float x, bool bf16) {
  return bf16 ? __bfloat16_as_ushort(__float2bfloat16_rn(x)) : __half_as_ushort(__float2half_rn(x));
}
__device__ __forceinline__ float f16b(uint16_t h, bool bf16) {
  return bf16 ? __bfloat162float(__ushort_as_bfloat16(h)) : __half2float(__ushort_as_half(h));
}

// Gershgorin bound per instance: gmax[i] = max_r sum_c |S_i[r][c]|.  One warp per row,
// grid.y = instance.
__global__ void k_b_rowabs(const BatchTables t, unsigned long long* gmax_bits) {
  const int i = blockIdx.y;
  const int n = t.n[i];
  const int row = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= n || t.Z0[i] != nullptr) return;
  const double* S = t.S[i] + (size_t)row * n;
  double s = 0.0;
  for (int c = lane; c < n; c += 32) s += fabs(S[c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) atomicMax(&gmax_bits[i], (unsigned long long)__double_as_longlong(s));
}

// Row statistics of every S_i for its FP64-accurate residual: g_i = max_r sum_c |S_i[r][c]|, and, for the moduli of
// its residue products (as launch_ozm_rho), rho2[i] = max_r sum_c (S_i[r][c] 2^-e_r)^2, e_r the row's exponent bound,
// FP32 bits, atomic maximum; +Inf for a row holding a NaN or Inf or whose largest entry is subnormal.  One warp
// per row, which reads it once for its sum and maximum and again (from L1) for the scaled sum, grid.y = instance.
__global__ void __launch_bounds__(256) k_b_rowstats(const BatchTables t, unsigned long long* gmax_bits,
                                                    unsigned int* rho2) {
  __shared__ double redg[8];
  __shared__ unsigned redr[8];
  const int i = blockIdx.y;
  const int n = t.n[i];
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (blockIdx.x * 8 >= n) return;  // the whole block (uniform)
  double g = 0.0;
  unsigned r = 0u;
  if (row < n) {
    const double* S = t.S[i] + (size_t)row * n;
    unsigned long long m = 0ull;
#pragma unroll 4
    for (int c = lane; c < n; c += 32) {
      const double x = S[c];
      g += fabs(x);
      m = max_bits(m, abs_bits(x));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      g += __shfl_xor_sync(0xffffffffu, g, o);
      m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
    if (m != 0ull) {
      if (col_no_bound(m)) {
        r = 0x7F800000u;
      } else {
        const int e = exp_of_bits(m);
        float acc = 0.0f;
#pragma unroll 4
        for (int c = lane; c < n; c += 32) {
          const float f = scaled_mag_f32(abs_bits(S[c]), e);
          acc = fmaf(f, f, acc);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        r = __float_as_uint(acc);
      }
    }
  }
  if (lane == 0) {
    redg[threadIdx.x >> 5] = g;
    redr[threadIdx.x >> 5] = r;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned long long gb = 0ull;  // (bits: a NaN above every number)
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    gb = max_bits(gb, (unsigned long long)__double_as_longlong(redg[w]));
    r = max(r, redr[w]);
  }
  atomicMax(&gmax_bits[i], gb);
  atomicMax(&rho2[i], r);
}

// Column statistics of every Z_i (the rows of the residual's first operand Z_i^T), grid.z = instance: colstats.cuh's
// blocks (block b of a column at b * rows + its packed position), then the exponents (packed like the rows), the
// largest rho^2 per instance and z_i = max |Z_i|.
__global__ void __launch_bounds__(256) k_b_colblocks(const BatchTables t, int rows, unsigned long long* pm, float* ps) {
  const int i = blockIdx.z, n = t.n[i];
  if (blockIdx.x * 32 >= n || blockIdx.y * kColRows >= n) return;
  const size_t o = (size_t)blockIdx.y * rows + t.row0[i] + blockIdx.x * 32 + threadIdx.x;
  col_block(t.Z[i], n, n, blockIdx.y * kColRows, pm + o, ps + o);
}

__global__ void k_b_colfin(const BatchTables t, int rows, const unsigned long long* pm, const float* ps, int* e,
                           unsigned int* rho2, unsigned long long* zmax_bits) {
  const int i = blockIdx.y, n = t.n[i], j = blockIdx.x * 64 + threadIdx.x;
  unsigned u = 0u;
  unsigned long long m = 0ull;
  if (j < n) {
    const size_t o = (size_t)t.row0[i] + j;
    m = col_fold(pm + o, ps + o, rows, (n + kColRows - 1) / kColRows, &u);
    e[o] = m ? exp_of_bits(m) : -2000000000;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    u = max(u, __shfl_xor_sync(0xffffffffu, u, o));
    m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
  }
  if ((threadIdx.x & 31) != 0) return;
  if (u) atomicMax(&rho2[i], u);
  if (m) atomicMax(&zmax_bits[i], m);
}

__device__ __forceinline__ void split_pair_b(float a, float b, bool bf16, uint32_t& h, uint32_t& l) {
  const uint16_t ha = r16b(a, bf16), hb = r16b(b, bf16);
  h = ha | ((uint32_t)hb << 16);
  l = r16b(a - f16b(ha, bf16), bf16) | ((uint32_t)r16b(b - f16b(hb, bf16), bf16) << 16);
}

// Pack instance i (grid.z) into the stacked buffers, 64 x 64 tiles, columns in pairs (the one past an odd size
// as zero: the K padding):
//   mode 0: S16 (hi[, lo]) from S_i
//   mode 1: Z master (FP32) + Z16 and Zt16 (hi[, lo]) from Z0_i, or from s_i I when Z0_i is null
// Bound: HBM.  32 clusters up to N = 2048: 165 us a matrix set (231 in 32 x 32 tiles with FP64 conversions).
__global__ void __launch_bounds__(256)
    k_b_pack(const BatchTables t, int mode, const unsigned long long* gmax_bits, int ld, int bf16, uint16_t* h16,
             uint16_t* l16, uint16_t* th16, uint16_t* tl16, float* m32) {
  __shared__ float tile[64][65];
  const int inst = blockIdx.z;
  const int n = t.n[inst];
  const int bi = blockIdx.y * 64, bj = blockIdx.x * 64, tx = threadIdx.x, ty = threadIdx.y;
  if (bi >= n || bj >= n) return;
  const size_t r0 = (size_t)t.row0[inst];
  const double* src = (mode == 0) ? t.S[inst] : t.Z0[inst];
  __shared__ float gs_shared;  // (an FP64 root and division in every thread would take longer than the pass)
  float gs = 0.0f;
  if (mode == 1 && !src) {
    if (tx == 0 && ty == 0) gs_shared = (float)(1.0 / sqrt(__longlong_as_double((long long)gmax_bits[inst])));
    __syncthreads();
    gs = gs_shared;
  }
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int r = ty + 8 * p, i = bi + r, j = bj + 2 * tx;
    float a = 0.0f, b = 0.0f;
    if (i < n && j < n) {
      const double* s = src + (size_t)i * n + j;
      a = src ? f32_of_f64(s[0], 0) : (i == j ? gs : 0.0f);
      if (j + 1 < n) b = src ? f32_of_f64(s[1], 0) : (i == j + 1 ? gs : 0.0f);
      uint32_t h, l;
      split_pair_b(a, b, bf16, h, l);
      const size_t o = (r0 + i) * ld + j;
      *reinterpret_cast<uint32_t*>(h16 + o) = h;
      if (l16) *reinterpret_cast<uint32_t*>(l16 + o) = l;
      if (mode == 1) *reinterpret_cast<float2*>(m32 + o) = make_float2(a, b);
    }
    if (mode == 1) {
      tile[r][2 * tx] = a;
      tile[r][2 * tx + 1] = b;
    }
  }
  if (mode == 0) return;
  __syncthreads();
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int r = ty + 8 * p, oi = bj + r, oj = bi + 2 * tx;  // transposed position
    if (oi < n && oj < n) {
      uint32_t h, l;
      split_pair_b(tile[2 * tx][r], tile[2 * tx + 1][r], bf16, h, l);
      const size_t o = (r0 + oi) * ld + oj;
      *reinterpret_cast<uint32_t*>(th16 + o) = h;
      if (tl16) *reinterpret_cast<uint32_t*>(tl16 + o) = l;
    }
  }
}

// Unpack the FP32 master of instance i (grid.z) into the caller's FP64 Z_i, 64 x 64 tiles.
__global__ void __launch_bounds__(256) k_b_unpack(const BatchTables t, const float* m32, int ld) {
  const int inst = blockIdx.z, n = t.n[inst];
  const int bi = blockIdx.y * 64, bj = blockIdx.x * 64;
  if (bi >= n || bj >= n) return;
  const float* src = m32 + (size_t)t.row0[inst] * ld;
  double* Z = t.Z[inst];
  float x[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    const int r = bi + (p >> 1) * 8 + threadIdx.y, c = bj + (p & 1) * 32 + threadIdx.x;
    x[p] = r < n && c < n ? src[(size_t)r * ld + c] : 0.0f;
  }
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    const int r = bi + (p >> 1) * 8 + threadIdx.y, c = bj + (p & 1) * 32 + threadIdx.x;
    if (r < n && c < n) Z[(size_t)r * n + c] = widen_pow2(x[p], 0);
  }
}

// Per-instance Err, history and stop test (Algorithm 2 with the guards of the single-instance
// path; Algorithm 1 with rule 1).  One block per instance; instances already done are left alone.
__global__ void k_b_finish(const double* __restrict__ partials, const BatchTables t, BatchState bs, int initial,
                           int rule, double tol, int check_stop, int limit) {
  __shared__ double red[256];
  const int i = blockIdx.x;
  if (!initial && bs.done[i]) return;
  const int p0 = t.part0[i], np = t.nparts[i];
  double s = 0.0;
  for (int p = threadIdx.x; p < np; p += blockDim.x) s += partials[p0 + p];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x != 0) return;
  const double err = sqrt(red[0]);
  const int it = initial ? 0 : bs.iters[i] + 1;
  if (!initial) bs.iters[i] = it;
  if (it < bs.cap) bs.hist[(size_t)i * bs.cap + it] = err;
  bs.hist_len[i] = it + 1;
  const double prev = bs.prev_err[i];
  bs.prev_err[i] = err;
  const double rn = sqrt((double)t.n[i]);
  int stop = 0;
  if (!isfinite(err)) {
    bs.nonfinite[i] = 1;
    stop = 1;
  } else if (initial) {
    stop = (check_stop && rule == 1 && err / rn <= tol) ? 1 : 0;
  } else {
    if (check_stop) {
      if (rule == 1)
        stop = err / rn <= tol;
      else
        stop = (err > prev * prev * prev) || (err >= prev);
    }
    if (it >= limit) stop = 1;
  }
  if (stop) {
    bs.done[i] = 1;
    atomicSub(bs.live, 1);
  }
}

}  // namespace

cudaError_t launch_b_gersh(const BatchTables& t, int count, int max_n, unsigned long long* gmax_bits,
                           cudaStream_t s) {
  cudaMemsetAsync(gmax_bits, 0, sizeof(unsigned long long) * count, s);
  dim3 grid((max_n + 7) / 8, count);
  k_b_rowabs<<<grid, 256, 0, s>>>(t, gmax_bits);
  return cudaGetLastError();
}

cudaError_t launch_b_stats(const BatchTables& t, int count, int max_n, int rows, unsigned long long* gmax_bits,
                           unsigned long long* zmax_bits, unsigned int* rho2, int* e_z, void* scratch, cudaStream_t s) {
  unsigned long long* pm = static_cast<unsigned long long*>(scratch);
  const int nb = col_blocks(max_n);
  float* ps = reinterpret_cast<float*>(pm + (size_t)nb * rows);
  cudaError_t e = cudaMemsetAsync(rho2, 0, sizeof(unsigned int) * 2 * (size_t)count, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(gmax_bits, 0, sizeof(unsigned long long) * count, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(zmax_bits, 0, sizeof(unsigned long long) * count, s);
  if (e != cudaSuccess) return e;
  k_b_rowstats<<<dim3((max_n + 7) / 8, count), 256, 0, s>>>(t, gmax_bits, rho2);
  k_b_colblocks<<<dim3((max_n + 31) / 32, nb, count), dim3(32, 8), 0, s>>>(t, rows, pm, ps);
  k_b_colfin<<<dim3((max_n + 63) / 64, count), 64, 0, s>>>(t, rows, pm, ps, e_z, rho2 + count, zmax_bits);
  return cudaGetLastError();
}

cudaError_t launch_b_pack(const BatchTables& t, int count, int max_n, int mode, const unsigned long long* gmax_bits,
                          int ld, bool bf16, uint16_t* h16, uint16_t* l16, uint16_t* th16, uint16_t* tl16, float* m32,
                          cudaStream_t s) {
  dim3 grid((max_n + 63) / 64, (max_n + 63) / 64, count), block(32, 8);
  k_b_pack<<<grid, block, 0, s>>>(t, mode, gmax_bits, ld, bf16 ? 1 : 0, h16, l16, th16, tl16, m32);
  return cudaGetLastError();
}

cudaError_t launch_b_unpack(const BatchTables& t, int count, int max_n, const float* m32, int ld, cudaStream_t s) {
  const dim3 grid((max_n + 63) / 64, (max_n + 63) / 64, count), block(32, 8);
  k_b_unpack<<<grid, block, 0, s>>>(t, m32, ld);
  return cudaGetLastError();
}

cudaError_t launch_b_finish(const double* partials, const BatchTables& t, const BatchState& bs, int count,
                            int initial, int rule, double tol, int check_stop, int limit, cudaStream_t s) {
  k_b_finish<<<count, 256, 0, s>>>(partials, t, bs, initial, rule, tol, check_stop, limit);
  return cudaGetLastError();
}

}  // namespace zf
