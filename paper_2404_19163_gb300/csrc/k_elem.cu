// Element-wise steps and reductions of the recursion: the Gershgorin start
// Z0 = I / sqrt(max_i sum_j |S_ij|) (Sec. 3: ||X0 - I||_2 < 1), the
// deterministic Frobenius-norm finish Err = ||I - X||_F, and the stop test of
// Algorithm 2 (Sec. 4.1, Eq. stopL2) evaluated on the device in FP64.
#include <math.h>

#include "kernels.h"

namespace zf {
namespace {

__global__ void k_rowabs_max(const double* __restrict__ S, int n, IterState* st) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= n) return;
  const double* row = S + (size_t)warp * n;
  double s = 0.0;
#pragma unroll 4
  for (int j = lane; j < n; j += 32) s += fabs(row[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  // non-negative doubles order like their bit patterns, and a NaN (or Inf) row sum orders above
  // every finite one, so a non-finite entry of S leaves a non-finite maximum
  if (lane == 0) atomicMax(reinterpret_cast<unsigned long long*>(&st->amax[0]), (unsigned long long)__double_as_longlong(s));
}

__global__ void k_gscale(IterState* st) { st->gscale = 1.0 / sqrt(st->amax[0]); }
__global__ void k_set_gscale(IterState* st, double s) { st->gscale = s; }

// Rows i = blockIdx.y, blockIdx.y + gridDim.y, ...; columns across blockIdx.x and the threads (no
// division per element).
__global__ void k_scaled_identity_f64(double* Z, int n, const IterState* st) {
  const double s = st->gscale;
  for (int i = blockIdx.y; i < n; i += gridDim.y) {
    double* zr = Z + (size_t)i * n;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) zr[j] = (i == j) ? s : 0.0;
  }
}

__device__ float pow2_for(double bound) {
  // largest power of two s with bound * s <= 2^14 (FP16 max is 65504 ~ 2^16: two bits of headroom)
  if (!(bound > 0.0) || !isfinite(bound)) return 1.0f;
  int e;
  frexp(bound, &e);  // bound in [2^(e-1), 2^e)
  int p = 14 - e;
  if (p > 60) p = 60;
  if (p < -60) p = -60;
  return ldexpf(1.0f, p);
}

__device__ float pow2_head(double bound, int headroom_log2) {
  if (!(bound > 0.0) || !isfinite(bound)) return 1.0f;
  int e;
  frexp(bound, &e);
  int p = 14 - headroom_log2 - e;
  if (p > 60) p = 60;
  if (p < -60) p = -60;
  return ldexpf(1.0f, p);
}

// One block sums the partials in a fixed order: 1024 threads with four loads in flight each, then shuffles (256
// threads one load after another took 28 us for the 16384 partials of N = 8192).  With f.on the FP16 scales of
// d and Q follow here.
__global__ void __launch_bounds__(1024)
    k_finish_err(const double* __restrict__ partials, int np, IterState* st, int idx, int rule, double tol, int n,
                 int check_stop, Fp16Scales f) {
  __shared__ double red[32];
  double s = 0.0;
#pragma unroll 4
  for (int p = threadIdx.x; p < np; p += 1024) s += partials[p];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  s = red[threadIdx.x];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) {
    const double err = sqrt(s);
    if (idx < 0) idx = st->loop_iter + 1;  // device-driven loop: the update this residual follows
    if (idx < kHistMax) st->hist[idx] = err;
    st->hist_len = idx + 1;
    if (!isfinite(err)) {
      st->nonfinite = 1;
      st->stop = 1;
    } else if (check_stop) {
      const double prev = st->prev_err;
      if (rule == 1) {
        if (err / sqrt((double)n) <= tol) st->stop = 1;
      } else if (err > prev * prev * prev || err >= prev) {
        st->stop = 1;
      }
    }
    st->prev_err = err;
    if (f.on) {
      const double ad = (double)__uint_as_float(st->amaxf[1]), e = idx < kHistMax ? err : ad;
      st->scale[0] = pow2_head(ad, f.head);
      st->scale[1] = pow2_head((double)f.c1 * ad + (double)f.c2 * e * e, f.head);
    }
  }
}

__device__ __forceinline__ uint16_t r16(float x, bool bf16) {
  return bf16 ? __bfloat16_as_ushort(__float2bfloat16_rn(x)) : __half_as_ushort(__float2half_rn(x));
}
__device__ __forceinline__ float f16v(uint16_t h, bool bf16) {
  return bf16 ? __bfloat162float(__ushort_as_bfloat16(h)) : __half2float(__ushort_as_half(h));
}

// The exponent of a positive power of two, else -2000.
__device__ __forceinline__ int pow2_exp(double s) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(s);
  const int e = (int)(b >> 52);
  return (b & 0xFFFFFFFFFFFFFull) == 0ull && e > 773 && e < 1273 ? e - 1023 : -2000;
}
// FP32[x sc], k = pow2_exp(sc)
__device__ __forceinline__ float scaled_f32(double x, double sc, int k) {
  return k > -2000 ? f32_of_f64(x, k) : (float)(x * sc);
}
__device__ __forceinline__ float scaled_f32(float x, double sc, int k) {
  return k > -2000 ? x * (float)sc : (float)((double)x * sc);
}
// hi = R16(x) and lo = R16(x - hi) of two values, packed (the first in the lower half)
__device__ __forceinline__ void split_pair(float a, float b, bool bf16, uint32_t& h, uint32_t& l) {
  const uint16_t ha = r16(a, bf16), hb = r16(b, bf16);
  h = ha | ((uint32_t)hb << 16);
  l = r16(a - f16v(ha, bf16), bf16) | ((uint32_t)r16(b - f16v(hb, bf16), bf16) << 16);
}

// 16-bit copies of a matrix's rows, eight columns a thread (columns n up to a multiple of eight as zeros: inside
// the leading dimension, a multiple of 64).  Bound: HBM (8 bytes in, 4 out) and issue
// alike; N = 4096: 37 us (73 with an FP64 product and conversion an entry and 2-byte stores, 53 with four columns
// a thread and subnormal results on the FP64 pipe).
template <typename T>
__global__ void __launch_bounds__(256)
    k_cvt16(const T* __restrict__ src, int n, int ld_src, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
            int ld16, double scale, const float* scale_ptr, int bf16) {
  const double sc = scale_ptr ? (double)*scale_ptr : scale;
  const int k = pow2_exp(sc), i = blockIdx.x, j = 8 * (blockIdx.y * blockDim.x + threadIdx.x);
  if (j >= n) return;
  const T* s = src + (size_t)i * ld_src + j;
  T v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = j + c < n ? s[c] : (T)0;
  uint32_t h[4], l[4];
#pragma unroll
  for (int c = 0; c < 4; ++c)
    split_pair(scaled_f32(v[2 * c], sc, k), scaled_f32(v[2 * c + 1], sc, k), bf16, h[c], l[c]);
  *reinterpret_cast<uint4*>(hi + (size_t)i * ld16 + j) = make_uint4(h[0], h[1], h[2], h[3]);
  if (lo) *reinterpret_cast<uint4*>(lo + (size_t)i * ld16 + j) = make_uint4(l[0], l[1], l[2], l[3]);
}

// The same transposed: 64 x 32 tiles through shared memory, two source rows to a 4-byte word, so that a warp
// stores 128 consecutive bytes of an output row.
template <typename T>
__global__ void __launch_bounds__(256)
    k_cvt16_t(const T* __restrict__ src, int n, int ld_src, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
              int ld16, double scale, const float* scale_ptr, int bf16) {
  __shared__ uint32_t th[32][33], tl[32][33];
  const double sc = scale_ptr ? (double)*scale_ptr : scale;
  const int k = pow2_exp(sc), bi = blockIdx.y * 64, bj = blockIdx.x * 32, tx = threadIdx.x, ty = threadIdx.y;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int u = ty + 8 * p, i = bi + 2 * u, j = bj + tx;
    const T* s = src + (size_t)i * ld_src + j;
    const float a = i < n && j < n ? scaled_f32(s[0], sc, k) : 0.0f;
    const float b = i + 1 < n && j < n ? scaled_f32(s[ld_src], sc, k) : 0.0f;
    split_pair(a, b, bf16, th[tx][u], tl[tx][u]);
  }
  __syncthreads();
  const int col = bi + 2 * tx;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q, row = bj + r;
    if (row >= n || col >= n) continue;
    *reinterpret_cast<uint32_t*>(hi + (size_t)row * ld16 + col) = th[r][tx];
    if (lo) *reinterpret_cast<uint32_t*>(lo + (size_t)row * ld16 + col) = tl[r][tx];
  }
}

__global__ void k_split_flat(const double* __restrict__ A, int64_t n, double scale, uint16_t* hi, uint16_t* lo,
                             int bf16) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const float x = (float)(A[e] * scale);
    const uint16_t h = r16(x, bf16);
    hi[e] = h;
    lo[e] = r16(x - f16v(h, bf16), bf16);
  }
}

// Row-by-row copies (grid.y strides over rows, grid.x * blockDim over columns): no per-element division.
__global__ void k_f64_to_f32(const double* __restrict__ src, int n, int ld64, float* dst, int ld32) {
  for (int i = blockIdx.y; i < n; i += gridDim.y) {
    const double* s = src + (size_t)i * ld64;
    float* d = dst + (size_t)i * ld32;
#pragma unroll 4
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) d[j] = f32_of_f64(s[j], 0);
  }
}

// With amax != null also max |x| into *amax (the bits of a non-negative double; the caller zeroes it).
__global__ void k_f32_to_f64(const float* __restrict__ src, int n, int ld32, double* dst, int ld64,
                             unsigned long long* amax) {
  unsigned long long m = 0ull;
  for (int i = blockIdx.y; i < n; i += gridDim.y) {
    const float* s = src + (size_t)i * ld32;
    double* d = dst + (size_t)i * ld64;
#pragma unroll 4
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
      const double x = widen_pow2(s[j], 0);
      d[j] = x;
      m = max_bits(m, abs_bits(x));
    }
  }
  if (amax) block_raise_max(amax, m);
}

// max |A_ij| on the integer pipes (abs_bits): a NaN orders above every number, so a NaN anywhere
// makes the maximum NaN and callers can test the result with isfinite.
__global__ void k_amax_f64(const double* __restrict__ A, size_t total, IterState* st, int slot) {
  unsigned long long m = 0ull;
#pragma unroll 4
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x)
    m = max_bits(m, abs_bits(A[e]));
  block_raise_max(reinterpret_cast<unsigned long long*>(&st->amax[slot]), m);
}

__global__ void k_pow2_scales(IterState* st, int idx, float c1, float c2) {
  const double ad = st->amax[1];
  const double err = (idx >= 0 && idx < kHistMax) ? st->hist[idx] : ad;
  st->scale[0] = pow2_for(ad);
  st->scale[1] = pow2_for((double)c1 * ad + (double)c2 * err * err);
  st->scale[2] = pow2_for(st->amax[2]);
}

// The scales that follow from max |Z| (amax[6], taken from the update's epilogue unless z0): A^T's, and that of the
// next iterate (slot next).  z0: a start, whose own scale goes to slot z0 (its maximum gscale when cold).
// head: extra headroom (log2) of every scale; an FP16 accumulator takes operands scaled to at most 1.
__global__ void k_fp16_scales(IterState* st, int z0, int cold, int next, int head) {
  if (!z0)
    st->amax[6] = (double)__uint_as_float(st->amaxf[2]);
  else if (cold)
    st->amax[6] = st->gscale;
  const double z = st->amax[6];
  if (z0) st->scale[z0] = pow2_head(z, 4 + head);
  st->scale[next] = pow2_head(z, 4 + head);
  st->scale[4] = pow2_head(st->amax[0] * z, head);
  st->amaxf[1] = st->amaxf[2] = 0u;  // for the next residual's and update's maxima
}

}  // namespace

cudaError_t launch_fp16_scales(IterState* st, int z0, bool cold, int next, int head, cudaStream_t s) {
  k_fp16_scales<<<1, 1, 0, s>>>(st, z0, cold ? 1 : 0, next, head);
  return cudaGetLastError();
}

namespace {
template <typename T>
cudaError_t cvt16(const T* src, int n, int ld_src, uint16_t* hi, uint16_t* lo, int ld16, double scale,
                  const float* scale_ptr, bool transpose, bool bf16, cudaStream_t s) {
  if (transpose)
    k_cvt16_t<T><<<dim3((n + 31) / 32, (n + 63) / 64), dim3(32, 8), 0, s>>>(src, n, ld_src, hi, lo, ld16, scale,
                                                                            scale_ptr, bf16 ? 1 : 0);
  else
    k_cvt16<T><<<dim3(n, (n + 2047) / 2048), n < 2048 ? ((n + 7) / 8 + 31) / 32 * 32 : 256, 0, s>>>(
        src, n, ld_src, hi, lo, ld16, scale, scale_ptr, bf16 ? 1 : 0);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_cvt16(const double* src, int n, int ld_src, uint16_t* hi, uint16_t* lo, int ld16, double scale,
                         const float* scale_ptr, bool transpose, bool bf16, cudaStream_t s) {
  return cvt16(src, n, ld_src, hi, lo, ld16, scale, scale_ptr, transpose, bf16, s);
}

cudaError_t launch_cvt16_f32(const float* src, int n, int ld_src, uint16_t* hi, uint16_t* lo, int ld16,
                             bool transpose, bool bf16, const float* scale_ptr, cudaStream_t s) {
  return cvt16(src, n, ld_src, hi, lo, ld16, 1.0, scale_ptr, transpose, bf16, s);
}

cudaError_t launch_split_flat(const double* A, int64_t n, double scale, uint16_t* hi, uint16_t* lo, bool bf16,
                              cudaStream_t s) {
  const int blocks = (int)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192);
  k_split_flat<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(A, n, scale, hi, lo, bf16);
  return cudaGetLastError();
}

// ---- cold start Z0 = s I (s = st->gscale, the Gershgorin scale of the start)
// The first residual needs no product: A^T = Z0^T S = s S and X0 = Z0^T A = s^2 S, so
// d0 = I - s^2 S, formed here from the upper triangle of S (X is defined by its upper triangle,
// mirrored).  Writes d0 in FP32 (D32, leading dimension ld) and, when hi != nullptr, its 16-bit
// hi (and lo, when lo != nullptr) copies; partials[block] = the block's sum of d0_ij^2 over the
// entries it owns (off-diagonal entries twice), amax_bits = max |d0| as FP32 bits.  Blocks of
// 32 x 8 threads walk the upper 32 x 32 tiles; the mirror goes through shared memory.
__global__ void k_cold_resid(const double* __restrict__ S, int n, const IterState* __restrict__ st,
                             float* __restrict__ D32, int ld, uint16_t* __restrict__ hi, uint16_t* __restrict__ lo,
                             int bf16, double* __restrict__ partials, unsigned int* amax_bits) {
  __shared__ float tile[32][33];
  __shared__ double red[8];
  const double s2 = st->gscale * st->gscale;
  const int tb = (n + 31) / 32;
  const int ntiles = tb * (tb + 1) / 2;
  const int tx = threadIdx.x, ty = threadIdx.y;
  double ss = 0.0, sd = 0.0;  // sums of d^2 off the diagonal and on it
  float am = 0.0f;
  int rb = 0, rem = blockIdx.x;  // tile t -> (rb, rb + rem), row by row of the upper triangle
  double v[4];                   // the tile's entries of this thread, loaded while the one before is written
  auto load = [&](int t) {
    if (t >= ntiles) return;
    while (rem >= tb - rb) {
      rem -= tb - rb;
      ++rb;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = rb * 32 + ty + 8 * q, j = (rb + rem) * 32 + tx;
      v[q] = i < n && j < n ? S[(size_t)i * n + j] : 0.0;
    }
  };
  load(blockIdx.x);
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int bi = rb * 32, bj = (rb + rem) * 32;
    double x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = v[q];
    rem += gridDim.x;
    load(t + gridDim.x);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = ty + 8 * q, i = bi + r, j = bj + tx;
      float d = 0.0f;
      if (i < n && j < n && j >= i) {
        const double dd = (i == j ? 1.0 : 0.0) - s2 * x[q];
        d = f32_of_f64(dd, 0);
        if (i == j)
          sd = fma(dd, dd, sd);
        else
          ss = fma(dd, dd, ss);
        am = fmaxf(am, fabsf(d));
        D32[(size_t)i * ld + j] = d;
        if (hi) {
          const uint16_t h = r16(d, bf16);
          hi[(size_t)i * ld + j] = h;
          if (lo) lo[(size_t)i * ld + j] = r16(d - f16v(h, bf16), bf16);
        }
      }
      tile[r][tx] = d;
    }
    __syncthreads();
    // mirror: (i, j) with j > i to (j, i): rows bj.., columns bi..
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = ty + 8 * q, oi = bj + r, oj = bi + tx;
      if (oi < n && oj < n && oi > oj) {
        const float d = tile[tx][r];
        D32[(size_t)oi * ld + oj] = d;
        if (hi) {
          const uint16_t h = r16(d, bf16);
          hi[(size_t)oi * ld + oj] = h;
          if (lo) lo[(size_t)oi * ld + oj] = r16(d - f16v(h, bf16), bf16);
        }
      }
    }
  }
  ss = fma(2.0, ss, sd);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
  }
  if (tx == 0) red[ty] = ss;
  if (amax_bits && tx == 0) atomicMax(amax_bits, __float_as_uint(am));
  __syncthreads();
  if (tx == 0 && ty == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red[w];
    partials[blockIdx.x] = t;
  }
}

// The first update from a cold start: Z1 = Z0 + Z0 Q0 = s (I + Q0), elementwise from the FP32 Q0
// (symmetric, both triangles written).  Writes the FP32 master Zm, the 16-bit copies of Z1
// (scaled by *out_scale when given, as the update epilogue does) and the same values as the
// transposed copy (Z1 is symmetric), and max |Z1| (FP32 bits) into amax_bits.
__global__ void k_cold_update(const float* __restrict__ Q, int n, int ld, const IterState* __restrict__ st,
                              float* __restrict__ Zm, uint16_t* zh, uint16_t* zl, uint16_t* th, uint16_t* tl,
                              const float* out_scale, int bf16, unsigned int* amax_bits) {
  const float s = (float)st->gscale;
  const float osc = out_scale ? *out_scale : 1.0f;
  float am = 0.0f;
  // rows across blockIdx.y, four columns a thread (columns n up to a multiple of four as zeros)
  const int j = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
  for (int i = blockIdx.y; j < n && i < n; i += gridDim.y) {
    const size_t o = (size_t)i * ld + j;
    const float4 q = *reinterpret_cast<const float4*>(Q + o);
    float z[4] = {q.x, q.y, q.z, q.w}, y[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      z[c] = j + c < n ? s * ((i == j + c ? 1.0f : 0.0f) + z[c]) : 0.0f;
      am = fmaxf(am, fabsf(z[c]));
      y[c] = z[c] * osc;
    }
    *reinterpret_cast<float4*>(Zm + o) = make_float4(z[0], z[1], z[2], z[3]);
    uint2 h, l;
    split_pair(y[0], y[1], bf16, h.x, l.x);
    split_pair(y[2], y[3], bf16, h.y, l.y);
    *reinterpret_cast<uint2*>(zh + o) = h;
    *reinterpret_cast<uint2*>(th + o) = h;
    if (zl) {
      *reinterpret_cast<uint2*>(zl + o) = l;
      *reinterpret_cast<uint2*>(tl + o) = l;
    }
  }
  if (!amax_bits) return;
  __shared__ float red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = am;
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int w = 1; w < 8; ++w) am = fmaxf(am, red[w]);
  atomicMax(amax_bits, __float_as_uint(am));
}

static int grid_for(size_t total) { return (int)((total + 255) / 256 < 8192 ? (total + 255) / 256 : 8192); }

static dim3 rows_grid(int n) {
  const int gx = (n + 255) / 256 < 4 ? (n + 255) / 256 : 4;
  return dim3(gx > 0 ? gx : 1, n < 2048 ? (n > 0 ? n : 1) : 2048);
}

cudaError_t launch_f64_to_f32(const double* src, int n, int ld64, float* dst, int ld32, cudaStream_t s) {
  k_f64_to_f32<<<rows_grid(n), 256, 0, s>>>(src, n, ld64, dst, ld32);
  return cudaGetLastError();
}

cudaError_t launch_f32_to_f64(const float* src, int n, int ld32, double* dst, int ld64, cudaStream_t s,
                              unsigned long long* amax) {
  if (amax) cudaMemsetAsync(amax, 0, sizeof(unsigned long long), s);
  k_f32_to_f64<<<rows_grid(n), 256, 0, s>>>(src, n, ld32, dst, ld64, amax);
  return cudaGetLastError();
}

cudaError_t launch_amax_f64(const double* A, int n, IterState* st, int slot, cudaStream_t s) {
  cudaMemsetAsync(&st->amax[slot], 0, sizeof(double), s);
  const size_t total = (size_t)n * n;
  k_amax_f64<<<grid_for(total) < 1024 ? grid_for(total) : 1024, 256, 0, s>>>(A, total, st, slot);
  return cudaGetLastError();
}

cudaError_t launch_pow2_scales(IterState* st, int idx, float c1, float c2, cudaStream_t s) {
  k_pow2_scales<<<1, 1, 0, s>>>(st, idx, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_gershgorin(const double* S, int n, IterState* st, cudaStream_t s) {
  cudaMemsetAsync(&st->amax[0], 0, sizeof(double), s);
  const int warps_per_block = 8;
  k_rowabs_max<<<(n + warps_per_block - 1) / warps_per_block, 32 * warps_per_block, 0, s>>>(S, n, st);
  k_gscale<<<1, 1, 0, s>>>(st);
  return cudaGetLastError();
}

namespace {
__global__ void k_loop_init(IterState* st, int iters, int limit) {
  st->loop_iter = iters;
  st->loop_limit = limit;
}

// The loop graph's first node: whether there is any update to do.  A cold start's first update ran before it was
// known whether the first residual is finite: if it is not, that update is taken back from the counts.
__global__ void k_loop_begin(IterState* st, cudaGraphConditionalHandle loop) {
  if (st->loop_iter > 0 && !isfinite(st->hist[0])) {
    st->loop_iter = 0;
    st->hist_len = 1;
  }
  cudaGraphSetConditional(loop, !st->stop && !st->nonfinite && st->error == 0 && st->loop_iter < st->loop_limit ? 1u : 0u);
}

// One update of the device-driven bulk loop is done (its residual's Err is in the history): count it and
// decide whether the loop goes on.  Every path ends the loop once loop_limit updates are done.
__global__ void k_loop_cond(IterState* st, cudaGraphConditionalHandle loop, cudaGraphConditionalHandle next,
                            int set_next) {
  const int it = st->loop_iter + 1;
  st->loop_iter = it;
  const unsigned go = (!st->stop && !st->nonfinite && st->error == 0 && it < st->loop_limit) ? 1u : 0u;
  cudaGraphSetConditional(loop, go);
  if (set_next) cudaGraphSetConditional(next, go);
}
}  // namespace

cudaError_t launch_loop_init(IterState* st, int iters, int limit, cudaStream_t s) {
  k_loop_init<<<1, 1, 0, s>>>(st, iters, limit);
  return cudaGetLastError();
}

cudaError_t launch_loop_begin(IterState* st, cudaGraphConditionalHandle loop, cudaStream_t s) {
  k_loop_begin<<<1, 1, 0, s>>>(st, loop);
  return cudaGetLastError();
}

cudaError_t launch_loop_cond(IterState* st, cudaGraphConditionalHandle loop, cudaGraphConditionalHandle next,
                             bool set_next, cudaStream_t s) {
  k_loop_cond<<<1, 1, 0, s>>>(st, loop, next, set_next ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_set_gscale(IterState* st, double scale, cudaStream_t s) {
  k_set_gscale<<<1, 1, 0, s>>>(st, scale);
  return cudaGetLastError();
}

cudaError_t launch_scaled_identity_f64(double* Z, int n, const IterState* st, cudaStream_t s) {
  k_scaled_identity_f64<<<rows_grid(n), 256, 0, s>>>(Z, n, st);
  return cudaGetLastError();
}

cudaError_t launch_finish_err(const double* partials, int nparts, IterState* st, int idx, int rule, double tol,
                              int n, int check_stop, cudaStream_t s, Fp16Scales f) {
  k_finish_err<<<1, 1024, 0, s>>>(partials, nparts, st, idx, rule, tol, n, check_stop, f);
  return cudaGetLastError();
}

}  // namespace zf

namespace zf {
int cold_resid_blocks(int n) {
  const int tb = (n + 31) / 32, t = tb * (tb + 1) / 2;
  return t < 1024 ? t : 1024;
}

cudaError_t launch_cold_resid(const double* S, int n, const IterState* st, float* D32, int ld, uint16_t* hi,
                              uint16_t* lo, bool bf16, double* partials, unsigned int* amax_bits, cudaStream_t s) {
  k_cold_resid<<<cold_resid_blocks(n), dim3(32, 8), 0, s>>>(S, n, st, D32, ld, hi, lo, bf16 ? 1 : 0, partials,
                                                           amax_bits);
  return cudaGetLastError();
}

cudaError_t launch_cold_update(const float* Q, int n, int ld, const IterState* st, float* Zm, uint16_t* zh,
                               uint16_t* zl, uint16_t* th, uint16_t* tl, const float* out_scale, bool bf16,
                               unsigned int* amax_bits, cudaStream_t s) {
  k_cold_update<<<dim3((n + 1023) / 1024, n < 1024 ? n : 1024), 256, 0, s>>>(Q, n, ld, st, Zm, zh, zl, th, tl, out_scale, bf16 ? 1 : 0, amax_bits);
  return cudaGetLastError();
}
}  // namespace zf
