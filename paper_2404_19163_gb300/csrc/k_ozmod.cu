// FP64-accurate products on the BF16 tensor cores by modular arithmetic (Ozaki scheme II:
// Ozaki, Uchino, Imamura, "Ozaki Scheme II: A GEMM-oriented emulation of floating-point matrix
// multiplication using an integer modular technique", 2025).
//
// Every row r of an FP64 operand is scaled by 2^(T - e_r) (e_r: the row's exponent bound) and
// rounded to an integer F with |F| <= 2^T.  The product C' = F_A F_B^T of two such integer
// matrices is exact and bounded by K 2^(T_A + T_B).  It is formed modulo pairwise coprime
// moduli m_i <= 256 (up to 24 of them, crt_wide.h, for rows of up to 83 bits): residues of F within 128 of
// zero (one FP32 reduction) are exact in BF16, a residue
// product over K <= 1024 terms stays an integer of at most 2^24 (exact in the FP32 accumulator;
// longer products are reduced modulo m_i every 1024 terms inside the product's epilogue), and
// the Chinese remainder theorem recovers C' from its residues once M = prod m_i > 4 |C'|.  The
// result is C_ij = 2^(eA_i + eB_j - T_A - T_B) C'_ij: the only errors are the two roundings to
// T-bit fixed point and the final conversion to FP64.  The moduli count grows linearly with the
// bits kept (about 7.9 bits per product), where slicing grows quadratically (s(s+1)/2 pairs).
#include <math.h>

#include "crt_wide.h"
#include "kernels.h"

namespace zf {

namespace {

// The NP signed 14-bit parts of round(x 2^(T - er)) for |x| < 2^er, from the bits of x (integer operations).
// NP = 4 holds rows of T <= 55 bits, 5 of T <= 62 and 6 of T <= 83 (for a normal x the shift is at most T - 53).
template <int NP>
__device__ __forceinline__ void parts_of(double x, int er, int T, float (&a)[NP]) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int eb = (int)((bits >> 52) & 0x7FF);
  const unsigned long long frac = bits & 0xFFFFFFFFFFFFFull, m = eb ? frac | (1ull << 52) : frac;
  const int sh = (eb ? eb - 1075 : -1074) - er + T;
  const unsigned sign = (unsigned)(bits >> 32) & 0x80000000u;
  unsigned long long lo = 0ull, hi = 0ull;
  if (er > -1000 && sh > -63) {
    if (sh < 0)
      lo = (m + (1ull << (-sh - 1))) >> (-sh);
    else if (NP < 6)
      lo = m << (sh < 11 ? sh : 11);
    else {
      const unsigned __int128 F = (unsigned __int128)m << (sh < 74 ? sh : 74);
      lo = (unsigned long long)F;
      hi = (unsigned long long)(F >> 64);
    }
  }
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    const int b = 14 * k;
    const unsigned long long v = b + 14 <= 64 ? lo >> b : b >= 64 ? hi >> (b - 64) : (lo >> b) | (hi << (64 - b));
    a[k] = crt_part_f((unsigned)v & 0x3FFFu, sign);
  }
}

// Eight neighbouring elements of an operand row, two to a register pair.
template <int NP>
struct Octet {
  f32x2 p[NP][4];
  __device__ __forceinline__ void set(const double (&v)[8], int er, int T) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float a[NP], b[NP];
      parts_of<NP>(v[2 * j], er, T, a);
      parts_of<NP>(v[2 * j + 1], er, T, b);
#pragma unroll
      for (int k = 0; k < NP; ++k) p[k][j] = pack2(a[k], b[k]);
    }
  }
};

// The octet's residues (crt_residue_step) for the moduli I, I + 1, ... < nmod, 16 bytes of BF16 a modulus (an
// integer |r| <= 128 has its low 16 FP32 bits zero, so its BF16 value is the upper half).
template <int NP, int I = 0>
__device__ __forceinline__ void octet_residues(const Octet<NP>& o, int nmod, uint16_t* out, size_t stride) {
  if constexpr (I < crtw::kMax) {
    if (I < nmod) {
      constexpr int m = crtw::modulus(I);
      constexpr float fm = (float)m, inv = 1.0f / (float)m;
      const f32x2 m2 = pack2(-fm, -fm), inv2 = pack2(inv, inv), big = pack2(12582912.0f, 12582912.0f),
                  nbig = pack2(-12582912.0f, -12582912.0f);
      unsigned w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f32x2 x = o.p[0][j];
#pragma unroll
        for (int k = 1; k < NP; ++k) {
          const float c = (float)crt_pow2_sym(m, 14 * k);
          x = fma2(o.p[k][j], pack2(c, c), x);
        }
        float r0, r1;
        unpack2(fma2(add2(fma2(x, inv2, big), nbig), m2, x), r0, r1);
        w[j] = __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
      }
      *reinterpret_cast<uint4*>(out + (size_t)I * stride) = make_uint4(w[0], w[1], w[2], w[3]);
      octet_residues<NP, I + 1>(o, nmod, out, stride);
    }
  }
}

// The products' epilogue carries two columns in a float (tc_kernel.cuh), so an odd size's last column meets the operand
// row after the last: an octet of zeros there.
__device__ __forceinline__ void zero_octet(int nmod, uint16_t* out, size_t stride) {
  for (int t = 0; t < nmod; ++t) *reinterpret_cast<uint4*>(out + (size_t)t * stride) = make_uint4(0, 0, 0, 0);
}
// A row's threads: the block, or one warp of it (TEAM = 32).
constexpr int kRowThreads = 256;
template <int TEAM>
__device__ __forceinline__ void team_sync() {
  if (TEAM == 32)
    __syncwarp();
  else
    __syncthreads();
}
template <int TEAM>
__device__ __forceinline__ void zero_row(int ncols, int nmod, uint16_t* orow, size_t stride) {
  const int tid = TEAM == 32 ? threadIdx.x & 31 : threadIdx.x, nt = TEAM == 32 ? 32 : blockDim.x;
  for (int c = 8 * tid; c < ncols; c += 8 * nt) zero_octet(nmod, orow + c, stride);
}

// Residues of one row xr of n elements (columns n ... up to a multiple of 8, or of 64 for `pad64`, as zeros): the
// row's largest magnitude, then octets.  Loads run along the row; octets are read from shared memory (element i at
// i + i / 8: two wavefronts for a warp's 8-byte reads, the least).
template <int NP, int TEAM>
__device__ __forceinline__ void row_residues(const double* __restrict__ xr, int n, bool pad64, int T, int nmod,
                                             int* __restrict__ e, uint16_t* __restrict__ orow, size_t stride) {
  __shared__ double sx_all[kRowThreads * 9];
  __shared__ unsigned long long red[kRowThreads / 32];
  const int tid = TEAM == 32 ? threadIdx.x & 31 : threadIdx.x, nt = TEAM == 32 ? 32 : blockDim.x, chunk = 8 * nt;
  double* sx = TEAM == 32 ? sx_all + (threadIdx.x >> 5) * 32 * 9 : sx_all;
  double v[8];
  unsigned long long m = 0ull;  // the row's largest magnitude, as a bit pattern (integer pipes)
  for (int c0 = (n - 1) / chunk * chunk; c0 >= 0; c0 -= chunk) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = c0 + tid + k * nt < n ? xr[c0 + tid + k * nt] : 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) m = max_bits(m, abs_bits(v[k]));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (TEAM != 32) {
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
    m = red[0];
    for (int w = 1; w < nt / 32; ++w) m = max_bits(m, red[w]);
  }
  const int er = m ? exp_of_bits(m) : -2000000000;
  if (tid == 0) *e = er;
  const int ncols = pad64 ? (n + 63) & ~63 : (n + 7) & ~7;
  for (int c0 = 0; c0 < ncols; c0 += chunk) {
    if (c0 > 0) {  // (the first chunk is the last the loop above read)
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = c0 + tid + k * nt < n ? xr[c0 + tid + k * nt] : 0.0;
      team_sync<TEAM>();
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int i = tid + k * nt;
      sx[i + (i >> 3)] = v[k];
    }
    team_sync<TEAM>();
    const int c = c0 + 8 * tid;
    if (c < ncols) {
      double x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = sx[9 * tid + k];
      Octet<NP> o;
      o.set(x, er, T);
      octet_residues<NP>(o, nmod, orow + c, stride);
    }
  }
}

// Rows of X, one block a row.  Bound: HBM (8 bytes in, 2 nmod out an element): an operand of N = 4096 over 14 moduli
// takes 105 us, 86% of the measured copy rate (140 with scalar arithmetic, 4-byte stores and loads of every other
// double).
template <int NP>
__global__ void __launch_bounds__(kRowThreads)
    k_ozm_rowres(const double* __restrict__ X, int n, int ld, int* __restrict__ e, int T, int nmod,
                 uint16_t* __restrict__ out, int ld16, int Rp) {
  const int row = blockIdx.x;
  uint16_t* orow = out + (size_t)row * ld16;
  if (row < n)
    row_residues<NP, kRowThreads>(X + (size_t)row * ld, n, false, T, nmod, e + row, orow, (size_t)Rp * ld16);
  else
    zero_row<kRowThreads>((n + 7) & ~7, nmod, orow, (size_t)Rp * ld16);
}

// Residues of a 64 x 32 tile of X^T (operand rows bj ... = columns of X, whose exponents e are known): row pairs of
// X go to shared memory as 16-byte units, unit u of operand row r at 33 r + 4 g + (k ^ (g >> 1)), g = u / 4 and
// k = u % 4, so that neither the stores (lanes along r) nor an octet's reads (lanes along g) meet in a bank.
template <int NP>
__device__ __forceinline__ void tile_residues(const double* __restrict__ X, int n, int ld, int ncols,
                                              const int* __restrict__ e, int T, int nmod, uint16_t* __restrict__ out,
                                              int ld16, size_t stride, int bi, int bj) {
  __shared__ double2 sx[32 * 33];
  const int tid = threadIdx.x;
  {
    const int r = tid & 31, j = bj + r;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int u = (tid >> 5) + 8 * p, i = bi + 2 * u, g = u >> 2;
      double2 t = make_double2(0.0, 0.0);
      if (j < n && i < n) t.x = X[(size_t)i * ld + j];
      if (j < n && i + 1 < n) t.y = X[(size_t)(i + 1) * ld + j];
      sx[33 * r + 4 * g + ((u & 3) ^ (g >> 1))] = t;
    }
  }
  __syncthreads();
  const int g = tid & 7, r = tid >> 3, row = bj + r, col = bi + 8 * g;
  if (col >= ncols) return;
  if (row >= n) {
    if (row == n && (n & 1)) zero_octet(nmod, out + (size_t)row * ld16 + col, stride);
    return;
  }
  double x[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 t = sx[33 * r + 4 * g + (k ^ (g >> 1))];
    x[2 * k] = t.x;
    x[2 * k + 1] = t.y;
  }
  Octet<NP> o;
  o.set(x, e[row], T);
  octet_residues<NP>(o, nmod, out + (size_t)row * ld16 + col, stride);
}

template <int NP>
__global__ void __launch_bounds__(256)
    k_ozm_tres(const double* __restrict__ X, int n, int ld, const int* __restrict__ e, int T, int nmod,
               uint16_t* __restrict__ out, int ld16, int Rp) {
  tile_residues<NP>(X, n, ld, (n + 7) & ~7, e, T, nmod, out, ld16, (size_t)Rp * ld16, blockIdx.y * 64, blockIdx.x * 32);
}

// rho_r^2 = sum_k (x_rk 2^-e_r)^2 of every row r of X (e_r the row's exponent bound, as in the
// residue kernels), and the largest of them as an FP32 bit pattern into *rho2 (atomic maximum:
// non-negative floats order like their bit patterns).  A row holding a NaN or Inf, or whose
// largest entry is subnormal, writes +Inf (no bound).
// One block of 256 threads per row; the sum runs in FP32 (its error is bounded by the caller).
__global__ void __launch_bounds__(256) k_ozm_rowrho(const double* __restrict__ X, int n, int ld,
                                                    unsigned int* __restrict__ rho2, unsigned long long* amax) {
  __shared__ unsigned long long redm[8];
  __shared__ float reds[8];
  const double* xr = X + (size_t)blockIdx.x * ld;
  const int tid = threadIdx.x;
  unsigned long long m = 0ull;
  for (int c = tid; c < n; c += 256) m = max_bits(m, abs_bits(xr[c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) == 0) redm[tid >> 5] = m;
  __syncthreads();
  m = redm[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = max_bits(m, redm[w]);
  if (amax && tid == 0) atomicMax(amax, m);
  if (m == 0ull) return;
  if (m >= 0x7FF0000000000000ull || m < (1ull << 52)) {
    // NaN or Inf, or a row of subnormals (their scaled values would all read as zero): no bound
    if (tid == 0) atomicMax(rho2, 0x7F800000u);
    return;
  }
  const int e = exp_of_bits(m);
  float acc = 0.0f;
  for (int c = tid; c < n; c += 256) {
    const float f = scaled_mag_f32(abs_bits(xr[c]), e);
    acc = fmaf(f, f, acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) reds[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += reds[w];
    atomicMax(rho2, __float_as_uint(t));
  }
}

// ---- grouped forms (the batched mode's final residuals): instance = blockIdx.y (rows) or blockIdx.z (tiles);
// columns n ... up to the K padding that the tensor-core loads read are zeros.  A warp a row: the rows of a group are
// enough warps, and sizes differ, so that blocks of the widest row's threads would idle on the others.
template <int NP>
__global__ void __launch_bounds__(kRowThreads)
    k_gozm_rowres(const GroupRes g, int nmod, uint16_t* __restrict__ out, int ld16, size_t plane) {
  const int inst = blockIdx.y, n = g.n[inst], row = blockIdx.x * (kRowThreads / 32) + (threadIdx.x >> 5);
  if (row >= n + (n & 1)) return;
  const int r0 = g.row0[inst];
  if (row == n) {
    zero_row<32>((n + 63) & ~63, nmod, out + (size_t)(r0 + row) * ld16, plane);
    return;
  }
  const double* xr = g.src ? g.src[inst] + (size_t)row * n : g.packed + (size_t)(r0 + row) * g.ldp;
  row_residues<NP, 32>(xr, n, true, g.T[inst], nmod, g.e + r0 + row, out + (size_t)(r0 + row) * ld16, plane);
}

template <int NP>
__global__ void __launch_bounds__(256)
    k_gozm_tres(const GroupRes g, int nmod, uint16_t* __restrict__ out, int ld16, size_t plane) {
  const int inst = blockIdx.z, n = g.n[inst], ncols = (n + 63) & ~63;
  const int bi = blockIdx.y * 64, bj = blockIdx.x * 32;
  if (bj >= n || bi >= ncols) return;  // the whole block (uniform)
  const int r0 = g.row0[inst];
  tile_residues<NP>(g.src[inst], n, n, ncols, g.e + r0, g.T[inst], nmod, out + (size_t)r0 * ld16, ld16, plane, bi, bj);
}

// rho2[inst] = max over the instance's packed rows of rho_r^2 (as k_ozm_rowrho).
__global__ void __launch_bounds__(256) k_gozm_rowrho(const GroupRes g, unsigned int* __restrict__ rho2) {
  __shared__ unsigned long long redm[8];
  __shared__ float reds[8];
  const int inst = blockIdx.y, n = g.n[inst], row = blockIdx.x;
  if (row >= n) return;
  const double* xr = g.packed + (size_t)(g.row0[inst] + row) * g.ldp;
  const int tid = threadIdx.x;
  unsigned long long m = 0ull;
  for (int c = tid; c < n; c += 256) m = max_bits(m, abs_bits(xr[c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_bits(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((tid & 31) == 0) redm[tid >> 5] = m;
  __syncthreads();
  m = redm[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = max_bits(m, redm[w]);
  if (m == 0ull) return;
  if (m >= 0x7FF0000000000000ull || m < (1ull << 52)) {
    if (tid == 0) atomicMax(&rho2[inst], 0x7F800000u);
    return;
  }
  const int e = exp_of_bits(m);
  float acc = 0.0f;
  for (int c = tid; c < n; c += 256) {
    const float f = scaled_mag_f32(abs_bits(xr[c]), e);
    acc = fmaf(f, f, acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((tid & 31) == 0) reds[tid >> 5] = acc;
  __syncthreads();
  if (tid == 0) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += reds[w];
    atomicMax(&rho2[inst], __float_as_uint(t));
  }
}

__global__ void k_gozm_finish(const double* __restrict__ partials, int nb, double* __restrict__ err) {
  __shared__ double red[256];
  const double* p = partials + (size_t)blockIdx.x * nb;
  double s = 0.0;
  for (int k = threadIdx.x; k < nb; k += 256) s += p[k];  // fixed order per thread
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) err[blockIdx.x] = sqrt(red[0]);
}

}  // namespace

namespace {
// f(parts) for rows of T bits, as an integral constant
template <int V>
struct Parts {
  static constexpr int value = V;
};
template <class F>
void with_parts(int T, F&& f) {
  if (T <= 55)
    f(Parts<4>{});
  else if (T <= 62)
    f(Parts<5>{});
  else
    f(Parts<6>{});
}
// threads of a row's block: the octets in as few equal chunks as whole warps allow
int row_threads(int n) {
  const int octets = (n + 7) / 8, chunks = (octets + kRowThreads - 1) / kRowThreads;
  return ((octets + chunks - 1) / chunks + 31) / 32 * 32;
}
}  // namespace

cudaError_t launch_ozm_residues(const double* X, int n, int ld, bool trans, int* e, int T, int nmod, uint16_t* out,
                                int ld16, int Rp, cudaStream_t s) {
  if (nmod < 1 || nmod > crtw::kMax || T < 1 || T > 83) return cudaErrorInvalidValue;
  with_parts(T, [&](auto np) {
    constexpr int NP = decltype(np)::value;
    if (trans)
      k_ozm_tres<NP><<<dim3((n + 31) / 32, (n + 63) / 64), 256, 0, s>>>(X, n, ld, e, T, nmod, out, ld16, Rp);
    else
      k_ozm_rowres<NP><<<n + (n & 1), row_threads(n), 0, s>>>(X, n, ld, e, T, nmod, out, ld16, Rp);
  });
  return cudaGetLastError();
}

cudaError_t launch_ozm_rho(const double* X, int n, int ld, unsigned int* rho2, cudaStream_t s,
                           unsigned long long* amax) {
  if (n < 1) return cudaErrorInvalidValue;
  k_ozm_rowrho<<<n, 256, 0, s>>>(X, n, ld, rho2, amax);
  return cudaGetLastError();
}

cudaError_t launch_gozm_rowres(const GroupRes& g, int nmod, uint16_t* out, int ld16, size_t plane, int maxT,
                               cudaStream_t s) {
  if (nmod < 1 || nmod > crtw::kMax || maxT < 1 || maxT > 83 || g.count < 1) return cudaErrorInvalidValue;
  with_parts(maxT, [&](auto np) {
    k_gozm_rowres<decltype(np)::value><<<dim3((g.max_n + 8) / 8, g.count), kRowThreads, 0, s>>>(g, nmod, out, ld16, plane);
  });
  return cudaGetLastError();
}

cudaError_t launch_gozm_tres(const GroupRes& g, int nmod, uint16_t* out, int ld16, size_t plane, int maxT,
                             cudaStream_t s) {
  if (nmod < 1 || nmod > crtw::kMax || maxT < 1 || maxT > 83 || g.count < 1 || !g.src) return cudaErrorInvalidValue;
  const dim3 grid((g.max_n + 31) / 32, (g.max_n + 63) / 64, g.count);
  with_parts(maxT, [&](auto np) { k_gozm_tres<decltype(np)::value><<<grid, 256, 0, s>>>(g, nmod, out, ld16, plane); });
  return cudaGetLastError();
}

cudaError_t launch_gozm_rowrho(const GroupRes& g, unsigned int* rho2, cudaStream_t s) {
  if (g.count < 1 || !g.packed) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(rho2, 0, sizeof(unsigned int) * (size_t)g.count, s);
  if (e != cudaSuccess) return e;
  k_gozm_rowrho<<<dim3(g.max_n, g.count), 256, 0, s>>>(g, rho2);
  return cudaGetLastError();
}

cudaError_t launch_gozm_finish(const double* partials, int nb, int count, double* err, cudaStream_t s) {
  if (count < 1 || nb < 1) return cudaErrorInvalidValue;
  k_gozm_finish<<<count, 256, 0, s>>>(partials, nb, err);
  return cudaGetLastError();
}

}  // namespace zf
