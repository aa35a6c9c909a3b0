// Reconstruction of the residue products (k_tc.cu's epilogue kEpiCrt8 leaves one digit plane per modulus):
// C 2^(eA_i + eB_j - TA - TB) in FP64 from the digits, by the byte arithmetic of crt_combine.h, with the
// residual d = I - C, its Err partials and max |d| fused where asked.
//
// Bound: integer issue.  An entry of a product over 14 moduli takes 64 four-way dot products, 8 permutes and about
// 60 other integer operations (the form with 32 x 32 -> 64-bit multiply-adds, a third of the dot products' rate
// on GB300 and two of them per modulus and limb pair, took about 400 instructions).  At N = 4096 over 14 moduli a full
// product takes 151 us (265 before; 55 for its bytes) and a symmetric one with d fused 130 (184); the group of 32
// clusters up to N = 2048 0.53 and 0.43 ms (1.63 and 0.98, where blocks past the smaller instances computed
// entries nobody stored).  A thread reads one 4-byte
// word per plane (four columns; a warp reads 128 consecutive bytes) and transposes four planes' words into
// the entries' digit words.  Values go through shared memory, so that rows and, for symmetric products, the
// mirrored columns are stored as whole segments.
#include "crt_combine.h"
#include "kernels.h"

namespace zf {
namespace {

// Column c of a staged row: the thread's four columns 36 doubles apart, so that neither its stores (lanes side
// by side), nor reads along a row, nor reads down a column (pitch 145) meet in a bank.
constexpr int kPitch = 145;
__device__ __forceinline__ int stage_col(int c) { return (c & 3) * 36 + (c >> 2); }

// One 8 R x 128 output tile at (bi, bj); 32 x 8 threads, each four columns of R rows.  out may be null (mode 2:
// only the tile's sum of d^2 into *partial_out).
template <int SH, int R>
__device__ __forceinline__ void combine_tile(const uint8_t* __restrict__ G, size_t gstride, int ld8,
                                             const CrtCombine& p, const int* __restrict__ eA,
                                             const int* __restrict__ eB, int Tsum, int n, double* __restrict__ out,
                                             int ld64, int mode, int sym, double* partial_out, int bi, int bj,
                                             unsigned long long* amax_out) {
  constexpr int Q = crt_shape_quads(SH), NB = crt_shape_bytes(SH), L = crt_shape_limbs(SH), ROWS = 8 * R;
  __shared__ double tile[ROWS * kPitch];
  __shared__ double red[8];
  __shared__ unsigned qtab[kCrtQRows * L];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * 32 + tx;
  // a tile past the matrix or below the diagonal holds nothing
  const bool active = bi < n && bj < n && (!sym || bj + 127 >= bi);
  double ss_off = 0.0, ss_diag = 0.0;  // sums of d_ij^2 over j > i and j = i
  unsigned long long am = 0ull;        // max |d_ij| (bits of a non-negative double) when amax_out is set
  if (active) {
    for (int e = tid; e < kCrtQRows * L; e += 256) qtab[e] = p.qM[e / L][e % L];
    __syncthreads();
    const int j0 = bj + 4 * tx;
    int eb[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) eb[k] = j0 + k < n ? eB[j0 + k] : -2000000000;
#pragma unroll 1
    for (int q = 0; q < R; ++q) {
      const int r = ty + 8 * q, i = bi + r;
      const bool rok = i < n && j0 < n;
      const uint8_t* g = G + (rok ? (size_t)i * ld8 + j0 : 0);
      unsigned w[4 * Q];
#pragma unroll
      for (int t = 0; t < 4 * Q; ++t)
        w[t] = (rok && t < p.nmod) ? __ldcs(reinterpret_cast<const unsigned*>(g + (size_t)t * gstride)) : 0u;
      // 4 x 4 byte transposes: word i of entry k holds its digits of moduli 4 i ... 4 i + 3
      unsigned d[4][Q];
#pragma unroll
      for (int x = 0; x < Q; ++x) {
        const unsigned a = __byte_perm(w[4 * x], w[4 * x + 1], 0x5140), b = __byte_perm(w[4 * x], w[4 * x + 1], 0x7362);
        const unsigned c = __byte_perm(w[4 * x + 2], w[4 * x + 3], 0x5140),
                       e = __byte_perm(w[4 * x + 2], w[4 * x + 3], 0x7362);
        d[0][x] = __byte_perm(a, c, 0x5410);
        d[1][x] = __byte_perm(a, c, 0x7632);
        d[2][x] = __byte_perm(b, e, 0x5410);
        d[3][x] = __byte_perm(b, e, 0x7632);
      }
      const int ea = i < n ? eA[i] : -2000000000;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        // (below the diagonal of a symmetric product the epilogue leaves digits unwritten: no entry is formed there)
        const int j = j0 + k;
        double v = 0.0;
        if (i < n && j < n && (!sym || j >= i)) {
          if (ea > -1000 && eb[k] > -1000) v = crt_combine_value<Q, NB, L>(p, d[k], qtab, L, ea + eb[k] - Tsum);
          if (mode == 2) {
            // d = I - C: a sign flip off the diagonal (no FP64 arithmetic), one subtraction on it
            if (i == j) {
              v = 1.0 - v;
              ss_diag = fma(v, v, ss_diag);
            } else {
              v = __longlong_as_double(__double_as_longlong(v) ^ (long long)0x8000000000000000ull);
              if (j > i) ss_off = fma(v, v, ss_off);
            }
            if (amax_out) am = max_bits(am, abs_bits(v));
          }
        }
        tile[r * kPitch + 36 * k + tx] = v;
      }
    }
    if (out) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int r = ty + 8 * q, i = bi + r;
        double* o = out + (size_t)i * ld64 + bj;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int c = 32 * x + tx, j = bj + c;
          if (i < n && j < n && (!sym || j >= i)) {
            const double v = tile[r * kPitch + stage_col(c)];
            if (mode == 1)
              o[c] += v;
            else
              o[c] = v;
          }
        }
      }
      if (sym && bj + 127 > bi) {
        // (i, j) with j > i also goes to (j, i): rows bj.. of the output, columns bi..
        for (int e = tid; e < 128 * ROWS; e += 256) {
          const int c = e / ROWS, r = e % ROWS, oi = bj + c, oj = bi + r;
          if (oi < n && oj < n && oi > oj) {
            double* o = out + (size_t)oi * ld64 + oj;
            const double v = tile[r * kPitch + stage_col(c)];
            if (mode == 1)
              *o += v;
            else
              *o = v;
          }
        }
      }
    }
  }
  if (mode == 2) {
    double ss = fma(2.0, ss_off, ss_diag);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if (tx == 0) red[ty] = ss;
    __syncthreads();
    if (ty == 0 && tx == 0) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) t += red[w];
      if (partial_out) *partial_out = t;
    }
    if (amax_out && active) block_raise_max(amax_out, am);
  }
}

template <int SH, int R>
__global__ void __launch_bounds__(256, SH > 4 ? 2 : 3)
    k_crt_combine(const uint8_t* __restrict__ G, size_t gstride, int ld8, const __grid_constant__ CrtCombine p,
                  const int* __restrict__ eA, const int* __restrict__ eB, int Tsum, int n, double* __restrict__ out,
                  int ld64, int mode, int sym, double* __restrict__ partials, unsigned long long* amax) {
  combine_tile<SH, R>(G, gstride, ld8, p, eA, eB, Tsum, n, out, ld64, mode, sym,
                      partials ? partials + blockIdx.y * gridDim.x + blockIdx.x : nullptr, blockIdx.y * 8 * R,
                      blockIdx.x * 128, amax);
}

// Every instance of a group (grid.z): its digits, exponents and output rows start at its packed row.
template <int SH, int R>
__global__ void __launch_bounds__(256, SH > 4 ? 2 : 3)
    k_gcrt_combine(const uint8_t* __restrict__ G, size_t gstride, int ld8, const __grid_constant__ CrtCombine p,
                   const GroupRes g, const int* __restrict__ eA, const int* __restrict__ eB, double* __restrict__ out,
                   int ld64, int mode, int sym, double* __restrict__ partials) {
  const int inst = blockIdx.z, r0 = g.row0[inst];
  const size_t nb = (size_t)gridDim.x * gridDim.y;
  combine_tile<SH, R>(G + (size_t)r0 * ld8, gstride, ld8, p, eA + r0, eB + r0, 2 * g.T[inst], g.n[inst],
                      out ? out + (size_t)r0 * ld64 : nullptr, ld64, mode, sym,
                      partials ? partials + inst * nb + blockIdx.y * gridDim.x + blockIdx.x : nullptr,
                      blockIdx.y * 8 * R, blockIdx.x * 128, nullptr);
}

// Rows of a tile in units of 8: 32-row tiles amortize a block's set-up, 8-row ones fill the SMs below N = 1536
// (32-row tiles number 576 there, 3.8 per SM; N = 256 takes 6 to 8 us, 21 to 26 on the 16 blocks of 32-row tiles).
int rows_of(int n) { return n < 1536 ? 1 : 4; }

// f(shape, rows) for the instantiation of `shape` and `rows`, as integral constants
template <int V>
struct Int {
  static constexpr int value = V;
};
template <int SH, class F>
void with_rows(int rows, F&& f) {
  if (rows == 1)
    f(Int<SH>{}, Int<1>{});
  else
    f(Int<SH>{}, Int<4>{});
}
template <class F>
void with_shape(int shape, int rows, F&& f) {
  switch (shape) {
    case 0: return with_rows<0>(rows, f);
    case 1: return with_rows<1>(rows, f);
    case 2: return with_rows<2>(rows, f);
    case 3: return with_rows<3>(rows, f);
    case 4: return with_rows<4>(rows, f);
    case 5: return with_rows<5>(rows, f);
    default: return with_rows<6>(rows, f);
  }
}

}  // namespace

int crt_combine_blocks(int n) {
  const int rows = 8 * rows_of(n);
  return ((n + 127) / 128) * ((n + rows - 1) / rows);
}

cudaError_t launch_crt_combine(const uint8_t* G, size_t gstride, int ld8, int nmod, const int* eA, const int* eB,
                               int TA, int TB, int n, double* out, int ld64, int mode, bool sym, double* partials,
                               cudaStream_t s, unsigned long long* amax) {
  const CrtCombine* p = crt_combine(nmod);
  if (!p || (ld8 % 4) != 0) return cudaErrorInvalidValue;
  with_shape(p->shape, rows_of(n), [&](auto sh, auto r) {
    constexpr int SH = decltype(sh)::value, R = decltype(r)::value;
    const dim3 grid((n + 127) / 128, (n + 8 * R - 1) / (8 * R));
    k_crt_combine<SH, R><<<grid, dim3(32, 8), 0, s>>>(G, gstride, ld8, *p, eA, eB, TA + TB, n, out, ld64, mode,
                                                      sym ? 1 : 0, partials, amax);
  });
  return cudaGetLastError();
}

cudaError_t launch_gcrt_combine(const uint8_t* G, size_t gstride, int ld8, int nmod, const GroupRes& g, const int* eA,
                                const int* eB, double* out, int ld64, int mode, bool sym, double* partials,
                                cudaStream_t s) {
  const CrtCombine* p = crt_combine(nmod);
  if (!p || (ld8 % 4) != 0 || g.count < 1) return cudaErrorInvalidValue;
  with_shape(p->shape, rows_of(g.max_n), [&](auto sh, auto r) {
    constexpr int SH = decltype(sh)::value, R = decltype(r)::value;
    const dim3 grid((g.max_n + 127) / 128, (g.max_n + 8 * R - 1) / (8 * R), g.count);
    k_gcrt_combine<SH, R><<<grid, dim3(32, 8), 0, s>>>(G, gstride, ld8, *p, g, eA, eB, out, ld64, mode, sym ? 1 : 0,
                                                       partials);
  });
  return cudaGetLastError();
}

}  // namespace zf
