// CUDA-core products of the recursion in FP64 (the paper's "double", Table I) and FP32
// ("single"),
// with the element-wise steps fused into the epilogues:
//   residual   d = I - Z^T (S Z), symmetric, upper tiles only   (Eq. np1, Algorithm 2's Err)
//   polynomial Q = c1 d + c2 d^2 (+ c_k d^k chains)               (delta-form of Eq. np1)
//   update     Z' = Z + Z Q                                       (Z_{n+1} = Z_n p(d_n))
// GB300's FP64 pipe is ~1.1 TFLOP/s (about 2 DFMA per SM per clock), so these
// kernels are bound by FP64 issue for every N of interest; a 64x64 tile with a
// 4x4 register micro-tile keeps the operand traffic far below that bound.
#include "kernels.h"

namespace zf {
namespace {

constexpr int BK = 16, NT = 256;

// Tile edge of the FP64 products: 64 x 64 tiles (4 x 4 outputs per thread) in general; 32 x 32 tiles (2 x 2 per
// thread) up to N = 1024, where 64-wide tiles leave most SMs idle (N = 256: 16 tiles on 152 SMs).  FP32: 64 x 64.
inline int tile_for(int n, bool fp32 = false) { return !fp32 && n <= 1024 ? 32 : 64; }

__device__ __forceinline__ void sym_tile_of(int b, int T, int& bi, int& bj) {
  // b-th tile of the upper triangle, row-major over (bi, bj >= bi)
  int row = 0, rem = b;
  while (rem >= T - row) {
    rem -= T - row;
    ++row;
  }
  bi = row;
  bj = row + rem;
}

template <int TE>
__global__ void __launch_bounds__(NT) k64_gemm(F64Gemm g) {
  using T = double;
  constexpr int BM = TE, BN = TE, R = TE / 16;  // R x R outputs per thread
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  __shared__ double red[NT / 32];
  const int n = g.n;
  const int TB = (n + BM - 1) / BM;
  int bi, bj;
  if (g.sym) {
    sym_tile_of(blockIdx.x, TB, bi, bj);
  } else {
    bi = blockIdx.y;
    bj = blockIdx.x;
  }
  const int i0 = bi * BM, j0 = bj * BN;
  const int t = threadIdx.x;
  const int ty = t / 16, tx = t % 16;
  T acc[R][R] = {};
  for (int k0 = 0; k0 < n; k0 += BK) {
#pragma unroll
    for (int e = 0; e < (BM * BK) / NT; ++e) {
      const int idx = t + e * NT;
      int ii, kk;
      T v = 0;
      if (g.transA) {
        kk = idx / BM;
        ii = idx % BM;
        const int gi = i0 + ii, gk = k0 + kk;
        if (gi < n && gk < n) v = g.A[(size_t)gk * n + gi];
      } else {
        ii = idx / BK;
        kk = idx % BK;
        const int gi = i0 + ii, gk = k0 + kk;
        if (gi < n && gk < n) v = g.A[(size_t)gi * n + gk];
      }
      As[kk][ii] = v;
    }
#pragma unroll
    for (int e = 0; e < (BK * BN) / NT; ++e) {
      const int idx = t + e * NT;
      const int kk = idx / BN, jj = idx % BN;
      const int gk = k0 + kk, gj = j0 + jj;
      Bs[kk][jj] = (gk < n && gj < n) ? g.B[(size_t)gk * n + gj] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      T a[R], b[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = As[kk][ty * R + r];
#pragma unroll
      for (int c = 0; c < R; ++c) b[c] = Bs[kk][tx * R + c];
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < R; ++c) acc[r][c] = fma(a[r], b[c], acc[r][c]);
    }
    __syncthreads();
  }
  double ss = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + ty * R + r;
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int j = j0 + tx * R + c;
      if (j >= n) continue;
      if (g.sym && j < i) continue;  // the (j, i) entry is written by the tile that owns it
      T v;
      if (g.resid) {
        v = (i == j ? T(1) : T(0)) - acc[r][c];
        ss += (i == j ? 1.0 : 2.0) * (double)v * (double)v;
      } else {
        v = (T)g.beta * acc[r][c];
        if (g.Add) v = fma((T)g.alpha, g.Add[(size_t)i * n + j], v);
        if (g.P) {
          g.P[(size_t)i * n + j] = acc[r][c];
          if (g.sym && j != i) g.P[(size_t)j * n + i] = acc[r][c];
        }
      }
      g.C[(size_t)i * n + j] = v;
      if (g.sym && j != i) g.C[(size_t)j * n + i] = v;
    }
  }
  if (g.resid) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((t & 31) == 0) red[t >> 5] = ss;
    __syncthreads();
    if (t == 0) {
      double s = 0.0;
      for (int w = 0; w < NT / 32; ++w) s += red[w];
      g.partials[blockIdx.x] = s;
    }
  }
}

// ---- FP32
// The same product with pairs of rows in packed FMAs (fma.rn.f32x2, each half an FP32 FMA), 8 x 4 outputs per
// thread, and the next K-block's loads in flight while one is multiplied (two shared-memory buffers).  Every
// entry adds its products in the order of k, as k64_gemm does.
// Bound: latency and shared memory (48 bytes a thread for 32 FMAs, 1.5 times what the FP32 pipe's time allows) at the
// three tiles an SM that N = 1331 gives.  The operands of the next k are read before the FMAs of this one (N = 1331:
// 1.95 ms a factorization, 2.04 without).  8 x 8 outputs ask shared memory for a third less but leave 64 threads a tile,
// too few to cover the latencies (2.32), on 128 x 128 tiles too few tiles (2.83); B's values stored twice, as the packed
// FMA takes them, ask for more (2.92); K-blocks of 32 gain below N = 1000 and lose above (N = 512: 652 us against 684,
// 2500: 9.4 ms against 8.9).  Factorizations on k64_gemm's scheme (2 x 2 outputs up to N = 1024, 4 x 4, and 8 x 8 from
// 2048) and here: N = 256 0.60 and 0.52 ms, 1000 2.07 and 1.21, 1331 3.07 and 1.95, 2047 10.4 and 5.0, 2500 15.6 and 8.9.
__global__ void __launch_bounds__(128) k32_gemm(F32Gemm g) {
  constexpr int TE = 64, RM = 8, RN = 4, T = (TE / RM) * (TE / RN), EL = TE * BK / T, TX = TE / RN, PITCH = TE + 4;
  __shared__ __align__(16) float As[2][BK][PITCH];
  __shared__ __align__(16) float Bs[2][BK][PITCH];
  __shared__ double red[T / 32];
  const int n = g.n, t = threadIdx.x;
  int bi, bj;
  if (g.sym) {
    sym_tile_of(blockIdx.x, (n + TE - 1) / TE, bi, bj);
  } else {
    bi = blockIdx.y;
    bj = blockIdx.x;
  }
  const int i0 = bi * TE, j0 = bj * TE, ty = t / TX, tx = t % TX;
  // Element e of the thread's share of a K-block: A^T's row k = t / TE + e T / TE, column t % TE (B's too), or A's
  // row t / BK + e T / BK, column k = t % BK.
  const bool ta = g.transA, cok = j0 + t % TE < n, rok = i0 + t % TE < n;
  const float* pb = g.B + (size_t)(t / TE) * n + (j0 + t % TE);
  const float* pa = ta ? g.A + (size_t)(t / TE) * n + (i0 + t % TE) : g.A + (size_t)(i0 + t / BK) * n + t % BK;
  const size_t step_k = (size_t)(T / TE) * n, step_i = (size_t)(T / BK) * n, adv = (size_t)BK * n;
  unsigned amask = 0u;
#pragma unroll
  for (int e = 0; e < EL; ++e) amask |= (i0 + t / BK + e * (T / BK) < n ? 1u : 0u) << e;
  float ra[EL], rb[EL];
  auto load = [&](int k0) {
    const bool whole = k0 + BK <= n;
#pragma unroll
    for (int e = 0; e < EL; ++e) {
      const bool kok = whole || k0 + t / TE + e * (T / TE) < n;
      if (ta)
        ra[e] = rok && kok ? pa[e * step_k] : 0.0f;
      else
        ra[e] = ((amask >> e) & 1u) && (whole || k0 + t % BK < n) ? pa[e * step_i] : 0.0f;
      rb[e] = cok && kok ? pb[e * step_k] : 0.0f;
    }
    pa += ta ? adv : BK;
    pb += adv;
  };
  auto store = [&](int b) {
#pragma unroll
    for (int e = 0; e < EL; ++e) {
      if (ta)
        As[b][t / TE + e * (T / TE)][t % TE] = ra[e];
      else
        As[b][t % BK][t / BK + e * (T / BK)] = ra[e];
      Bs[b][t / TE + e * (T / TE)][t % TE] = rb[e];
    }
  };
  f32x2 acc[RM / 2][RN];
#pragma unroll
  for (int r = 0; r < RM / 2; ++r)
#pragma unroll
    for (int c = 0; c < RN; ++c) acc[r][c] = pack2(0.0f, 0.0f);
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < n; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < n;
    if (more) load(k0 + BK);
    f32x2 a[2][RM / 2], b[2][RN];
    auto frag = [&](int kk, int f) {
#pragma unroll
      for (int r = 0; r < RM / 4; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(&As[buf][kk][ty * RM + 4 * r]);
        a[f][2 * r] = pack2(v.x, v.y);
        a[f][2 * r + 1] = pack2(v.z, v.w);
      }
      const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * RN]);
      b[f][0] = pack2(v.x, v.x);
      b[f][1] = pack2(v.y, v.y);
      b[f][2] = pack2(v.z, v.z);
      b[f][3] = pack2(v.w, v.w);
    };
    frag(0, 0);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      if (kk + 1 < BK) frag(kk + 1, (kk + 1) & 1);
#pragma unroll
      for (int r = 0; r < RM / 2; ++r)
#pragma unroll
        for (int c = 0; c < RN; ++c) acc[r][c] = fma2(a[kk & 1][r], b[kk & 1][c], acc[r][c]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
  }
  double ss = 0.0;
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    const int i = i0 + ty * RM + r;
    if (i >= n) continue;
#pragma unroll
    for (int c = 0; c < RN; ++c) {
      const int j = j0 + tx * RN + c;
      if (j >= n || (g.sym && j < i)) continue;  // the (j, i) entry is written by the tile that owns it
      float x0, x1;
      unpack2(acc[r / 2][c], x0, x1);
      const float x = r % 2 ? x1 : x0;
      float v;
      if (g.resid) {
        v = (i == j ? 1.0f : 0.0f) - x;
        ss += (i == j ? 1.0 : 2.0) * (double)v * (double)v;
      } else {
        v = (float)g.beta * x;
        if (g.Add) v = fmaf((float)g.alpha, g.Add[(size_t)i * n + j], v);
        if (g.P) {
          g.P[(size_t)i * n + j] = x;
          if (g.sym && j != i) g.P[(size_t)j * n + i] = x;
        }
      }
      g.C[(size_t)i * n + j] = v;
      if (g.sym && j != i) g.C[(size_t)j * n + i] = v;
    }
  }
  if (g.resid) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    if ((t & 31) == 0) red[t >> 5] = ss;
    __syncthreads();
    if (t == 0) {
      double s = 0.0;
      for (int w = 0; w < T / 32; ++w) s += red[w];
      g.partials[blockIdx.x] = s;
    }
  }
}

}  // namespace

int f64_num_blocks(int n, bool sym, bool fp32) {
  const int te = tile_for(n, fp32);
  const int T = (n + te - 1) / te;
  return sym ? T * (T + 1) / 2 : T * T;
}

static dim3 grid_of(int n, bool sym, int te) {
  const int tb = (n + te - 1) / te;
  return sym ? dim3(tb * (tb + 1) / 2) : dim3(tb, tb);
}

cudaError_t launch_f64_gemm(const F64Gemm& g, cudaStream_t s) {
  const int te = tile_for(g.n);
  if (te == 32)
    k64_gemm<32><<<grid_of(g.n, g.sym, te), NT, 0, s>>>(g);
  else
    k64_gemm<64><<<grid_of(g.n, g.sym, te), NT, 0, s>>>(g);
  return cudaGetLastError();
}

cudaError_t launch_f32_gemm(const F32Gemm& g, cudaStream_t s) {
  k32_gemm<<<grid_of(g.n, g.sym, tile_for(g.n, true)), 128, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace zf
