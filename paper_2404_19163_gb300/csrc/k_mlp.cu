// Learned start proposal (not in the paper; its warm-start motivation is Sec. 6):
// features of an overlap matrix and a 16 -> 64 -> 64 -> 5 GELU MLP (FP32) with its
// forward, backward and Adam kernels.  Gradients are reduced over the batch in a fixed
// order (per chunk of samples and per parameter the sum over the chunk, then over the chunks), so training is
// deterministic.
#include <math.h>

#include "mlp.h"

namespace zf {
namespace {

constexpr int I0 = 16, H = 64, O = 5;
// per-sample values (feature index of each block) a block keeps in shared memory, and its samples
constexpr int A_X = 0, A_GZ1 = A_X + I0, A_H1 = A_GZ1 + H, A_GZ2 = A_H1 + H, A_H2 = A_GZ2 + H, A_GY = A_H2 + H,
              A_N = A_GY + O;
constexpr int kChunk = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + H * I0, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H,
              OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + O * H, NPAR = OFF_B3 + O;
static_assert(NPAR == kMlpParams, "parameter layout");

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

constexpr int kPitch = kChunk + 4;     // feature f of sample q at F[f * kPitch + q]: 16-byte rows, distinct banks
constexpr int kParFloats = NPAR + 3;   // parameters, padded to 16 bytes
constexpr int kMlpSmem = (kParFloats + A_N * kPitch) * (int)sizeof(float) + kChunk * (int)sizeof(double);

// A block takes a chunk of 64 samples through the forward pass and, with TRAIN, through the gradient of
// l_b = (y0 - t)^2 + w CE(softmax(y1..4), m) divided by the batch size, and sums every parameter's gradient over
// the chunk in sample order (part), and the losses (lpart).  Parameters and the chunk's values stay in shared
// memory.  A thread holds 16 neurons of one sample (weights are broadcast reads of 16 bytes, values one
// conflict-free read for 16 FMAs) and a 4 x 4 tile of a weight gradient (8 reads of 16 bytes for 64 FMAs).
// Bound: FP32 issue and latency at two blocks an SM.  One thread a sample with its values in local memory, whose
// factors went out (22 MB) and back in by a second kernel, and a serial chain of 5440 FMAs for a single sample, took
// 241 us for a training step over 20000 rows (130 now) and 304 us for a proposal at N = 1500 (168 now).
template <bool TRAIN>
__global__ void __launch_bounds__(256, 2)
    k_mlp(const float* __restrict__ P, const float* __restrict__ mean, const float* __restrict__ stdv,
          const float* __restrict__ X, int batch, float* __restrict__ Y, const float* __restrict__ tgt,
          const int* __restrict__ ord, float w, float* __restrict__ part, double* __restrict__ lpart) {
  extern __shared__ __align__(16) float sm[];
  float* F = sm + kParFloats;
  double* ls = reinterpret_cast<double*>(F + A_N * kPitch);
  const int tid = threadIdx.x, q = tid & 63, n0 = (tid >> 6) * 16;  // sample; first of the thread's 16 neurons
  const int b0 = blockIdx.x * kChunk, nb = min(kChunk, batch - b0);
  for (int e = tid; e < NPAR; e += 256) sm[e] = P[e];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int f = n0 / 4 + k;
    F[(A_X + f) * kPitch + q] = q < nb ? (X[(size_t)(b0 + q) * I0 + f] - mean[f]) / stdv[f] : 0.0f;
  }
  __syncthreads();
  float g1[16], g2[16];  // GELU's derivatives at the thread's neurons
  {
    float x[I0];
#pragma unroll
    for (int k = 0; k < I0; ++k) x[k] = F[(A_X + k) * kPitch + q];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int j = n0 + r;
      float s = sm[OFF_B1 + j];
#pragma unroll
      for (int k = 0; k < I0; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&sm[OFF_W1 + j * I0 + k]);
        s = fmaf(v.w, x[k + 3], fmaf(v.z, x[k + 2], fmaf(v.y, x[k + 1], fmaf(v.x, x[k], s))));
      }
      F[(A_H1 + j) * kPitch + q] = gelu(s);
      if (TRAIN) g1[r] = gelu_grad(s);
    }
  }
  __syncthreads();
  {
    float z[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) z[r] = sm[OFF_B2 + n0 + r];
#pragma unroll 2
    for (int k = 0; k < H; k += 4) {
      float h[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) h[x] = F[(A_H1 + k + x) * kPitch + q];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const float4 v = *reinterpret_cast<const float4*>(&sm[OFF_W2 + (n0 + r) * H + k]);
        z[r] = fmaf(v.w, h[3], fmaf(v.z, h[2], fmaf(v.y, h[1], fmaf(v.x, h[0], z[r]))));
      }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      F[(A_H2 + n0 + r) * kPitch + q] = gelu(z[r]);
      if (TRAIN) g2[r] = gelu_grad(z[r]);
    }
  }
  __syncthreads();
  for (int e = tid; e < O * kChunk; e += 256) {
    const int o = e / kChunk, b = e % kChunk;
    float s = sm[OFF_B3 + o];
#pragma unroll 16
    for (int k = 0; k < H; ++k) s = fmaf(sm[OFF_W3 + o * H + k], F[(A_H2 + k) * kPitch + b], s);
    if (TRAIN) F[(A_GY + o) * kPitch + b] = s;
    if (Y && b < nb) Y[(size_t)(b0 + b) * O + o] = s;
  }
  if (!TRAIN) return;
  __syncthreads();
  if (tid < kChunk) {
    // loss and output gradient (samples past the batch: none)
    float y[O], gy[O];
#pragma unroll
    for (int o = 0; o < O; ++o) {
      y[o] = F[(A_GY + o) * kPitch + q];
      gy[o] = 0.0f;
    }
    if (q < nb) {
      const float r = y[0] - tgt[b0 + q];
      float mx = y[1];
#pragma unroll
      for (int k = 2; k < O; ++k) mx = fmaxf(mx, y[k]);
      float e[O - 1], se = 0.0f;
#pragma unroll
      for (int k = 0; k < O - 1; ++k) {
        e[k] = expf(y[1 + k] - mx);
        se += e[k];
      }
      const int m = ord[b0 + q];
      float ym = 0.0f;
#pragma unroll
      for (int k = 0; k < O - 1; ++k)
        if (k == m) ym = y[1 + k];
      ls[q] = (double)(r * r) + (double)w * ((double)logf(se) + (double)mx - (double)ym);
      const float inv_b = 1.0f / (float)batch;
      gy[0] = 2.0f * r * inv_b;
#pragma unroll
      for (int k = 0; k < O - 1; ++k) gy[1 + k] = w * (e[k] / se - (k == m ? 1.0f : 0.0f)) * inv_b;
    }
#pragma unroll
    for (int o = 0; o < O; ++o) F[(A_GY + o) * kPitch + q] = gy[o];
  }
  __syncthreads();
  {
    float gy[O];
#pragma unroll
    for (int o = 0; o < O; ++o) gy[o] = F[(A_GY + o) * kPitch + q];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      float s = 0.0f;
#pragma unroll
      for (int o = 0; o < O; ++o) s = fmaf(sm[OFF_W3 + o * H + n0 + r], gy[o], s);
      F[(A_GZ2 + n0 + r) * kPitch + q] = s * g2[r];
    }
  }
  __syncthreads();
  {
    float s[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) s[r] = 0.0f;
#pragma unroll 4
    for (int j = 0; j < H; ++j) {
      const float g = F[(A_GZ2 + j) * kPitch + q];
#pragma unroll
      for (int r = 0; r < 16; r += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&sm[OFF_W2 + j * H + n0 + r]);
        s[r] = fmaf(v.x, g, s[r]);
        s[r + 1] = fmaf(v.y, g, s[r + 1]);
        s[r + 2] = fmaf(v.z, g, s[r + 2]);
        s[r + 3] = fmaf(v.w, g, s[r + 3]);
      }
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) F[(A_GZ1 + n0 + r) * kPitch + q] = s[r] * g1[r];
  }
  __syncthreads();
  // the gradients: sum_b row(a)[b] row(c)[b] over the chunk's samples in order
  float* out = part + (size_t)blockIdx.x * NPAR;
  const int jt = tid >> 4, it = tid & 15, full = nb & ~3;
  {
    float s[4][4] = {}, t[4] = {};
    for (int b = 0; b < full; b += 4) {
      float4 a[4], c[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        a[r] = *reinterpret_cast<const float4*>(&F[(A_GZ2 + jt + 16 * r) * kPitch + b]);
        c[r] = *reinterpret_cast<const float4*>(&F[(A_H1 + it + 16 * r) * kPitch + b]);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int x = 0; x < 4; ++x)
          s[r][x] = fmaf(a[r].w, c[x].w, fmaf(a[r].z, c[x].z, fmaf(a[r].y, c[x].y, fmaf(a[r].x, c[x].x, s[r][x]))));
      const float4 xv = *reinterpret_cast<const float4*>(&F[(A_X + it) * kPitch + b]);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float4 g = *reinterpret_cast<const float4*>(&F[(A_GZ1 + jt + 16 * r) * kPitch + b]);
        t[r] = fmaf(g.w, xv.w, fmaf(g.z, xv.z, fmaf(g.y, xv.y, fmaf(g.x, xv.x, t[r]))));
      }
    }
    for (int b = full; b < nb; ++b)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
#pragma unroll
        for (int x = 0; x < 4; ++x)
          s[r][x] = fmaf(F[(A_GZ2 + jt + 16 * r) * kPitch + b], F[(A_H1 + it + 16 * x) * kPitch + b], s[r][x]);
        t[r] = fmaf(F[(A_GZ1 + jt + 16 * r) * kPitch + b], F[(A_X + it) * kPitch + b], t[r]);
      }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
#pragma unroll
      for (int x = 0; x < 4; ++x) out[OFF_W2 + (jt + 16 * r) * H + it + 16 * x] = s[r][x];
      out[OFF_W1 + (jt + 16 * r) * I0 + it] = t[r];
    }
  }
  for (int e = tid; e < O * H; e += 256) {
    const float *a = &F[(A_GY + e / H) * kPitch], *c = &F[(A_H2 + e % H) * kPitch];
    float s = 0.0f;
    for (int b = 0; b < nb; ++b) s = fmaf(a[b], c[b], s);
    out[OFF_W3 + e] = s;
  }
  if (tid < 2 * H + O) {
    const int f = tid < H ? A_GZ1 + tid : tid < 2 * H ? A_GZ2 + tid - H : A_GY + tid - 2 * H;
    float s = 0.0f;
    for (int b = 0; b < nb; ++b) s += F[f * kPitch + b];
    out[tid < H ? OFF_B1 + tid : tid < 2 * H ? OFF_B2 + tid - H : OFF_B3 + tid - 2 * H] = s;
  }
  if (tid == 255) {
    double l = 0.0;
    for (int b = 0; b < nb; ++b) l += ls[b];
    lpart[blockIdx.x] = l;
  }
}

// grad[p] = sum over chunks of the chunk sums, in chunk order; the last block: loss = the mean of the losses.
// 16 loads in flight a thread (the sum itself is a chain).
__global__ void __launch_bounds__(64) k_mlp_reduce(const float* __restrict__ part, int nchunks, int batch,
                                                   float* __restrict__ grad, const double* __restrict__ lpart,
                                                   double* __restrict__ loss_out) {
  if (blockIdx.x == gridDim.x - 1) {
    if (threadIdx.x != 0 || !loss_out) return;
    double l = 0.0;
#pragma unroll 16
    for (int c = 0; c < nchunks; ++c) l += lpart[c];
    *loss_out = l / batch;
    return;
  }
  const int p = blockIdx.x * 64 + threadIdx.x;
  if (p >= NPAR) return;
  float s = 0.0f;
#pragma unroll 16
  for (int c = 0; c < nchunks; ++c) s += part[(size_t)c * NPAR + p];
  grad[p] = s;
}

__global__ void k_adam(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M,
                       float* __restrict__ V, int n, float c1, float c2, float lr, float b1, float b2, float eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float g = G[i];
  const float m = b1 * M[i] + (1.0f - b1) * g;
  const float v = b2 * V[i] + (1.0f - b2) * g * g;
  M[i] = m;
  V[i] = v;
  P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

// ---- features
// Per row r: diagonal, off-diagonal absolute sum, absolute row sum.
__global__ void k_feat_rows(const double* __restrict__ S, int n, double* __restrict__ rows) {
  const int r = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= n) return;
  double s = 0.0;
  for (int c = lane; c < n; c += 32) s += fabs(S[(size_t)r * n + c]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) {
    const double d = S[(size_t)r * n + r];
    rows[3 * r] = d;
    rows[3 * r + 1] = s - fabs(d);
    rows[3 * r + 2] = s;
  }
}

// Row statistics in a fixed order: st[0] g_hi, st[1] g_lo, st[2] mean d, st[3] min d,
// st[4] mean row sum, st[5] min row sum.
__global__ void k_feat_rowstats(const double* __restrict__ rows, int n, double* st) {
  __shared__ double sh[6][256];
  double ghi = -INFINITY, glo = INFINITY, sd = 0, md = INFINITY, sr = 0, mr = INFINITY;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const double d = rows[3 * r], off = rows[3 * r + 1], rs = rows[3 * r + 2];
    ghi = fmax(ghi, d + off);
    glo = fmin(glo, d - off);
    sd += d;
    md = fmin(md, d);
    sr += rs;
    mr = fmin(mr, rs);
  }
  sh[0][threadIdx.x] = ghi;
  sh[1][threadIdx.x] = glo;
  sh[2][threadIdx.x] = sd;
  sh[3][threadIdx.x] = md;
  sh[4][threadIdx.x] = sr;
  sh[5][threadIdx.x] = mr;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      sh[0][threadIdx.x] = fmax(sh[0][threadIdx.x], sh[0][threadIdx.x + w]);
      sh[1][threadIdx.x] = fmin(sh[1][threadIdx.x], sh[1][threadIdx.x + w]);
      sh[2][threadIdx.x] += sh[2][threadIdx.x + w];
      sh[3][threadIdx.x] = fmin(sh[3][threadIdx.x], sh[3][threadIdx.x + w]);
      sh[4][threadIdx.x] += sh[4][threadIdx.x + w];
      sh[5][threadIdx.x] = fmin(sh[5][threadIdx.x], sh[5][threadIdx.x + w]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    st[0] = sh[0][0];
    st[1] = sh[1][0];
    st[2] = sh[2][0] / n;
    st[3] = sh[3][0];
    st[4] = sh[4][0] / n;
    st[5] = sh[5][0];
  }
}

// E = d0 - t1 I = (1 - t1) I - S / g_hi, with t1 = tr(d0)/N = 1 - mean(S_ii)/g_hi: the spectrum of
// d0 centred, so that the central moments tr(E^k)/N come out without cancellation.
// With max |E_ij| (the bits of a double, a NaN above Inf; the caller zeroes it).
__global__ void k_feat_d0(const double* __restrict__ S, int n, const double* __restrict__ st, double* __restrict__ D0,
                          unsigned long long* amax) {
  __shared__ double c[2];  // (an FP64 division in every thread would take longer than the pass)
  if (threadIdx.x == 0) {
    c[0] = 1.0 / st[0];
    c[1] = 1.0 - st[2] * c[0];
  }
  __syncthreads();
  unsigned long long m = 0ull;
  const double inv = c[0], t1 = c[1];
  for (int i = blockIdx.y; i < n; i += gridDim.y) {
    const double* r = S + (size_t)i * n;
#pragma unroll 4
    for (int j = blockIdx.x * 256 + threadIdx.x; j < n; j += gridDim.x * 256) {
      const double x = (i == j ? 1.0 - t1 : 0.0) - r[j] * inv;
      D0[(size_t)i * n + j] = x;
      m = max_bits(m, abs_bits(x));
    }
  }
  block_raise_max(amax, m);
}

// Per-block partial sums of tr E, sum E^2, sum (E^2) o E, sum (E^2)^2 (E symmetric, P = E^2).
__global__ void k_feat_traces(const double* __restrict__ D0, const double* __restrict__ P, int n,
                              double* __restrict__ part) {
  __shared__ double sh[4][256];
  double a = 0, b = 0, c = 0, d = 0;
  const size_t total = (size_t)n * n, stride = (size_t)gridDim.x * blockDim.x;
  const size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (size_t r = t; r < (size_t)n; r += stride) a += D0[r * (n + 1)];
  for (size_t e = t; e < total; e += stride) {
    const double x = D0[e], p = P[e];
    b = fma(x, x, b);
    c = fma(p, x, c);
    d = fma(p, p, d);
  }
  sh[0][threadIdx.x] = a;
  sh[1][threadIdx.x] = b;
  sh[2][threadIdx.x] = c;
  sh[3][threadIdx.x] = d;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int q = 0; q < 4; ++q) part[4 * blockIdx.x + q] = sh[q][0];
}

// The block partials summed in a fixed order (thread t takes blocks t, t + 256, ..., then a tree), and
// the 16 features.
__global__ void __launch_bounds__(256) k_feat_final(const double* __restrict__ part, int nblocks,
                                                    const double* __restrict__ st, int n, float* __restrict__ f) {
  __shared__ double sh[4][256];
  double v[4] = {0, 0, 0, 0};
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x)
    for (int q = 0; q < 4; ++q) v[q] += part[4 * b + q];
  for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w)
      for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + w];
    __syncthreads();
  }
  // a feature and the one eight after it to each warp (in one thread, the 16 features' FP64 divisions, roots and
  // logarithms are one chain)
  if (threadIdx.x & 31) return;
  const double g = st[0];
  // central moments of the spectrum of d0 from E = d0 - t1 I, then the raw moments t_k
  auto t1 = [&] { return 1.0 - st[2] / g; };
  auto m = [&](int k) { return sh[k - 1][0] / n; };
  auto t2 = [&] { return m(2) + t1() * t1(); };
  const int q = threadIdx.x >> 5;
  switch (q) {
    case 0:
      f[0] = (float)log((double)n);
      f[8] = (float)t2();
      break;
    case 1: {
      const double t = t1(), m2 = m(2);
      f[1] = (float)log(g);
      f[9] = (float)(m(3) + 3 * t * m2 + t * t * t);
      break;
    }
    case 2: {
      const double t = t1(), m2 = m(2), m3 = m(3);
      f[2] = (float)(st[1] / g);
      f[10] = (float)(m(4) + 4 * t * m3 + 6 * t * t * m2 + t * t * t * t);
      break;
    }
    case 3:
      f[3] = (float)(st[2] / g);
      f[11] = (float)sqrt(t2());
      break;
    case 4:
      f[4] = (float)(st[3] / g);
      f[12] = (float)m(2);
      break;
    case 5:
      f[5] = (float)(st[4] / g);
      f[13] = (float)m(3);
      break;
    case 6:
      f[6] = (float)(st[5] / g);
      f[14] = (float)m(4);
      break;
    default:
      f[7] = (float)t1();
      f[15] = (float)log(sqrt(t2() * n));
      break;
  }
}

}  // namespace

int mlp_chunks(int batch) { return (batch + kChunk - 1) / kChunk; }

cudaError_t launch_mlp(const float* P, const float* mean, const float* stdv, const float* X, int batch, float* Y,
                       cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmem);
  if (e != cudaSuccess) return e;
  k_mlp<false><<<mlp_chunks(batch), 256, kMlpSmem, s>>>(P, mean, stdv, X, batch, Y, nullptr, nullptr, 0.0f, nullptr,
                                                        nullptr);
  return cudaGetLastError();
}

cudaError_t launch_mlp_backward(const float* P, const float* mean, const float* stdv, const float* X, int batch,
                                const float* tgt, const int* ord, float w, float* part, double* lpart, float* grad,
                                double* loss, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmem);
  if (e != cudaSuccess) return e;
  const int nc = mlp_chunks(batch);
  k_mlp<true><<<nc, 256, kMlpSmem, s>>>(P, mean, stdv, X, batch, nullptr, tgt, ord, w, part, lpart);
  k_mlp_reduce<<<(NPAR + 63) / 64 + 1, 64, 0, s>>>(part, nc, batch, grad, lpart, loss);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* P, const float* G, float* M, float* V, int n, int step, float lr, float b1, float b2,
                        float eps, cudaStream_t s) {
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adam<<<(n + 255) / 256, 256, 0, s>>>(P, G, M, V, n, c1, c2, lr, b1, b2, eps);
  return cudaGetLastError();
}

cudaError_t launch_feat_rows(const double* S, int n, double* rows, double* st, cudaStream_t s) {
  k_feat_rows<<<(n + 7) / 8, 256, 0, s>>>(S, n, rows);
  k_feat_rowstats<<<1, 256, 0, s>>>(rows, n, st);
  return cudaGetLastError();
}

cudaError_t launch_feat_d0(const double* S, int n, const double* st, double* D0, unsigned long long* amax,
                           cudaStream_t s) {
  k_feat_d0<<<dim3((n + 1023) / 1024, n < 2048 ? n : 2048), 256, 0, s>>>(S, n, st, D0, amax);
  return cudaGetLastError();
}

int feat_trace_blocks(int n) {
  const size_t total = (size_t)n * n;
  return (int)((total + 255) / 256 < 1024 ? (total + 255) / 256 : 1024);
}

cudaError_t launch_feat_traces(const double* D0, const double* P, int n, double* part, const double* st, float* f,
                               cudaStream_t s) {
  const int nb = feat_trace_blocks(n);
  k_feat_traces<<<nb, 256, 0, s>>>(D0, P, n, part);
  k_feat_final<<<1, 256, 0, s>>>(part, nb, st, n, f);
  return cudaGetLastError();
}

}  // namespace zf
