// tcgen05 GEMM engine for the recursion's products on GB300 (sm_103a).
//
// Persistent CTAs (or CTA pairs) walk a list of output tiles.  Warp 0 streams K-blocks of the operands
// into a ring of shared-memory stages with TMA (128-byte swizzle); one thread of warp 1 issues tcgen05.mma
// (kind::f16, FP32 accumulation in tensor memory) and releases each stage with tcgen05.commit; warps 2-9
// read the accumulator back with tcgen05.ld and run the fused epilogue while the next tile accumulates in
// the other half of the tensor memory (two accumulator buffers).  Two epilogue warps share each 32-lane
// quadrant of the accumulator (a warp may only read its own quadrant), one for each half of the tile's
// columns.  Each epilogue is its own instantiation of the kernel, so no epilogue pays for another's
// registers.
//
// Tiles (tc_pick_tile chooses): 256 x 256 formed by a pair of CTAs (cta_group::2: each CTA holds 128 rows
// of the accumulator and loads 128 rows of A and half of B's rows; rank 0 issues the instructions), and
// 128 x 128, 128 x 64 and 128 x 32 by one CTA, for products with too few wide tiles to fill the SMs.  A
// 128 x 256 tile of one CTA asks shared memory for 192 bytes per clock (operand reads and TMA writes)
// where it gives 128; the pair halves B's share.  Residue products at N = 4096: 1748 TFLOP/s on 128 x 256
// tiles, 2263 on the pair's; the split Z^T S: 1525 and 1877 (3.37 rounds of tiles, so 2230 within a
// round).  256 x 128 tiles of a pair were no faster than 128 x 128 of one CTA.  At N = 256 the residual and
// update epilogues took 39 and 33 us on two 128 x 256 tiles and take 14 us on 32-wide ones.
// Every tile shape adds the K-blocks of an entry in the same order, so the results do not depend on it.
//
// Epilogues write through a 4 KiB buffer per warp, so that global accesses run along rows (full sectors)
// although a thread holds a row of the accumulator; transposed and mirrored copies go out from registers,
// where neighbouring lanes are neighbouring addresses (16-bit ones as pairs).
//
// A product may consist of up to four K-concatenated segments accumulated
// into one accumulator: the split scheme (h)(h)+(h)(l)+(l)(h) of Sec. 3.2
// (Eqs. SZn, Xn, Xsq) is three segments.  Symmetric products (X = Z^T S Z and
// the powers of d) form only the tiles that touch the upper triangle and
// write every entry (i, j), i <= j, to both (i, j) and (j, i).
//
// Every wait on an mbarrier is bounded; a wait that gives up raises a flag in
// the device state and the CTA winds down (no trap).
#pragma once
#include <stdio.h>

#include "crt_wide.h"
#include "tc_gemm.h"

namespace zf {
namespace {

constexpr int BM = 128, BK = 64, UK = 16, NEPI_WARPS = 8, NTHREADS = 64 + 32 * NEPI_WARPS;
constexpr int EPI_WARP_BYTES = 4096;  // staging buffer of one epilogue warp: 32 rows of 128 bytes

// CG CTAs form a tile of 128 CG x BN.
template <int BN, int CG>
struct Cfg {
  static constexpr int A_BYTES = BM * BK * 2;
  static constexpr int B_ROWS = BN / CG;
  static constexpr int B_BYTES = B_ROWS * BK * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int STAGES = STAGE > 24576 ? 6 : 8;
  static constexpr int TMEM_COLS = 2 * BN;
  static constexpr int SMEM = STAGES * STAGE + NEPI_WARPS * EPI_WARP_BYTES + 1024 + 256;
  static constexpr int NCHUNK = BN / 32;                 // 32-column chunks of a tile
  static constexpr int HCHUNK = (NCHUNK + 1) / 2;        // chunks per column half
};

__host__ __device__ inline int tiles_of(int M, int N, int sym, int bm_size, int bn_size) {
  const int tm = (M + bm_size - 1) / bm_size, tn = (N + bn_size - 1) / bn_size;
  if (!sym) return tm * tn;
  int total = 0;
  for (int r = 0; r < tm; ++r) total += tn - (r * bm_size) / bn_size;
  return total;
}

__host__ __device__ inline int units_of(const TcArgs& a, int bm_size, int bn_size) {
  if (a.ninst > 0) return a.M;  // grouped: total units passed in M by the host
  const int t = tiles_of(a.M, a.N, a.sym, bm_size, bn_size);
  return a.oz_s > 0 ? t * a.oz_s * a.oz_nch : t;
}

// Work of one unit: `npairs` operand pairs over K-blocks [kb0, kb1) of the output tile `tile`
// of a problem of size n whose rows start at row0 (grouped mode) or 0.
struct UnitPlan {
  int tile, group, npairs, p0, t, kb0, kb1;
  int inst, n, row0, skip;
};

template <int BN, int CG>
__device__ __forceinline__ UnitPlan plan_unit(int u, const TcArgs& a, int kblocks_all) {
  UnitPlan pl;
  pl.inst = 0;
  pl.row0 = 0;
  pl.n = a.N;
  pl.skip = 0;
  int kblocks = kblocks_all;
  if (a.ninst > 0) {
    int lo = 0, hi = a.ninst - 1;  // slot j with g_prefix[j] <= u < g_prefix[j+1]
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.g_prefix[mid] <= u)
        lo = mid;
      else
        hi = mid - 1;
    }
    pl.inst = a.g_inst[lo];
    pl.n = a.g_n[pl.inst];
    pl.row0 = a.g_row0[pl.inst];
    pl.skip = (a.g_done && a.g_done[pl.inst]) ? 1 : 0;
    u -= a.g_prefix[lo];
    kblocks = (pl.n + BK - 1) / BK;
  }
  if (a.oz_s > 0) {
    // group-major order: the CTAs running at the same time form different tiles of the same
    // (group, K-chunk) and so read the same slice panels, which then stay in L2
    // (grouped residue products: the instance's own tile count; its units are tiles x moduli x chunks)
    const int ntiles = a.ninst > 0 ? tiles_of(pl.n, pl.n, a.sym, BM * CG, BN) : a.oz_tiles;
    pl.group = u / ntiles;
    pl.tile = u % ntiles;
    pl.t = pl.group / a.oz_nch;
    const int c = pl.group % a.oz_nch;
    if (a.oz_diag) {
      // residue products: group t is the single pair (t, t)
      pl.p0 = pl.t;
      pl.npairs = 1;
    } else {
      pl.p0 = pl.t - (a.oz_s - 1) > 0 ? pl.t - (a.oz_s - 1) : 0;
      const int p1 = pl.t < a.oz_s - 1 ? pl.t : a.oz_s - 1;
      pl.npairs = p1 - pl.p0 + 1;
    }
    pl.kb0 = (a.oz_c0 + c) * a.oz_chunk_kb;
    pl.kb1 = pl.kb0 + a.oz_chunk_kb < kblocks ? pl.kb0 + a.oz_chunk_kb : kblocks;
  } else {
    pl.tile = u;
    pl.group = 0;
    pl.t = 0;
    pl.p0 = 0;
    pl.npairs = a.nseg;
    pl.kb0 = 0;
    pl.kb1 = kblocks;
  }
  return pl;
}

__device__ __forceinline__ void decode_unit(int u, const TcArgs& a, int n_inst, int bm_size, int bn_size, int& bm,
                                            int& bn) {
  const int M = a.ninst > 0 ? n_inst : a.M, N = a.ninst > 0 ? n_inst : a.N;
  const int tm = (M + bm_size - 1) / bm_size, tn = (N + bn_size - 1) / bn_size;
  if (!a.sym) {
    bm = u % tm;
    bn = u / tm;
    return;
  }
  for (int r = 0; r < tm; ++r) {
    const int first = (r * bm_size) / bn_size, cnt = tn - first;
    if (u < cnt) {
      bm = r;
      bn = first + u;
      return;
    }
    u -= cnt;
  }
  bm = tm;
  bn = tn;
}

// ---------------------------------------------------------------- epilogue stores
// The warp's staging buffer holds 32 rows of 128 bytes; 16-byte unit u of row r sits at unit u ^ (r & 7),
// so that both a thread writing its own row and eight threads reading one row touch distinct banks.
__device__ __forceinline__ uint4* stage_unit(uint8_t* st, int r, int u) {
  return reinterpret_cast<uint4*>(st + r * 128 + ((u ^ (r & 7)) << 4));
}

__device__ __forceinline__ uint4 as_uint4(float a, float b, float c, float d) {
  return make_uint4(__float_as_uint(a), __float_as_uint(b), __float_as_uint(c), __float_as_uint(d));
}

// x (the thread's row i0 + lane, 32 columns from col0) into rows of an FP32 matrix, four rows of 128 bytes
// per instruction.  Columns up to col0 + 32 are inside the row (leading dimensions are multiples of 64).
__device__ __forceinline__ void rows32(float* base, int ld, int i0, int nrows, int col0, uint8_t* st, int lane,
                                       const float (&x)[32]) {
#pragma unroll
  for (int u = 0; u < 8; ++u) *stage_unit(st, lane, u) = as_uint4(x[4 * u], x[4 * u + 1], x[4 * u + 2], x[4 * u + 3]);
  __syncwarp();
  const int r0 = lane >> 3, u = lane & 7;
  float* p = base + (size_t)(i0 + r0) * ld + col0 + 4 * u;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if (i0 + r0 + 4 * k < nrows) *reinterpret_cast<uint4*>(p + (size_t)(4 * k) * ld) = *stage_unit(st, r0 + 4 * k, u);
  __syncwarp();
}

// The thread's row of 32 columns of an FP32 matrix (rows past nrows read as 0), read four rows at a time.
__device__ __forceinline__ void load_rows32(const float* base, int ld, int i0, int nrows, int col0, uint8_t* st,
                                            int lane, float (&x)[32]) {
  const int r0 = lane >> 3, u = lane & 7;
  const float* p = base + (size_t)(i0 + r0) * ld + col0 + 4 * u;
  uint4 t[8];
#pragma unroll
  for (int k = 0; k < 8; ++k)
    t[k] = i0 + r0 + 4 * k < nrows ? *reinterpret_cast<const uint4*>(p + (size_t)(4 * k) * ld) : make_uint4(0, 0, 0, 0);
#pragma unroll
  for (int k = 0; k < 8; ++k) *stage_unit(st, r0 + 4 * k, u) = t[k];
  __syncwarp();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const uint4 w = *stage_unit(st, lane, q);
    x[4 * q] = __uint_as_float(w.x);
    x[4 * q + 1] = __uint_as_float(w.y);
    x[4 * q + 2] = __uint_as_float(w.z);
    x[4 * q + 3] = __uint_as_float(w.w);
  }
  __syncwarp();
}

// Element jj of the thread's row i to (col0 + jj, i): 128 consecutive bytes per instruction.
__device__ __forceinline__ void cols32(float* base, int ld, int i, int nrows, int col0, int n, const float (&x)[32]) {
  if (i >= nrows) return;
  float* p = base + (size_t)col0 * ld + i;
#pragma unroll
  for (int jj = 0; jj < 32; ++jj)
    if (col0 + jj < n) p[(size_t)jj * ld] = x[jj];
}

// 16-bit hi (and lo) values, packed two columns to a word, into rows.
__device__ __forceinline__ void rows16(uint16_t* bh, uint16_t* bl, int ld, int i0, int nrows, int col0, uint8_t* st,
                                       int lane, const uint32_t (&h)[16], const uint32_t (&l)[16]) {
#pragma unroll
  for (int u = 0; u < 4; ++u) *stage_unit(st, lane, u) = make_uint4(h[4 * u], h[4 * u + 1], h[4 * u + 2], h[4 * u + 3]);
  if (bl) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      *stage_unit(st, lane, 4 + u) = make_uint4(l[4 * u], l[4 * u + 1], l[4 * u + 2], l[4 * u + 3]);
    __syncwarp();
    const int r0 = lane >> 3, u = lane & 7;
    uint16_t* p = (u < 4 ? bh : bl) + (size_t)(i0 + r0) * ld + col0 + 8 * (u & 3);
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (i0 + r0 + 4 * k < nrows) *reinterpret_cast<uint4*>(p + (size_t)(4 * k) * ld) = *stage_unit(st, r0 + 4 * k, u);
  } else {
    __syncwarp();
    const int r0 = lane >> 2, u = lane & 3;
    uint16_t* p = bh + (size_t)(i0 + r0) * ld + col0 + 8 * u;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i0 + r0 + 8 * k < nrows) *reinterpret_cast<uint4*>(p + (size_t)(8 * k) * ld) = *stage_unit(st, r0 + 8 * k, u);
  }
  __syncwarp();
}

// The packed 16-bit values transposed: column c of rows i (even), i + 1 as one word of row c.  Neighbouring
// threads exchange halves: the even one stores column 2q, the odd one column 2q + 1.  A pair whose second
// row is past nrows writes that row's value (0) into the row's padding column.
__device__ __forceinline__ void cols16(uint16_t* base, int ld, int i, int nrows, int col0, int n, int lane,
                                       const uint32_t (&w)[16]) {
  const int odd = lane & 1, ie = i & ~1;
  uint16_t* p = base + (size_t)(col0 + odd) * ld + ie;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, w[q], 1);
    const uint32_t v = odd ? __byte_perm(o, w[q], 0x7632) : __byte_perm(w[q], o, 0x5410);
    if (ie < nrows && col0 + 2 * q + odd < n) *reinterpret_cast<uint32_t*>(p + (size_t)(2 * q) * ld) = v;
  }
}

// h = R16(x sc), l = R16(x sc - h), two columns to a word.
__device__ __forceinline__ void split32(const float (&x)[32], float sc, int bf16, bool want_lo, uint32_t (&h)[16],
                                        uint32_t (&l)[16]) {
  if (bf16) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const float a = x[2 * q] * sc, b = x[2 * q + 1] * sc;
      const __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
      h[q] = *reinterpret_cast<const uint32_t*>(&t);
      if (want_lo) {
        const __nv_bfloat162 r =
            __floats2bfloat162_rn(a - __uint_as_float(h[q] << 16), b - __uint_as_float(h[q] & 0xFFFF0000u));
        l[q] = *reinterpret_cast<const uint32_t*>(&r);
      }
    }
  } else {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const float a = x[2 * q] * sc, b = x[2 * q + 1] * sc;
      const __half2 t = __floats2half2_rn(a, b);
      h[q] = *reinterpret_cast<const uint32_t*>(&t);
      if (want_lo) {
        const float2 f = __half22float2(t);
        const __half2 r = __floats2half2_rn(a - f.x, b - f.y);
        l[q] = *reinterpret_cast<const uint32_t*>(&r);
      }
    }
  }
}

// 16 doubles of the thread's row into rows of an FP64 matrix of any leading dimension (columns c0 .. c0 + 15,
// those past n skipped): two rows of 128 bytes per instruction.
__device__ __forceinline__ void rows64(double* base, int ld, int i0, int nrows, int c0, int n, uint8_t* st, int lane,
                                       const double (&x)[16]) {
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    double2 t = make_double2(x[2 * u], x[2 * u + 1]);
    *stage_unit(st, lane, u) = *reinterpret_cast<uint4*>(&t);
  }
  __syncwarp();
  const int r0 = lane >> 4, c = lane & 15;
  double* p = base + (size_t)(i0 + r0) * ld + c0 + c;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int r = r0 + 2 * k;
    const double t = *(reinterpret_cast<const double*>(stage_unit(st, r, c >> 1)) + (c & 1));
    if (i0 + r < nrows && c0 + c < n) p[(size_t)(2 * k) * ld] = t;
  }
  __syncwarp();
}

// Adding and subtracting 1.5 2^23 rounds |x| < 2^22 to the nearest integer.
constexpr float kRint = 12582912.0f;

// One chunk of the epilogue: the warp's rows i0 .. i0 + 31 (row i0 + lane in this thread) and columns
// col0 .. col0 + 31 of an output of nrows x n (instance rows start at row0 of every buffer).  Symmetric
// outputs get chunks on the diagonal (made symmetric here, from their upper half) and above it (mirrored).
template <int EPI>
__device__ __forceinline__ void epi_chunk(const TcArgs& a, uint8_t* stg, int lane, int i0, int col0, float (&v)[32],
                                          double& ss, float& amax, float osc, float us, int uk, int group, int nrows,
                                          int n, int row0) {
  // grouped problems are stacked along rows: shift every output/input base to the instance
  const size_t r16 = (size_t)row0 * a.ld16, r32 = (size_t)row0 * a.ld32, r64 = (size_t)row0 * a.ld64;
  uint16_t* o16h = a.o16h ? a.o16h + r16 : nullptr;
  uint16_t* t16h = a.t16h ? a.t16h + r16 : nullptr;
  float* f32 = a.f32 ? a.f32 + r32 : nullptr;
  double* f64 = a.f64 ? a.f64 + r64 : nullptr;
  const bool lo = a.split_out != 0;
  uint16_t* o16l = lo && a.o16l ? a.o16l + r16 : nullptr;
  uint16_t* t16l = lo && a.t16l ? a.t16l + r16 : nullptr;
  const int i = i0 + lane;
  const bool sym = a.sym != 0, mirror = sym && col0 > i0;
  uint32_t h[16], l[16];
  // rows and columns past the matrix hold zeros (a NaN of the operands would reach them through 0 x NaN):
  // padding columns of the outputs are written with them
  if (i0 + 32 > nrows || col0 + 32 > n) {
#pragma unroll
    for (int jj = 0; jj < 32; ++jj)
      if (i >= nrows || col0 + jj >= n) v[jj] = 0.0f;
  }
  if (EPI != kEpiG32 && sym && col0 == i0) {
    // the diagonal chunk: entry (i, j), j < i, from (j, i)
#pragma unroll
    for (int u = 0; u < 8; ++u)
      *stage_unit(stg, lane, u) = as_uint4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
    __syncwarp();
#pragma unroll
    for (int jj = 0; jj < 32; ++jj) {
      const float t = *(reinterpret_cast<const float*>(stage_unit(stg, jj, lane >> 2)) + (lane & 3));
      if (jj < lane) v[jj] = t;
    }
    __syncwarp();
  }
  switch (EPI) {
    case kEpiStore16: {
#pragma unroll
      for (int jj = 0; jj < 32; ++jj) v[jj] *= us;
      split32(v, osc, a.bf16, lo, h, l);
      rows16(o16h, o16l, a.ld16, i0, nrows, col0, stg, lane, h, l);
      break;
    }
    case kEpiResid: {
      // the chunk's sum of squares in FP32 (32 terms: relative error below 2^-19), then one FP64 add:
      // GB300's FP64 pipe would otherwise set the pace of this epilogue
      float cs = 0.0f;
#pragma unroll
      for (int jj = 0; jj < 32; ++jj) {
        const int j = col0 + jj;
        const float d = (i == j && i < nrows ? 1.0f : 0.0f) - v[jj] * us;
        v[jj] = d;
        if (j < n && j >= i) {
          cs = fmaf(i == j ? d : 2.0f * d, d, cs);
          amax = fmaxf(amax, fabsf(d));
        }
      }
      ss += (double)cs;
      rows32(f32, a.ld32, i0, nrows, col0, stg, lane, v);
      if (mirror) cols32(f32, a.ld32, i, nrows, col0, n, v);
      if (o16h) {
        split32(v, osc, a.bf16, lo, h, l);
        rows16(o16h, o16l, a.ld16, i0, nrows, col0, stg, lane, h, l);
        if (mirror) cols16(o16h, a.ld16, i, nrows, col0, n, lane, h);
        if (mirror && o16l) cols16(o16l, a.ld16, i, nrows, col0, n, lane, l);
      }
      break;
    }
    case kEpiPoly: {
      // r = c1 * f32_in + c2 * v: the running sum of c_k d^k.  Outputs: the running sum in
      // FP32 (f32), its 16-bit copy (o16, the final Q), and the raw power v (t16, P_k for
      // the next product of the chain), all at (i, j) and (j, i).
      float r[32];
      load_rows32(a.f32_in + r32, a.ld32, i0, nrows, col0, stg, lane, r);
#pragma unroll
      for (int jj = 0; jj < 32; ++jj) {
        v[jj] *= us;
        r[jj] = col0 + jj < n ? a.c1 * r[jj] + a.c2 * v[jj] : 0.0f;
      }
      if (f32) {
        rows32(f32, a.ld32, i0, nrows, col0, stg, lane, r);
        if (mirror) cols32(f32, a.ld32, i, nrows, col0, n, r);
      }
      if (o16h) {
        split32(r, osc, a.bf16, lo, h, l);
        rows16(o16h, o16l, a.ld16, i0, nrows, col0, stg, lane, h, l);
        if (mirror) cols16(o16h, a.ld16, i, nrows, col0, n, lane, h);
        if (mirror && o16l) cols16(o16l, a.ld16, i, nrows, col0, n, lane, l);
      }
      if (t16h) {
        split32(v, a.p_scale ? *a.p_scale : 1.0f, a.bf16, lo, h, l);
        rows16(t16h, t16l, a.ld16, i0, nrows, col0, stg, lane, h, l);
        if (mirror) cols16(t16h, a.ld16, i, nrows, col0, n, lane, h);
        if (mirror && t16l) cols16(t16l, a.ld16, i, nrows, col0, n, lane, l);
      }
      break;
    }
    case kEpiZupd: {
      float zo[32];
      load_rows32(f32, a.ld32, i0, nrows, col0, stg, lane, zo);
#pragma unroll
      for (int jj = 0; jj < 32; ++jj) {
        const float z = (col0 + jj < n) ? zo[jj] + v[jj] * us : 0.0f;
        v[jj] = z;
        amax = fmaxf(amax, fabsf(z));
      }
      rows32(f32, a.ld32, i0, nrows, col0, stg, lane, v);
      split32(v, osc, a.bf16, lo, h, l);
      rows16(o16h, o16l, a.ld16, i0, nrows, col0, stg, lane, h, l);
      cols16(t16h, a.ld16, i, nrows, col0, n, lane, h);
      if (t16l) cols16(t16l, a.ld16, i, nrows, col0, n, lane, l);
      break;
    }
    case kEpiF64: {
      const double* fin = a.f64_in ? a.f64_in + r64 : nullptr;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int c0 = col0 + 16 * p;
        double x[16];
        if (uk > -1000) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) x[jj] = widen_pow2(v[16 * p + jj], uk);
        } else {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) x[jj] = (double)v[16 * p + jj] * (double)us;
        }
        if (fin) {
          // f64_in is symmetric (as the output is): entry (j, i) for (i, j), along rows of neighbouring threads
          double d[16];
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) d[jj] = (i < nrows && c0 + jj < n) ? fin[(size_t)(c0 + jj) * a.ld64 + i] : 0.0;
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) x[jj] = fma((double)a.c1, d[jj], (double)a.c2 * x[jj]);
        }
        rows64(f64, a.ld64, i0, nrows, c0, n, stg, lane, x);
        if (mirror && i < nrows) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj)
            if (c0 + jj < n) f64[(size_t)(c0 + jj) * a.ld64 + i] = x[jj];
        }
      }
      break;
    }
    case kEpiG32: {
      rows32(f32 + (size_t)group * a.g_stride, a.ld32, i0, nrows, col0, stg, lane, v);
      break;
    }
    case kEpiZupd64: {
      if (i < nrows) {
        double* zrow = f64 + (size_t)i * a.ld64;
#pragma unroll
        for (int jj = 0; jj < 32; ++jj) {
          const int j = col0 + jj;
          if (j < n) {
            const double z = zrow[j] + (double)v[jj] * (double)us;
            zrow[j] = z;
            amax = fmaxf(amax, fabsf((float)z));
          }
        }
      }
      break;
    }
    default:
      break;
  }
}

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

template <int BN, int CG, int EPI>
__global__ void __launch_bounds__(NTHREADS, 1) k_tc_gemm(const __grid_constant__ TcMaps maps, const TcArgs a) {
  using C = Cfg<BN, CG>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* epi_stage = smem + C::STAGES * C::STAGE;
  uint64_t* full = reinterpret_cast<uint64_t*>(epi_stage + NEPI_WARPS * EPI_WARP_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* done_bar = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done_bar + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)cluster_rank() : 0;
  const int unit0 = blockIdx.x / CG, ustride = gridDim.x / CG;
  const int units = units_of(a, BM * CG, BN);
  const int kblocks = (a.K + BK - 1) / BK;

  // In a pair the leader's (rank 0) full and tempty barriers count both CTAs' transfers and epilogues, and
  // the commits of the leader's instructions arrive at the empty and tfull barriers of both.
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], NEPI_WARPS * CG);
    }
    mbar_init(done_bar, 1);
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc<CG>(tmem_slot, C::TMEM_COLS);
    tmem_relinquish<CG>();
  }
  if (warp == 0 && lane == 0) {
    for (int s = 0; s < a.nseg; ++s) {
      tma_prefetch_desc(&maps.a[s]);
      tma_prefetch_desc(&maps.b[s]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // The streaming and the issuing warp run their loops converged, with one lane elected at each
  // instruction that takes one thread: stages, phases, addresses and descriptors then live in uniform
  // registers, where TMA and tcgen05.mma take their operands.  (As loops of a single thread they cost about 600
  // cycles a K-block, more than the 512 that the widest tile's instructions take.)
  const uint32_t smem0 = smem_u32(smem), full0 = smem_u32(full), empty0 = smem_u32(empty);
  if (warp == 0) {
    uint32_t st = 0, ph = 1;  // ph: parity of the empty barrier to wait for
    // the pair's transfers are counted on the leader's barrier
    const uint32_t sig0 = CG == 2 ? map_rank0(full0) : full0;
    bool ok = true;
    for (int u = unit0; u < units && ok; u += ustride) {
      const UnitPlan pl = plan_unit<BN, CG>(u, a, kblocks);
      if (uniform(pl.skip)) continue;
      int bm, bn;
      decode_unit(pl.tile, a, pl.n, BM * CG, BN, bm, bn);
      const int npairs = uniform(pl.npairs), x0 = uniform(pl.kb0 * BK), x1 = uniform(pl.kb1 * BK);
      const int ra = uniform(pl.row0 + (bm * CG + rank) * BM), rb = uniform(pl.row0 + bn * BN + rank * C::B_ROWS);
      const int p0 = uniform(pl.p0), t = uniform(pl.t);
      for (int pi = 0; pi < npairs && ok; ++pi) {
        int mi = pi, ya = ra, yb = rb;
        if (a.oz_s > 0) {
          const int p = p0 + pi, q = a.oz_diag ? p : t - p;
          mi = 0;
          ya += p * a.oz_ra;
          yb += q * a.oz_rb;
        }
        const CUtensorMap *ma = &maps.a[mi], *mb = &maps.b[mi];
        for (int x = x0; x < x1; x += BK) {
          if (!mbar_wait_warp(empty0 + 8 * st, ph, a.err_flag, 1)) {
            ok = false;
            break;
          }
          const uint32_t sa = smem0 + st * C::STAGE;
          if (elect_one()) {
            if (CG == 1) {
              mbar_arrive_expect_tx_at(full0 + 8 * st, C::STAGE);
              tma_load_2d(sa, ma, x, ya, full0 + 8 * st);
              tma_load_2d(sa + C::A_BYTES, mb, x, yb, full0 + 8 * st);
            } else {
              if (rank == 0) mbar_arrive_expect_tx_at(full0 + 8 * st, 2 * C::STAGE);
              tma_load_2d_pair(sa, ma, x, ya, sig0 + 8 * st);
              tma_load_2d_pair(sa + C::A_BYTES, mb, x, yb, sig0 + 8 * st);
            }
          }
          __syncwarp();
          if (++st == C::STAGES) {
            st = 0;
            ph ^= 1u;
          }
        }
      }
    }
    // every release of a stage has arrived here before this CTA ends (stages never used pass at once)
    for (int s = 0; s < C::STAGES && ok; ++s) {
      ok = mbar_wait_warp(empty0 + 8 * st, ph, a.err_flag, 1);
      if (++st == C::STAGES) {
        st = 0;
        ph ^= 1u;
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = idesc_f16(BM * CG, BN, a.bf16 != 0, a.acc16 != 0);
      const uint64_t desc0 = smem_desc_sw128(smem0);
      const uint32_t tfull0 = smem_u32(tfull), tempty0 = smem_u32(tempty);
      const uint32_t tmem0 = (uint32_t)uniform((int)tmem_base);
      uint32_t st = 0, ph = 0;
      int ui = 0;
      bool ok = true;
      for (int u = unit0; u < units && ok; u += ustride) {
        const UnitPlan pl = plan_unit<BN, CG>(u, a, kblocks);
        if (uniform(pl.skip)) continue;
        // the residue products hand the accumulator to the epilogue every `sub` K-blocks (an exact
        // FP32 sum of at most that many blocks), each time in the other tensor-memory buffer
        const int sub = (EPI == kEpiCrt8 && a.oz_sub_kb > 0) ? a.oz_sub_kb : (1 << 30);
        int left = uniform(pl.npairs * (pl.kb1 - pl.kb0));
        while (left > 0 && ok) {
          const int buf = ui & 1, cnt = left < sub ? left : sub;
          if (!mbar_wait_warp(tempty0 + 8 * buf, ((uint32_t)(ui >> 1) & 1u) ^ 1u, a.err_flag, 2)) {
            ok = false;
            break;
          }
          ++ui;
          tc_fence_after();
          const uint32_t dtm = tmem0 + (uint32_t)(buf * BN);
          for (int kb = 0; kb < cnt; ++kb) {
            if (!mbar_wait_warp(full0 + 8 * st, ph, a.err_flag, 3)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t da = desc0 + (uint64_t)(st * (C::STAGE >> 4)), db = da + (C::A_BYTES >> 4);
            if (elect_one()) {
#pragma unroll
              for (int k = 0; k < BK / UK; ++k)
                // advance the start address by k * 16 elements * 2 bytes inside the swizzle atom
                tc_mma_f16<CG>(dtm, da + (uint64_t)((k * UK * 2) >> 4), db + (uint64_t)((k * UK * 2) >> 4), idesc,
                               (kb | k) != 0 ? 1u : 0u);
              tc_commit<CG>(empty0 + 8 * st);
            }
            __syncwarp();
            if (++st == C::STAGES) {
              st = 0;
              ph ^= 1u;
            }
          }
          if (ok && elect_one()) tc_commit<CG>(tfull0 + 8 * buf);
          __syncwarp();
          left -= cnt;
        }
      }
      if (elect_one()) tc_commit<CG>(smem_u32(done_bar));
      __syncwarp();
    }
  } else {
    const int q = warp & 3;                  // TMEM lane quadrant this warp may access
    const int half = (warp - 2) / 4;         // which half of the tile's columns it handles
    constexpr int CH = C::HCHUNK;            // 32-column chunks per half
    const int c_lo = half * CH, c_hi = (c_lo + CH < C::NCHUNK) ? c_lo + CH : C::NCHUNK;
    uint8_t* stg = epi_stage + (warp - 2) * EPI_WARP_BYTES;
    int ui = 0;
    const float osc = a.out_scale ? *a.out_scale : 1.0f;
    float us = a.unscale;
    if (a.sa_ptr) us /= *a.sa_ptr;
    if (a.sb_ptr) us /= *a.sb_ptr;
    // the exponent of a power-of-two us (widen_pow2), else -2000
    const uint32_t ub = __float_as_uint(us), ue = ub >> 23;
    const int uk = ((ub & 0x7FFFFFu) == 0u && ue > 0u && ue < 255u) ? (int)ue - 127 : -2000;
    float amax = 0.0f;
    // hand the accumulator buffer back to the issuing thread
    auto release = [&](int buf) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 1)
          mbar_arrive(&tempty[buf]);
        else
          mbar_arrive_rank0(&tempty[buf]);
      }
    };
    for (int u = unit0; u < units; u += ustride) {
      const UnitPlan pl = plan_unit<BN, CG>(u, a, kblocks);
      if (pl.skip) continue;
      int bm, bn;
      decode_unit(pl.tile, a, pl.n, BM * CG, BN, bm, bn);
      const int i0 = (bm * CG + rank) * BM + q * 32;
      const int nrows = a.ninst > 0 ? pl.n : a.M;
      if constexpr (EPI == kEpiCrt8) {
        // The unit's accumulator arrives in sub-chunks (as many as the MMA issuer hands over), exact integers
        // of at most 2^24.  Each is reduced modulo m (crt_step) and added to the running residue sums, two
        // columns to a float; products longer than kCrtFoldSub sub-chunks fold the sums modulo m.  In pairs
        // of columns this is five instructions a pair where integer sums took eleven, two of them
        // conversions at a quarter of the rate: the epilogue has to keep up with the 8192 tensor-core cycles
        // of a sub-chunk (1.80 against 1.62 PFLOP/s at N = 4096 before the loops above were made uniform).
        const int sub = a.oz_sub_kb > 0 ? a.oz_sub_kb : (1 << 30);
        const int total_kb = pl.npairs * (pl.kb1 - pl.kb0);
        const int nsub = (int)(((long long)total_kb + sub - 1) / sub);
        const float m = (float)crtw::modulus(pl.t), inv = 1.0f / m;
        float wt = 0.0f;
#pragma unroll
        for (int t = 0; t < 32; ++t)
          if (t == pl.t) wt = a.crt_w[t];
        const f32x2 m2 = pack2(-m, -m), inv2 = pack2(inv, inv), big = pack2(kRint, kRint), nbig = pack2(-kRint, -kRint);
        float racc[CH][16];
#pragma unroll
        for (int cc = 0; cc < CH; ++cc)
#pragma unroll
          for (int p2 = 0; p2 < 16; ++p2) racc[cc][p2] = 0.0f;
        bool got = true;
        for (int sc = 0; sc < nsub; ++sc) {
          const int buf = ui & 1;
          const uint32_t uph = (uint32_t)(ui >> 1) & 1u;
          ++ui;
          if (!mbar_wait(&tfull[buf], uph, a.err_flag, 5)) {
            got = false;
            break;
          }
          tc_fence_after();
#pragma unroll
          for (int cc = 0; cc < CH; ++cc) {
            const int c = c_lo + cc;
            if (c >= c_hi || (a.sym && bn * BN + c * 32 < i0)) continue;  // chunk entirely below the diagonal
            float v[32];
            tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c * 32), v);
#pragma unroll
            for (int p2 = 0; p2 < 16; ++p2) {
              const f32x2 x = pack2(v[2 * p2], v[2 * p2 + 1]);
              float r0, r1;
              unpack2(fma2(add2(fma2(x, inv2, big), nbig), m2, x), r0, r1);
              racc[cc][p2] = fmaf(r1, 4096.0f, racc[cc][p2] + r0);
            }
          }
          release(buf);
          if (sc % kCrtFoldSub == kCrtFoldSub - 1) {
#pragma unroll
            for (int cc = 0; cc < CH; ++cc)
#pragma unroll
              for (int p2 = 0; p2 < 16; ++p2) {
                float s0, s1;
                crt_unpack2(racc[cc][p2], &s0, &s1);
                racc[cc][p2] = fmaf(crt_step(s1, m, inv), 4096.0f, crt_step(s0, m, inv));
              }
          }
        }
        if (!got) break;
        // Every entry's sum to its CRT digit in [0, m) < 2^8 (crt_digit_sum), which is all the reconstruction
        // needs.  The digits of a row, 32 bytes a chunk, go out as whole segments through the staging buffer
        // (16-byte unit x of row r at unit x ^ (r & (UPR - 1)) of the row's UPR).
        constexpr int UPR = 2 * CH;
        uint4* sd = reinterpret_cast<uint4*>(stg);
        const f32x2 w2 = pack2(wt, wt), off = pack2(0.5f * inv - 0.5f, 0.5f * inv - 0.5f);
        const f32x2 byte0 = pack2(8388608.0f, 8388608.0f);
#pragma unroll
        for (int cc = 0; cc < CH; ++cc) {
          if (c_lo + cc >= c_hi || (a.sym && bn * BN + (c_lo + cc) * 32 < i0)) continue;
          uint32_t w[8];
#pragma unroll
          for (int x = 0; x < 8; ++x) {
            float y[4];
#pragma unroll
            for (int b = 0; b < 4; b += 2) {
              float s0, s1;
              crt_unpack2(racc[cc][2 * x + b / 2], &s0, &s1);
              const f32x2 xs = mul2(pack2(s0, s1), w2);
              const f32x2 fl = add2(add2(fma2(xs, inv2, off), big), nbig);
              unpack2(add2(fma2(fl, m2, xs), byte0), y[b], y[b + 1]);
            }
            w[x] = __byte_perm(__byte_perm(__float_as_uint(y[0]), __float_as_uint(y[1]), 0x0040),
                               __byte_perm(__float_as_uint(y[2]), __float_as_uint(y[3]), 0x0040), 0x5410);
          }
          sd[lane * UPR + ((2 * cc) ^ (lane & (UPR - 1)))] = make_uint4(w[0], w[1], w[2], w[3]);
          sd[lane * UPR + ((2 * cc + 1) ^ (lane & (UPR - 1)))] = make_uint4(w[4], w[5], w[6], w[7]);
        }
        __syncwarp();
        uint8_t* dst = a.d8 + (size_t)pl.group * a.g_stride + (size_t)(pl.row0 + i0) * a.ld32;
#pragma unroll
        for (int k = 0; k < UPR; ++k) {
          const int r = (k * 32 + lane) / UPR, x = lane % UPR, c = c_lo + x / 2, col = bn * BN + c * 32 + 16 * (x & 1);
          if (i0 + r < nrows && c < c_hi && col < a.ld32 && !(a.sym && bn * BN + c * 32 < i0))
            *reinterpret_cast<uint4*>(dst + (size_t)r * a.ld32 + col) = sd[r * UPR + (x ^ (r & (UPR - 1)))];
        }
        __syncwarp();
      } else {
        const int buf = ui & 1;
        const uint32_t uph = (uint32_t)(ui >> 1) & 1u;
        ++ui;
        if constexpr (EPI == kEpiPoly || EPI == kEpiZupd) {
          // the FP32 input row segments of this half (one 128-byte line per chunk) into L2's nearer
          // side and L1 while the products run
          const float* src = (EPI == kEpiPoly) ? a.f32_in : a.f32;
          if (i0 + lane < nrows) {
            const float* r = src + ((size_t)pl.row0 + i0 + lane) * a.ld32 + (size_t)bn * BN;
#pragma unroll
            for (int cc = 0; cc < CH; ++cc)
              if (c_lo + cc < c_hi && bn * BN + (c_lo + cc) * 32 < pl.n)
                asm volatile("prefetch.global.L1 [%0];" ::"l"(r + (c_lo + cc) * 32));
          }
        }
        if (!mbar_wait(&tfull[buf], uph, a.err_flag, 5)) break;
        tc_fence_after();
        double ss = 0.0;
#pragma unroll 1
        for (int c = c_lo; c < c_hi; ++c) {
          const int col0 = bn * BN + c * 32;
          // past the last column, past the last row, or entirely below the diagonal: nothing to write
          if (col0 >= pl.n || i0 >= nrows || (a.sym && col0 < i0)) continue;
          float v[32];
          tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN + c * 32), v);
          if (a.acc16) widen_acc16(v);
          epi_chunk<EPI>(a, stg, lane, i0, col0, v, ss, amax, osc, us, uk, pl.group, nrows, pl.n, pl.row0);
        }
        release(buf);
        if constexpr (EPI == kEpiResid) {
          // fixed-order warp reduction; one partial per (tile, CTA, quadrant, half), summed in order later
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
          const size_t t = a.ninst > 0 ? (size_t)pl.tile : (size_t)u;
          const size_t p0 = a.ninst > 0 ? (size_t)a.g_part0[pl.inst] : 0;
          if (lane == 0) a.partials[p0 + (t * CG + rank) * kTcPartsPerCta + half * 4 + q] = ss;
        }
      }
    }
    if (a.amax_bits) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
      if (lane == 0) atomicMax(a.amax_bits, __float_as_uint(amax));
    }
  }
  tc_fence_before();
  __syncthreads();
  // The leader's last commit arrives in both CTAs, so each waits for its own: a CTA that left before would have it
  // arrive in the shared memory of the SM's next block.
  if (warp == 1) mbar_wait(done_bar, 0, a.err_flag, 4);
  if (CG == 2) cluster_sync();  // neither CTA leaves while the other may still signal or read it
  __syncwarp();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc<CG>(tmem_base, C::TMEM_COLS);
  }
}

template <int BN, int CG, int EPI>
cudaError_t launch_epi(const TcArgs& a, const TcMaps& maps, int num_sms, cudaStream_t s) {
  static bool attr_set = false;
  using C = Cfg<BN, CG>;
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(k_tc_gemm<BN, CG, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int units = units_of(a, BM * CG, BN), workers = num_sms / CG;
  const int grid = (units < workers ? units : workers) * CG;
  if (grid <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(NTHREADS);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CG;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = CG > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_tc_gemm<BN, CG, EPI>, maps, a);
}

}  // namespace

template <int BN, int CG>
cudaError_t tc_launch_tile(const TcArgs& a, const TcMaps& maps, int num_sms, cudaStream_t s) {
  switch (a.epi) {
    case kEpiStore16: return launch_epi<BN, CG, kEpiStore16>(a, maps, num_sms, s);
    case kEpiResid: return launch_epi<BN, CG, kEpiResid>(a, maps, num_sms, s);
    case kEpiPoly: return launch_epi<BN, CG, kEpiPoly>(a, maps, num_sms, s);
    case kEpiZupd: return launch_epi<BN, CG, kEpiZupd>(a, maps, num_sms, s);
    case kEpiF64: return launch_epi<BN, CG, kEpiF64>(a, maps, num_sms, s);
    case kEpiZupd64: return launch_epi<BN, CG, kEpiZupd64>(a, maps, num_sms, s);
    case kEpiG32: return launch_epi<BN, CG, kEpiG32>(a, maps, num_sms, s);
    case kEpiCrt8: return launch_epi<BN, CG, kEpiCrt8>(a, maps, num_sms, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zf
