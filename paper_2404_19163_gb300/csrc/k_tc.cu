// Host side of the tcgen05 engine (tc_kernel.cuh): tensor maps, the choice of the tile shape, and the
// launches on CTA pairs.  The narrower tiles are instantiated in k_tc_128.cu, k_tc_64.cu and k_tc_32.cu.
#include <math.h>

#include "tc_kernel.cuh"

namespace zf {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);


// cuTensorMapEncodeTiled is resolved through the runtime's driver entry-point query, so the
// library carries no link-time dependency on libcuda (it loads on machines without a driver).
static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

int tc_make_map(CUtensorMap* m, const void* base, int rows, int cols, int ld, int box_rows, bool bf16) {
  if ((ld % 8) != 0 || (reinterpret_cast<uintptr_t>(base) & 15) != 0) return -1;
  EncodeTiledFn enc = encode_fn();
  if (!enc) return -2;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                   const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)r;
}

int tc_tiles(int m, int n, bool sym, int tile) {
  return tiles_of(m, n, sym ? 1 : 0, BM * tc_tile_ctas(tile), tc_tile_width(tile));
}

int tc_num_units(const TcArgs& a, int tile) { return units_of(a, BM * tc_tile_ctas(tile), tc_tile_width(tile)); }

// ---- the tile shape of a product
// Microseconds of a unit's K-block (streaming and issuing; nearly the same for every width, see
// tc_kernel.cuh) and of one 32-column chunk of an epilogue (what an SM can write per microsecond; the FP64
// epilogues by their pipe), measured at N = 128 ... 4096.  A wide tile spends its K-blocks best, a narrow one
// spreads a small product's epilogues over more SMs: the rule takes the shape whose rounds of units, each the
// longer of its K-blocks and its epilogue, plus the last epilogue, are shortest.  With three segments
// the line between 32- and 128-wide tiles lies near N = 1100, and the pair takes over from about
// N = 2300 (full) and 3600 (symmetric); residue products, with a unit per modulus and tile, go to the
// pair from N = 700.
namespace {
constexpr double kUsPerKb[kTiles] = {0.199, 0.205, 0.222, 0.286};
// 32-column chunks each column half writes (a 32-wide tile has one chunk, so half an SM's writes)
constexpr double kChunks[kTiles] = {0.5, 1, 2, 4};

double us_per_chunk(int epi) {
  switch (epi) {
    case kEpiStore16:
    case kEpiG32: return 1.0;
    case kEpiCrt8: return 0.8;
    case kEpiF64:
    case kEpiZupd64: return 7.0;
    default: return 3.0;  // kEpiResid, kEpiPoly, kEpiZupd: two copies of FP32 and 16-bit values
  }
}

// kbs: K-blocks of a unit; returns the time of a unit and its epilogue's.
double unit_us(int tile, double kbs, int epi, double* tail) {
  *tail = kChunks[tile] * us_per_chunk(epi);
  const double t = kbs * kUsPerKb[tile];
  return t > *tail ? t : *tail;
}
}  // namespace

int tc_pick_tile(const TcArgs& a, int num_sms) {
  const double kblocks = (a.K + BK - 1) / BK;
  double groups = 1.0, kbs = kblocks * a.nseg;
  if (a.oz_s > 0) {
    groups = (double)a.oz_s * a.oz_nch;
    kbs = a.oz_chunk_kb < kblocks ? a.oz_chunk_kb : kblocks;
    if (!a.oz_diag) kbs *= 0.5 * (a.oz_s + 1);  // slice pairs of a group, on average
  }
  int best = kTilePair;
  double best_us = 1e30;
  for (int t : {kTilePair, kTile128, kTile64, kTile32}) {
    double tail;
    const double us = unit_us(t, kbs, a.epi, &tail);
    const int workers = num_sms / tc_tile_ctas(t);
    const double total = ceil(tc_tiles(a.M, a.N, a.sym != 0, t) * groups / (workers > 0 ? workers : 1)) * us + tail;
    if (total < best_us) {
      best_us = total;
      best = t;
    }
  }
  return best;
}

// Units of different sizes keep the persistent CTAs evenly loaded: the work over the workers, half the
// longest unit on average, and the last epilogue.
int tc_pick_tile_grouped(const int* n, int count, bool sym, int pairs, int epi, int num_sms) {
  int best = kTilePair;
  double best_us = 1e30;
  for (int t : {kTilePair, kTile128, kTile64, kTile32}) {
    double sum = 0.0, longest = 0.0, tail = 0.0;
    for (int i = 0; i < count; ++i) {
      const double kblocks = (n[i] + BK - 1) / BK, tiles = tc_tiles(n[i], n[i], sym, t);
      const bool crt = epi == kEpiCrt8;
      const double us = unit_us(t, crt ? kblocks : kblocks * pairs, epi, &tail);
      sum += tiles * us * (crt ? pairs : 1);
      longest = us > longest ? us : longest;
    }
    const int workers = num_sms / tc_tile_ctas(t);
    const double total = sum / (workers > 0 ? workers : 1) + 0.5 * longest + tail;
    if (total < best_us) {
      best_us = total;
      best = t;
    }
  }
  return best;
}

template cudaError_t tc_launch_tile<256, 2>(const TcArgs&, const TcMaps&, int, cudaStream_t);
extern template cudaError_t tc_launch_tile<128, 1>(const TcArgs&, const TcMaps&, int, cudaStream_t);
extern template cudaError_t tc_launch_tile<64, 1>(const TcArgs&, const TcMaps&, int, cudaStream_t);
extern template cudaError_t tc_launch_tile<32, 1>(const TcArgs&, const TcMaps&, int, cudaStream_t);

cudaError_t launch_tc_gemm(const TcArgs& a, const TcMaps& maps, int tile, int num_sms, cudaStream_t s) {
  if (a.oz_s <= 0 && (a.nseg < 1 || a.nseg > kTcMaxSeg)) return cudaErrorInvalidValue;
  switch (tile) {
    case kTilePair: return tc_launch_tile<256, 2>(a, maps, num_sms, s);
    case kTile128: return tc_launch_tile<128, 1>(a, maps, num_sms, s);
    case kTile64: return tc_launch_tile<64, 1>(a, maps, num_sms, s);
    case kTile32: return tc_launch_tile<32, 1>(a, maps, num_sms, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zf
