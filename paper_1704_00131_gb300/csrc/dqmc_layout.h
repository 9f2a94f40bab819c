// Sizes of the digit planes of the split products and of a CTA's dynamic shared memory:
// arithmetic that the host and the kernels share (this header needs no CUDA).
#pragma once
#include <cstddef>

#ifdef __CUDACC__
#define DQMC_HD __host__ __device__
#else
#define DQMC_HD
#endif

namespace dqmc {

// Digit planes of the split tensor-core products: blocks of digits x rows x kPlaneK
// bf16, one block per (tile, 16-wide K chunk), copied to shared memory by one
// tiled tensor copy each.  Float pairs have kPlaneDigits digits, FP64 operands
// kPlaneDigits64; a right operand's tiles have kPlaneRowsB rows, a left operand's
// umma_rows(N).
constexpr int kPlaneDigits = 7, kPlaneDigits64 = 8, kPlaneMaxRows = 128, kPlaneRowsB = 32, kPlaneK = 16;
constexpr int kPlaneRowElems = 256;  // bf16 per row of the copies' 2D view of a plane buffer
// row tiles of an N-row left operand: equal, at most kPlaneMaxRows, rounded to 16
DQMC_HD inline int umma_row_tiles(int n) { return (n + kPlaneMaxRows - 1) / kPlaneMaxRows; }
DQMC_HD inline int umma_rows(int n) {
  const int t = umma_row_tiles(n);
  return ((n + t - 1) / t + 15) / 16 * 16;
}
// bf16 elements of the left and right operands' planes of N x K matrices
DQMC_HD inline size_t plane_elems(int digits, int n, int k, bool right) {
  const size_t rows = right ? (size_t)(n + kPlaneRowsB - 1) / kPlaneRowsB * kPlaneRowsB
                            : (size_t)umma_rows(n) * umma_row_tiles(n);
  return (size_t)digits * rows * ((k + kPlaneK - 1) / kPlaneK * kPlaneK);
}

// The first kSmemCounterBytes of the dynamic shared memory hold thread 0's
// cycle counters of the sweep kernel (fixed addresses, no registers).
constexpr int kSmemCounterBytes = 16 * 8;
// Dynamic shared memory a CTA can have on this architecture.
constexpr size_t kMaxSmemBytes = 227 * 1024;

// exponent entries per operand of the split products: rows padded to whole tiles
DQMC_HD inline int exp_len(int ld) { return ld + kPlaneMaxRows; }

// Layout: the vectors and barriers, then (128-byte aligned) the SIMT products'
// panels and, in the sweep kernel, the delayed vectors.  The tensor-core products
// stage their operands over both: neither is live inside a product (a flush has
// cut its delayed vectors into digits before the first copy lands).
// (The panels also hold the QR's, two of `qr_cols` columns.)
constexpr int kGemmMaxTile = 80;  // widest SIMT tile, 16 * 5
constexpr int kGemmRegionBytes = 2 * 16 * kGemmMaxTile * 8;
constexpr int kPanel = 4;  // columns per panel of the QR (the reason stands at qr_blocked's panels)
DQMC_HD inline size_t gemm_region_bytes(int ld, int qr_cols = kPanel) {
  const size_t qr = (size_t)2 * qr_cols * (ld + 1) * 8;
  return ((qr > (size_t)kGemmRegionBytes ? qr : (size_t)kGemmRegionBytes) + 127) / 128 * 128;
}

DQMC_HD inline size_t smem_stage_offset(int ld, int MV) {
  size_t b = kSmemCounterBytes;
  b += 6 * (size_t)ld * 8;        // v, ev, d, hv, xdiag, spare
  b += 3 * (size_t)MV * 8;        // u2, delta, gam
  b += 8 * 8 + 32 * 8 + 32 * 4;   // xs, red, ired
  b += (size_t)MV * 4;            // qsite
  b += (size_t)ld * 4;            // qinv
  b += 2 * (size_t)MV + 16;       // fnew, fslice
  b = (b + 15) / 16 * 16;
  b += 8 * 128 * 8;               // qred
  b += 2 * (size_t)exp_len(ld) * 4;  // expA, expB
  b = (b + 15) / 16 * 16;
  b += 128;                       // mbarriers and the TMEM slot of the tensor-core products
  return (b + 127) / 128 * 128 + 128;  // room to align the panels
}
// ... without split products: the QR's panels get the kPanel columns where they fit,
// fewer from 1441 sites (2) and 1821 (1); the kernels read the width off the size.
DQMC_HD inline size_t smem_bytes_for(int ld, int MV) {
  size_t b = 0;
  for (int w = kPanel; w >= 1; w >>= 1) {
    b = smem_stage_offset(ld, MV) + gemm_region_bytes(ld, w);
    if (b <= kMaxSmemBytes) break;
  }
  return b;
}
// columns per panel of the QR of N columns in a region of `bytes`
DQMC_HD inline int qr_panel_cols(int N, size_t bytes) {
  int w = kPanel;
  while (w > 1 && (size_t)2 * w * (N | 1) * 8 > bytes) w >>= 1;
  return w;
}

// One stage of the split products of matrices of up to maxN sites.
inline size_t split_stage_bytes(int maxN, int digits) {
  size_t stage = 0;  // the tile height is not monotonic in N
  for (int n = 1; n <= maxN; ++n) {
    const size_t b = (size_t)digits * kPlaneK * 2 * (umma_rows(n) + kPlaneRowsB);
    stage = b > stage ? b : stage;
  }
  return stage;
}
// The split products need two stages: where a CTA cannot have them beside the vectors
// (FP64 from 1561 sites, float pairs from 1673) the products keep the register tiles.
inline bool split_fits(int maxld, int maxMV, int maxN, int digits) {
  return smem_stage_offset(maxld, maxMV) + 2 * split_stage_bytes(maxN, digits) <= kMaxSmemBytes;
}
// Dynamic shared memory with `ab_bytes` of delayed vectors; digits > 0: also room to stage
// the split products of matrices of up to maxN sites (split_fits).  They want three
// stages; two where three would leave room for one CTA per SM instead of two (a second
// CTA hides more than a third stage), or for none (FP64 from 1105 sites).
inline size_t smem_total(int maxld, int maxMV, size_t ab_bytes, int maxN, int digits) {
  const size_t off = smem_stage_offset(maxld, maxMV), half = 113 * 1024;
  const size_t plain = ab_bytes ? off + gemm_region_bytes(maxld) + ab_bytes : smem_bytes_for(maxld, maxMV);
  if (!digits) return plain;
  const size_t stage = split_stage_bytes(maxN, digits);
  const size_t two = off + 2 * stage > plain ? off + 2 * stage : plain;
  const size_t three = off + 3 * stage > plain ? off + 3 * stage : plain;
  // every CTA of these kernels holds half of the SM's tensor memory (256 of 512
  // columns): at least 78 KB of shared memory per CTA keeps three of them from
  // sharing an SM, so an allocation never waits
  const size_t need = (three <= half || (two > half && three <= kMaxSmemBytes)) ? three : two;
  return need > 78 * 1024 ? need : 78 * 1024;
}

}  // namespace dqmc
