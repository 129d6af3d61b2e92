// Shared layout constants of the tensor-core H_eff path (heff_tc.cu, tc_host.cu).
#pragma once
#include <stdint.h>

namespace mrd {

// Tensor-core precisions: complex operands, or real ones (the sine / cosine machine of Eq. rot
// with real environments and theta: imaginary planes dropped, the result's imaginary parts 0).
enum { TC_TF32 = 1, TC_BF16X3 = 2, TC_TF32_REAL = 3, TC_BF16X3_REAL = 4 };
__host__ __device__ constexpr bool tc_is_tf32(int prec) { return prec == TC_TF32 || prec == TC_TF32_REAL; }
__host__ __device__ constexpr bool tc_is_real(int prec) { return prec == TC_TF32_REAL || prec == TC_BF16X3_REAL; }

// Panels. A K step is what one MMA multiplies: 32 bytes per row, 16 BF16 or 8 TF32 values. A tile
// (128 rows of an A panel, the last one padded to 8; ntile rows of a B panel, the last one padded
// to 16) holds its K steps one after another, each step its planes, each plane rows x 32 bytes in
// the 32-byte swizzle of the tcgen05 descriptors. Consecutive steps of a tile are contiguous, so
// one bulk copy brings any run of them, and K is padded to one step only.
__host__ __device__ constexpr int tc_kstep(int prec) { return tc_is_tf32(prec) ? 8 : 16; }
__host__ __device__ constexpr int tc_aplanes(int prec) {
  return prec == TC_TF32 ? 2 : prec == TC_BF16X3 ? 4 : prec == TC_TF32_REAL ? 1 : 2;
}
// accumulator column groups of one output tile: (re, im) TF32, (re_hi, re_lo, im_hi, im_lo) BF16X3,
// (re) and (hi, lo) for real operands
__host__ __device__ constexpr int tc_groups(int prec) { return tc_aplanes(prec); }
// Planes of a B tile of nrow rows. A complex product C_re = A_re B_re - A_im B_im, C_im = A_re B_im +
// A_im B_re over the tile's column groups takes, with planes S = [re, im] (each hi and lo in BF16X3):
//   A_re x S into both groups (N = 2 x width), then -A_im x S[im] into C_re and A_im x S[re] into
//   C_im (the sign from the instruction's A-negate bit);
// or, with the negated imaginary planes as well, S = [-im, re, im]: A_re x [re, im] and
//   A_im x [-im, re], one MMA each. An MMA costs N / 2 cycles but at least 48 (measured), so the
// second form is for narrow tiles: half of the group width (2 nrow BF16X3, nrow TF32) up to 96
// columns. Both sum every element in the same order and give the same bits.
__host__ __device__ constexpr bool tc_neg_planes(int prec, int nrow) {
  return !tc_is_real(prec) && tc_aplanes(prec) / 2 * nrow <= 96;
}
__host__ __device__ constexpr int tc_bplanes(int prec, int nrow) {
  return tc_aplanes(prec) + (tc_neg_planes(prec, nrow) ? tc_aplanes(prec) / 2 : 0);
}
__host__ __device__ constexpr int64_t tc_apad(int64_t rows) { return (rows + 7) / 8 * 8; }
__host__ __device__ constexpr int64_t tc_bpad(int64_t rows) { return (rows + 15) / 16 * 16; }

// K segment of a task: panel byte offsets (multiples of 256) and K steps, b = offset / 256 << 16 | steps.
struct TcSeg {
  int64_t a, b;
};
// One output tile (128 x ntile at most).
struct alignas(16) TcItem {
  int32_t nrow, mrow;      // padded columns (B rows) and rows (A rows) of the tile
  int32_t rows, cols;      // outputs
  int32_t seg0, nseg;
  int32_t rt, nt;
  int64_t out, ld;         // packed Z output: first entry of the tile in the row map, K steps of the
                           // Z panels; FP64 output: element offset of the tile, leading dimension
  int32_t row0, nks;       // rows below row0 are not stored; K steps of all segments
  int64_t pad;
  TcSeg seg[2];            // the first two segments (all that a step-1 task has)
};
// Row map entry of a stacked step-1 row: (byte offset of its Z tile / 256) << 12 | (padded rows of that
// tile / 8 - 1) << 7 | row in the tile.
inline int64_t tc_rowmap(int64_t tile_off, int64_t mrow, int64_t row) { return tile_off / 256 << 12 | (mrow / 8 - 1) << 7 | row; }

// pack job row (int64): src_off ld trans rows K panel_byte_offset rowtile (0: A panel) steps
// panel_rows first_piece row0; element (r, k) = src[r ld + k], or src[k ld + r] if trans, goes to row
// row0 + r of the panel. Units: pairs of K (not trans) or 16-byte chunks of K (trans) times rows.
enum { TCJ = 11 };
constexpr int kPackPiece = 256;

// Tile configuration of the grouped GEMM, picked per problem class by the autotuner
// (tc_host.cu): B rows (output columns) per tile, pipeline depth in 128-byte K tiles (4 K steps),
// task order (0: charge order, 1: largest work first) among tiles of equal K.
struct TcCfg {
  int ntile, stages, order;
};
// A pipeline slot holds up to tc_group K steps of a tile (8 A planes together: 32 KB), whichever
// segments they come from: about 1000 cycles of MMAs. Handing a slot over costs the producer ~400
// and the MMA thread ~200 cycles: with half of it (16 KB of A) both were slower than the tensor cores
// (0.86 against 0.71 ms per BF16X3 application at Ly = 10, chi = 3200, before their loops were
// shortened).
__host__ __device__ constexpr int tc_group(int prec) { return 8 / tc_aplanes(prec); }
constexpr int kTcABytes = 32768;
constexpr int kTcMaxSlots = 8;
// dynamic shared memory; with the kernel's static shared memory (below 1 KB) it stays below the
// 227 KB a block may use
constexpr int kTcMaxSmem = 225 * 1024;
__host__ __device__ constexpr int tc_slot_bytes(int prec, int ntile) {
  const int wide = tc_bplanes(prec, ntile) * ntile;   // narrower tiles may have more planes
  const int edge = tc_is_real(prec) ? 0 : tc_is_tf32(prec) ? 3 * (ntile < 96 ? ntile : 96) : 6 * (ntile < 48 ? ntile : 48);
  return kTcABytes + tc_group(prec) * (wide > edge ? wide : edge) * 32;
}
__host__ __device__ constexpr int tc_slots(int prec, TcCfg c) { return c.stages * 4 / tc_group(prec); }
__host__ __device__ constexpr int tc_smem_bytes(int prec, TcCfg c) { return tc_slots(prec, c) * tc_slot_bytes(prec, c.ntile) + 1024; }
// the accumulator of one tile spans groups x ntile FP32 columns: at most 256, so that two
// tiles (two slots) fit the 512 columns of tensor memory
__host__ __device__ constexpr bool tc_cfg_ok(int prec, TcCfg c) {
  return c.stages >= 1 && tc_slots(prec, c) >= 2 && tc_slots(prec, c) <= kTcMaxSlots && c.ntile >= 16 && c.ntile <= 128 &&
         c.ntile % 16 == 0 && tc_groups(prec) * c.ntile <= 256 && tc_smem_bytes(prec, c) <= kTcMaxSmem;
}
// default configuration (also the first candidate of the autotuner)
inline TcCfg tc_default_cfg(int prec) {
  return prec == TC_TF32 ? TcCfg{128, 3, 0} : prec == TC_BF16X3 ? TcCfg{64, 2, 0} : prec == TC_TF32_REAL ? TcCfg{128, 6, 0} : TcCfg{128, 3, 0};
}

}  // namespace mrd
