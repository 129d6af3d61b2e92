// Digit-split grouped complex GEMM on the tcgen05 tensor cores (digits.cu, digits_host.cu): the
// arithmetic of the FP64 and float-float products of the library.
//
// Method (error-free splitting: Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012). Every
// row of the left and every column of the right operand is scaled by a power of two to
// |x| < 1 and rounded to an integer T, |T| < 2^t, which is written in 8 balanced digits of
// `beta` bits, T = sum_i d_i 2^(beta (7 - i)), -2^(beta-1) <= d_i < 2^(beta-1). Digits are exact
// in BF16 and products of digits are integers, so a tensor-core product with FP32 accumulation
// is exact while its sums stay within 2^24. A product needs the pairs i + j <= 7 (36 of 64):
// digit i of A multiplies the window of digits 0 .. 7 - i of B with one MMA, whose N columns are
// the accumulator levels i .. 7 (level l collects i + j = l). The levels are flushed to integers
// in registers before they can pass 2^24 and added exactly; one rounding makes the FP64 result.
//   beta = 8 (t = 62, the FP64 products): 62-bit fixed point against the largest entry of the row
//     / column. Error against quadruple precision, relative to the result's norm: 8e-17 on uniform
//     random operands, 7e-17 on converged MPS environments (the FP64 CUDA-core kernel: 6-9e-16,
//     4-7e-16).
//   beta = 7 (t = 55, the float-float products): fewer flushes; 4e-16 and 2-4e-15 (the float-float
//     CUDA-core kernel: 2-4e-14, 0.6-1.4e-14).
// Entries far below the largest of their row or column keep fewer bits than a floating-point
// product would give them: a term is off by at most 2^-58 (FP64; 2^-51.8 float-float) of its row's
// times its column's bound: two roundings of 2^-63 (2^-56), seven dropped digit pairs of 2^-62 (2^-56)
// on the first level, and twice that in a complex product. K FMAs in FP64 may be off by
// 2 K 2^-53 (float-float: 2 K 2^-46) of the sum of the terms' magnitudes, so a result block is kept when
// that sum reaches 2^-6 (float-float: 2^-6.8) of the largest row times the largest column somewhere in it: the
// error is then below what FMAs may be off in the block. The largest result is a lower bound of the sum and costs
// nothing; where it is too small, the terms of the largest row and column are added up. The other blocks
// (operands graded against each other along K) are computed again in FP64, or in float-float for the
// float-float products. On states of the cylinders
// under 1% of the blocks fail the first test, and of those most pass the second.
//
// Measured on H_eff applications (Hofstadter cylinder, mid-ring sites, random operands): FP64 at
// Ly = 8, chi = 1024 0.49 ms (CUDA cores 11.2 ms); loading environments and one float-float
// application at Ly = 10, chi = 3200 7.6 ms (31.9 ms). The product kernel is bound by the tensor
// pipe: 26 complex multiply-adds per cycle and SM at full tiles, against 0.21 for FP64 FMAs.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "mrd_internal.h"

namespace mrd {

constexpr int kDgRows = 128;      // rows of a left (tall) tile
constexpr int kDgCols = 32;       // columns of a tile: 8 levels x 32 x (re, im) = 512 TMEM columns
constexpr int kDgDigits = 8;
constexpr int kDgStep = 16;       // K of one MMA, one panel step
constexpr int kDgRedoTile = 8;    // tiles of blocks that are computed again
constexpr int kDgSpread = 6;      // bits a block's largest result may lie below its operands' bounds
// the same of the sum of the terms' magnitudes: 2^-6 (FP64), 2^-6.8 (float-float), with 1% for its rounding.
// With 2^-6 for both step 2 of the refinement that repeats most (Ly = 10, chi = 3200) took 5.3 instead of 4.0 ms (repeats and their check together).
constexpr float kDgLine64 = 1.01f / 64.f, kDgLineFF = 1.01f / 111.4f;
__host__ __device__ inline int dg_planes(bool real) { return real ? kDgDigits : 2 * kDgDigits; }
__host__ __device__ inline int dg_tbits(int beta) { return beta == 8 ? 62 : 55; }
// K steps between flushes. Level l sums 2 (l + 1) digit products of at most 2^(2 beta - 2) per
// K: beta = 7 stays within 2^24 on every level for 256 values of K; beta = 8 for 96 on the
// levels 0 .. 4, and what rounding could touch above that weighs at most 2^-54 of the operands'
// largest product.
__host__ __device__ inline int dg_flush(int beta) { return beta == 8 ? 6 : 16; }

// One operand block of a group's panel: rows x K values at src (element (r, k) at off + r ld + k
// when kcontig, else at off + k ld + r; conjugated if conj; off < 0: zeros), written to rows
// row0 .. of the panel at K positions k0 .. k0 + kpad - 1 (zeros beyond K).
struct DgJob {
  int64_t off, ld, panel;
  int32_t rows, K, kpad, row0, k0, prows, nks, exp0;   // prows: rows of the whole panel
  int32_t flags, pad;                                  // DGJ_*
};
enum { DGJ_KCONTIG = 1, DGJ_CONJ = 2, DGJ_TALL = 4 };   // TALL: 128-row tiles, else 32-column tiles
// One stacked product: R x N outputs (R: tall side), nks K steps. Every task's operands are the
// blocks of buffer 0 (tasks' A) or 1 (tasks' B); tall_op says which one is tall here.
struct DgGroup {
  int64_t a_off, b_off;        // panels of the tall and the other side (bytes, in their buffers)
  int32_t R, N, nks, ea, eb;   // ea, eb: first row's / column's exponent
  int32_t tall_op;
  int32_t cm, cm_rows;         // C map: first entry; indexed by rows (1) or by columns (0)
  int32_t job, n_jobs;         // the shared operand's blocks in its job list
};
// C map entries of one task: entry r is (off + r step, other), the C offset of its r-th stacked
// row (column) and the stride along the shared side. job: its first block in the stacked operand's
// job list (one per block of the group, in the same order).
struct DgMember {
  int64_t off, step, other;
  int32_t first, rows;
  int32_t group, job;
};
// K steps ks0 .. ks1 - 1 of a tile; split >= 0: one part of a tile cut along K (split * 64 + part).
struct DgItem {
  int32_t group, tile, ks, split;   // ks = ks0 | ks1 << 16
};

// Host tables of one grouped product.
struct DgPlan {
  std::vector<DgJob> jobs[2];        // per operand buffer
  std::vector<int2> pieces[2];       // (job, first unit) per CTA pass of the pack kernel
  std::vector<int2> mpieces[2];      // the same for the exponent kernel
  std::vector<DgGroup> groups;
  std::vector<DgItem> items;         // longest first
  std::vector<int64_t> item0;        // first item of every group, + total (group-major plans only)
  std::vector<int2> splits;          // per split tile: first partial slot, parts
  std::vector<DgMember> members;
  int64_t cmap = 0;                  // entries of the C map (expanded on the device)
  int64_t bytes[2] = {0, 0};         // panels
  int64_t rows[2] = {0, 0};          // exponents
  int64_t slots = 0;                 // partial sums of split tiles
  int64_t redo = 0;                  // tiles of kDgRedoTile x kDgRedoTile of all tasks
  int max_tiles = 0;                 // of one task
  int sop = 0;                       // the stacked operand
  double cost = 0.0;                 // estimated cycles of the product
  bool real = false;
};

// How tasks (plan.cuh rows) share panels: tasks that multiply the same right blocks are
// stacked along their rows (BY_B), tasks given the same id are (BY_ID: the union of their right
// blocks, zeros where a task lacks one), tasks that share their left blocks are stacked along
// their columns (BY_A).
enum DgStack { DG_BY_B = 0, DG_BY_ID = 1, DG_BY_A = 2 };

// group_major: items in group order (for launches of one group each), no tile cut along K.
void dg_plan(DgPlan& p, const int64_t* tasks, const int64_t* segs, int64_t n_tasks, DgStack how, const int32_t* ids,
             bool real, int beta, int n_sm, bool group_major = false);
// Estimated cycles of the CUDA-core kernels on the same tasks.
double dg_cost_cores(const int64_t* tasks, const int64_t* segs, int64_t n_tasks, bool ff, bool real, int n_sm);

// Device side of a plan: tables in one allocation, panels, exponents, partial sums.
struct DgDev {
  uint8_t* tab = nullptr;            // uploaded tables
  size_t tab_bytes = 0;
  DgJob* jobs[2] = {nullptr, nullptr};
  int2* pieces[2] = {nullptr, nullptr};
  int2* mpieces[2] = {nullptr, nullptr};
  int n_pieces[2] = {0, 0}, n_mpieces[2] = {0, 0};
  DgGroup* groups = nullptr;
  DgItem* items = nullptr;
  int2* splits = nullptr;
  DgMember* members = nullptr;
  longlong2* cmap = nullptr;         // follows the uploaded tables
  int n_items = 0, n_splits = 0, n_members = 0;
  uint8_t* panel[2] = {nullptr, nullptr};
  int* expo[2] = {nullptr, nullptr};
  int64_t rows[2] = {0, 0};
  uint8_t* partial = nullptr;        // dg_partial_bytes
  int* tickets = nullptr;            // 8 per split tile, zeroed before each product
  int* res = nullptr;                // largest exponent field of each stacked row's results; zeroed likewise
  int* redo_count = nullptr;         // tiles to be computed again, zeroed likewise
  int2* redo = nullptr;              // (task, tile)
  int max_tiles = 0;
  int sop = 0;
  bool real = false;
};
// Partial sums of a split tile: 128 x 32 complex numbers of 12-byte sums, per part.
constexpr int64_t kDgSlotBytes = 128 * 32 * 2 * 12;

// Bytes of the uploaded tables, and of the device allocation that holds them and the C map.
size_t dg_table_bytes(const DgPlan& p);
size_t dg_device_table_bytes(const DgPlan& p);
// Fill `host` (dg_table_bytes) with the plan's tables and point d's tables into `dev`; after the
// upload dg_expand forms the C map.
void dg_tables(const DgPlan& p, uint8_t* host, uint8_t* dev, DgDev& d);
cudaError_t dg_expand(const DgDev& d, cudaStream_t s);
// Zeroed words of a product besides its exponents: tickets, result exponents, count of tiles to redo.
inline int64_t dg_state_words(const DgPlan& p) { return 8 * (int64_t)p.splits.size() + p.cmap + 1; }
inline void dg_state(const DgPlan& p, int* words, DgDev& d) {
  d.tickets = words;
  d.res = words + 8 * p.splits.size();
  d.redo_count = d.res + p.cmap;
}
// Scratch words shared by the products of a handle (device ints): item counter, error flag.
enum { DG_CTR = 0, DG_ERR = 1, DG_WORDS = 4 };
// Units of a pack / exponent piece (see the kernels).
constexpr int kDgPairPiece = 2048;   // kcontig pack: (row, pair of K) units
constexpr int kDgChunkPiece = 512;   // row-contiguous pack: (chunk of 8 K, row) units
constexpr int kDgMaxRows = 64;       // kcontig exponents: rows
constexpr int kDgMaxK = 32;          // row-contiguous exponents: K
// Exponents and digits of operand buffer `op` (0: tasks' A, 1: tasks' B) from `src`; the caller has
// zeroed expo[op] and the product's state. Resets the item counter for the next dg_gemm.
cudaError_t dg_pack(const DgDev& d, int op, const double2* src, int beta, int* words, cudaStream_t s);
// The product; first / count: a sub-range of the items (per-group launches), count < 0: all.
cudaError_t dg_gemm(const DgDev& d, double2* C, int beta, int* words, int n_sm, uint64_t wait_ns, cudaStream_t s,
                    int first = 0, int count = -1);
// After the product: the tasks whose operands or results have an infinity or NaN, which has no
// fixed-point form, or for which the fixed point was too coarse, are computed again in FP64 (float-float
// where the product is and their range allows it) from the operands themselves (buffers 0 and 1).
cudaError_t dg_redo(const DgDev& d, const double2* a, const double2* b, double2* C, int beta, const int* words, int n_sm, cudaStream_t s);
cudaError_t dg_init();

}  // namespace mrd
