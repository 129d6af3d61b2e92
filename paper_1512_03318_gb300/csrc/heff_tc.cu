// Tensor-core (tcgen05 / TMEM) grouped complex GEMMs of the two-site H_eff in reduced
// precision with FP32 accumulation.
//
// Same two steps as the FP64 path (step 1: Z_{w'} = LW_{w'} theta; step 2:
// theta' = sum_{w'} Z_{w'} WR_{w'}). Precisions:
//   TF32    operands rounded to TF32 (planes re, im).
//   BF16X3  every operand x split as x_hi = bf16(x), x_lo = bf16(x - x_hi) (planes re_hi,
//           re_lo, im_hi, im_lo); (A_hi + A_lo) x (B_hi + B_lo) per real product (the
//           split-precision scheme of Henry, Tang & Heinecke 2019; the lo x lo product comes with
//           the MMA's columns and is kept).
//
// Operands live in HBM as panels of K steps (tc.cuh). LW and WR are packed once per environment
// load, theta once per matvec, and the step-1 epilogue writes Z directly in the packed A format of
// step 2: a warp's 32 rows x 16 columns are 1 KB runs of every plane.
//
// Kernel: persistent, one CTA per SM, 10 warps: warp 0 takes tiles (longest K first) from a global
// counter and issues the bulk copies, warp 1 owns TMEM (512 columns: two accumulator slots) and
// issues the MMAs from one thread, warps 2-9 drain the accumulators (warp w reads TMEM lanes
// 32 (w % 4) ..). Shared-memory slots of tc_group K steps are handed over with mbarriers together
// with a word that tells the MMA thread what they hold, so that thread reads no global memory; every
// wait is bounded (global-timer limit set by the host) and sets an error flag when it gives up.
// Before the CTA frees its tensor memory and exits, the producer waits for the last fill of every
// slot and the MMA thread for all its MMAs (commit to a drain barrier), so a CTA whose waits gave
// up leaves no copy or MMA in flight.
//
// What bounds it: the serial work between MMAs. A full BF16X3 K step (128 x 64 x 16) is 512 tensor
// cycles, and the tensor core queues only one or two MMAs, so what the issuing thread does between two
// slots (a wait, a table row, a commit) leaves it idle for 200 - 300 of ~1300 cycles per slot; leaving
// the copies out changes nothing. The sectors of an MPS are small (tens of rows), so padding counts as
// much: K is padded to one MMA (16 or 8 values), and step 2 stacks the rows of both spin values. With
// K in tiles of 64 (BF16) and 32 values, two stages, a table lookup per K segment on the copying thread
// and a tile per (s1', s2'): 0.97 ms per BF16X3 application at Ly = 10, chi = 3200 (step 1 0.41, step 2
// 0.53), TF32 Ly = 8, chi = 2049 0.39 ms, real BF16X3 Ly = 6, chi = 777 0.115 ms; now 0.55 (0.23 +
// 0.29), 0.20 and 0.058 ms, the same bits.
#include <cuda_bf16.h>

#include "mrd_internal.h"
#include "tc.cuh"

namespace mrd {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t sw32(uint32_t off) { return off ^ (((off >> 7) & 1u) << 4); }

// Shared-memory descriptor of a K-major operand in the 32-byte swizzle: the low word holds the address
// in units of 16 bytes (and LBO, unused here), the high word is the same for every operand: SBO 256 (8
// rows x 32 bytes), version 1, swizzle 6.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFF) >> 4) | 1u << 16; }
#define TC_DESC_HI "0xC0004010"   // 256 >> 4 | 1 << 14 | 6 << 29

__device__ __forceinline__ constexpr uint32_t make_idesc(int prec, int n, bool neg_a) {
  uint32_t d = 0;
  d |= 1u << 4;                                        // D: FP32
  if (tc_is_tf32(prec)) { d |= 2u << 7; d |= 2u << 10; }  // A, B: TF32
  else { d |= 1u << 7; d |= 1u << 10; }                // A, B: BF16
  if (neg_a) d |= 1u << 13;
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(128 >> 4) << 24;
  return d;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t mbar_probe(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done;
}

// Wait for the phase of `parity` of an mbarrier to complete, for at most limit_ns nanoseconds
// of the global timer; limit_ns = 0 gives up without probing. On giving up, records `code` in
// the error flag (first failure wins) and returns false.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int code, uint64_t limit_ns) {
  if (limit_ns > 0) {
    if (mbar_probe(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (global_ns() - t0 < limit_ns)
      if (mbar_probe(bar, parity)) return true;
  }
  atomicCAS(err, 0, code);
  return false;
}

// Limit of the waits that drain a CTA's own copies and MMAs before it frees its tensor memory
// and exits, whatever limit the work's waits had.
constexpr uint64_t kDrainNs = 2000000000ull;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

template <int PREC>
__device__ __forceinline__ void mma(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
#define TC_MMA(kind)                                                                            \
  asm volatile("{\n.reg .pred p;\n.reg .b64 da, db;\nsetp.ne.b32 p, %4, 0;\n"                 \
               "mov.b64 da, {%1, " TC_DESC_HI "};\nmov.b64 db, {%2, " TC_DESC_HI "};\n"         \
               "tcgen05.mma.cta_group::1.kind::" kind " [%0], da, db, %3, p;\n}\n"              \
               ::"r"(d), "r"(a), "r"(b), "r"(idesc), "r"(acc))
  if (tc_is_tf32(PREC)) TC_MMA("tf32");
  else TC_MMA("f16");
#undef TC_MMA
}

// Per-tile operands of the MMAs: accumulator, instruction descriptors of N = AP nrow, AP / 2 nrow and that
// with A negated, and strides in 16-byte units (planes of A and B, steps of both).
struct TcMma {
  uint32_t d, dh, wide, half, neg, pa, pb, sa, sb;
};

// The MMAs of `steps` K steps (tc.cuh: the two forms of a complex product). a, b: low descriptor words of
// the first planes; acc = 0 starts the accumulator of the tile.
template <int PREC, bool NEG>
__device__ __forceinline__ void mma_steps(const TcMma& m, uint32_t a, uint32_t b, int steps, uint32_t acc) {
  constexpr int AP = tc_aplanes(PREC), H = AP / 2, G = tc_group(PREC);   // H: planes of one part (complex)
#pragma unroll
  for (int k = 0; k < G; ++k) {
    if (k >= steps) break;
    if (tc_is_real(PREC)) {
#pragma unroll
      for (int p = 0; p < AP; ++p) mma<PREC>(m.d, a + p * m.pa, b, m.wide, p == 0 && k == 0 ? acc : 1u);
    } else {
#pragma unroll
      for (int p = 0; p < H; ++p) mma<PREC>(m.d, a + p * m.pa, NEG ? b + H * m.pb : b, m.wide, p == 0 && k == 0 ? acc : 1u);
#pragma unroll
      for (int p = H; p < AP; ++p) {
        if (NEG) {
          mma<PREC>(m.d, a + p * m.pa, b, m.wide, 1u);
        } else {
          mma<PREC>(m.d, a + p * m.pa, b + H * m.pb, m.neg, 1u);
          mma<PREC>(m.dh, a + p * m.pa, b, m.half, 1u);
        }
      }
    }
    a += m.sa;
    b += m.sb;
  }
}

// 16 consecutive FP32 columns of the warp's 32 TMEM lanes (one row per lane); the caller waits
// with tcgen05.wait::ld before reading the registers.
__device__ __forceinline__ void tmem_ld16(uint32_t* v, uint32_t taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                 "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
               : "r"(taddr));
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

}  // namespace

// ---------------------------------------------------------------- packing kernels

// Planes of N consecutive K values of one row: 4-byte words of the BF16 planes (re_hi, re_lo, im_hi,
// im_lo) or of the TF32 planes (re, im). The BF16 split is done in FP32 after one conversion of each
// value (hi = bf16(x), lo = bf16(x - hi), with x - hi exact in FP32): the split's error, ~2^-17 |x|
// from rounding lo, is the same as splitting in FP64, and the FP64 pipe (2 ops per clock per SM) only
// converts. Negation is exact in both formats. Returns whether an infinity or NaN was met.
template <bool TF32, int N>
__device__ __forceinline__ bool split_row(const double2* v, uint32_t (*w)[N * (TF32 ? 4 : 2) / 4]) {
  constexpr uint32_t kInf = 0x7f800000u;
  uint32_t top = 0;   // largest exponent field: all ones for an infinity or NaN
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const float xr = __double2float_rn(v[q].x), xi = __double2float_rn(v[q].y);
    if (TF32) {
      w[0][q] = __float_as_uint(tf32_rna(xr));
      w[1][q] = __float_as_uint(tf32_rna(xi));
      top = max(top, max(w[0][q] & kInf, w[1][q] & kInf));
    } else {
      const __nv_bfloat16 rh = __float2bfloat16_rn(xr), ih = __float2bfloat16_rn(xi);
      ((__nv_bfloat16*)w[0])[q] = rh;
      ((__nv_bfloat16*)w[1])[q] = __float2bfloat16_rn(__fsub_rn(xr, __bfloat162float(rh)));
      ((__nv_bfloat16*)w[2])[q] = ih;
      ((__nv_bfloat16*)w[3])[q] = __float2bfloat16_rn(__fsub_rn(xi, __bfloat162float(ih)));
      top = max(top, max(__float_as_uint(__bfloat162float(rh)) & kInf, __float_as_uint(__bfloat162float(ih)) & kInf));
    }
  }
  return top == kInf;
}

__device__ __forceinline__ void store_words(uint8_t* p, const uint32_t (&w)[1]) { *(uint32_t*)p = w[0]; }
__device__ __forceinline__ void store_words(uint8_t* p, const uint32_t (&w)[2]) { *(uint2*)p = make_uint2(w[0], w[1]); }
__device__ __forceinline__ void store_words(uint8_t* p, const uint32_t (&w)[4]) {
  *(uint4*)p = make_uint4(w[0], w[1], w[2], w[3]);
}

// N consecutive K values of one row into every plane of its tile.
template <int PREC, int N>
__device__ __forceinline__ bool put_row(uint8_t* p, int64_t plane, bool neg, const double2* v) {
  constexpr bool TF32 = tc_is_tf32(PREC), REAL = tc_is_real(PREC);
  constexpr int AP = tc_aplanes(PREC), H = AP / 2, W = N * (TF32 ? 4 : 2) / 4;
  uint32_t w[TF32 ? 2 : 4][W];
  const bool bad = split_row<TF32, N>(v, w);
  if (neg) {   // [-im, re, im]
#pragma unroll
    for (int q = 0; q < H; ++q) {
      uint32_t m[W];
#pragma unroll
      for (int e = 0; e < W; ++e) m[e] = w[(REAL ? 0 : H) + q][e] ^ (TF32 ? 0x80000000u : 0x80008000u);
      store_words(p + q * plane, m);
    }
    p += H * plane;
  }
#pragma unroll
  for (int q = 0; q < AP; ++q) store_words(p + q * plane, w[q]);
  return bad;
}

// Pack FP64 complex blocks into panels (job rows: tc.cuh). A CTA takes one piece (kPackPiece units of
// one job) at a time, so large blocks spread over the whole grid. Blocks contiguous along K: a unit
// is a pair of K values of a row, consecutive threads along K (a row's 32 bytes of a plane per 8 or 4
// threads, whole rows next to each other); blocks contiguous along the rows: a unit is a 16-byte
// chunk of a row, consecutive threads along the rows, so each of the chunk's reads is coalesced. K
// beyond the block, up to a whole step, is written as zeros. The first thread also resets the tile
// counters of the two products that follow (ctr, or null); *bad (or null) is set when an infinity or
// NaN was packed.
template <int PREC>
__global__ void __launch_bounds__(256) k_pack(const double2* __restrict__ src, uint8_t* __restrict__ dst,
                                              const int64_t* __restrict__ jobs, int njobs, int64_t npieces,
                                              int* __restrict__ ctr, int* __restrict__ bad) {
  constexpr int STEP = tc_kstep(PREC), CH = STEP / 2, VB = tc_is_tf32(PREC) ? 4 : 2;
  if (ctr && blockIdx.x == 0 && threadIdx.x < 2) ctr[threadIdx.x] = 0;
  for (int64_t pc = blockIdx.x; pc < npieces; pc += gridDim.x) {
    int lo = 0, hi = njobs - 1;                  // the last job whose first piece is <= pc
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (jobs[TCJ * mid + 9] <= pc) lo = mid; else hi = mid - 1;
    }
    const int64_t* d = jobs + TCJ * lo;
    const int64_t s_off = d[0], ld = d[1];
    const bool trans = d[2] != 0;
    const int rows = (int)d[3], K = (int)d[4], rowtile = (int)d[6], nks = (int)d[7], prows = (int)d[8], row0 = (int)d[10];
    const int64_t p_off = d[5];
    const int per = trans ? nks * 2 : nks * CH;  // units per row
    const int64_t e64 = (pc - d[9]) * kPackPiece + threadIdx.x;
    if (e64 >= (int64_t)rows * per) continue;
    int r, u;
    if (e64 < 0x7fffffff) {
      const uint32_t e = (uint32_t)e64, q = (uint32_t)(trans ? rows : per);
      const uint32_t a = e / q, b = e - a * q;
      r = (int)(trans ? b : a);
      u = (int)(trans ? a : b);
    } else {
      r = (int)(trans ? e64 % rows : e64 / per);
      u = (int)(trans ? e64 / rows : e64 % per);
    }
    const int pr = row0 + r;
    const int rt = rowtile ? pr / rowtile : pr >> 7, tile_rows = rowtile ? rowtile : 128;
    const int left = prows - rt * tile_rows;
    const int nrow = left >= tile_rows ? tile_rows : (int)(rowtile ? tc_bpad(left) : tc_apad(left));
    const int full = rowtile ? tc_bplanes(PREC, tile_rows) : tc_aplanes(PREC);      // planes of a whole tile
    const int planes = rowtile ? tc_bplanes(PREC, nrow) : tc_aplanes(PREC);
    const bool neg = rowtile && tc_neg_planes(PREC, nrow);
    const int k0 = trans ? u * CH : u * 2, ks = k0 / STEP;
    uint8_t* p = dst + p_off + ((int64_t)rt * tile_rows * nks * full + (int64_t)ks * planes * nrow) * 32 +
                 sw32((uint32_t)((pr - rt * tile_rows) * 32 + (k0 - ks * STEP) * VB));
    const int64_t plane = (int64_t)nrow * 32;
    if (trans) {
      double2 v[CH];
      const double2* x = src + s_off + r;
#pragma unroll
      for (int q = 0; q < CH; ++q) v[q] = k0 + q < K ? x[(int64_t)(k0 + q) * ld] : make_double2(0.0, 0.0);
      if (put_row<PREC, CH>(p, plane, neg, v) && bad) *bad = 1;
    } else {
      double2 v[2];
      const double2* x = src + s_off + (int64_t)r * ld + k0;
#pragma unroll
      for (int q = 0; q < 2; ++q) v[q] = k0 + q < K ? x[q] : make_double2(0.0, 0.0);
      if (put_row<PREC, 2>(p, plane, neg, v) && bad) *bad = 1;
    }
  }
}

// ---------------------------------------------------------------- grouped GEMM

struct TcArgs {
  const uint8_t* a_base;   // packed A panels
  const uint8_t* b_base;   // packed B panels
  const TcItem* items;     // longest first
  const TcSeg* segs;
  const int64_t* rowmap;   // packed Z output (z_out), one entry per output row
  uint8_t* z_out;          // packed Z output, or null:
  double2* f_out;          // FP64 output
  int* ctr;                // item counter (zeroed before the launch), or null: CTA c runs items c, c + gridDim.x, ..
  int* err;
  const TcItem* alt;       // tiles to run instead if *bad (or null)
  const int* bad;
  int count, alt_count;
  int ntile;               // B rows of a whole tile
  int nslots, slot_bytes;
  uint64_t wait_ns;        // limit of each pipeline wait (ns); 0: the first wait gives up
};

constexpr int kAccSlots = 2;   // accumulator slots in TMEM, 256 columns each
constexpr int kTcRing = 8;     // items handed from the producer to the epilogue
constexpr int kTcEpi = 8;      // epilogue warps

// 32 bytes in one store.
__device__ __forceinline__ void store32(void* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

// One row's 32 bytes of a plane at p (its first 16 bytes at offset 0 or 16 by the row's swizzle).
__device__ __forceinline__ void store_plane(uint8_t* p, uint32_t row, const uint32_t* v) {
  const bool sw = (row >> 2) & 1;
  uint32_t o[8];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    o[e] = sw ? v[4 + e] : v[e];
    o[4 + e] = sw ? v[e] : v[4 + e];
  }
  store32(p + row * 32, o);
}

// 16 consecutive output values of one row (zeros from nvalid on) into a packed A panel: rm its row map
// entry, nks the panel's K steps, col the first value's K.
template <int PREC>
__device__ __forceinline__ void put_packed16(uint8_t* z, int64_t rm, int nks, int col, const float* re, const float* im,
                                             int nvalid) {
  constexpr int AP = tc_aplanes(PREC);
  const uint32_t row = (uint32_t)rm & 127u;
  const int64_t plane = (((rm >> 7) & 15) + 1) * 256;
  uint8_t* tile = z + (rm >> 12) * 256;
  if (tc_is_tf32(PREC)) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {   // two steps of 8
      const int ks = col / 8 + h;
      if (ks >= nks) break;
      uint32_t v[2][8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int j = 8 * h + e;
        v[0][e] = __float_as_uint(j < nvalid ? tf32_rna(re[j]) : 0.f);
        v[1][e] = __float_as_uint(j < nvalid ? tf32_rna(im[j]) : 0.f);
      }
#pragma unroll
      for (int p = 0; p < AP; ++p) store_plane(tile + ((int64_t)ks * AP + p) * plane, row, v[p]);
    }
  } else {
    uint32_t v[4][8];
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float x = e < nvalid ? re[e] : 0.f, y = e < nvalid ? im[e] : 0.f;
      const __nv_bfloat16 xh = __float2bfloat16_rn(x), yh = __float2bfloat16_rn(y);
      ((__nv_bfloat16*)v[0])[e] = xh;
      ((__nv_bfloat16*)v[1])[e] = __float2bfloat16_rn(x - __bfloat162float(xh));
      ((__nv_bfloat16*)v[2])[e] = yh;
      ((__nv_bfloat16*)v[3])[e] = __float2bfloat16_rn(y - __bfloat162float(yh));
    }
#pragma unroll
    for (int p = 0; p < AP; ++p) store_plane(tile + ((int64_t)(col / 16) * AP + p) * plane, row, v[p]);   // real: [hi, lo]
  }
}

// What a shared-memory slot holds, for the MMA thread: (word, low descriptor words of A and B). Word:
// steps (4 bits), first (16) and last (32) slot of the tile, nrow / 16 from bit 8, mrow / 8 from bit
// 16; first and no steps: no more work.
__device__ __forceinline__ uint32_t slot_word(int steps, bool first, bool last, int nrow, int mrow) {
  return (uint32_t)steps | (first ? 16u : 0u) | (last ? 32u : 0u) | (uint32_t)(nrow / 16) << 8 | (uint32_t)(mrow / 8) << 16;
}

template <int PREC>
__global__ void __launch_bounds__(320, 1) k_tc_gemm(TcArgs g) {
  constexpr int AP = tc_aplanes(PREC), G = tc_group(PREC), GROUPS = tc_groups(PREC);
  constexpr bool REAL = tc_is_real(PREC);
  extern __shared__ uint8_t dyn[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t bar_full[kTcMaxSlots], bar_empty[kTcMaxSlots], bar_acc_full[kAccSlots],
      bar_acc_empty[kAccSlots], bar_it_full[kTcRing], bar_it_empty[kTcRing], bar_drain;
  __shared__ uint4 s_slot[kTcMaxSlots];
  __shared__ int s_item[kTcRing];
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nslots = g.nslots;
  if (g.alt && *g.bad) {
    g.items = g.alt;
    g.count = g.alt_count;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < nslots; ++s) {
      mbar_init(smem_u32(&bar_full[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int b = 0; b < kAccSlots; ++b) {
      mbar_init(smem_u32(&bar_acc_full[b]), 1);
      mbar_init(smem_u32(&bar_acc_empty[b]), kTcEpi);
    }
    for (int r = 0; r < kTcRing; ++r) {
      mbar_init(smem_u32(&bar_it_full[r]), 1);
      mbar_init(smem_u32(&bar_it_empty[r]), kTcEpi);
    }
    mbar_init(smem_u32(&bar_drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  const uint32_t s0 = smem_u32(smem);

  if (warp == 0 && lane == 0) {
    // ---------------- producer
    int slot = 0;
    uint32_t phase = 0;
    int64_t fills = 0;   // slot fills issued
    bool ok = true;
    // Fixed deal: item rows are loaded one tile ahead. Counter: the next tile is claimed when the last
    // copy of this one is issued (a claim ahead of time would be tiles that another CTA could start
    // now); the slots in flight cover the latency.
    const bool fixed = g.ctr == nullptr;
    int cur = fixed ? (int)blockIdx.x : atomicAdd(g.ctr, 1);
    TcItem it = g.items[cur < g.count ? cur : 0];
    for (int n = 0;; ++n) {
      // hand the item to the epilogue (-1: no more)
      const int r = n % kTcRing;
      ok = mbar_wait(smem_u32(&bar_it_empty[r]), ((n / kTcRing) & 1) ^ 1, g.err, 10, g.wait_ns);
      if (!ok) break;
      s_item[r] = cur < g.count ? cur : -1;
      mbar_arrive(smem_u32(&bar_it_full[r]));   // release: the epilogue reads the item after it
      if (cur >= g.count) {   // and tell the MMA thread
        if (mbar_wait(smem_u32(&bar_empty[slot]), phase ^ 1, g.err, 11, g.wait_ns)) {
          s_slot[slot] = make_uint4(16u, 0u, 0u, 0u);
          mbar_arrive(smem_u32(&bar_full[slot]));
          ++fills;
        }
        break;
      }
      const int nxt = cur + (int)gridDim.x;
      TcItem itn = it;
      if (fixed) itn = g.items[nxt < g.count ? nxt : 0];
      const uint32_t ab = (uint32_t)(AP * it.mrow * 32), bb = (uint32_t)(tc_bplanes(PREC, it.nrow) * it.nrow * 32);   // bytes per step
      const int64_t at = (int64_t)it.rt * 128 * AP * 32, bt = (int64_t)it.nt * g.ntile * tc_bplanes(PREC, g.ntile) * 32;
      int left = it.nks, in = 0, cap = 0;   // steps still to copy; steps in the slot, and how many it gets
      uint32_t dst = 0, full = 0;
      TcSeg sg = it.seg[0], sg1 = it.seg[1];
      for (int s = 0; s < it.nseg && ok; ++s) {
        TcSeg sg2 = sg1;   // two ahead
        if (s + 2 < it.nseg) sg2 = g.segs[it.seg0 + s + 2];
        const int nks = (int)(sg.b & 0xffff);
        const uint8_t* a = g.a_base + sg.a + at * nks;
        const uint8_t* b = g.b_base + (sg.b >> 16) * 256 + bt * nks;
        for (int ks = 0; ks < nks;) {
          if (in == 0) {
            ok = mbar_wait(smem_u32(&bar_empty[slot]), phase ^ 1, g.err, 11, g.wait_ns);
            if (!ok) break;
            cap = left < G ? left : G;
            dst = s0 + slot * g.slot_bytes;
            s_slot[slot] = make_uint4(slot_word(cap, left == it.nks, left == cap, it.nrow, it.mrow), desc_lo(dst),
                                      desc_lo(dst + kTcABytes), 0u);
            full = smem_u32(&bar_full[slot]);
            mbar_expect_tx(full, cap * (ab + bb));
          }
          const int run = nks - ks < cap - in ? nks - ks : cap - in;
          bulk_g2s(dst + in * ab, a, run * ab, full);
          bulk_g2s(dst + kTcABytes + in * bb, b, run * bb, full);
          a += run * ab;
          b += run * bb;
          ks += run;
          left -= run;
          in += run;
          if (in == cap) {
            in = 0;
            ++fills;
            if (++slot == nslots) { slot = 0; phase ^= 1; }
          }
        }
        sg = sg1;
        sg1 = sg2;
      }
      if (!ok) break;
      if (fixed) {
        cur = nxt;
        it = itn;
      } else {
        cur = atomicAdd(g.ctr, 1);
        it = g.items[cur < g.count ? cur : 0];
      }
    }
    // drain: the last fills of every slot have landed before the CTA may exit (after normal
    // work they have, since the MMAs consumed them; after a wait gave up they may not have)
    for (int64_t f = fills - 1; f >= 0 && f >= fills - nslots; --f)
      mbar_wait(smem_u32(&bar_full[f % nslots]), (uint32_t)((f / nslots) & 1), g.err, 15, kDrainNs);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer. The tensor core queues only one or two MMAs, so every instruction of
    // this thread between the last MMA of a slot and the first of the next leaves it idle (a loop that
    // decoded the tile at every slot: 400 of 1500 cycles): the producer prepares the descriptors, and
    // what a tile's slots share is kept.
    constexpr int H = AP / 2;
    uint32_t bar = smem_u32(&bar_full[0]), rec = smem_u32(&s_slot[0]);   // of the slot
    const uint32_t to_empty = smem_u32(&bar_empty[0]) - smem_u32(&bar_full[0]), bar_end = bar + 8 * nslots;
    uint32_t phase = 0, acc_phase = 0;   // acc_phase bit b: phase of accumulator slot b
    int acc_slot = 0;
    TcMma m{};
    bool neg = false;
    for (;;) {
      if (!mbar_wait(bar, phase, g.err, 13, g.wait_ns)) break;
      uint32_t w, a, b;
      asm volatile("{\n.reg .b32 t;\nld.shared.v4.u32 {%0, %1, %2, t}, [%3];\n}\n" : "=r"(w), "=r"(a), "=r"(b) : "r"(rec) : "memory");
      if (w & 16u) {   // a tile's first slot
        if ((w & 15u) == 0) break;
        const int nrow = (int)((w >> 8) & 255u) * 16;
        neg = tc_neg_planes(PREC, nrow);
        m.pa = (w >> 16) * 16;
        m.pb = (uint32_t)nrow * 2;
        m.sa = AP * m.pa;
        m.sb = (uint32_t)tc_bplanes(PREC, nrow) * m.pb;
        m.wide = make_idesc(PREC, AP * nrow, false);
        m.half = make_idesc(PREC, H * nrow, false);
        m.neg = make_idesc(PREC, H * nrow, true);
        m.d = tmem + 256 * acc_slot;   // GROUPS x nrow <= 256 columns
        m.dh = m.d + H * nrow;
        if (!mbar_wait(smem_u32(&bar_acc_empty[acc_slot]), ((acc_phase >> acc_slot) & 1) ^ 1, g.err, 12, g.wait_ns)) break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t acc = w & 16u ? 0u : 1u;
      if (!tc_is_real(PREC) && neg) mma_steps<PREC, true>(m, a, b, (int)(w & 15u), acc);
      else mma_steps<PREC, false>(m, a, b, (int)(w & 15u), acc);
      mma_commit(bar + to_empty);
      if (w & 32u) {
        mma_commit(smem_u32(&bar_acc_full[acc_slot]));
        acc_phase ^= 1u << acc_slot;
        acc_slot ^= 1;
      }
      bar += 8;
      rec += 16;
      if (bar == bar_end) {
        bar -= 8 * nslots;
        rec -= 16 * nslots;
        phase ^= 1;
      }
    }
    // drain: every MMA this thread issued has completed before the tensor memory is freed
    mma_commit(smem_u32(&bar_drain));
    mbar_wait(smem_u32(&bar_drain), 0, g.err, 16, kDrainNs);
  } else if (warp >= 2) {
    // ---------------- epilogue
    const int quad = warp & 3, half = (warp - 2) >> 2;   // TMEM lanes 32*quad .. 32*quad+31
    uint32_t acc_phase = 0;   // bit b: phase of slot b
    int slot = 0;
    bool ok = true;
    for (int n = 0; ok; ++n) {
      const int r = n % kTcRing;
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_it_full[r]), (n / kTcRing) & 1, g.err, 17, g.wait_ns));
      if (!ok) break;
      const int item = s_item[r];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_it_empty[r]));
      if (item < 0) break;
      const TcItem it = g.items[item];
      const int row = quad * 32 + lane;
      int64_t rm = 0;
      if (g.z_out && row < it.rows) rm = g.rowmap[it.out + row];
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bar_acc_full[slot]), (acc_phase >> slot) & 1, g.err, 14, g.wait_ns));
      acc_phase ^= 1u << slot;
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t tacc = tmem + 256 * slot + ((uint32_t)(quad * 32) << 16);
      for (int cb = half * 16; cb < it.cols; cb += 32) {
        // group q of the accumulator sits at columns q * nrow; split BF16 adds the hi and lo
        // groups of each part
        uint32_t v[GROUPS][16];
#pragma unroll
        for (int q = 0; q < GROUPS; ++q) tmem_ld16(v[q], tacc + q * it.nrow + cb);
        asm volatile("tcgen05.wait::ld.sync.aligned;");
        if (row < it.rows && row >= it.row0) {
          const int nvalid = it.cols - cb < 16 ? it.cols - cb : 16;
          float re[16], im[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            re[j] = __uint_as_float(v[0][j]);
            im[j] = 0.f;
            if (PREC == TC_BF16X3_REAL) re[j] = __fadd_rn(re[j], __uint_as_float(v[GROUPS > 1 ? 1 : 0][j]));
            if (PREC == TC_TF32) im[j] = __uint_as_float(v[GROUPS > 1 ? 1 : 0][j]);
            if (PREC == TC_BF16X3) {
              re[j] = __fadd_rn(re[j], __uint_as_float(v[GROUPS > 1 ? 1 : 0][j]));
              im[j] = __fadd_rn(__uint_as_float(v[GROUPS > 2 ? 2 : 0][j]), __uint_as_float(v[GROUPS > 2 ? 3 : 0][j]));
            }
          }
          if (g.z_out) {
            put_packed16<PREC>(g.z_out, rm, (int)it.ld, it.nt * g.ntile + cb, re, im, nvalid);
          } else {
            double2* dst = g.f_out + it.out + row * it.ld + cb;
            if (nvalid == 16 && ((uintptr_t)dst & 31) == 0) {
#pragma unroll
              for (int j = 0; j < 16; j += 2) {
                const double o[4] = {(double)re[j], (double)im[j], (double)re[j + 1], (double)im[j + 1]};
                uint32_t u[8];
#pragma unroll
                for (int e = 0; e < 4; ++e) { u[2 * e] = (uint32_t)__double2loint(o[e]); u[2 * e + 1] = (uint32_t)__double2hiint(o[e]); }
                store32(dst + j, u);
              }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (j < nvalid) dst[j] = make_double2((double)re[j], (double)im[j]);
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_acc_empty[slot]));
      slot ^= 1;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// Kernel attributes (dynamic shared memory above 48 KB); called before any capture.
cudaError_t tc_gemm_init() {
  static DeviceOnce once;
  return once.run([] {
    cudaError_t e = cudaSuccess;
    for (const void* f : {(const void*)k_tc_gemm<TC_TF32>, (const void*)k_tc_gemm<TC_BF16X3>,
                          (const void*)k_tc_gemm<TC_TF32_REAL>, (const void*)k_tc_gemm<TC_BF16X3_REAL>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcMaxSmem);
    return e;
  });
}

cudaError_t tc_pack(const double2* src, uint8_t* dst, const int64_t* jobs, int njobs, int64_t npieces, int prec, int* ctr,
                    int* bad, cudaStream_t s) {
  if (njobs <= 0 || npieces <= 0) return cudaSuccess;
  auto k = prec == TC_TF32 ? k_pack<TC_TF32> : prec == TC_BF16X3 ? k_pack<TC_BF16X3>
           : prec == TC_TF32_REAL ? k_pack<TC_TF32_REAL> : k_pack<TC_BF16X3_REAL>;
  k<<<(unsigned)(npieces < 16384 ? npieces : 16384), 256, 0, s>>>(src, dst, jobs, njobs, npieces, ctr, bad);
  mrd::count_launch();
  return cudaGetLastError();
}

// From this many tiles per CTA on, they are dealt round robin instead of from a counter: short tiles,
// sorted, so that a CTA's share differs by about one of them, and their table rows can be loaded
// ahead (a claim, the row and the copies one after another take ~1500 cycles of the producer).
constexpr int kTcFixed = 4;

cudaError_t tc_gemm(const uint8_t* a_base, const uint8_t* b_base, const TcItem* items, int count, const TcItem* alt,
                    int alt_count, const int* bad, const TcSeg* segs,
                    const int64_t* rowmap, uint8_t* z_out, double2* f_out, int prec, TcCfg cfg, int ntile, int* ctr, int* err, int n_sm,
                    uint64_t wait_ns, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  cudaError_t ea = tc_gemm_init();
  if (ea != cudaSuccess) return ea;
  if (!tc_cfg_ok(prec, cfg) || ntile < 16 || ntile > cfg.ntile || ntile % 16) return cudaErrorInvalidValue;
  TcArgs g{a_base, b_base, items, segs, rowmap, z_out, f_out, ctr, err, alt, bad, count, alt_count, ntile, tc_slots(prec, cfg),
           tc_slot_bytes(prec, cfg.ntile), wait_ns};
  auto k = prec == TC_TF32 ? k_tc_gemm<TC_TF32> : prec == TC_BF16X3 ? k_tc_gemm<TC_BF16X3>
           : prec == TC_TF32_REAL ? k_tc_gemm<TC_TF32_REAL> : k_tc_gemm<TC_BF16X3_REAL>;
  if (count >= kTcFixed * n_sm) g.ctr = nullptr;
  k<<<(unsigned)(count < n_sm ? count : n_sm), 320, tc_smem_bytes(prec, cfg), s>>>(g);
  mrd::count_launch();
  return cudaGetLastError();
}

}  // namespace mrd
