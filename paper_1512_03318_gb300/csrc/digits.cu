// Device side of the digit-split grouped GEMM (digits.cuh): exponents, digit panels, and the
// persistent tcgen05 kernel.
//
// Panels: a left tile is 128 rows (the last one padded to 8), a right tile 32 columns (the last
// one padded to 16); per K step of 16 a tile holds its planes (digit 0 .. 7 of the real parts,
// then of the imaginary parts) back to back, each plane rows x 32 bytes in the 32-byte swizzle
// of the tcgen05 shared-memory descriptors, so that one cp.async.bulk brings the half of a
// step (one part's 8 planes) and a window of right digits is a run of consecutive rows.
#include <cuda_bf16.h>

#include "digits.cuh"
#include "ff.cuh"

namespace mrd {

namespace {

__device__ __forceinline__ uint32_t sw32(uint32_t off) { return off ^ (((off >> 7) & 1u) << 4); }

__device__ __forceinline__ int expo_field(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff); }

// Integer T = x 2^(t - e), e = emax - 1022 the exponent that bounds the row (|x| < 2^e), rounded
// to nearest: the mantissa shifted, in integer arithmetic (the FP64 pipe has 2 lanes per SM).
template <int BETA>
__device__ __forceinline__ long long fixed_of(double x, int emax) {
  constexpr int UP = (BETA == 8 ? 62 : 55) - 53;   // t - 53
  const long long b = __double_as_longlong(x);
  const int f = (int)(b >> 52) & 0x7ff;
  unsigned long long m = (unsigned long long)b & 0xfffffffffffffull;
  if (f) m |= 0x10000000000000ull;
  m <<= UP;
  const int d = min(emax - (f ? f : 1), 63);       // emax >= f: the row's largest (0 only if the row is denormal)
  if (d < 0) m <<= 1;
  else m = (m + ((1ull << d) >> 1)) >> d;
  const long long sg = b >> 63;
  return ((long long)m ^ sg) - sg;
}

// The 8 balanced digits of Ta and Tb as pairs of BF16 (a in the low half): w[i] = digit i.
// Adding half a base to every digit makes them unsigned bit fields of the sum; the fields are
// placed into the mantissa of a floating-point constant and the offset is subtracted (exact).
template <int BETA>
__device__ __forceinline__ void digit_pairs(long long Ta, long long Tb, uint32_t* w) {
  if (BETA == 8) {
    const unsigned long long a = (unsigned long long)Ta + 0x8080808080808080ull, b = (unsigned long long)Tb + 0x8080808080808080ull;
#pragma unroll
    for (int i = 0; i < kDgDigits; ++i) {
      const int y = kDgDigits - 1 - i;   // byte of digit i
      const uint32_t wa = y < 4 ? (uint32_t)a : (uint32_t)(a >> 32), wb = y < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
      const float fa = __uint_as_float(__byte_perm(wa, 0x4B000000u, 0x7540 | (y & 3))) - 8388736.f;   // 2^23 + 128
      const float fb = __uint_as_float(__byte_perm(wb, 0x4B000000u, 0x7540 | (y & 3))) - 8388736.f;
      w[i] = __byte_perm(__float_as_uint(fa), __float_as_uint(fb), 0x7632);
    }
  } else {
    constexpr unsigned long long H = 64ull * (1ull + (1ull << 7) + (1ull << 14) + (1ull << 21) + (1ull << 28) + (1ull << 35) +
                                              (1ull << 42) + (1ull << 49));
    const unsigned long long a = (unsigned long long)Ta + H, b = (unsigned long long)Tb + H;
    const __nv_bfloat162 off = __floats2bfloat162_rn(192.f, 192.f);   // 128 + 64
#pragma unroll
    for (int i = 0; i < kDgDigits; ++i) {
      const int sh = 7 * (kDgDigits - 1 - i);
      const uint32_t mask = i == 0 ? 0xffu : 0x7fu;   // the top field reaches 128
      const uint32_t fa = ((uint32_t)(a >> sh) & mask) | 0x43004300u, fb = (uint32_t)(b >> sh) & mask;
      uint32_t v = fa + (fb << 16);
      __nv_bfloat162 q = __hsub2(*(__nv_bfloat162*)&v, off);
      w[i] = *(uint32_t*)&q;
    }
  }
}

// ---------------------------------------------------------------- exponents

// expo[row] = largest exponent field of the row's real and imaginary parts. kcontig pieces: 64
// rows, 8 lanes per row along K; row-contiguous pieces: 32 values of K, lanes along the rows.
// Memory bound: 16 bytes read per element.
__global__ void __launch_bounds__(256) k_dg_expo(const double2* __restrict__ src, const DgJob* __restrict__ jobs,
                                                 const int2* __restrict__ pieces, int n_pieces, int* __restrict__ expo) {
  for (int pc = blockIdx.x; pc < n_pieces; pc += gridDim.x) {
    const int2 pi = pieces[pc];
    const DgJob& j = jobs[pi.x];
    if (j.off < 0) continue;
    const int rows = j.rows, K = j.K;
    const int64_t ld = j.ld;
    const double2* x = src + j.off;
    int* out = expo + j.exp0;
    if (j.flags & DGJ_KCONTIG) {
      const int sub = threadIdx.x >> 3, lane = threadIdx.x & 7;
      for (int r = pi.y + sub; r < rows && r < pi.y + kDgMaxRows; r += 32) {
        int e = 0;
#pragma unroll 4
        for (int k = lane; k < K; k += 8) {
          const double2 v = x[r * ld + k];
          e = max(e, max(expo_field(v.x), expo_field(v.y)));
        }
        const unsigned m = 0xffu << (threadIdx.x & 24);
        e = max(e, __shfl_xor_sync(m, e, 4));
        e = max(e, __shfl_xor_sync(m, e, 2));
        e = max(e, __shfl_xor_sync(m, e, 1));
        if (lane == 0 && e > 0) atomicMax(out + r, e);
      }
    } else {
      const int nr = rows < 256 ? rows : 256, kg = 256 / nr;
      const int kend = pi.y + kDgMaxK < K ? pi.y + kDgMaxK : K;
      const int r0 = threadIdx.x % nr, g = threadIdx.x / nr;
      if (g < kg)
        for (int r = r0; r < rows; r += nr) {
          int e = 0;
#pragma unroll 4
          for (int k = pi.y + g; k < kend; k += kg) {
            const double2 v = x[k * ld + r];
            e = max(e, max(expo_field(v.x), expo_field(v.y)));
          }
          if (e > 0) atomicMax(out + r, e);
        }
    }
  }
}

// ---------------------------------------------------------------- digits

// Position of (row pr, K position k) in a panel of prows rows: byte offset of plane 0; the
// plane stride (bytes) in *pstride. Tiles of 128 rows padded to 8 (tall) or of 32 padded to 16.
__device__ __forceinline__ int64_t panel_pos(bool tall, int prows, int nks, int planes, int pr, int k, int* pstride) {
  const int lg = tall ? 7 : 5, H = 1 << lg, pad = tall ? 7 : 15;
  const int t = pr >> lg, rin = pr & (H - 1);
  const int left = prows - (t << lg);
  const int nrow = left < H ? (left + pad) & ~pad : H;
  *pstride = nrow * 32;
  return ((int64_t)(t << lg) * nks + (int64_t)(k >> 4) * nrow) * (planes * 32) + sw32((uint32_t)(rin * 32 + (k & 15) * 2));
}

// Digits of every job's block. kcontig pieces: units (row, pair of K values), consecutive
// threads along K, one 4-byte store per plane (a row's 32-byte segment per 8 threads);
// row-contiguous pieces: units (chunk of 8 K values, row), consecutive threads along the rows,
// one 16-byte store per plane. K positions beyond the block are written as zeros.
// 16 bytes read and 32 written per complex element; the digits take ~45 instructions per real.
// Ly = 10, chi = 3200: LW (51 M elements) 0.52 ms, WR 0.76, Z (78 M) 0.81, 0.4-0.7 of the copy
// bandwidth. Units of 4 K values (8-byte stores) and of a whole panel step (32-byte stores) hold
// twice the registers: 0.52, 0.85 and 0.76 ms there, but 120 against 93 us for Z at chi = 1024.
template <int BETA, bool REAL>
__global__ void __launch_bounds__(256) k_dg_pack(const double2* __restrict__ src, uint8_t* __restrict__ dst,
                                                 const DgJob* __restrict__ jobs, const int2* __restrict__ pieces,
                                                 int n_pieces, const int* __restrict__ expo, int* __restrict__ words) {
  constexpr int P = REAL ? kDgDigits : 2 * kDgDigits;
  if (blockIdx.x == 0 && threadIdx.x == 0) words[DG_CTR] = 0;
  for (int pc = blockIdx.x; pc < n_pieces; pc += gridDim.x) {
    const int2 pi = pieces[pc];
    const DgJob& j = jobs[pi.x];
    const int rows = j.rows, K = j.off < 0 ? 0 : j.K, row0 = j.row0, k0 = j.k0, prows = j.prows, nks = j.nks;
    const int64_t ld = j.ld;
    const double2* x = src + j.off;
    uint8_t* panel = dst + j.panel;
    const int* ex = expo + j.exp0;
    const bool conj = (j.flags & DGJ_CONJ) != 0, tall = (j.flags & DGJ_TALL) != 0;
    if (j.flags & DGJ_KCONTIG) {
      const unsigned kc = (unsigned)j.kpad >> 1, n = (unsigned)rows * kc;
      const unsigned end = min(n, (unsigned)pi.y + kDgPairPiece);
      for (unsigned u = pi.y + threadIdx.x; u < end; u += 256) {
        const int r = (int)(u / kc), k = (int)(u - (unsigned)r * kc) * 2;
        double2 v0 = make_double2(0.0, 0.0), v1 = v0;
        if (k < K) v0 = x[r * ld + k];
        if (k + 1 < K) v1 = x[r * ld + k + 1];
        if (conj) { v0.y = -v0.y; v1.y = -v1.y; }
        const int e = ex[r];
        int ps;
        uint8_t* q = panel + panel_pos(tall, prows, nks, P, row0 + r, k0 + k, &ps);
        uint32_t w[kDgDigits];
        digit_pairs<BETA>(fixed_of<BETA>(v0.x, e), fixed_of<BETA>(v1.x, e), w);
#pragma unroll
        for (int i = 0; i < kDgDigits; ++i) *(uint32_t*)(q + i * ps) = w[i];
        if (!REAL) {
          digit_pairs<BETA>(fixed_of<BETA>(v0.y, e), fixed_of<BETA>(v1.y, e), w);
#pragma unroll
          for (int i = 0; i < kDgDigits; ++i) *(uint32_t*)(q + (kDgDigits + i) * ps) = w[i];
        }
      }
    } else {
      const unsigned n = (unsigned)rows * ((unsigned)j.kpad >> 3);
      const unsigned end = min(n, (unsigned)pi.y + kDgChunkPiece);
      for (unsigned u = pi.y + threadIdx.x; u < end; u += 256) {
        const int ch = (int)(u / (unsigned)rows), r = (int)(u - (unsigned)ch * rows);
        double2 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int k = ch * 8 + q;
          v[q] = k < K ? x[k * ld + r] : make_double2(0.0, 0.0);
          if (conj) v[q].y = -v[q].y;
        }
        const int e = ex[r];
        int ps;
        uint8_t* q = panel + panel_pos(tall, prows, nks, P, row0 + r, k0 + ch * 8, &ps);
#pragma unroll
        for (int part = 0; part < (REAL ? 1 : 2); ++part) {
          uint32_t w[4][kDgDigits];
#pragma unroll
          for (int h = 0; h < 4; ++h)
            digit_pairs<BETA>(fixed_of<BETA>(part ? v[2 * h].y : v[2 * h].x, e),
                              fixed_of<BETA>(part ? v[2 * h + 1].y : v[2 * h + 1].x, e), w[h]);
#pragma unroll
          for (int i = 0; i < kDgDigits; ++i)
            *(uint4*)(q + (part * kDgDigits + i) * ps) = make_uint4(w[0][i], w[1][i], w[2][i], w[3][i]);
        }
      }
    }
  }
}

// C map of every member (one warp each).
__global__ void __launch_bounds__(256) k_dg_cmap(const DgMember* __restrict__ members, int n, longlong2* __restrict__ cmap) {
  for (int i = (blockIdx.x * 256 + threadIdx.x) >> 5; i < n; i += gridDim.x * 8) {
    const DgMember m = members[i];
    for (int r = threadIdx.x & 31; r < m.rows; r += 32) cmap[m.first + r] = {m.off + r * m.step, m.other};
  }
}

// ---------------------------------------------------------------- tcgen05 helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-major operand of 32-byte rows in the 32-byte swizzle: 8-row atoms of 256 bytes
__device__ __forceinline__ uint64_t dg_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;                // leading offset (unused for swizzled K-major)
  d |= (uint64_t)(256 >> 4) << 32;       // stride between 8-row atoms
  d |= (uint64_t)1 << 46;                // descriptor version
  d |= (uint64_t)6 << 61;                // 32-byte swizzle
  return d;
}

// BF16 x BF16 -> FP32, M = 128, N = n; neg: A negated
__device__ __forceinline__ uint32_t dg_idesc(int n, bool neg) {
  return 1u << 4 | 1u << 7 | 1u << 10 | (neg ? 1u << 13 : 0u) | (uint32_t)(n >> 3) << 17 | (uint32_t)(kDgRows >> 4) << 24;
}

__device__ __forceinline__ void dg_mma(uint32_t tacc, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tacc), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t bar_probe(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done;
}

// Bounded wait for the phase of `parity`: gives up after limit_ns (0: at once, without probing)
// and records `code` in the error flag (the first one stays).
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity, int* err, int code, uint64_t limit_ns) {
  if (limit_ns > 0) {
    if (bar_probe(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (global_ns() - t0 < limit_ns)
      if (bar_probe(bar, parity)) return true;
  }
  atomicCAS(err, 0, code);
  return false;
}

constexpr uint64_t kDgDrainNs = 2000000000ull;   // limit of the waits that drain a CTA's own work

__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void dg_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t* v, uint32_t taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr));
}

// (hi 2^(4 BETA) + lo) 2^ex as a double, rounded to nearest, in integer arithmetic (the FP64 pipe
// would take 4 operations per number at 2 lanes per SM); lo in [0, 2^(4 BETA)). Without branches,
// so that the 32 conversions of a thread overlap: with the rare cases inside, a tile's conversions
// and stores took 12,000 cycles. `odd` is set when the result is outside the normal range (the value
// returned is then meaningless; the task is computed again in FP64).
template <int BETA>
__device__ __forceinline__ double to_double(long long hi, uint32_t lo, int ex, bool& odd) {
  const uint32_t sg = (uint32_t)(hi >> 63);   // 0 or all ones
  uint32_t c = lo << (32 - 4 * BETA);         // value = (a b c) 2^(ex + 4 BETA - 32) as 96 bits
  uint32_t b = (uint32_t)hi, a = (uint32_t)((unsigned long long)hi >> 32);
  const unsigned long long low = (((unsigned long long)b << 32 | c) ^ ((unsigned long long)sg << 32 | sg)) + (sg & 1);
  a = (a ^ sg) + (low == 0 ? (sg & 1) : 0u);
  b = (uint32_t)(low >> 32);
  c = (uint32_t)low;
  int e2 = ex + 4 * BETA - 32 + 95;           // exponent of bit 95
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool z = a == 0;
    a = z ? b : a;
    b = z ? c : b;
    c = z ? 0 : c;
    e2 -= z ? 32 : 0;
  }
  const int lz = __clz((int)a);
  const uint32_t m1 = __funnelshift_l(b, a, lz), m0 = __funnelshift_l(c, b, lz);
  e2 -= lz;
  const unsigned long long m = (unsigned long long)m1 << 32 | m0, r = (m >> 11) + ((m >> 10) & 1);
  const bool zero = (hi | (long long)lo) == 0;
  odd = odd || (!zero && (unsigned)(e2 + 1022) >= 2045u);
  const unsigned long long bits = ((unsigned long long)(uint32_t)(e2 + 1022) << 52) + r + ((unsigned long long)(sg & 1) << 63);
  return __longlong_as_double(zero ? 0ll : (long long)bits);
}

}  // namespace

// ---------------------------------------------------------------- the product

struct DgArgs {
  const uint8_t *a, *b;      // panels of operand buffers 0 and 1
  const DgGroup* groups;
  const DgItem* items;
  int first, count;
  const longlong2* cmap;
  const int *ea, *eb;        // exponents of operand buffers 0 and 1
  const int2* splits;
  uint8_t* partial;
  int *tickets, *res;
  double2* c;
  int* words;
  uint64_t wait_ns;
};

constexpr int kDgASlots = 5;                    // half steps of the left operand (32 KB each)
constexpr int kDgBSlots = 3;                    // steps of the right operand (16 KB each)
constexpr int kDgASlot = kDgRows * 32 * kDgDigits;
constexpr int kDgBSlot = kDgCols * 32 * 2 * kDgDigits;
constexpr int kDgSmem = kDgASlots * kDgASlot + kDgBSlots * kDgBSlot + 1024;
constexpr int kDgRing = 4;                      // items handed from the producer to the other roles
constexpr int kDgEpi = 8;                       // epilogue warps

// Persistent, one CTA per SM, 10 warps: warp 0 takes items (longest K first) from a global
// counter and issues the bulk copies, warp 1 owns TMEM (all 512 columns: 8 levels x 32 columns
// x re, im) and issues the MMAs, warps 2 .. 9 flush the levels (warp w reads TMEM lanes
// 32 (w % 4) .. and half of the columns) and write the tile.
// The left operand moves in half steps (the 8 planes of one part) through a ring of 5, the
// right one in steps through a ring of 3. One step of a full complex tile is 32 MMAs of
// N = 256, 224, .. 32: 2510 cycles at the measured N / 2 (at least 48) cycles per MMA for 80 KB of
// operands.
template <int BETA, bool REAL>
__global__ void __launch_bounds__(320, 1) k_dg_gemm(DgArgs g) {
  constexpr int FLUSH = BETA == 8 ? 6 : 16;
  constexpr int PARTS = REAL ? 1 : 2;
  constexpr int PB = 32 * kDgDigits * PARTS;    // panel bytes per row and step
  extern __shared__ uint8_t dyn[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)dyn + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t a_full[kDgASlots], a_empty[kDgASlots], b_full[kDgBSlots], b_empty[kDgBSlots],
      acc_full, acc_empty, it_full[kDgRing], it_empty[kDgRing], drain;
  __shared__ int s_item[kDgRing];
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* err = g.words + DG_ERR;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDgASlots; ++s) { bar_init(smem_u32(&a_full[s]), 1); bar_init(smem_u32(&a_empty[s]), 1); }
    for (int s = 0; s < kDgBSlots; ++s) { bar_init(smem_u32(&b_full[s]), 1); bar_init(smem_u32(&b_empty[s]), 1); }
    for (int s = 0; s < kDgRing; ++s) { bar_init(smem_u32(&it_full[s]), 1); bar_init(smem_u32(&it_empty[s]), 1 + kDgEpi); }
    bar_init(smem_u32(&acc_full), 1);
    bar_init(smem_u32(&acc_empty), kDgEpi);
    bar_init(smem_u32(&drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  const uint32_t sa0 = smem_u32(smem), sb0 = sa0 + kDgASlots * kDgASlot;

  if (warp == 0 && lane == 0) {
    // ---------------- producer
    int as = 0, bs = 0, n = 0;
    uint32_t ap = 0, bp = 0;
    bool ok = true;
    int64_t fa = 0, fb = 0;   // fills issued
    int next = atomicAdd(g.words + DG_CTR, 1);
    for (;;) {
      const int item = next;
      const int slot = n % kDgRing;
      ok = bar_wait(smem_u32(&it_empty[slot]), ((n / kDgRing) & 1) ^ 1, err, 21, g.wait_ns);
      if (!ok) break;
      s_item[slot] = item < g.count ? g.first + item : -1;
      bar_arrive(smem_u32(&it_full[slot]));   // release: the roles read the item after it
      ++n;
      if (item >= g.count) break;
      next = atomicAdd(g.words + DG_CTR, 1);
      const DgItem it = g.items[g.first + item];
      const DgGroup& q = g.groups[it.group];
      const int tn = (q.N + kDgCols - 1) / kDgCols, rt = it.tile / tn, ct = it.tile % tn;
      const int ml = q.R - rt * kDgRows, nl = q.N - ct * kDgCols, nks = q.nks;
      const uint32_t mrow = ml < kDgRows ? (ml + 7) / 8 * 8 : kDgRows, nrow = nl < kDgCols ? (nl + 15) / 16 * 16 : kDgCols;
      const uint8_t* a = (q.tall_op ? g.b : g.a) + q.a_off + (int64_t)rt * kDgRows * nks * PB;
      const uint8_t* b = (q.tall_op ? g.a : g.b) + q.b_off + (int64_t)ct * kDgCols * nks * PB;
      const uint32_t ab = mrow * 32 * kDgDigits, bb = nrow * PB;
      for (int ks = it.ks & 0xffff, ke = it.ks >> 16; ks < ke && ok; ++ks) {
        ok = bar_wait(smem_u32(&b_empty[bs]), bp ^ 1, err, 22, g.wait_ns);
        if (!ok) break;
        bar_expect(smem_u32(&b_full[bs]), bb);
        bulk_load(sb0 + bs * kDgBSlot, b + (int64_t)ks * bb, bb, smem_u32(&b_full[bs]));
        ++fb;
        if (++bs == kDgBSlots) { bs = 0; bp ^= 1; }
        for (int h = 0; h < PARTS && ok; ++h) {
          ok = bar_wait(smem_u32(&a_empty[as]), ap ^ 1, err, 23, g.wait_ns);
          if (!ok) break;
          bar_expect(smem_u32(&a_full[as]), ab);
          bulk_load(sa0 + as * kDgASlot, a + ((int64_t)ks * PARTS + h) * ab, ab, smem_u32(&a_full[as]));
          ++fa;
          if (++as == kDgASlots) { as = 0; ap ^= 1; }
        }
      }
      if (!ok) break;
    }
    // drain: every copy of this CTA has landed before it may exit
    for (int64_t f = fa - 1; f >= 0 && f >= fa - kDgASlots; --f)
      bar_wait(smem_u32(&a_full[f % kDgASlots]), (uint32_t)((f / kDgASlots) & 1), err, 24, kDgDrainNs);
    for (int64_t f = fb - 1; f >= 0 && f >= fb - kDgBSlots; --f)
      bar_wait(smem_u32(&b_full[f % kDgBSlots]), (uint32_t)((f / kDgBSlots) & 1), err, 25, kDgDrainNs);
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer
    int as = 0, bs = 0;
    uint32_t ap = 0, bp = 0, flushes = 0;
    bool ok = true;
    for (int n = 0; ok; ++n) {
      const int slot = n % kDgRing;
      ok = bar_wait(smem_u32(&it_full[slot]), (n / kDgRing) & 1, err, 31, g.wait_ns);
      if (!ok) break;
      const int item = s_item[slot];
      bar_arrive(smem_u32(&it_empty[slot]));
      if (item < 0) break;
      const DgItem it = g.items[item];
      const DgGroup& q = g.groups[it.group];
      const int tn = (q.N + kDgCols - 1) / kDgCols, rt = it.tile / tn, ct = it.tile % tn;
      const int ml = q.R - rt * kDgRows, nl = q.N - ct * kDgCols, nks = (it.ks >> 16) - (it.ks & 0xffff);
      const uint32_t mrow = ml < kDgRows ? (ml + 7) / 8 * 8 : kDgRows, nrow = nl < kDgCols ? (nl + 15) / 16 * 16 : kDgCols;
      const uint64_t pa = (mrow * 32) >> 4, pb = (nrow * 32) >> 4;   // plane strides (descriptor units)
      for (int ks = 0; ks < nks && ok; ++ks) {
        const bool fresh = ks % FLUSH == 0;
        if (fresh) {   // the levels of the previous flush have been read
          ok = bar_wait(smem_u32(&acc_empty), (flushes & 1) ^ 1, err, 32, g.wait_ns);
          if (!ok) break;
          ++flushes;
          asm volatile("tcgen05.fence::after_thread_sync;");
        }
        ok = bar_wait(smem_u32(&b_full[bs]), bp, err, 33, g.wait_ns);
        if (!ok) break;
        const uint64_t b0 = dg_desc(sb0 + bs * kDgBSlot), b1 = b0 + kDgDigits * pb;
        for (int h = 0; h < PARTS && ok; ++h) {
          ok = bar_wait(smem_u32(&a_full[as]), ap, err, 34, g.wait_ns);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
          const uint64_t a0 = dg_desc(sa0 + as * kDgASlot);
          // real part A_re: C_re += A_re B_re, C_im += A_re B_im; imaginary part A_im:
          // C_re -= A_im B_im, C_im += A_im B_re
#pragma unroll
          for (int i = 0; i < kDgDigits; ++i) {
            const int nn = (kDgDigits - i) * (int)nrow;
            const uint32_t acc = fresh && h == 0 && i == 0 ? 0u : 1u;
            const uint32_t d = tmem + i * nrow;
            if (REAL) {
              dg_mma(d, a0 + i * pa, b0, dg_idesc(nn, false), acc);
            } else {
              dg_mma(d, a0 + i * pa, h == 0 ? b0 : b1, dg_idesc(nn, h != 0), acc);
              dg_mma(d + 256, a0 + i * pa, h == 0 ? b1 : b0, dg_idesc(nn, false), acc);
            }
          }
          dg_commit(smem_u32(&a_empty[as]));
          if (++as == kDgASlots) { as = 0; ap ^= 1; }
        }
        if (!ok) break;
        dg_commit(smem_u32(&b_empty[bs]));
        if (++bs == kDgBSlots) { bs = 0; bp ^= 1; }
        if (ks % FLUSH == FLUSH - 1 || ks == nks - 1) dg_commit(smem_u32(&acc_full));
      }
    }
    // drain: every MMA this thread issued has completed before the tensor memory is freed
    dg_commit(smem_u32(&drain));
    bar_wait(smem_u32(&drain), 0, err, 35, kDgDrainNs);
  } else if (warp >= 2) {
    // ---------------- epilogue
    const int quad = warp & 3, half = (warp - 2) >> 2;
    uint32_t flushes = 0;
    bool ok = true;
    for (int n = 0; ok; ++n) {
      const int slot = n % kDgRing;
      ok = __all_sync(0xffffffffu, bar_wait(smem_u32(&it_full[slot]), (n / kDgRing) & 1, err, 41, g.wait_ns));
      if (!ok) break;
      const int item = s_item[slot];
      __syncwarp();
      if (lane == 0) bar_arrive(smem_u32(&it_empty[slot]));
      if (item < 0) break;
      const DgItem it = g.items[item];
      const DgGroup& q = g.groups[it.group];
      const int N = q.N, R = q.R, nks = (it.ks >> 16) - (it.ks & 0xffff);
      const int tn = (N + kDgCols - 1) / kDgCols, rt = it.tile / tn, ct = it.tile % tn;
      const int nl = N - ct * kDgCols;
      const int nrow = nl < kDgCols ? (nl + 15) / 16 * 16 : kDgCols;
      const int w = nrow / 2;                       // columns of this warp's half: 8 or 16
      const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + half * w;
      const int row = rt * kDgRows + quad * 32 + lane, col0 = ct * kDgCols + half * w;
      // this lane's row exponent and (lanes 0 .. 15) column exponent and C map entries, fetched
      // while the MMAs run
      const int* ea = q.tall_op ? g.eb : g.ea;
      const int* eb = q.tall_op ? g.ea : g.eb;
      const bool by_row = q.cm_rows;
      int er = 0, ec = 0;
      longlong2 map = {0, 0};
      if (row < R) er = ea[q.ea + row];
      if (lane < w && col0 + lane < N) ec = eb[q.eb + col0 + lane];
      if (by_row ? row < R : lane < w && col0 + lane < N) map = g.cmap[q.cm + (by_row ? row : col0 + lane)];
      // sums of the tile: hi 2^(4 BETA) + lo (96 bits) per real number
      long long hi[PARTS][16];
      uint32_t lo[PARTS][16];
#pragma unroll
      for (int p = 0; p < PARTS; ++p)
#pragma unroll
        for (int c = 0; c < 16; ++c) { hi[p][c] = 0; lo[p][c] = 0; }
      for (int f = 0; f < nks; f += FLUSH) {
        ok = __all_sync(0xffffffffu, bar_wait(smem_u32(&acc_full), flushes & 1, err, 42, g.wait_ns));
        ++flushes;
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
        for (int p = 0; p < PARTS; ++p)
#pragma unroll
          for (int cb = 0; cb < 16; cb += 4) {
            if (cb >= w) continue;
            uint32_t v[kDgDigits][4];
#pragma unroll
            for (int l = 0; l < kDgDigits; ++l) tmem_ld4(v[l], tq + p * 256 + l * nrow + cb);
            asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              long long th = 0, tl = lo[p][cb + c];
#pragma unroll
              for (int l = 0; l < 4; ++l) {
                th += (long long)__float2int_rn(__uint_as_float(v[l][c])) << (BETA * (3 - l));
                tl += (long long)__float2int_rn(__uint_as_float(v[4 + l][c])) << (BETA * (3 - l));
              }
              hi[p][cb + c] += th + (tl >> (4 * BETA));
              lo[p][cb + c] = (uint32_t)tl & (uint32_t)((1ull << (4 * BETA)) - 1);
            }
          }
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncwarp();
        if (lane == 0) bar_arrive(smem_u32(&acc_empty));
      }
      if (!ok) break;
      if (it.split >= 0) {
        // a part of a tile cut along K: every part but the last to arrive leaves its sums in its
        // slot, the last one adds them (integers: the order does not matter) and goes on
        const int2 sp = g.splits[it.split >> 6];
        const int part = it.split & 63;
        auto slot_of = [&](int pt) { return g.partial + (int64_t)(sp.x + pt) * kDgSlotBytes + (warp - 2) * (kDgSlotBytes / kDgEpi); };
        long long* sh = (long long*)slot_of(part);              // [part of the number][column][lane]
        uint32_t* sl = (uint32_t*)(sh + PARTS * 16 * 32);
#pragma unroll
        for (int p = 0; p < PARTS; ++p)
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (c < w) {
              sh[(p * 16 + c) * 32 + lane] = hi[p][c];
              sl[(p * 16 + c) * 32 + lane] = lo[p][c];
            }
        __threadfence();
        __syncwarp();
        int* tk = g.tickets + (it.split >> 6) * kDgEpi + (warp - 2);
        int t = 0;
        if (lane == 0) t = atomicAdd(tk, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t != sp.y - 1) continue;
        __threadfence();
        for (int o = 0; o < sp.y; ++o) {
          if (o == part) continue;
          const long long* oh = (const long long*)slot_of(o);
          const uint32_t* ol = (const uint32_t*)(oh + PARTS * 16 * 32);
#pragma unroll
          for (int p = 0; p < PARTS; ++p)
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (c < w) {
                const unsigned long long l = (unsigned long long)lo[p][c] + __ldcg(ol + (p * 16 + c) * 32 + lane);
                hi[p][c] += __ldcg(oh + (p * 16 + c) * 32 + lane) + (long long)(l >> (4 * BETA));
                lo[p][c] = (uint32_t)l & (uint32_t)((1ull << (4 * BETA)) - 1);
              }
        }
      }
      const int exr = er - 2 * 1022 + (BETA == 8 ? -68 : -61);
      int top[16];   // upper word of the larger part of each result; the largest number outside the normal range
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int eg = __shfl_sync(0xffffffffu, ec, c);
        const long long at = by_row ? map.x + (long long)(col0 + c) * map.y
                                    : __shfl_sync(0xffffffffu, map.x, c) + (long long)row * __shfl_sync(0xffffffffu, map.y, c);
        bool odd = false;
        const double2 o = make_double2(to_double<BETA>(hi[0][c], lo[0][c], exr + eg, odd),
                                       REAL ? 0.0 : to_double<BETA>(hi[PARTS - 1][c], lo[PARTS - 1][c], exr + eg, odd));
        const bool valid = row < R && c < w && col0 + c < N;
        top[c] = !valid ? 0 : odd ? 0x7fffffff : max(__double2hiint(o.x) & 0x7fffffff, __double2hiint(o.y) & 0x7fffffff);
        if (valid) g.c[at] = o;
      }
      // the largest of this lane's row, or (lanes 0 .. 15) column, of the C map
      int most = 0;
      if (by_row) {
#pragma unroll
        for (int c = 0; c < 16; ++c) most = max(most, top[c]);
      } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int v = __reduce_max_sync(0xffffffffu, top[c]);
          if (lane == c) most = v;
        }
      }
      if (most > 0) atomicMax(g.res + q.cm + (by_row ? row : col0 + lane), most >> 20);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // (k_dg_check waits for this grid's results)
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// ---------------------------------------------------------------- products that are computed again

constexpr int kDgFF = 1 << 30;   // mark of a listed tile that float-float arithmetic can do

// sum_k |s_rk| |u_ck| over the bounds 2^(er - 1022) of row r and 2^(ec - 1022) of column c, in the part (real or
// imaginary) where it is larger; NW warps, 8 lanes per block, the lanes along K. In FP32 from truncated
// magnitudes, so that the FP64 pipe has no part in it: low by 2^-20 at most, and right to 2^-10 in a sum
// of 10^4 terms. FP64 application at Ly = 4, chi = 48 70.1 -> 68.0 us, at Ly = 8, chi = 1024 488 -> 485.
__device__ __forceinline__ float mag_over(double x, int e) {   // |x| / 2^(e - 1022), truncated, below 1
  const int hi = __double2hiint(x) & 0x7fffffff, f = (hi >> 20) - e + 126;
  return f <= 0 ? 0.f : __int_as_float(f << 23 | (hi & 0xfffff) << 3 | (int)((unsigned)__double2loint(x) >> 29));
}
template <int NW>
__device__ __forceinline__ float terms_sum(const DgJob* sj, const DgJob* uj, int n, const double2* ssrc, const double2* usrc, int r,
                                           int c, int er, int ec, int lane, int warp) {
  float re = 0.f, im = 0.f;
  for (int f = warp * 4 + (lane >> 3); f < n; f += 4 * NW) {
    const DgJob &x = sj[f], &y = uj[f];
    if (x.off < 0) continue;
    const int64_t x0 = x.off + (x.flags & DGJ_KCONTIG ? r * x.ld : r), xs = x.flags & DGJ_KCONTIG ? 1 : x.ld;
    const int64_t y0 = y.off + (y.flags & DGJ_KCONTIG ? c * y.ld : c), ys = y.flags & DGJ_KCONTIG ? 1 : y.ld;
    const int K = y.K;
#pragma unroll 4
    for (int k = lane & 7; k < K; k += 8) {
      const double2 p = ssrc[x0 + k * xs], q = usrc[y0 + k * ys];
      const float px = mag_over(p.x, er), py = mag_over(p.y, er), qx = mag_over(q.x, ec), qy = mag_over(q.y, ec);
      re = fmaf(px, qx, fmaf(py, qy, re));
      im = fmaf(px, qy, fmaf(py, qx, im));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    re += __shfl_xor_sync(0xffffffffu, re, o);
    im += __shfl_xor_sync(0xffffffffu, im, o);
  }
  if constexpr (NW > 1) {
    __shared__ float2 part[NW];
    if (lane == 0) part[warp] = make_float2(re, im);
    __syncthreads();
    re = im = 0.f;
    for (int w = 0; w < NW; ++w) {
      re += part[w].x;
      im += part[w].y;
    }
    __syncthreads();
  }
  return fmaxf(re, im);
}

// Whether a task has to be computed again (0: no, 1: in FP64, 2: in float-float): a row or column of its
// operands is not finite (exponent field 2047), a result is outside the normal range (marked likewise), or
// the fixed point was too coarse: no result within 2^kDgSpread of the largest row times the largest
// column, and not for want of large terms (sums that cancel are as inexact in FMAs): the terms of the
// largest row and column tell. NW warps, all with the same answer.
template <int NW>
__device__ __forceinline__ int task_form(const DgGroup& g, const DgMember& m, const DgJob* sjobs, const DgJob* ujobs, const double2* ssrc,
                                         const double2* usrc, const int* e0, const int* e1, const int* res, bool ff, int lane, int warp) {
  const int *tall = g.tall_op ? e1 : e0, *flat = g.tall_op ? e0 : e1;
  const int* stacked = (g.cm_rows ? tall + g.ea : flat + g.eb) + (m.first - g.cm);
  const int* shared = g.cm_rows ? flat + g.eb : tall + g.ea;
  const int ns = g.cm_rows ? g.N : g.R;
  int a = 0, b = 0, o = 0, ra = 0, cb = 0;   // largest exponents, and a row and a column that have them
  for (int r = lane; r < m.rows; r += 32) {
    const int e = stacked[r];
    if (e > a) { a = e; ra = r; }
    o = max(o, res[m.first + r]);
  }
  for (int c = lane; c < ns; c += 32) {
    const int e = shared[c];
    if (e > b) { b = e; cb = c; }
  }
  const int am = __reduce_max_sync(0xffffffffu, a), bm = __reduce_max_sync(0xffffffffu, b);
  o = __reduce_max_sync(0xffffffffu, o);
  if (am == 2047 || bm == 2047 || o == 2047) return 1;
  // bounds of rows and columns 2^(field - 1022), result >= 2^(field - 1023)
  if (am == 0 || bm == 0 || am + bm - o <= 1021 + kDgSpread) return 0;
  const int r = __shfl_sync(0xffffffffu, ra, __ffs(__ballot_sync(0xffffffffu, a == am)) - 1);
  const int c = __shfl_sync(0xffffffffu, cb, __ffs(__ballot_sync(0xffffffffu, b == bm)) - 1);
  const float line = ff ? kDgLineFF : kDgLine64;
  if (terms_sum<NW>(sjobs + m.job, ujobs + g.job, g.n_jobs, ssrc, usrc, r, c, am, bm, lane, warp) >= line) return 0;
  // float-float products take operands within the FP32 range only
  return ff && abs(am - 1022) <= 30 && abs(bm - 1022) <= 30 ? 2 : 1;
}

// One listed tile: 8 stacked rows x 8 of the shared side, FP64 FMAs or float-float (REAL: imaginary parts taken
// and returned as zeros). Few blocks are computed again, so what counts is the time of one: the FP64 pipe
// has 2 lanes per SM, and a tile is small so that a block spreads over many SMs (32 x 32 tiles: 17 us
// per 16 values of K, FP64 update at Ly = 8, chi = 1024 208 ms, with these 181, for 12 blocks in 40 products). Four groups of 64
// threads take the chunks of 16 values of K in turn, each with buffers and a barrier of its own, so that
// their loads overlap; their sums are added in a fixed order. Float-float operands are split from
// their bits, which the FP64 pipe has no part in: step 2 of the refinement in the update that repeats most
// (Ly = 10, chi = 3200) 6.2 -> 5.3 ms.
constexpr int kRedoTile = kDgRedoTile, kRedoK = 16, kRedoGroups = 4, kRedoJobs = 64;
struct RedoJob {
  int64_t so, uo, sl, ul;   // offsets and strides of the blocks; so < 0: a block this task does not multiply
  int K, flags;             // flags: stacked operand's, shared operand's << 4
};
template <bool FFM, bool REAL>
struct RedoSmem {
  RedoJob jobs[kRedoJobs];
  alignas(16) uint8_t a[kRedoGroups][kRedoTile * (kRedoK + 1) * 16], b[kRedoGroups][kRedoK * (kRedoTile + 1) * 16];
  float2 as[kRedoGroups][FFM && !REAL ? kRedoTile * (kRedoK + 1) : 1], bs[kRedoGroups][FFM && !REAL ? kRedoK * (kRedoTile + 1) : 1];
  double2 sum[kRedoGroups][kRedoTile * kRedoTile];
};

template <bool FFM, bool REAL, class Smem>
__device__ __forceinline__ void redo_tile(const DgGroup& g, const DgMember& m, int tile, const DgJob* __restrict__ sjobs,
                                          const DgJob* __restrict__ ujobs, const double2* __restrict__ ssrc,
                                          const double2* __restrict__ usrc, double2* __restrict__ C, Smem& sm) {
  const int tid = threadIdx.x, grp = tid >> 6, t = tid & 63, orow = t >> 3, ocol = t & 7;
  const int ns = g.cm_rows ? g.N : g.R, tn = (ns + kRedoTile - 1) / kRedoTile;
  const int r0 = tile / tn * kRedoTile, c0 = tile % tn * kRedoTile;
  auto group_sync = [&] { asm volatile("bar.sync %0, 64;" ::"r"(1 + grp) : "memory"); };
  auto put = [&](uint8_t* s, float2* sum, int at, double2 v, bool conj) {   // stage one element
    if (conj) v.y = -v.y;
    if (REAL) v.y = 0.0;
    if constexpr (FFM) {
      const FF re = ff_from_bits(v.x), im = ff_from_bits(v.y);
      const float4 x = make_float4(re.hi, im.hi, re.lo, im.lo);
      ((float4*)s)[at] = x;
      if (!REAL) sum[at] = cff_sum(x);
    } else {
      ((double2*)s)[at] = v;
    }
  };
  double2 acc = make_double2(0.0, 0.0);
  CAcc fac = {};
  int chunk = 0;   // of the whole product
  for (int f0 = 0; f0 < g.n_jobs; f0 += kRedoJobs) {
    const int nf = g.n_jobs - f0 < kRedoJobs ? g.n_jobs - f0 : kRedoJobs;
    __syncthreads();
    if (tid < nf) {
      const DgJob &x = sjobs[m.job + f0 + tid], &y = ujobs[g.job + f0 + tid];
      sm.jobs[tid] = {x.off, y.off, x.ld, y.ld, y.K, x.flags | y.flags << 4};
    }
    __syncthreads();
    for (int f = 0; f < nf; ++f) {
      const RedoJob& j = sm.jobs[f];
      if (j.so < 0) continue;
      const int K = j.K, nc = (K + kRedoK - 1) / kRedoK;
      const bool sk = j.flags & DGJ_KCONTIG, uk = (j.flags >> 4) & DGJ_KCONTIG;
      for (int i = (grp - chunk) & (kRedoGroups - 1); i < nc; i += kRedoGroups) {
        const int k0 = i * kRedoK;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int e = t + q * 64;
          const int sr = sk ? e >> 4 : e & 7, sc = sk ? e & 15 : e >> 3;
          double2 v = make_double2(0.0, 0.0), w = v;
          if (r0 + sr < m.rows && k0 + sc < K) v = ssrc[j.so + (sk ? (r0 + sr) * j.sl + k0 + sc : (k0 + sc) * j.sl + r0 + sr)];
          const int ur = uk ? e >> 4 : e & 7, uc = uk ? e & 15 : e >> 3;
          if (c0 + ur < ns && k0 + uc < K) w = usrc[j.uo + (uk ? (c0 + ur) * j.ul + k0 + uc : (k0 + uc) * j.ul + c0 + ur)];
          put(sm.a[grp], sm.as[grp], sr * (kRedoK + 1) + sc, v, j.flags & DGJ_CONJ);
          put(sm.b[grp], sm.bs[grp], uc * (kRedoTile + 1) + ur, w, (j.flags >> 4) & DGJ_CONJ);
        }
        group_sync();
        const int kn = K - k0 < kRedoK ? K - k0 : kRedoK;
        for (int k = 0; k < kn; ++k) {
          const int p = orow * (kRedoK + 1) + k, q = k * (kRedoTile + 1) + ocol;
          if constexpr (FFM) {
            const float4 x = ((const float4*)sm.a[grp])[p], y = ((const float4*)sm.b[grp])[q];
            if (REAL) ff_mac(fac.rr, FF{x.x, x.z}, FF{y.x, y.z});
            else cff_mac(fac, x, sm.as[grp][p], y, sm.bs[grp][q]);
          } else {
            const double2 x = ((const double2*)sm.a[grp])[p], y = ((const double2*)sm.b[grp])[q];
            acc.x = fma(-x.y, y.y, fma(x.x, y.x, acc.x));
            acc.y = fma(x.y, y.x, fma(x.x, y.y, acc.y));
          }
        }
        if constexpr (FFM) {   // as the float-float GEMM: errors collected over 16 products at most
          fac.rr = ff_renorm(fac.rr);
          if (!REAL) {
            fac.ii = ff_renorm(fac.ii);
            fac.ss = ff_renorm(fac.ss);
          }
        }
        group_sync();
      }
      chunk += nc;
    }
  }
  if constexpr (FFM) {
    FF re = ff_norm(fac.rr), im = {0.f, 0.f};
    if (!REAL) cff_result(fac, re, im);
    acc = make_double2((double)re.hi + (double)re.lo, (double)im.hi + (double)im.lo);
  }
  sm.sum[grp][t] = acc;
  __syncthreads();
  if (grp == 0 && r0 + orow < m.rows && c0 + ocol < ns) {
#pragma unroll
    for (int q = 1; q < kRedoGroups; ++q) {
      acc.x += sm.sum[q][t].x;
      acc.y += sm.sum[q][t].y;
    }
    C[m.off + (r0 + orow) * m.step + (c0 + ocol) * m.other] = make_double2(acc.x, REAL ? 0.0 : acc.y);
  }
}

// Tiles of a task.
__device__ __forceinline__ int redo_tiles(const DgGroup& g, const DgMember& m) {
  const int ns = g.cm_rows ? g.N : g.R;
  return ((m.rows + kRedoTile - 1) / kRedoTile) * ((ns + kRedoTile - 1) / kRedoTile);
}

// NW warps per task: the tiles of those to be computed again join the list. Not after a wait gave up, when
// nothing is valid. A CTA per task where there are few: adding up the terms of a task's largest row and column
// is a chain of loads along K (step 2 at Ly = 10, chi = 3200, 260 tasks: a warp each
// 322 us, a CTA each 74).
template <int NW>
__global__ void __launch_bounds__(256) k_dg_check(const DgGroup* __restrict__ groups, const DgMember* __restrict__ members, int n,
                                                  const DgJob* __restrict__ sjobs, const DgJob* __restrict__ ujobs,
                                                  const double2* __restrict__ ssrc, const double2* __restrict__ usrc,
                                                  const int* __restrict__ e0, const int* __restrict__ e1,
                                                  const int* __restrict__ res, int* __restrict__ count, int2* __restrict__ list,
                                                  const int* __restrict__ err, bool ff) {
  const int lane = threadIdx.x & 31, warp = NW > 1 ? threadIdx.x >> 5 : 0;
  int i = NW > 1 ? (int)blockIdx.x : (int)(blockIdx.x * 256 + threadIdx.x) >> 5;
  DgMember m = members[min(i, n - 1)];
  DgGroup g = groups[m.group];
  // launched as a programmatic dependent of the product: above are tables, below its results
  asm volatile("griddepcontrol.wait;\ngriddepcontrol.launch_dependents;" ::: "memory");
  if (*err) return;
  for (; i < n; i += gridDim.x * (8 / NW), m = members[min(i, n - 1)], g = groups[m.group]) {
    const int form = task_form<NW>(g, m, sjobs, ujobs, ssrc, usrc, e0, e1, res, ff, lane, warp);
    if (form == 0 || warp > 0) continue;
    const int tiles = redo_tiles(g, m), mark = form == 2 ? kDgFF : 0;
    int at = 0;
    if (lane == 0) at = atomicAdd(count, tiles);
    at = __shfl_sync(0xffffffffu, at, 0);
    for (int t = lane; t < tiles; t += 32) list[at + t] = make_int2(i, t | mark);
  }
}

// The listed tiles. Usually the list is empty and the launch returns at once.
template <bool FFM, bool REAL>
__global__ void __launch_bounds__(256) k_dg_redo(const DgGroup* __restrict__ groups, const DgMember* __restrict__ members,
                                                 const DgJob* __restrict__ sjobs, const DgJob* __restrict__ ujobs,
                                                 const double2* __restrict__ ssrc, const double2* __restrict__ usrc,
                                                 double2* __restrict__ C, const int* __restrict__ count,
                                                 const int2* __restrict__ list) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // (dependent of k_dg_check)
  const int total = *count;
  __shared__ RedoSmem<FFM, REAL> sm;
  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    const int2 it = list[item];
    const DgMember m = members[it.x];
    const DgGroup g = groups[m.group];
    if (FFM && (it.y & kDgFF)) redo_tile<FFM, REAL>(g, m, it.y & ~kDgFF, sjobs, ujobs, ssrc, usrc, C, sm);
    else redo_tile<false, REAL>(g, m, it.y & ~kDgFF, sjobs, ujobs, ssrc, usrc, C, sm);
  }
}

// Both in one launch, for products of small tasks: a CTA checks a task and computes its few tiles if it must.
template <bool FFM, bool REAL>
__global__ void __launch_bounds__(256) k_dg_redo_tasks(const DgGroup* __restrict__ groups, const DgMember* __restrict__ members,
                                                       const DgJob* __restrict__ sjobs, const DgJob* __restrict__ ujobs,
                                                       const double2* __restrict__ ssrc, const double2* __restrict__ usrc,
                                                       double2* __restrict__ C, const int* __restrict__ e0,
                                                       const int* __restrict__ e1, const int* __restrict__ res,
                                                       const int* __restrict__ err) {
  const DgMember m = members[blockIdx.x];
  const DgGroup g = groups[m.group];
  __shared__ RedoSmem<FFM, REAL> sm;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // (dependent of the product)
  if (*err) return;
  const int form = task_form<8>(g, m, sjobs, ujobs, ssrc, usrc, e0, e1, res, FFM, threadIdx.x & 31, threadIdx.x >> 5);
  if (form == 0) return;
  for (int t = 0; t < redo_tiles(g, m); ++t) {
    if (FFM && form == 2) redo_tile<FFM, REAL>(g, m, t, sjobs, ujobs, ssrc, usrc, C, sm);
    else redo_tile<false, REAL>(g, m, t, sjobs, ujobs, ssrc, usrc, C, sm);
  }
}

// Products whose tasks have few tiles, up to this many tasks, take the one-launch form: 2 to 3 us less per product
// (FP64 application at Ly = 4, chi = 48 74.4 -> 69.0 us, float-float at Ly = 5, chi = 112 in real arithmetic
// 66 -> 58). With larger tasks the tiles of one would follow each other.
constexpr int kDgRedoTiles = 4, kDgRedoTasks = 4096;

cudaError_t dg_redo(const DgDev& d, const double2* a, const double2* b, double2* C, int beta, const int* words, int n_sm, cudaStream_t s) {
  if (d.n_members <= 0) return cudaSuccess;
  const int grid = (d.n_members + 7) / 8, u = 1 - d.sop;
  // as programmatic dependents of the launch before them, so that they cost little when there is
  // nothing to do: 4 us per product less than in plain stream order
  cudaLaunchAttribute pdl;
  pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  pdl.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t lc{};
  lc.blockDim = dim3(256);
  lc.stream = s;
  lc.attrs = &pdl;
  lc.numAttrs = 1;
  const DgGroup* gr = d.groups;
  const DgMember* me = d.members;
  const DgJob *sj = d.jobs[d.sop], *uj = d.jobs[u];
  const double2 *ss = d.sop ? b : a, *us = d.sop ? a : b;
  const int *e0 = d.expo[0], *e1 = d.expo[1], *res = d.res, *err = words + DG_ERR;
  if (d.max_tiles <= kDgRedoTiles && d.n_members <= kDgRedoTasks) {
    lc.gridDim = dim3(d.n_members);
    auto k = beta == 8 ? k_dg_redo_tasks<false, false> : d.real ? k_dg_redo_tasks<true, true> : k_dg_redo_tasks<true, false>;
    count_launch();
    return cudaLaunchKernelEx(&lc, k, gr, me, sj, uj, ss, us, C, e0, e1, res, err);
  }
  const bool wide = d.n_members <= 4 * n_sm;   // (that many CTAs run at once)
  lc.gridDim = dim3(wide ? d.n_members : grid < 2048 ? grid : 2048);
  cudaError_t e = cudaLaunchKernelEx(&lc, wide ? k_dg_check<8> : k_dg_check<1>, gr, me, d.n_members, sj, uj, ss, us, e0, e1, res, d.redo_count, d.redo, err, beta != 8);
  if (e != cudaSuccess) return e;
  lc.gridDim = dim3(4 * n_sm);
  auto k = beta == 8 ? k_dg_redo<false, false> : d.real ? k_dg_redo<true, true> : k_dg_redo<true, false>;
  e = cudaLaunchKernelEx(&lc, k, gr, me, sj, uj, ss, us, C, (const int*)d.redo_count, (const int2*)d.redo);
  count_launches(2);
  return e;
}

cudaError_t dg_init() {
  static DeviceOnce once;
  return once.run([] {
    cudaError_t r = cudaSuccess;
    for (const void* f : {(const void*)k_dg_gemm<7, false>, (const void*)k_dg_gemm<7, true>,
                          (const void*)k_dg_gemm<8, false>, (const void*)k_dg_gemm<8, true>})
      if (r == cudaSuccess) r = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kDgSmem);
    return r;
  });
}

cudaError_t dg_expand(const DgDev& d, cudaStream_t s) {
  if (d.n_members <= 0) return cudaSuccess;
  const int grid = (d.n_members + 7) / 8;
  k_dg_cmap<<<grid < 2048 ? grid : 2048, 256, 0, s>>>(d.members, d.n_members, d.cmap);
  count_launch();
  return cudaGetLastError();
}

cudaError_t dg_pack(const DgDev& d, int op, const double2* src, int beta, int* words, cudaStream_t s) {
  if (d.n_mpieces[op] > 0) {
    k_dg_expo<<<d.n_mpieces[op] < 16384 ? d.n_mpieces[op] : 16384, 256, 0, s>>>(src, d.jobs[op], d.mpieces[op],
                                                                               d.n_mpieces[op], d.expo[op]);
    count_launch();
  }
  if (d.n_pieces[op] > 0) {
    const unsigned grid = d.n_pieces[op] < 16384 ? d.n_pieces[op] : 16384;
    auto k = beta == 8 ? (d.real ? k_dg_pack<8, true> : k_dg_pack<8, false>)
                       : (d.real ? k_dg_pack<7, true> : k_dg_pack<7, false>);
    k<<<grid, 256, 0, s>>>(src, d.panel[op], d.jobs[op], d.pieces[op], d.n_pieces[op], d.expo[op], words);
    count_launch();
  }
  return cudaGetLastError();
}

cudaError_t dg_gemm(const DgDev& d, double2* C, int beta, int* words, int n_sm, uint64_t wait_ns, cudaStream_t s,
                    int first, int count) {
  if (count < 0) count = d.n_items;
  if (count <= 0) return cudaSuccess;
  cudaError_t e = dg_init();
  if (e != cudaSuccess) return e;
  DgArgs g{d.panel[0], d.panel[1], d.groups, d.items, first, count, d.cmap, d.expo[0], d.expo[1],
           d.splits, d.partial, d.tickets, d.res, C, words, wait_ns};
  auto k = beta == 8 ? (d.real ? k_dg_gemm<8, true> : k_dg_gemm<8, false>)
                     : (d.real ? k_dg_gemm<7, true> : k_dg_gemm<7, false>);
  k<<<count < n_sm ? count : n_sm, 320, kDgSmem, s>>>(g);
  count_launch();
  return cudaGetLastError();
}

}  // namespace mrd
