// FP64 kernels of the two-site H_eff application.
//
// theta' = H_eff theta is evaluated as
//   step 1   Z_{w'}[(s1',a'), (s2,b)] = sum_{s1,a} LW_{w'}^{(s1',s1)}[a',a] theta[(s1,a),(s2,b)]
//   step 2   theta'[(s1',a'), (s2',b')] = sum_{w',s2,b} Z_{w'}[(s1',a'),(s2,b)] WR_{w'}^{(s2,s2')}[b,b']
// with LW_{w'}^{(s1',s1)} = sum_w W_i[w,w',s1',s1] L_w and
//      WR_{w'}^{(s2,s2')}  = sum_{w''} W_{i+1}[w',w'',s2',s2] R_{w''},
// which is the definition L W_i W_{i+1} R theta with the MPO sums folded into the
// environments once per environment load. Both steps are grouped complex GEMMs over the task
// lists built in plan.cu; every output block is owned by exactly one task, so there are no
// atomics and the result is deterministic.
//
// On GB300 FP64 runs on the CUDA cores at about 1.2 TFLOP/s, far below what shared memory or
// HBM can feed, so a small 32 x 32 complex tile per 256-thread CTA (2 x 2 outputs per
// thread) keeps every DFMA pipe busy while wasting little work on ragged blocks.
#include "mrd_internal.h"
#include "plan.cuh"

namespace mrd {

namespace {

constexpr int kT = 32;   // output tile (complex elements per side)
constexpr int kK = 16;   // K chunk

__device__ __forceinline__ int64_t find_task(const int64_t* prefix, int64_t n, int64_t item) {
  // largest t with prefix[t] <= item (prefix[0] = 0, prefix[n] = total > item)
  int64_t lo = 0, hi = n - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void cmac(double2& c, const double2 a, const double2 b) {
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
}

}  // namespace

__global__ void __launch_bounds__(256) k_cgemm_fp64(const double2* __restrict__ A, const double2* __restrict__ B,
                                                    double2* __restrict__ C, const int64_t* __restrict__ tasks,
                                                    const int64_t* __restrict__ segs,
                                                    const int64_t* __restrict__ prefix, int64_t n_tasks) {
  __shared__ double2 As[kT][kK + 1];
  __shared__ double2 Bs[kK][kT + 1];
  const int tid = threadIdx.x;
  const int ty = tid >> 4, tx = tid & 15;
  const int64_t total = prefix[n_tasks];
  for (int64_t item = blockIdx.x; item < total; item += gridDim.x) {
    const int64_t t = find_task(prefix, n_tasks, item);
    const int64_t* task = tasks + TF * t;
    const int64_t M = task[0], N = task[1], c_off = task[2], ldc = task[3];
    const int64_t seg0 = task[4], nseg = task[5];
    const int64_t tiles_n = (N + kT - 1) / kT;
    const int64_t local = item - prefix[t];
    const int64_t m0 = (local / tiles_n) * kT, n0 = (local % tiles_n) * kT;
    double2 acc[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] = make_double2(0.0, 0.0);
    for (int64_t s = 0; s < nseg; ++s) {
      const int64_t* sg = segs + SF * (seg0 + s);
      const int64_t a_off = sg[0], lda = sg[1], b_off = sg[2], ldb = sg[3], K = sg[4];
      const int64_t flags = sg[5];
      for (int64_t k0 = 0; k0 < K; k0 += kK) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int e = tid + r * 256;
          if (!(flags & 1)) {                           // A[m, k] at a_off + m * lda + k
            const int ar = e >> 4, ak = e & 15;
            const int64_t gr = m0 + ar, gk = k0 + ak;
            As[ar][ak] = (gr < M && gk < K) ? A[a_off + gr * lda + gk] : make_double2(0.0, 0.0);
          } else {                                      // A[m, k] = conj(A[a_off + k * lda + m])
            const int ar = e & 31, ak = e >> 5;
            const int64_t gr = m0 + ar, gk = k0 + ak;
            double2 v = (gr < M && gk < K) ? A[a_off + gk * lda + gr] : make_double2(0.0, 0.0);
            v.y = -v.y;
            As[ar][ak] = v;
          }
          if (!(flags & 2)) {                           // B[k, n] at b_off + k * ldb + n
            const int bk = e >> 5, bc = e & 31;
            const int64_t gk2 = k0 + bk, gc = n0 + bc;
            Bs[bk][bc] = (gk2 < K && gc < N) ? B[b_off + gk2 * ldb + gc] : make_double2(0.0, 0.0);
          } else {                                      // B[k, n] = conj(B[b_off + n * ldb + k])
            const int bk = e & 15, bc = e >> 4;
            const int64_t gk2 = k0 + bk, gc = n0 + bc;
            double2 v = (gk2 < K && gc < N) ? B[b_off + gc * ldb + gk2] : make_double2(0.0, 0.0);
            v.y = -v.y;
            Bs[bk][bc] = v;
          }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kK; ++k) {
          const double2 a0 = As[2 * ty][k], a1 = As[2 * ty + 1][k];
          const double2 b0 = Bs[k][2 * tx], b1 = Bs[k][2 * tx + 1];
          cmac(acc[0][0], a0, b0);
          cmac(acc[0][1], a0, b1);
          cmac(acc[1][0], a1, b0);
          cmac(acc[1][1], a1, b1);
        }
        __syncthreads();
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int64_t r = m0 + 2 * ty + i, c = n0 + 2 * tx + j;
        if (r < M && c < N) C[c_off + r * ldc + c] = acc[i][j];
      }
  }
}

// LW / WR fold: out block = sum over its contributing MPO entries of value * env block.
// rows: LW or WR table (10 int64 per row); env_map: [channel][sector] -> env offset;
// perm/idx/val: sorted MPO entries; chan_field: index of the env channel in an entry
// (0 = w for W_i, 1 = w'' for W_{i+1}); sec_field: row field holding the env sector.
//
// The blocks lie one after another in `out`, and a CTA takes a chunk of consecutive elements of it,
// whichever blocks they belong to, so that the few large blocks spread over the GPU like the many
// small ones; the search for the first block and a block's entry tables (a chain of dependent
// loads) are paid once per CTA and block. Most entries are real, and most blocks one entry of
// value 1 (a channel that passes through): those take 2 and 0 of the 6 FP64 operations of a general
// complex entry (the FP64 pipe has 2 lanes per SM), with the same rounding. Ly = 10, chi = 3200
// (LW, WR: 0.82 GB written each): 0.49 + 0.40 ms; one CTA per block with every entry taken as
// complex needed 1.4 + 0.9. (Testing every element for infinities inside its own branch instead
// of four at once: 0.83 + 0.93.)
constexpr int kFoldPer = 4, kFoldSub = kFoldPer * 256, kFoldTerms = 32;
// Elements per CTA: 8192 where that gives four CTAs per SM, else fewer (down to one per thread).
inline int64_t fold_chunk(int64_t len, int n_sm) {
  const int64_t c = (len / (4 * n_sm) + 255) / 256 * 256;
  return c < 256 ? 256 : c > 8192 ? 8192 : c;
}

// An infinity or NaN takes the full product, zero times it included.
__device__ __forceinline__ bool fold_odd(double2 x) {
  constexpr int kExp = 0x7ff00000;
  const int a = __double2hiint(x.x) & kExp, b = __double2hiint(x.y) & kExp;
  return (a > b ? a : b) == kExp;
}

__device__ __forceinline__ void fold_full(double2& acc, double2 x, double2 v) {
  acc.x += v.x * x.x - v.y * x.y;
  acc.y += v.x * x.y + v.y * x.x;
}

__device__ __forceinline__ void fold_real(double2& acc, double2 x, double v, bool first) {
  if (v == -1.0) x = make_double2(-x.x, -x.y);
  else if (v != 1.0) x = make_double2(__dmul_rn(v, x.x), __dmul_rn(v, x.y));
  acc = first ? x : make_double2(__dadd_rn(acc.x, x.x), __dadd_rn(acc.y, x.y));
}

// Blocks of a few elements: one CTA each, so that its chain of dependent loads is paid once
// per block, side by side with those of the other blocks. At Ly = 5, chi = 61 the flat form in chunks of
// 8192 elements took ~100 us, in chunks of 256 10, this one 9 and 6 (LW, WR).
constexpr int64_t kFoldSmall = 128;   // mean elements per block up to which this form runs

__global__ void __launch_bounds__(256) k_fold_small(const double2* __restrict__ env, double2* __restrict__ out,
                                                   const int64_t* __restrict__ rows, int nrows,
                                                   const int64_t* __restrict__ env_map, int n_sec,
                                                   const int32_t* __restrict__ perm, const int32_t* __restrict__ idx,
                                                   const double* __restrict__ val, int chan_field) {
  for (int r = blockIdx.x; r < nrows; r += gridDim.x) {
    const int64_t* row = rows + (int64_t)LWF * r;
    const int64_t sec = row[3], n = row[5] * row[6], off = row[7], cb = row[8], ce = row[9];
    for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
      double2 acc = make_double2(0.0, 0.0);
      for (int64_t c = cb; c < ce; ++c) {
        const int ent = perm[c];
        const double2 x = env[env_map[(int64_t)idx[4 * ent + chan_field] * n_sec + sec] + e];
        fold_full(acc, x, make_double2(val[2 * ent], val[2 * ent + 1]));
      }
      out[off + e] = acc;
    }
  }
}

__global__ void __launch_bounds__(256) k_fold_env(const double2* __restrict__ env, double2* __restrict__ out,
                                                  const int64_t* __restrict__ rows, int nrows, int64_t len,
                                                  const int64_t* __restrict__ env_map, int n_sec,
                                                  const int32_t* __restrict__ perm, const int32_t* __restrict__ idx,
                                                  const double* __restrict__ val, int chan_field, int chunk) {
  __shared__ int64_t s_off[257];
  __shared__ const double2* s_src[kFoldTerms];
  __shared__ double2 s_val[kFoldTerms];
  const int tid = threadIdx.x;
  const int64_t base = (int64_t)blockIdx.x * chunk, stop = base + chunk < len ? base + chunk : len;
  // the last block that starts at or before the chunk, by 256-way search
  int lo = 0, hi = nrows;
  while (hi - lo > 1) {
    const int step = (hi - lo + 255) / 256, i = lo + tid * step;
    const int k = __syncthreads_count(i < hi && rows[(int64_t)LWF * i + 7] <= base);
    lo += (k - 1) * step;
    hi = hi < lo + step ? hi : lo + step;
  }
  for (int i = tid; i < 257; i += 256) s_off[i] = lo + i < nrows ? rows[(int64_t)LWF * (lo + i) + 7] : len;
  __syncthreads();
  int cur = -1;          // block whose terms are staged
  int terms = 0;
  int64_t cur_off = 0, cur_n = 0;
  for (int64_t e0 = base; e0 < stop; e0 += kFoldSub) {
    int r = 0, top = 257;                // the last staged block that starts at or before e0
    while (top - r > 1) {
      const int m = (r + top) >> 1;
      if (s_off[m] <= e0) r = m; else top = m;
    }
    const int64_t end = e0 + kFoldSub < stop ? e0 + kFoldSub : stop;
    if (r < 256 && s_off[r + 1] >= end) {   // one block
      if (r != cur) {
        const int64_t* row = rows + (int64_t)LWF * (lo + r);
        const int64_t cb = row[8];
        __syncthreads();                    // the staged terms have been used
        terms = (int)(row[9] - cb);
        cur_off = row[7];
        cur_n = row[5] * row[6];
        cur = r;
        if (tid < terms && tid < kFoldTerms) {
          const int ent = perm[cb + tid];
          s_src[tid] = env + env_map[(int64_t)idx[4 * ent + chan_field] * n_sec + row[3]];
          s_val[tid] = make_double2(val[2 * ent], val[2 * ent + 1]);
        }
        __syncthreads();
      }
      if (terms <= kFoldTerms) {
        const int64_t f = e0 - cur_off + tid, n = end - cur_off < cur_n ? end - cur_off : cur_n;
        double2 acc[kFoldPer];
#pragma unroll
        for (int q = 0; q < kFoldPer; ++q) acc[q] = make_double2(0.0, 0.0);
        for (int c = 0; c < terms; ++c) {
          const double2* src = s_src[c];
          const double2 v = s_val[c];
          double2 x[kFoldPer];
#pragma unroll
          for (int q = 0; q < kFoldPer; ++q) x[q] = f + q * 256 < n ? src[f + q * 256] : make_double2(0.0, 0.0);
          bool full = v.y != 0.0;
#pragma unroll
          for (int q = 0; q < kFoldPer; ++q) full |= fold_odd(x[q]);
          if (full) {
#pragma unroll
            for (int q = 0; q < kFoldPer; ++q) fold_full(acc[q], x[q], v);
          } else {
#pragma unroll
            for (int q = 0; q < kFoldPer; ++q) fold_real(acc[q], x[q], v.x, c == 0);
          }
        }
#pragma unroll
        for (int q = 0; q < kFoldPer; ++q)
          if (f + q * 256 < n) out[cur_off + f + q * 256] = acc[q];
        continue;
      }
    }
    for (int64_t e = e0 + tid; e < end; e += 256) {   // several blocks: every element finds its own
      int b = 0;
      top = 257;
      while (top - b > 1) {
        const int m = (b + top) >> 1;
        if (s_off[m] <= e) b = m; else top = m;
      }
      b += lo;
      while (b + 1 < nrows && rows[(int64_t)LWF * (b + 1) + 7] <= e) ++b;   // beyond the staged ones
      const int64_t* row = rows + (int64_t)LWF * b;
      const int64_t off = row[7], sec = row[3], cb = row[8], ce = row[9];
      if (e - off >= row[5] * row[6]) continue;
      double2 acc = make_double2(0.0, 0.0);
      for (int64_t c = cb; c < ce; ++c) {
        const int ent = perm[c];
        const double2* src = env + env_map[(int64_t)idx[4 * ent + chan_field] * n_sec + sec];
        const double2 x = src[e - off], v = make_double2(val[2 * ent], val[2 * ent + 1]);
        if (v.y != 0.0 || fold_odd(x)) fold_full(acc, x, v);
        else fold_real(acc, x, v.x, c == cb);
      }
      out[e] = acc;
    }
  }
}

cudaError_t launch_cgemm_fp64(const double2* A, const double2* B, double2* C, const int64_t* tasks,
                              const int64_t* segs, const int64_t* prefix, int64_t n_tasks, int64_t total_tiles,
                              int n_sm, cudaStream_t s) {
  if (total_tiles <= 0) return cudaSuccess;
  int64_t grid = (int64_t)n_sm * 8;
  if (grid > total_tiles) grid = total_tiles;
  k_cgemm_fp64<<<(unsigned)grid, 256, 0, s>>>(A, B, C, tasks, segs, prefix, n_tasks);
  mrd::count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fold_env(const double2* env, double2* out, const int64_t* rows, int64_t nrows,
                            const int64_t* env_map, int n_sec, const int32_t* perm, const int32_t* idx,
                            const double* val, int chan_field, int64_t len, int n_sm, cudaStream_t s) {
  if (nrows <= 0 || len <= 0) return cudaSuccess;
  if (len <= kFoldSmall * nrows) {
    k_fold_small<<<(unsigned)(nrows < 65535 ? nrows : 65535), 256, 0, s>>>(env, out, rows, (int)nrows, env_map, n_sec, perm, idx, val,
                                                                       chan_field);
    mrd::count_launch();
    return cudaGetLastError();
  }
  const int64_t chunk = fold_chunk(len, n_sm);
  k_fold_env<<<(unsigned)((len + chunk - 1) / chunk), 256, 0, s>>>(env, out, rows, (int)nrows, len, env_map, n_sec, perm, idx, val,
                                                                   chan_field, (int)chunk);
  mrd::count_launch();
  return cudaGetLastError();
}

}  // namespace mrd
