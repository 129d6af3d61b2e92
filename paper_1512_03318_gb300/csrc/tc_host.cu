// Host side of the tensor-core H_eff: packed-panel tables (derived on the host from the
// device-built charge tables of plan.cu), packing of the folded environments and of theta,
// and the two grouped-GEMM launches.
#include <algorithm>
#include <map>
#include <new>
#include <thread>
#include <vector>

#include "heff_internal.h"
#include "tc.cuh"

namespace mrd {
cudaError_t tc_pack(const double2* src, uint8_t* dst, const int64_t* jobs, int njobs, int64_t npieces, int prec, int* ctr,
                    int* bad, cudaStream_t s);
cudaError_t tc_gemm_init();
cudaError_t tc_gemm(const uint8_t* a_base, const uint8_t* b_base, const TcItem* items, int count, const TcItem* alt,
                    int alt_count, const int* bad, const TcSeg* segs,
                    const int64_t* rowmap, uint8_t* z_out, double2* f_out, int prec, TcCfg cfg, int ntile, int* ctr, int* err, int n_sm,
                    uint64_t wait_ns, cudaStream_t s);
}  // namespace mrd

struct Tc {
  int prec = 0;
  TcCfg cfg{0, 0, 0};
  int cfg_source = 0;   // 0: default, 1: tuned on this H_eff, 2: tuned earlier on this context
  bool env_dirty = true;
  Arena mem;
  uint8_t *lw = nullptr, *wr = nullptr, *th = nullptr, *z = nullptr;
  TcItem *it1 = nullptr, *it2 = nullptr;   // tiles of the two steps, longest first
  TcSeg *s1 = nullptr, *s2 = nullptr;
  int n_it1 = 0, n_it2 = 0, ntile2 = 0;
  TcItem* alt2 = nullptr;                  // step-2 tiles that keep each row to its own K segments
  int n_alt2 = 0;
  std::vector<int32_t> task1, task2, taska; // first tile of every task, + total (per-task launches)
  int64_t* rmap1 = nullptr;                // step-1 row map (tc_rowmap)
  int64_t *j_lw = nullptr, *j_wr = nullptr, *j_th = nullptr;
  int n_lw = 0, n_wr = 0, n_th = 0;
  int64_t pc_lw = 0, pc_wr = 0, pc_th = 0; // pack pieces of each job list
  bool zero_out = true;                    // some output blocks receive no product
  int* words = nullptr;                    // tile counters of the two steps, error flag, WR not finite
  int* err() const { return words + 2; }
  int* bad() const { return words + 3; }
};

void tc_free(Tc* t) { delete t; }

// Tensor-core precision of an application: complex, or real when the H_eff is declared real
// (MRD_OPT_REAL).
int tc_prec_of(const mrd_heff* h, int32_t prec) {
  if (prec == MRD_PREC_TF32) return h->real ? TC_TF32_REAL : TC_TF32;
  return h->real ? TC_BF16X3_REAL : TC_BF16X3;
}

namespace {

int64_t round_up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

struct Panel {
  int64_t off, nks;
};

// Panels keyed by the FP64 element offset of their block: appended in build order, sorted once
// (stably, so that of equal keys, e.g. an empty block and the one after it, the last appended
// wins), then found by binary search. Tens of thousands of lookups per H_eff: a sorted vector
// avoids the per-node allocations and pointer chasing of a tree map.
struct PanelIndex {
  std::vector<std::pair<int64_t, Panel>> v;
  void add(int64_t key, Panel p) { v.push_back({key, p}); }
  void finish() {
    auto lt = [](const std::pair<int64_t, Panel>& a, const std::pair<int64_t, Panel>& b) { return a.first < b.first; };
    if (!std::is_sorted(v.begin(), v.end(), lt)) std::stable_sort(v.begin(), v.end(), lt);
  }
  const Panel* find(int64_t key) const {
    auto it = std::upper_bound(v.begin(), v.end(), key,
                               [](int64_t k, const std::pair<int64_t, Panel>& e) { return k < e.first; });
    if (it == v.begin()) return nullptr;
    --it;
    return it->first == key ? &it->second : nullptr;
  }
};

// bytes of an A panel (128-row tiles) or a B panel (ntile-row tiles)
int64_t a_bytes(int64_t rows, int64_t nks, int prec) { return tc_apad(rows) * nks * tc_aplanes(prec) * 32; }
int64_t b_bytes(int64_t rows, int64_t nks, int prec, int ntile) {
  const int64_t full = rows / ntile, rest = tc_bpad(rows - full * ntile);
  return (full * ntile * tc_bplanes(prec, ntile) + rest * tc_bplanes(prec, (int)rest)) * nks * 32;
}

// Host tables of the tensor-core path for one precision and tile configuration: panel
// layouts, pack jobs, tasks, segments, row map and the per-CTA item deal. Built without any
// device call, so that a host thread can build them while the device works (tc_prebuild).
struct TcTables {
  int prec = 0;
  TcCfg cfg{0, 0, 0};
  int n_sm = 0;
  std::vector<int64_t> j_lw, j_wr, j_th, rowmap;
  std::vector<TcSeg> s1, s2;
  int ntile2 = 0;              // columns per tile of step 2 (WR panels), at most cfg.ntile
  std::vector<TcItem> i1, i2, ia;
  std::vector<int32_t> task1, task2, taska;
  int64_t lw_b = 0, wr_b = 0, th_b = 0, z_b = 0, pc_lw = 0, pc_wr = 0, pc_th = 0;
  bool zero_z = false, zero_out = false;   // rows of Z that are read but not written; blocks of the output
  const char* err = nullptr;   // why the tables could not be built
};

// A stacked product: M x N outputs, K segments seg0 .. seg0 + nseg - 1 of nks steps in all. Rows from
// `cut` on may have other segments than the ones before (part 0 and 1: psg0, pseg, pnks; their union is the
// task's): 0 if all rows have the same.
struct TcTask {
  int64_t M, N, out, ld;   // out, ld: TcItem (of the task's first tile)
  int32_t seg0, nseg;
  int64_t nks;
  int64_t cut;
  int32_t psg0[2], pseg[2];
  int64_t pnks[2];
};

// Tiles of the tasks, tasks by decreasing K steps (equal ones in task order, or, for order 1, by
// decreasing work), which is the order in which the CTAs take them. alt: the tiles that compute the
// same outputs with every row's own segments only.
void cut_tiles(std::vector<TcTask>& tasks, int ntile, int order, bool z_out, const std::vector<TcSeg>& segs, std::vector<TcItem>& items,
               std::vector<int32_t>& first, std::vector<TcItem>* alt = nullptr, std::vector<int32_t>* afirst = nullptr) {
  const int64_t nt = ntile;
  auto tiles = [&](const TcTask& t) { return ((t.M + 127) / 128) * ((t.N + nt - 1) / nt); };
  if (order == 1)
    std::stable_sort(tasks.begin(), tasks.end(),
                     [&](const TcTask& a, const TcTask& b) { return tiles(a) * a.nks > tiles(b) * b.nks; });
  std::stable_sort(tasks.begin(), tasks.end(), [](const TcTask& a, const TcTask& b) { return a.nks > b.nks; });
  int64_t n = 0;
  for (const TcTask& t : tasks) n += tiles(t);
  items.reserve((size_t)n);
  auto cut = [&](std::vector<TcItem>& v, const TcTask& t, int64_t lo, int64_t hi, int32_t seg0, int32_t nseg, int64_t nks) {
    if (nseg == 0) return;
    for (int64_t r = lo / 128 * 128; r < hi; r += 128)
      for (int64_t c = 0; c < t.N; c += nt) {
        const int64_t rows = std::min<int64_t>(hi - r, 128), cols = std::min<int64_t>(t.N - c, nt);
        v.push_back({(int32_t)tc_bpad(cols), (int32_t)tc_apad(std::min<int64_t>(t.M - r, 128)), (int32_t)rows, (int32_t)cols,
                     seg0, nseg, (int32_t)(r / 128), (int32_t)(c / nt), z_out ? t.out + r : t.out + r * t.ld + c, t.ld,
                     (int32_t)std::max<int64_t>(lo - r, 0), (int32_t)nks, 0,
                     {segs[(size_t)seg0], segs[(size_t)(nseg > 1 ? seg0 + 1 : seg0)]}});
      }
  };
  for (const TcTask& t : tasks) {
    first.push_back((int32_t)items.size());
    cut(items, t, 0, t.M, t.seg0, t.nseg, t.nks);
    if (!alt) continue;
    afirst->push_back((int32_t)alt->size());
    if (t.cut == 0) {
      cut(*alt, t, 0, t.M, t.seg0, t.nseg, t.nks);
    } else {
      cut(*alt, t, 0, t.cut, t.psg0[0], t.pseg[0], t.pnks[0]);
      cut(*alt, t, t.cut, t.M, t.psg0[1], t.pseg[1], t.pnks[1]);
    }
  }
  first.push_back((int32_t)items.size());
  if (alt) afirst->push_back((int32_t)alt->size());
}

// Columns per tile of step 2. Its tiles have long and unequal K (every channel of an output sector),
// and K is not cut (the FP32 sums keep their order), so with few sectors the longest tile sets the
// time: narrower tiles finish it sooner, and cost more in all (the 128 rows of A are multiplied for
// fewer columns). Estimated cycles: per K step of a tile its MMAs (max(48, N / 2) each) and a share of
// the slots' hand-over; the choice minimises the larger of the longest tile and the average load of a
// CTA, plus half of the latter for the uneven rest. Measured us of step 2 (16 / 32 / 48 / 64 columns):
// BF16X3 Ly = 8, chi = 1024 68 / 60 / 65 / 64, Ly = 10, chi = 3200 632 / 348 / 317 / 292; TF32 Ly = 8,
// chi = 2049 222 / 146 / 111 / 115; real BF16X3 Ly = 6, chi = 777 32.8 / 32.8 / 34.6 / 34.9 (128: 37.0).
int step2_columns(const mrd_heff* h, int prec, int ntile) {
  auto cost = [&](int64_t n) {   // cycles per K step of a tile of n columns (padded to 16)
    const double wide = std::max(48.0, tc_aplanes(prec) * n / 2.0), half = std::max(48.0, tc_aplanes(prec) * n / 4.0);
    const int ap = tc_aplanes(prec);
    const double m = tc_is_real(prec) || tc_neg_planes(prec, (int)n) ? ap * wide : ap / 2 * wide + ap * half;
    return m + 600.0 / tc_group(prec);
  };
  const int kst = tc_kstep(prec);
  int best = ntile;
  double best_t = -1.0;
  for (int n = ntile; n >= 16; n = n > 64 ? 64 : n - 16) {
    double longest = 0.0, total = 0.0;
    for (int64_t m = 0; m < h->counts[C_NMID]; ++m) {
      const int64_t* rout = &h->mid_host[MIDF * m];
      for (int s2p = 0; s2p < 2; ++s2p) {
        if (rout[8 + s2p] < 0) continue;
        int64_t ks = 0;
        for (int s1p = 0; s1p < 2; ++s1p) {   // (about the union of the two lists)
          const int64_t* t = &h->t2_host[TF * ((m * 2 + s1p) * 2 + s2p)];
          int64_t k = 0;
          for (int64_t q = 0; q < t[5]; ++q) k += (h->s2_host[SF * (t[4] + q) + 4] + kst - 1) / kst;
          ks = std::max(ks, k);
        }
        const int64_t N = h->right[3 * rout[8 + s2p] + 2], rows = (rout[2] + 127) / 128;
        const int64_t rest = tc_bpad(N % n);
        total += rows * ks * ((N / n) * cost(n) + (rest ? cost(rest) : 0.0));
        longest = std::max(longest, ks * cost(std::min<int64_t>(n, tc_bpad(N))));
      }
    }
    const double load = total / std::max(h->n_sm, 1), t = std::max(longest, load) + 0.5 * load;
    if (best_t < 0.0 || t < best_t) { best_t = t; best = n; }
  }
  return best;
}

bool tables(const mrd_heff* h, int prec, TcCfg cfg, TcTables& o) {
  auto fail = [&](const char* m) { o.err = m; return false; };
  o.prec = prec;
  o.cfg = cfg;
  o.n_sm = h->n_sm;
  if (!tc_cfg_ok(prec, cfg)) return fail("tc: tile configuration does not fit");
  const int kst = tc_kstep(prec), ntile = cfg.ntile, ntile2 = step2_columns(h, prec, cfg.ntile);
  o.ntile2 = ntile2;
  auto steps = [&](int64_t K) { return (K + kst - 1) / kst; };
  const int64_t* c = h->counts;
  PanelIndex wr_map, th_map, z_map;
  wr_map.v.reserve(c[C_NWR]);
  std::vector<int64_t>&j_lw = o.j_lw, &j_wr = o.j_wr, &j_th = o.j_th;
  int64_t &lw_b = o.lw_b, &wr_b = o.wr_b, &th_b = o.th_b, &z_b = o.z_b;
  // (the folded left operand LW is packed below, stacked by input middle sector)
  // folded right operand WR(w', s2, s2', b): B panel of its transpose, rows d_b', K d_b
  j_wr.reserve((size_t)c[C_NWR] * TCJ);
  for (int64_t k = 0; k < c[C_NWR]; ++k) {
    const int64_t* r = &h->wr_host[WRF * k];
    const int64_t K = r[5], rows = r[6], nks = steps(K);
    wr_map.add(r[7], {wr_b, nks});
    j_wr.insert(j_wr.end(), {r[7], rows, 1, rows, K, wr_b, ntile2, nks, rows, 0, 0});
    wr_b += b_bytes(rows, nks, prec, ntile2);
  }
  // theta block (s1, a) x (s2, b) of every middle sector: B panel of its transpose, rows d_b, K d_a
  const std::vector<int64_t>& mid = h->mid_host;
  for (int64_t m = 0; m < c[C_NMID]; ++m) {
    const int64_t* r = &mid[MIDF * m];
    for (int s1 = 0; s1 < 2; ++s1) {
      if (r[5 + s1] < 0) continue;
      const int64_t K = h->left[3 * r[5 + s1] + 2], nks = steps(K);
      for (int s2 = 0; s2 < 2; ++s2) {
        if (r[8 + s2] < 0) continue;
        const int64_t rows = h->right[3 * r[8 + s2] + 2];
        const int64_t src = r[4] + (s1 ? r[7] : 0) * r[3] + (s2 ? r[10] : 0);
        th_map.add(src, {th_b, nks});
        j_th.insert(j_th.end(), {src, r[3], 1, rows, K, th_b, ntile, nks, rows, 0, 0});
        th_b += b_bytes(rows, nks, prec, ntile);
      }
    }
  }
  // Z(w', m_in), columns s2: A panels with the rows of both s1' under each other, keyed by their FP64
  // element offset (row 0). Rows that no LW block feeds (s1mask) are zeros.
  const std::vector<int64_t>& z = h->z_host;   // downloaded with the other tables at creation
  if ((int64_t)z.size() < ZF * c[C_NZ]) return fail("tc: Z table missing");
  const int64_t nmid = c[C_NMID];
  z_map.v.reserve((size_t)c[C_NZ] * 2);
  for (int64_t k = 0; k < c[C_NZ]; ++k) {
    const int64_t* zr = &z[ZF * k];
    const int64_t* rin = &mid[MIDF * zr[1]];
    const int64_t* rout = &mid[MIDF * zr[2]];
    for (int s1p = 0; s1p < 2; ++s1p)
      if (rout[5 + s1p] >= 0 && h->t1_host[TF * ((zr[0] * nmid + zr[1]) * 2 + s1p) + 5] == 0) o.zero_z = true;
    for (int s2 = 0; s2 < 2; ++s2) {
      if (rin[8 + s2] < 0) continue;
      const int64_t nks = steps(h->right[3 * rin[8 + s2] + 2]);
      z_map.add(zr[5] + (s2 ? rin[10] : 0), {z_b, nks});
      z_b += a_bytes(zr[3], nks, prec);
    }
  }
  wr_map.finish();
  th_map.finish();
  z_map.finish();
  for (const PanelIndex* m : {&wr_map, &th_map, &z_map})
    for (const auto& e : m->v)
      if (e.second.nks > 0xffff) return fail("tc: sector dimension too large");
  auto seg = [](const Panel& a, const Panel& b) { return TcSeg{a.off, b.off / 256 << 16 | b.nks}; };
  // step-2 tasks (theta' = sum Z WR), built on a second host thread while this one builds the
  // step-1 tasks: the two loops share only the finished (read-only) panel indexes. A task is an
  // output block column (m_out, s2') with the rows of both s1' (twice the rows per tile for the same
  // WR): its segments are those of either, in the tables' order (w', s2), which both lists have;
  // rows that lack one meet zeros of Z there. Zero times an infinity or NaN of WR would not be
  // nothing: when WR holds one, the kernel runs the tiles of the two lists by themselves.
  bool step2_ok = true;
  std::vector<TcTask> tasks1, tasks2;
  auto build_step2 = [&] {
    std::vector<TcSeg> part[2];
    for (int64_t m = 0; m < nmid; ++m) {
      const int64_t* rout = &mid[MIDF * m];
      for (int s2p = 0; s2p < 2; ++s2p) {
        if (rout[8 + s2p] < 0) continue;
        const int64_t *t[2], *sg[2];
        int64_t n[2];
        for (int s1p = 0; s1p < 2; ++s1p) {
          t[s1p] = &h->t2_host[TF * ((m * 2 + s1p) * 2 + s2p)];
          n[s1p] = t[s1p][0] && t[s1p][1] ? t[s1p][5] : 0;
          sg[s1p] = h->s2_host.data() + SF * t[s1p][4];
          part[s1p].clear();
        }
        const int64_t N = h->right[3 * rout[8 + s2p] + 2];
        TcTask k{rout[2], N, rout[4] + (s2p ? rout[10] : 0), rout[3], (int32_t)o.s2.size(), 0, 0, 0, {0, 0}, {0, 0}, {0, 0}};
        int64_t last = -1, i[2] = {0, 0};
        while (i[0] < n[0] || i[1] < n[1]) {
          int64_t key[2] = {INT64_MAX, INT64_MAX};   // Z panel of either list's next segment
          for (int q = 0; q < 2; ++q)
            if (i[q] < n[q]) key[q] = sg[q][SF * i[q]] - (q ? rout[7] : 0) * sg[q][SF * i[q] + 1];
          const int64_t next = std::min(key[0], key[1]), wr = sg[key[0] == next ? 0 : 1][SF * i[key[0] == next ? 0 : 1] + 2];
          const Panel* a = z_map.find(next);
          const Panel* b = wr_map.find(wr);
          if (!a || !b || a->nks != b->nks || next <= last) { step2_ok = false; return; }
          last = next;
          for (int q = 0; q < 2; ++q) {
            if (key[q] != next) continue;
            if (sg[q][SF * i[q] + 2] != wr) { step2_ok = false; return; }
            if (a->nks > 0) part[q].push_back(seg(*a, *b));
            ++i[q];
          }
          if (a->nks == 0) continue;
          o.s2.push_back(seg(*a, *b));
          ++k.nseg;
          k.nks += a->nks;
        }
        const bool lo = rout[5] >= 0 && rout[7] > 0, hi = rout[6] >= 0 && rout[7] < k.M;   // rows of either s1'
        if (lo && hi && (part[0].size() != (size_t)k.nseg || part[1].size() != (size_t)k.nseg)) {
          k.cut = rout[7];
          for (int q = 0; q < 2; ++q) {
            k.psg0[q] = (int32_t)o.s2.size();
            k.pseg[q] = (int32_t)part[q].size();
            for (const TcSeg& e : part[q]) k.pnks[q] += e.b & 0xffff;
            o.s2.insert(o.s2.end(), part[q].begin(), part[q].end());
            if (part[q].empty()) o.zero_out = true;   // (only the separate lists leave these rows out)
          }
        }
        if (k.nks > 0 && k.M > 0 && k.N > 0) tasks2.push_back(k);
        else if (k.M > 0 && k.N > 0) o.zero_out = true;
      }
    }
  };
  std::thread step2;
  try {
    step2 = std::thread([&] {
      try {
        build_step2();
      } catch (...) {   // out of host memory
        step2_ok = false;
      }
    });
  } catch (...) {   // no thread to be had: build it here, before step 1
    build_step2();
  }
  struct Join {
    std::thread& t;
    ~Join() { if (t.joinable()) t.join(); }
  } join_step2{step2};
  // step-1 tasks (Z = LW theta), stacked: for every input middle sector m_in, the output rows
  // (w', s1', a') of all its Z blocks are stacked along M into one GEMM per column part s2, so
  // that small blocks share 128-row tiles instead of each filling one. Rows are grouped in
  // three classes by the LW blocks that feed them (s1 = 0 only, s1 = 1 only, both), each
  // class a task of its own with the K segments it needs, so no zero block is multiplied.
  // The stacked LW of a class and K segment s1 is one A panel; each output row is scattered to
  // its Z panel through a row map.
  std::vector<int64_t>& rowmap = o.rowmap;
  {
    std::vector<int64_t> zrow_of((size_t)c[C_NMID] > 0 ? (size_t)h->d.d_m * nmid : 0, -1);
    for (int64_t k = 0; k < c[C_NZ]; ++k) zrow_of[(size_t)(z[ZF * k] * nmid + z[ZF * k + 1])] = k;
    struct Member { int64_t wp, s1p, rows, row0, lw[2]; };
    for (int64_t mi = 0; mi < nmid; ++mi) {
      const int64_t* rin = &mid[MIDF * mi];
      std::vector<Member> cls[3];
      for (int64_t wp = 0; wp < h->d.d_m; ++wp)
        for (int s1p = 0; s1p < 2; ++s1p) {
          const int64_t ti = (wp * nmid + mi) * 2 + s1p;
          const int64_t* t = &h->t1_host[TF * ti];
          if (t[5] == 0 || t[0] == 0 || t[1] == 0) continue;
          Member mb{wp, s1p, t[0], 0, {-1, -1}};
          for (int64_t k = 0; k < t[5]; ++k) {
            const int64_t* sg = &h->s1_host[SF * (t[4] + k)];
            int q1 = sg[2] == rin[4] + rin[7] * rin[3] ? 1 : 0;   // theta rows of the s1 = 1 part
            if (rin[5] < 0) q1 = 1;
            if (rin[6] < 0) q1 = 0;
            mb.lw[q1] = sg[0];
          }
          const int k = mb.lw[0] >= 0 && mb.lw[1] >= 0 ? 2 : (mb.lw[0] >= 0 ? 0 : 1);
          cls[k].push_back(mb);
        }
      for (int k = 0; k < 3; ++k) {
        if (cls[k].empty()) continue;
        int64_t R = 0;
        for (Member& mb : cls[k]) { mb.row0 = R; R += mb.rows; }
        // the class's stacked A panels, one per K segment s1
        int64_t aoff[2] = {-1, -1}, ank[2] = {0, 0};
        for (int q1 = 0; q1 < 2; ++q1) {
          if (k != 2 && k != q1) continue;
          if (rin[5 + q1] < 0) return fail("tc: LW block without its theta rows");
          const int64_t K = h->left[3 * rin[5 + q1] + 2];
          ank[q1] = steps(K);
          aoff[q1] = lw_b;
          for (const Member& mb : cls[k])
            j_lw.insert(j_lw.end(), {mb.lw[q1], K, 0, mb.rows, K, lw_b, 0, ank[q1], R, 0, mb.row0});
          lw_b += a_bytes(R, ank[q1], prec);
        }
        for (int s2p = 0; s2p < 2; ++s2p) {
          if (rin[8 + s2p] < 0) continue;
          const int64_t N = h->right[3 * rin[8 + s2p] + 2], coff = s2p ? rin[10] : 0, nks_z = steps(N);
          if (N == 0) continue;
          TcTask task{R, N, (int64_t)rowmap.size(), nks_z, (int32_t)o.s1.size(), 0, 0, 0, {0, 0}, {0, 0}, {0, 0}};
          for (int q1 = 0; q1 < 2; ++q1) {
            if (aoff[q1] < 0) continue;
            const Panel* b = th_map.find(rin[4] + (q1 ? rin[7] : 0) * rin[3] + coff);
            if (!b || b->nks != ank[q1]) return fail("tc: step-1 operand not packed");
            if (ank[q1] == 0) continue;
            o.s1.push_back(seg({aoff[q1], ank[q1]}, *b));
            ++task.nseg;
            task.nks += ank[q1];
          }
          if (task.nks == 0) { o.zero_z = true; continue; }
          for (const Member& mb : cls[k]) {
            const int64_t zk = zrow_of[(size_t)(mb.wp * nmid + mi)];
            if (zk < 0) return fail("tc: step-1 output block missing");
            const int64_t* zr = &z[ZF * zk];
            const int64_t* rout = &mid[MIDF * zr[2]];
            const Panel* q = z_map.find(zr[5] + coff);
            if (!q || q->nks != nks_z) return fail("tc: step-1 output panel missing");
            const int64_t row0 = mb.s1p ? rout[7] : 0;
            if (row0 + mb.rows > zr[3]) return fail("tc: step-1 output rows outside their panel");
            for (int64_t r = row0; r < row0 + mb.rows; ++r) {
              const int64_t rt = r / 128, mrow = tc_apad(std::min<int64_t>(zr[3] - rt * 128, 128));
              rowmap.push_back(tc_rowmap(q->off + rt * a_bytes(128, nks_z, prec), mrow, r % 128));
            }
          }
          tasks1.push_back(task);
        }
      }
    }
  }
  if (step2.joinable()) step2.join();
  if (!step2_ok) return fail("tc: step-2 operand not packed");
  // every tile the kernel reads must lie inside its buffer (the Z rows it writes: checked above)
  {
    auto chk = [&](const std::vector<TcTask>& tk, const std::vector<TcSeg>& sg, int64_t alen, int64_t blen, int nt) {
      for (const TcTask& t : tk)
        for (int64_t k = 0; k < t.nseg; ++k) {   // (the parts' segments are among them)
          const TcSeg& q = sg[(size_t)(t.seg0 + k)];
          const int64_t nks = q.b & 0xffff, b = (q.b >> 16) * 256;
          if (nks < 1 || q.a < 0 || q.a % 256 || q.a + a_bytes(t.M, nks, prec) > alen) return false;
          if (b < 0 || b + b_bytes(t.N, nks, prec, nt) > blen) return false;
        }
      return true;
    };
    if (!chk(tasks1, o.s1, lw_b, th_b, ntile) || !chk(tasks2, o.s2, z_b, wr_b, ntile2)) return fail("tc: internal panel table check failed");
  }
  cut_tiles(tasks1, ntile, cfg.order, true, o.s1, o.i1, o.task1);
  cut_tiles(tasks2, o.ntile2, cfg.order, false, o.s2, o.i2, o.task2, &o.ia, &o.taska);
  // first piece of every pack job (field 9) and the pieces of each list
  auto pieces = [&](std::vector<int64_t>& j) {
    int64_t n = 0;
    for (size_t k = 0; k < j.size(); k += TCJ) {
      j[k + 9] = n;
      n += (j[k + 3] * j[k + 7] * (j[k + 2] ? 2 : kst / 2) + kPackPiece - 1) / kPackPiece;
    }
    return n;
  };
  o.pc_lw = pieces(j_lw);
  o.pc_wr = pieces(j_wr);
  o.pc_th = pieces(j_th);
  return true;
}

// Device buffers of the tables in `o` (which must have been built for this H_eff): allocation
// and upload; replaces the H_eff's tensor-core state. Synchronises the stream.
int upload(mrd_heff* h, const TcTables& o) {
  mrd_ctx* ctx = h->ctx;
  delete h->tc;
  Tc* T = h->tc = new Tc();
  T->prec = o.prec;
  T->cfg = o.cfg;
  T->ntile2 = o.ntile2;
  Arena& A = T->mem;
  A.stream = ctx->stream;
  cudaError_t e = cudaSuccess;
#define TALLOC(ptr, n) if (e == cudaSuccess) e = A.alloc(&(ptr), (size_t)std::max<int64_t>((n), 1))
  TALLOC(T->lw, o.lw_b); TALLOC(T->wr, o.wr_b); TALLOC(T->th, o.th_b); TALLOC(T->z, o.z_b);
  TALLOC(T->it1, o.i1.size()); TALLOC(T->it2, o.i2.size()); TALLOC(T->alt2, o.ia.size());
  TALLOC(T->s1, o.s1.size()); TALLOC(T->s2, o.s2.size());
  TALLOC(T->rmap1, o.rowmap.size());
  TALLOC(T->j_lw, o.j_lw.size()); TALLOC(T->j_wr, o.j_wr.size()); TALLOC(T->j_th, o.j_th.size());
  TALLOC(T->words, 4);
#undef TALLOC
  if (e != cudaSuccess) {   // nothing half-built stays: the next application builds anew
    delete h->tc;
    h->tc = nullptr;
    return mrd_cuda_fail(ctx, e, "tc: device buffers");
  }
  T->n_it1 = (int)o.i1.size(); T->n_it2 = (int)o.i2.size();
  T->n_alt2 = (int)o.ia.size();
  T->task1 = o.task1; T->task2 = o.task2; T->taska = o.taska;
  T->n_lw = (int)(o.j_lw.size() / TCJ); T->n_wr = (int)(o.j_wr.size() / TCJ); T->n_th = (int)(o.j_th.size() / TCJ);
  T->pc_lw = o.pc_lw; T->pc_wr = o.pc_wr; T->pc_th = o.pc_th;
  T->zero_out = o.zero_out;
  cudaStream_t s = ctx->stream;
  auto up = [&](void* d, const void* v, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(d, v, bytes, cudaMemcpyHostToDevice, s);
  };
  for (auto pr : {std::make_pair(T->j_lw, &o.j_lw), std::make_pair(T->j_wr, &o.j_wr), std::make_pair(T->j_th, &o.j_th),
                  std::make_pair(T->rmap1, &o.rowmap)})
    up(pr.first, pr.second->data(), pr.second->size() * 8);
  up(T->it1, o.i1.data(), o.i1.size() * sizeof(TcItem));
  up(T->it2, o.i2.data(), o.i2.size() * sizeof(TcItem));
  up(T->alt2, o.ia.data(), o.ia.size() * sizeof(TcItem));
  up(T->s1, o.s1.data(), o.s1.size() * sizeof(TcSeg));
  up(T->s2, o.s2.data(), o.s2.size() * sizeof(TcSeg));
  // Packing and the Z epilogue write whole K steps; rows that only pad a tile reach only outputs that
  // are not stored. Only Z rows that no product feeds have to be zeros.
  if (e == cudaSuccess && o.zero_z && T->z) e = cudaMemsetAsync(T->z, 0, (size_t)o.z_b, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(T->words, 0, 16, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the host tables may be released after this
  if (e != cudaSuccess) {
    delete h->tc;
    h->tc = nullptr;
    return mrd_cuda_fail(ctx, e, "tc: upload");
  }
  return MRD_OK;
}

int build(mrd_heff* h, int prec, TcCfg cfg) {
  TcTables o;
  if (!tables(h, prec, cfg, o)) return mrd_fail(h->ctx, MRD_E_STATE, o.err);
  return upload(h, o);
}

}  // namespace

namespace {

// Candidate tile configurations per precision (all fit the 227 KB of shared memory).
std::vector<TcCfg> candidates(int prec) {
  if (prec == TC_TF32) return {{128, 3, 0}, {64, 4, 0}, {128, 3, 1}, {64, 4, 1}};
  if (prec == TC_BF16X3) return {{64, 2, 0}, {48, 2, 0}, {64, 2, 1}, {48, 2, 1}};
  if (prec == TC_TF32_REAL) return {{128, 6, 0}, {64, 8, 0}, {128, 6, 1}, {64, 8, 1}};
  return {{128, 3, 0}, {64, 4, 0}, {128, 3, 1}, {64, 4, 1}};
}

// Problem class of an H_eff for the tuning cache: precision, size of theta (powers of two)
// and number of tensor-core step-2 tasks (powers of two).
uint64_t tune_key(const mrd_heff* h, int prec) {
  auto lg = [](int64_t v) { uint64_t b = 0; while (v > 1) { v >>= 1; ++b; } return b; };
  return (uint64_t)prec << 56 | lg(h->counts[C_THETA]) << 40 | lg(h->counts[C_NT2]) << 24 | (uint64_t)h->n_sm;
}

// The two grouped products on the packed operands (the tile counters are zero).
cudaError_t products(const mrd_heff* h, double2* out, cudaStream_t s, cudaEvent_t between = nullptr, bool cap = false) {
  const Tc* T = h->tc;
  cudaError_t e = tc_gemm(T->lw, T->th, T->it1, T->n_it1, nullptr, 0, nullptr, T->s1, T->rmap1, T->z, nullptr, T->prec, T->cfg, T->cfg.ntile, T->words, T->err(),
                          h->n_sm, h->wait_ns, s);
  if (e == cudaSuccess && between) e = record_event(between, s, cap);
  if (e == cudaSuccess)
    e = tc_gemm(T->z, T->wr, T->it2, T->n_it2, T->alt2, T->n_alt2, T->bad(), T->s2, nullptr, nullptr, out, T->prec, T->cfg, T->ntile2, T->words + 1, T->err(), h->n_sm,
                h->wait_ns, s);
  return e;
}

// Kernel time (ms) of steps 1 and 2 with the built configuration, on the packed operands
// (values do not change the time): 1 warm-up, 3 timed applications.
int time_cfg(mrd_heff* h, double* ms) {
  mrd_ctx* ctx = h->ctx;
  Tc* T = h->tc;
  cudaStream_t s = ctx->stream;
  cudaEvent_t a = nullptr, b = nullptr;
  MRD_CUDA(ctx, cudaEventCreate(&a));
  cudaError_t e = cudaEventCreate(&b);
  if (e != cudaSuccess) { cudaEventDestroy(a); return mrd_cuda_fail(ctx, e, "autotune: event"); }
  double2* out = nullptr;   // scratch output of the timing runs
  e = cache_alloc((void**)&out, (size_t)std::max<int64_t>(h->counts[C_THETA], 1) * 16, s);
  for (int r = 0; r < 4 && e == cudaSuccess; ++r) {
    if (r == 1) e = cudaEventRecord(a, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(T->words, 0, 8, s);
    if (e == cudaSuccess) e = products(h, out, s);
  }
  float f = 0.f;
  if (e == cudaSuccess) e = cudaEventRecord(b, s);
  if (e == cudaSuccess) e = cudaEventSynchronize(b);
  if (e == cudaSuccess) e = cudaEventElapsedTime(&f, a, b);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cache_free(out, s);
  if (e != cudaSuccess) return mrd_cuda_fail(ctx, e, "autotune: timing");
  *ms = f / 3.0;
  return tc_status(h);
}

}  // namespace

// Tables being built on a host thread for a known configuration (tc_prebuild).
struct TcPre {
  std::thread th;
  TcTables tab;
  bool ok = false;
  ~TcPre() {
    if (th.joinable()) th.join();
  }
};

void tc_pre_free(TcPre* t) { delete t; }

namespace {

// The configuration a build of `prec` would use without timing anything: the default when
// tuning is off, the tuned one when this problem class is in the context's cache; false when
// it would have to be tuned.
bool known_cfg(const mrd_heff* h, int prec, TcCfg* cfg) {
  if (!h->autotune) {
    *cfg = tc_default_cfg(prec);
    return true;
  }
  auto it = h->ctx->tc_tuned.find(tune_key(h, prec));
  if (it == h->ctx->tc_tuned.end()) return false;
  *cfg = TcCfg{it->second[0], it->second[1], it->second[2]};
  return true;
}

// Build for (prec, cfg), from the host thread's tables when it built exactly these (its thread
// is joined and its tables released either way).
int build_known(mrd_heff* h, int prec, TcCfg cfg) {
  if (TcPre* pre = h->tc_pre) {
    h->tc_pre = nullptr;
    if (pre->th.joinable()) pre->th.join();
    const TcTables& o = pre->tab;
    const bool same = pre->ok && o.prec == prec && o.n_sm == h->n_sm && o.cfg.ntile == cfg.ntile &&
                      o.cfg.stages == cfg.stages && o.cfg.order == cfg.order;
    int rc = same ? upload(h, o) : MRD_OK;
    delete pre;
    if (same) return rc;
  }
  return build(h, prec, cfg);
}

}  // namespace

// Starts building the tensor-core tables of `prec` on a host thread when their configuration
// is known without timing (tuning off, or this problem class tuned earlier on the context),
// so that the host work (milliseconds at large bond dimension) overlaps device work queued
// meanwhile; the next tc_prepare joins it. Does nothing otherwise, or when the thread cannot be
// started (tc_prepare then builds the tables itself). The host tables of h must not change
// until the thread is joined (tc_prepare, or freeing h).
void tc_prebuild(mrd_heff* h, int32_t prec) {
  const int tp = tc_prec_of(h, prec);
  TcCfg cfg{0, 0, 0};
  if ((h->tc && h->tc->prec == tp) || h->tc_pre || !known_cfg(h, tp, &cfg)) return;
  TcPre* pre = new (std::nothrow) TcPre();
  if (!pre) return;
  try {
    pre->th = std::thread([h, pre, tp, cfg] {
      try {
        pre->ok = tables(h, tp, cfg, pre->tab);
      } catch (...) {   // out of host memory: tc_prepare builds the tables itself
        pre->ok = false;
      }
    });
  } catch (...) {
    delete pre;
    return;
  }
  h->tc_pre = pre;
}

// Pick the tile configuration: from the context's tuning cache for this problem class, else
// by timing every candidate on this H_eff (MRD_OPT_AUTOTUNE, default on), else the default.
int autotune(mrd_heff* h, int prec) {
  mrd_ctx* ctx = h->ctx;
  const uint64_t key = tune_key(h, prec);
  TcCfg known{0, 0, 0};
  if (known_cfg(h, prec, &known)) {
    int rc = build_known(h, prec, known);
    if (rc == MRD_OK) h->tc->cfg_source = h->autotune ? 2 : 0;
    return rc;
  }
  if (h->tc_pre) {   // tables of another precision
    tc_pre_free(h->tc_pre);
    h->tc_pre = nullptr;
  }
  TcCfg best{0, 0, 0};
  double best_ms = 1e300;
  for (const TcCfg& c : candidates(prec)) {
    int rc = build(h, prec, c);
    if (rc != MRD_OK) return rc;
    Tc* T = h->tc;
    MRD_CUDA(ctx, tc_pack(h->lw, T->lw, T->j_lw, T->n_lw, T->pc_lw, prec, nullptr, nullptr, ctx->stream));
    MRD_CUDA(ctx, tc_pack(h->wr, T->wr, T->j_wr, T->n_wr, T->pc_wr, prec, nullptr, T->bad(), ctx->stream));
    double ms = 0.0;
    if ((rc = time_cfg(h, &ms)) != MRD_OK) return rc;
    if (ms < best_ms) { best_ms = ms; best = c; }
  }
  ctx->tc_tuned[key] = {best.ntile, best.stages, best.order};
  const TcCfg last = candidates(prec).back();
  if (best.ntile != last.ntile || best.stages != last.stages || best.order != last.order) {
    int rc = build(h, prec, best);
    if (rc != MRD_OK) return rc;
  }
  h->tc->cfg_source = 1;
  h->tc->env_dirty = true;
  return MRD_OK;
}

void tc_env_changed(mrd_heff* h) {
  if (h->tc) h->tc->env_dirty = true;
}

int tc_status(mrd_heff* h) {
  if (!h->tc || !h->tc->words) return MRD_OK;
  int herr = 0;
  MRD_CUDA(h->ctx, cudaMemcpyAsync(&herr, h->tc->err(), 4, cudaMemcpyDeviceToHost, h->ctx->stream));
  MRD_CUDA(h->ctx, cudaStreamSynchronize(h->ctx->stream));
  if (herr) {   // reported once: the flag is cleared for the next launches
    MRD_CUDA(h->ctx, cudaMemsetAsync(h->tc->err(), 0, 4, h->ctx->stream));
    MRD_CUDA(h->ctx, cudaStreamSynchronize(h->ctx->stream));
    return mrd_fail(h->ctx, MRD_E_TIMEOUT, "tensor-core GEMM: a bounded wait gave up (code " + std::to_string(herr) + ")");
  }
  return MRD_OK;
}

// Panel tables and buffers for `prec` (host work, allocation, synchronisation) and the packed
// environments; a no-op when both are current.
int tc_prepare(mrd_heff* h, int32_t prec) {
  mrd_ctx* ctx = h->ctx;
  const int tp = tc_prec_of(h, prec);
  int rc;
  MRD_CUDA(ctx, tc_gemm_init());
  if (!h->tc || h->tc->prec != tp) {
    if (!h->tc) h->tc = new Tc();
    if ((rc = autotune(h, tp)) != MRD_OK) return rc;
    ++h->gen;
  }
  Tc* T = h->tc;
  cudaStream_t s = ctx->stream;
  if (T->env_dirty) {
    MRD_CUDA(ctx, cudaMemsetAsync(T->bad(), 0, 4, s));
    MRD_CUDA(ctx, tc_pack(h->lw, T->lw, T->j_lw, T->n_lw, T->pc_lw, tp, nullptr, nullptr, s));
    MRD_CUDA(ctx, tc_pack(h->wr, T->wr, T->j_wr, T->n_wr, T->pc_wr, tp, nullptr, T->bad(), s));
    T->env_dirty = false;
  }
  return MRD_OK;
}

int tc_config(const mrd_heff* h, int32_t* cfg4) {
  if (!h->tc) {
    cfg4[0] = cfg4[1] = cfg4[2] = cfg4[3] = -1;
    return MRD_OK;
  }
  cfg4[0] = h->tc->cfg.ntile;
  cfg4[1] = h->tc->cfg.stages;
  cfg4[2] = h->tc->cfg.order;
  cfg4[3] = h->tc->cfg_source;
  return MRD_OK;
}

int tc_apply(mrd_heff* h, const double* in, double* out, int32_t prec) {
  mrd_ctx* ctx = h->ctx;
  const int tp = tc_prec_of(h, prec);
  int rc = tc_prepare(h, prec);
  if (rc != MRD_OK) return rc;
  Tc* T = h->tc;
  cudaStream_t s = ctx->stream;
  cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
  bool cap = false;
  if (h->timing && !apply_events(h, s, ev, &cap)) return mrd_fail(ctx, MRD_E_CUDA, "mrd_heff_apply: cudaEventCreate");
  const cudaEvent_t e0 = ev[0], e1 = ev[1], e2 = ev[2];
  if (T->zero_out) MRD_CUDA(ctx, cudaMemsetAsync(out, 0, (size_t)h->counts[C_THETA] * 16, s));
  MRD_CUDA(ctx, tc_pack((const double2*)in, T->th, T->j_th, T->n_th, T->pc_th, tp, T->words, nullptr, s));
  MRD_CUDA(ctx, record_event(e0, s, cap));
  if (!h->per_task) {
    MRD_CUDA(ctx, products(h, (double2*)out, s, e1, cap));
  } else {   // one launch per task: the per-block baseline of the grouped persistent launch
    for (size_t t = 0; t + 1 < T->task1.size(); ++t)
      MRD_CUDA(ctx, tc_gemm(T->lw, T->th, T->it1 + T->task1[t], T->task1[t + 1] - T->task1[t], nullptr, 0, nullptr, T->s1, T->rmap1, T->z, nullptr, tp, T->cfg,
                            T->cfg.ntile, nullptr, T->err(), h->n_sm, h->wait_ns, s));
    MRD_CUDA(ctx, record_event(e1, s, cap));
    for (size_t t = 0; t + 1 < T->task2.size(); ++t)
      MRD_CUDA(ctx, tc_gemm(T->z, T->wr, T->it2 + T->task2[t], T->task2[t + 1] - T->task2[t], T->alt2 + T->taska[t],
                            T->taska[t + 1] - T->taska[t], T->bad(), T->s2, nullptr, nullptr, (double2*)out, tp, T->cfg, T->ntile2, nullptr, T->err(), h->n_sm, h->wait_ns, s));
  }
  MRD_CUDA(ctx, record_event(e2, s, cap));
  return MRD_OK;
}
