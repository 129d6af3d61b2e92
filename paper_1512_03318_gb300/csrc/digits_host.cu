// Host side of the digit-split grouped GEMM (digits.cuh): stacking of the tasks of plan.cuh's
// tables into panels, and the two products of an H_eff application.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <exception>
#include <memory>
#include <thread>

#include "digits.cuh"
#include "heff_internal.h"

namespace mrd {

namespace {

int64_t up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

// Cycles of one K step of a complex tile of `nrow` columns (32 MMAs of N = 8 nrow .. nrow, at
// least 48 cycles each, else N / 2: measured 2510 and 1669), of one flush of the accumulators and
// of a tile's ends.
double step_cycles(int nrow, bool real) { return (nrow > 16 ? 2510.0 : 1669.0) / (real ? 4 : 1); }
constexpr double kFlushCycles = 3000.0, kTileCycles = 3000.0;

// Cycles per K step of all tiles of a group whose tall side has R rows.
double group_step_cycles(int R, int N, bool real) {
  const int full = N / kDgCols, rest = N % kDgCols;
  const double c = full * step_cycles(32, real) + (rest ? step_cycles(rest > 16 ? 32 : 16, real) : 0.0);
  return (R + kDgRows - 1) / kDgRows * c;
}

}  // namespace

void dg_plan(DgPlan& p, const int64_t* tasks, const int64_t* segs, int64_t n_tasks, DgStack how, const int32_t* ids,
             bool real, int beta, int n_sm, bool group_major) {
  p.real = real;
  // the stacked operand (members one under the other) and the shared one
  const int sop = how == DG_BY_A ? 1 : 0, uop = 1 - sop;
  p.sop = sop;
  const int sf = sop ? 2 : 0, uf = uop ? 2 : 0;        // first segment field of their blocks (off, ld)
  const int64_t sbit = sop ? 2 : 1, ubit = uop ? 2 : 1;   // their flag bits (conjugate-transposed)
  struct Entry {   // a shared block of a group
    int64_t off, ld;
    int32_t K, k0, kpad;
    bool ct;
  };
  struct Member {
    int64_t task;
    int32_t rows, row0;
  };
  struct Group {
    int32_t N, R, kp;   // shared and stacked extents, padded K
    std::vector<Entry> e;
    std::vector<Member> m;
    bool rising;        // the blocks' offsets rise from one to the next, here and in every member's list
  };
  std::vector<Group> gs;
  gs.reserve((size_t)std::min<int64_t>(n_tasks, 1024));
  // open addressing over the groups' signatures (an id, or the shared blocks)
  size_t cells = 64;
  while (cells < (size_t)n_tasks * 2 && cells < ((size_t)1 << 20)) cells *= 2;
  std::vector<std::pair<uint64_t, int32_t>> index(cells, {0, -1});
  int64_t n_segs = 0;
  for (int64_t i = 0; i < n_tasks; ++i) {
    const int64_t* t = tasks + 6 * i;
    const int64_t ns = t[5];
    if (ns <= 0 || t[0] <= 0 || t[1] <= 0) continue;
    n_segs += ns;
    const int64_t* sg = segs + 6 * t[4];
    const int32_t rows = (int32_t)t[sop], N = (int32_t)t[uop];
    uint64_t h = 0x9E3779B97F4A7C15ull * (uint64_t)(N + 1);
    if (how == DG_BY_ID) {
      h = 0x9E3779B97F4A7C15ull * (uint64_t)(ids[i] + 1);
    } else {
      for (int64_t k = 0; k < ns; ++k) {
        h = (h ^ (uint64_t)sg[6 * k + uf]) * 0xBF58476D1CE4E5B9ull;
        h ^= h >> 29;
        h = (h + (uint64_t)sg[6 * k + 4]) * 0x94D049BB133111EBull;
        h ^= h >> 31;
      }
    }
    int32_t gi = -1;
    for (size_t at = (size_t)(h >> 20) & (cells - 1);; at = (at + 1) & (cells - 1)) {
      if (index[at].second < 0) {
        if (gs.size() + 1 >= cells) {   // more groups than cells: not this kind of problem
          p.items.clear();
          return;
        }
        index[at] = {h, gi = (int32_t)gs.size()};
        break;
      }
      if (index[at].first != h) continue;
      const Group& g = gs[(size_t)index[at].second];
      bool same = how == DG_BY_ID || (g.N == N && (int64_t)g.e.size() == ns);
      for (int64_t k = 0; same && how != DG_BY_ID && k < ns; ++k)
        same = g.e[(size_t)k].off == sg[6 * k + uf] && g.e[(size_t)k].ld == sg[6 * k + uf + 1] &&
               g.e[(size_t)k].K == sg[6 * k + 4] && g.e[(size_t)k].ct == ((sg[6 * k + 5] & ubit) != 0);
      if (same) {
        gi = index[at].second;
        break;
      }
    }
    if (gi == (int32_t)gs.size()) gs.push_back(Group{N, 0, 0, {}, {}, true});
    Group& g = gs[(size_t)gi];
    if (g.m.empty() || how == DG_BY_ID) {   // collect the shared blocks (members list them in one order)
      size_t cur = 0;
      int64_t before = -1;
      if (g.m.empty()) g.e.reserve((size_t)ns);
      for (int64_t k = 0; k < ns; ++k) {
        const int64_t off = sg[6 * k + uf];
        const size_t n = g.e.size();
        g.rising = g.rising && off > before;
        before = off;
        size_t f = n;
        if (cur < n && g.e[cur].off == off) {
          f = cur;
        } else if (!g.rising || (n > 0 && off <= g.e[n - 1].off)) {   // from the cursor on, around to it
          for (size_t q = 0; q < n && f == n; ++q) {
            const size_t at = cur + q < n ? cur + q : cur + q - n;
            if (g.e[at].off == off) f = at;
          }
        }
        if (f == n) {
          g.rising = g.rising && (n == 0 || off > g.e[n - 1].off);
          g.e.push_back({off, sg[6 * k + uf + 1], (int32_t)sg[6 * k + 4], 0, 0, (sg[6 * k + 5] & ubit) != 0});
        }
        cur = f + 1;
      }
    }
    g.m.push_back({i, rows, g.R});
    g.R += rows;
  }
  for (Group& g : gs) {
    int32_t k = 0;
    for (Entry& e : g.e) {
      e.k0 = k;
      e.kpad = (int32_t)up(e.K, 8);
      k += e.kpad;
    }
    if (k % kDgStep) {   // the last block also writes the step's zeros
      g.e.back().kpad += 8;
      k += 8;
    }
    g.kp = k;
    if (k / kDgStep >= 32768) {   // outside the items' K field: left to the other kernels
      p.items.clear();
      return;
    }
  }
  const int64_t pb = 32 * dg_planes(real);
  const int fl = dg_flush(beta);
  auto tile_cost = [&](int nks, int nrow) {
    return nks * step_cycles(nrow, real) + (nks + fl - 1) / fl * kFlushCycles + kTileCycles;
  };
  double total = 0.0;
  size_t nu = 0, nst = 0, nm = 0;
  for (const Group& g : gs) {
    nu += g.e.size();
    nst += g.e.size() * g.m.size();
    nm += g.m.size();
  }
  p.groups.reserve(gs.size());
  p.jobs[uop].reserve(nu);
  p.jobs[sop].reserve(nst);
  p.members.reserve(nm);
  for (const Group& g : gs) {
    const int32_t nks = g.kp / kDgStep;
    // the side whose padding to 128 rows wastes less is the tall one (the stacked one on ties:
    // its results are written along the shared side)
    const bool s_tall = group_step_cycles(g.R, g.N, real) <= group_step_cycles(g.N, g.R, real);
    const int32_t es = (int32_t)p.rows[sop], eu = (int32_t)p.rows[uop];
    const int64_t os = p.bytes[sop], ou = p.bytes[uop];
    DgGroup d;
    d.R = s_tall ? g.R : g.N;
    d.N = s_tall ? g.N : g.R;
    d.nks = nks;
    d.a_off = s_tall ? os : ou;
    d.b_off = s_tall ? ou : os;
    d.ea = s_tall ? es : eu;
    d.eb = s_tall ? eu : es;
    d.tall_op = s_tall ? sop : uop;
    d.cm = (int32_t)p.cmap;
    d.cm_rows = s_tall ? 1 : 0;
    d.job = (int32_t)p.jobs[uop].size();
    d.n_jobs = (int32_t)g.e.size();
    const int32_t s_flag = s_tall ? DGJ_TALL : 0, u_flag = s_tall ? 0 : DGJ_TALL;
    auto kind = [](int op, bool ct) { return ((op ? ct : !ct) ? DGJ_KCONTIG : 0) | (ct ? DGJ_CONJ : 0); };
    for (const Entry& e : g.e)
      p.jobs[uop].push_back({e.off, e.ld, ou, g.N, e.K, e.kpad, 0, e.k0, g.N, nks, eu, kind(uop, e.ct) | u_flag, 0});
    for (const Member& m : g.m) {
      const int64_t* t = tasks + 6 * m.task;
      const int64_t* sg = segs + 6 * t[4];
      const int32_t job0 = (int32_t)p.jobs[sop].size();
      int64_t k = 0;
      for (size_t f = 0; f < g.e.size(); ++f) {
        const Entry& e = g.e[f];
        // the member's segment of this shared block (both list them in one order; a member of a
        // DG_BY_ID group may lack some or, rarely, list them otherwise)
        int64_t hit = -1;
        if (k < t[5] && sg[6 * k + uf] == e.off) {
          hit = k++;
        } else if (how == DG_BY_ID && !(g.rising && (k == t[5] || sg[6 * k + uf] > e.off))) {
          for (int64_t q = 0; q < t[5]; ++q)
            if (sg[6 * q + uf] == e.off) {
              hit = q;
              k = q + 1;
              break;
            }
        }
        const int64_t* s = sg + 6 * (hit >= 0 ? hit : 0);
        const bool ct = hit >= 0 && (s[5] & sbit) != 0;
        p.jobs[sop].push_back({hit >= 0 ? s[sf] : -1, s[sf + 1], os, m.rows, e.K, e.kpad, m.row0, e.k0, g.R, nks,
                               es + m.row0, kind(sop, ct) | s_flag, 0});
      }
      p.members.push_back({t[2], sop ? 1 : t[3], sop ? t[3] : 1, (int32_t)p.cmap + m.row0, m.rows, (int32_t)p.groups.size(), job0});
      const int64_t tiles = up(m.rows, kDgRedoTile) / kDgRedoTile * (up(g.N, kDgRedoTile) / kDgRedoTile);
      p.redo += tiles;
      p.max_tiles = (int)std::max<int64_t>(p.max_tiles, tiles);
    }
    p.cmap += g.R;
    p.bytes[sop] += up(g.R, s_tall ? 8 : 16) * nks * pb;
    p.bytes[uop] += up(g.N, s_tall ? 16 : 8) * nks * pb;
    p.rows[sop] += g.R;
    p.rows[uop] += g.N;
    p.groups.push_back(d);
    const int tm = (d.R + kDgRows - 1) / kDgRows, tn = (d.N + kDgCols - 1) / kDgCols;
    total += tm * (tn - 1) * tile_cost(nks, 32) + tm * tile_cost(nks, d.N - (tn - 1) * kDgCols);
  }
  // Items. A tile longer than a third of an SM's share is cut along K into parts (their integer
  // sums add exactly), so that a few long tiles neither leave SMs idle nor end the launch alone. A part
  // writes its 96-bit sums and the last one reads those of all others, one after another (~20,000
  // cycles for each), so parts stay above 100,000 cycles or 1.6 shares where the shares are short. us of
  // step 2 (parts from a third of a share or 9,000 cycles on / these): float-float Ly = 5, chi = 301
  // 128 / 70, Ly = 8, chi = 1024 418 / 333, Ly = 10, chi = 400 303 / 125; FP64 85 / 67, 338 / 331, 155 / 110.
  const double share = total / n_sm, cap = std::max({9000.0, std::min(1.6 * share, 100000.0), share / 3.0});
  struct Cls {   // tiles of a group with the same number of columns
    double cost;
    int32_t group, parts, ct0, ct1;
  };
  std::vector<Cls> cls;
  cls.reserve(gs.size() * 2);
  double longest = 0.0;
  for (size_t i = 0; i < p.groups.size(); ++i) {
    const DgGroup& d = p.groups[i];
    const int tn = (d.N + kDgCols - 1) / kDgCols, last = d.N - (tn - 1) * kDgCols;
    const int cut = last > 16 ? tn : tn - 1;   // column tiles of 32
    for (int z = 0; z < 2; ++z) {
      const int c0 = z ? cut : 0, c1 = z ? tn : cut;
      if (c0 >= c1) continue;
      const double c = tile_cost(d.nks, z ? 16 : 32);
      int parts = 1;
      if (!group_major && c > cap) parts = std::max(1, std::min({(int)std::ceil(c / cap), d.nks / 3, 60}));
      const double each = tile_cost((d.nks + parts - 1) / parts, z ? 16 : 32);
      longest = std::max(longest, each);
      cls.push_back({each, (int32_t)i, parts, c0, c1});
    }
  }
  if (!group_major) std::stable_sort(cls.begin(), cls.end(), [](const Cls& a, const Cls& b) { return a.cost > b.cost; });
  for (const Cls& c : cls) {
    const DgGroup& d = p.groups[(size_t)c.group];
    const int tm = (d.R + kDgRows - 1) / kDgRows, tn = (d.N + kDgCols - 1) / kDgCols;
    if (group_major)
      while ((int32_t)p.item0.size() <= c.group) p.item0.push_back((int64_t)p.items.size());
    // the tiles of one K range follow each other: CTAs that run together then read the same rows and
    // columns of the panels, which come from DRAM once
    const int sid = (int)p.splits.size(), wide = c.ct1 - c.ct0;
    if (c.parts > 1)
      for (int q = 0; q < tm * wide; ++q, p.slots += c.parts) p.splits.push_back(make_int2((int)p.slots, c.parts));
    for (int q = 0; q < c.parts; ++q) {
      const int k0 = (int)((int64_t)d.nks * q / c.parts), k1 = (int)((int64_t)d.nks * (q + 1) / c.parts);
      for (int r = 0; r < tm; ++r)
        for (int ct = c.ct0; ct < c.ct1; ++ct)
          p.items.push_back({c.group, r * tn + ct, k0 | k1 << 16,
                             c.parts > 1 ? (sid + r * wide + ct - c.ct0) * 64 + q : -1});
    }
  }
  if (group_major) p.item0.push_back((int64_t)p.items.size());
  p.cost = total / n_sm + 0.5 * longest + 12000.0;
  for (int op = 0; op < 2; ++op) {
    p.pieces[op].reserve(p.jobs[op].size() * 2);
    p.mpieces[op].reserve(p.jobs[op].size() * 2);
    for (size_t j = 0; j < p.jobs[op].size(); ++j) {
      const DgJob& b = p.jobs[op][j];
      const bool kc = (b.flags & DGJ_KCONTIG) != 0;
      const int64_t units = (int64_t)b.rows * (kc ? b.kpad / 2 : b.kpad / 8);
      const int64_t per = kc ? kDgPairPiece : kDgChunkPiece;
      for (int64_t u = 0; u < units; u += per) p.pieces[op].push_back(make_int2((int)j, (int)u));
      if (b.off < 0) continue;
      const int n = kc ? b.rows : b.K, q = kc ? kDgMaxRows : kDgMaxK;
      for (int u = 0; u < n; u += q) p.mpieces[op].push_back(make_int2((int)j, u));
    }
  }
}

// The 32 x 32 tile kernels: K multiply-adds of 1024 outputs per tile (FP64: 4 FMAs at 1.7 per
// cycle and SM; float-float: 36 instructions, 12 when real, at 75% of 128 lanes), no shorter than
// the longest tile's chain of K chunks (~3 us each when few tiles run).
double dg_cost_cores(const int64_t* tasks, const int64_t* segs, int64_t n_tasks, bool ff, bool real, int n_sm) {
  double sum = 0.0, longest = 0.0;
  const double per_k = ff ? (real ? 12 : 36) * 1024.0 / 96.0 : 2400.0;
  for (int64_t i = 0; i < n_tasks; ++i) {
    const int64_t* t = tasks + 6 * i;
    if (t[5] <= 0 || t[0] <= 0 || t[1] <= 0) continue;
    double k = 0.0, chunks = 0.0;
    for (int64_t q = 0; q < t[5]; ++q) {
      const int64_t K = segs[6 * (t[4] + q) + 4];
      k += (double)K;
      chunks += (double)((K + 15) / 16);
    }
    sum += (double)(((t[0] + 31) / 32) * ((t[1] + 31) / 32)) * k * per_k;
    longest = std::max(longest, chunks * 5500.0);
  }
  return std::max(sum / n_sm, longest) + 8000.0;
}

namespace {
template <class T>
size_t vbytes(const std::vector<T>& v) { return (size_t)up((int64_t)(v.size() * sizeof(T)), 16); }
template <class T>
void place(const std::vector<T>& v, uint8_t* host, uint8_t* dev, size_t& off, T** out) {
  if (!v.empty()) std::memcpy(host + off, v.data(), v.size() * sizeof(T));
  *out = (T*)(dev + off);
  off += vbytes(v);
}
}  // namespace

size_t dg_table_bytes(const DgPlan& p) {
  size_t n = vbytes(p.groups) + vbytes(p.items) + vbytes(p.splits) + vbytes(p.members);
  for (int s = 0; s < 2; ++s) n += vbytes(p.jobs[s]) + vbytes(p.pieces[s]) + vbytes(p.mpieces[s]);
  return n;
}

size_t dg_device_table_bytes(const DgPlan& p) { return dg_table_bytes(p) + (size_t)p.cmap * sizeof(longlong2); }

void dg_tables(const DgPlan& p, uint8_t* host, uint8_t* dev, DgDev& d) {
  size_t off = 0;
  d.tab = dev;
  for (int s = 0; s < 2; ++s) {
    place(p.jobs[s], host, dev, off, &d.jobs[s]);
    place(p.pieces[s], host, dev, off, &d.pieces[s]);
    place(p.mpieces[s], host, dev, off, &d.mpieces[s]);
    d.n_pieces[s] = (int)p.pieces[s].size();
    d.n_mpieces[s] = (int)p.mpieces[s].size();
    d.rows[s] = p.rows[s];
  }
  place(p.groups, host, dev, off, &d.groups);
  place(p.items, host, dev, off, &d.items);
  place(p.splits, host, dev, off, &d.splits);
  place(p.members, host, dev, off, &d.members);
  d.cmap = (longlong2*)(dev + off);
  d.n_members = (int)p.members.size();
  d.n_items = (int)p.items.size();
  d.n_splits = (int)p.splits.size();
  d.tab_bytes = off;
  d.max_tiles = p.max_tiles;
  d.sop = p.sop;
  d.real = p.real;
}

}  // namespace mrd

// ---------------------------------------------------------------- H_eff

// The two products of an H_eff in one form: a precision, with or without imaginary parts, grouped or
// one launch per stacked block. Plans, device buffers and packed environments stay until the handle is
// freed, so that a program that changes precisions on it plans and packs once for each.
struct DgForm {
  int32_t prec = 0;
  int beta = 0;
  bool real = false, major = false;
  bool decided = false, planned = false;   // whether digits are cheaper is known; the plans are made
  bool refused = false;                    // dimensions beyond the tables' fields: there can be no plans
  bool cheaper = false, built = false, env_dirty = true;
  bool captured = false;   // a caller's graph reads the panels
  bool no_room = false;    // the panels found no memory since the last environment load
  DgPlan p1, p2;
  DgDev d1, d2;
  int* words = nullptr;   // DG_WORDS, then the exponents of theta and Z and the products' states (zeroed
  size_t zero_bytes = 0;  // together before each application)
  Arena mem;
};
// Digit-split state of an H_eff. A form's plans may be built on a host thread (dg_prebuild) while the
// device works.
struct DgHeff {
  std::vector<std::unique_ptr<DgForm>> forms;
  DgForm* cur = nullptr;   // of the last prepared application
  std::thread th;
  ~DgHeff() {
    if (th.joinable()) th.join();
  }
  DgForm* form(int32_t prec, bool real, bool major) {
    for (auto& f : forms)
      if (f->prec == prec && f->real == real && f->major == major) return f.get();
    forms.push_back(std::make_unique<DgForm>());
    DgForm* f = forms.back().get();
    f->prec = prec;
    f->beta = prec == MRD_PREC_FP64 ? 8 : 7;
    f->real = real;
    f->major = major;
    return f;
  }
};

void dg_heff_free(DgHeff* g) { delete g; }

namespace {

// Cycles of planning, uploading and packing the environments of a small H_eff (~50 us: what the
// applications of one environment load must save together; the other way needs next to no
// setup). On the 4 x 4 cylinder (chi = 64, 6 applications per load) a sweep takes 53 ms with this
// line, 62 ms with twice the value and 90 ms on the CUDA cores alone.
constexpr double kSetupCycles = 100000.0;

double cores_cost(const mrd_heff* h, bool ff, bool real) {
  return dg_cost_cores(h->t1_host.data(), h->s1_host.data(), h->counts[C_NT1], ff, real, h->n_sm) +
         dg_cost_cores(h->t2_host.data(), h->s2_host.data(), h->counts[C_NT2], ff, real, h->n_sm);
}

// K of the segments over their K in the panels: dg_plan pads each to 8 (and a group's total to 16).
double k_padding(const mrd_heff* h) {
  double padded = 0.0, k = 0.0;
  auto add = [&](const std::vector<int64_t>& t, const std::vector<int64_t>& sg, int64_t n) {
    for (int64_t i = 0; i < n; ++i)
      for (int64_t q = 0; q < t[(size_t)(TF * i + 5)]; ++q) {
        const int64_t K = sg[(size_t)(SF * (t[(size_t)(TF * i + 4)] + q) + 4)];
        k += (double)K;
        padded += (double)up(K, 8);
      }
  };
  add(h->t1_host, h->s1_host, h->counts[C_NT1]);
  add(h->t2_host, h->s2_host, h->counts[C_NT2]);
  return k > 0.0 ? padded / k : 1.0;
}

// Float-float products whose segments are mostly padding stay on the CUDA cores, which take their K as it
// is: dg_cost_cores counts whole chunks of 16 there and would call them too dear (FP64 ones do not, that
// pipe is 12 times slower). First application on a new handle / every further one, us, digits | CUDA cores:
// padding 2.3 (Ly = 10, chi = 100) 916 / 116 | 340 / 165, 2.2 (Ly = 4, chi = 40) 239 / 85 | 117 / 58, 2.1 (Ly = 6, chi
// = 64) 390 / 96 | 178 / 91, 1.9 (Ly = 5, chi = 61) 278 / 90 | 141 / 79; 1.4 (Ly = 5, chi = 301) 500 / 123 |
// 280 / 191, 1.2 (Ly = 10, chi = 400) 717 / 183 | 699 / 520.
constexpr double kMaxPadding = 1.55;

// Decides whether the digit products of a form are the cheaper way (the same for grouped and per-task launches,
// which give the same bits), with the plans of both unless it is plain without; force: the plans in any case.
void plan_both(const mrd_heff* h, DgForm* g, bool force) {
  const int64_t n1 = h->counts[C_NT1], n2 = h->counts[C_NT2];
  const bool ff = g->prec == MRD_PREC_FF, real = g->real;
  const int beta = g->beta;
  const double cores = cores_cost(h, ff, real);
  const bool worth = cores * h->dg_uses >= kSetupCycles && !(ff && k_padding(h) > kMaxPadding);
  g->cheaper = false;
  g->decided = true;
  if (!worth && !force) return;
  std::vector<int32_t> ids((size_t)n2);   // step 2: the two row parts s1' of an output sector
  for (int64_t i = 0; i < n2; ++i) ids[(size_t)i] = (int32_t)(i >> 2 << 1 | (i & 1));   // share (nearly) all WR blocks
  // the two plans are independent: the second on a host thread of its own where that pays for starting
  // one (~60 us with its first use of the tables; a plan takes ~40 ns per segment)
  int64_t segs2 = 0;
  for (int64_t i = 0; i < n2; ++i) segs2 += h->t2_host[(size_t)(TF * i + 5)];
  auto both = [&](bool gm) {
    g->p1 = DgPlan();
    g->p2 = DgPlan();
    auto second = [&] {
      dg_plan(g->p2, h->t2_host.data(), h->s2_host.data(), n2, DG_BY_ID, ids.data(), real, beta, h->n_sm, gm);
    };
    std::exception_ptr failed;
    std::thread th;
    if (segs2 > 2500) {
      try {
        th = std::thread([&] {
          try {
            second();
          } catch (...) {
            failed = std::current_exception();
          }
        });
      } catch (...) {   // no thread to be had
      }
    }
    struct Join {
      std::thread& t;
      ~Join() { if (t.joinable()) t.join(); }
    } join{th};
    const bool split = th.joinable();
    dg_plan(g->p1, h->t1_host.data(), h->s1_host.data(), n1, DG_BY_B, nullptr, real, beta, h->n_sm, gm);
    if (!split) return second();
    th.join();
    if (failed) std::rethrow_exception(failed);
  };
  both(false);
  // the exponent and digit passes move ~80 bytes per element of theta and Z
  const double pass = (double)(h->counts[C_THETA] + h->counts[C_ZLEN]) * 80.0 / 5.0e12 * 1.9e9 + 25000.0;
  const double mine = g->p1.cost + g->p2.cost + pass;
  const bool fits = !g->p1.items.empty() && !g->p2.items.empty();   // (else dimensions beyond the tables' fields)
  g->cheaper = worth && fits && mine * h->dg_uses + kSetupCycles < cores * h->dg_uses;
  if (fits && g->major) both(true);
  g->planned = fits;
  g->refused = !fits;
}

}  // namespace

// Start planning on a host thread (the host tables of h must not change until dg_prepare or
// until h is freed); does nothing when no thread can be had.
void dg_prebuild(mrd_heff* h, int32_t prec) {
  const bool ff = prec == MRD_PREC_FF;
  if (h->dg || h->dg_mode != 1 || cores_cost(h, ff, h->real && ff) * h->dg_uses < 2 * kSetupCycles)
    return;   // planned on demand (or not at all) where that is a matter of microseconds
  DgHeff* g = new DgHeff();
  h->dg = g;
  DgForm* f = g->form(prec, h->real && ff, h->per_task);
  try {
    g->th = std::thread([h, f] {
      try {
        plan_both(h, f, false);
      } catch (...) {   // out of host memory: planned on demand instead
        f->decided = f->planned = false;
      }
    });
  } catch (...) {
  }
}

// Plans, tables, panels and packed environments for `prec`; *use tells whether the digit-split
// products take this H_eff (else the CUDA-core kernels do: very small problems, or no memory for
// the panels).
int dg_prepare(mrd_heff* h, int32_t prec, bool* use) {
  mrd_ctx* ctx = h->ctx;
  cudaStream_t s = ctx->stream;
  // In a caller's capture nothing can be allocated, and what is packed now would be old when the graph is
  // replayed after another environment load. The FP64 kernel needs no preparation and reads LW and WR
  // themselves; float-float products run in the form that an earlier application has built.
  const bool cap = !h->in_lanczos && stream_capturing(s);
  *use = false;
  h->dg_form = 0;
  if (h->dg_mode == 0 || (cap && prec == MRD_PREC_FP64)) return MRD_OK;
  if (!h->dg) h->dg = new DgHeff();
  if (h->dg->th.joinable()) h->dg->th.join();
  DgForm* g = h->dg->cur = h->dg->form(prec, h->real && prec == MRD_PREC_FF, h->per_task);
  const int beta = g->beta;
  if (cap && !g->built) return MRD_OK;
  const bool force = h->dg_mode == 2;
  if (!g->decided || (force && !g->planned && !g->refused)) {
    plan_both(h, g, force);
    ++h->gen;
  }
  if (!g->planned || !(g->cheaper || force)) return MRD_OK;
  if (!g->built && g->no_room) {
    h->dg_form = 2;
    return MRD_OK;
  }
  if (!g->built) {
    Arena& A = g->mem;
    A.stream = s;
    const size_t b1 = dg_table_bytes(g->p1), b2 = dg_table_bytes(g->p2), d1 = dg_device_table_bytes(g->p1);
    uint8_t* tab = nullptr;
    int* env_expo = nullptr;
    uint8_t* partial = nullptr;
    const int64_t ne = g->p1.rows[0] + g->p2.rows[1], ns1 = dg_state_words(g->p1);
    const int64_t nz = g->p1.rows[1] + g->p2.rows[0] + ns1 + dg_state_words(g->p2);
    int2* redo = nullptr;
    cudaError_t e = A.alloc(&tab, d1 + dg_device_table_bytes(g->p2) + 16);
    if (e == cudaSuccess) e = A.alloc(&g->words, (size_t)(DG_WORDS + nz));
    if (e == cudaSuccess) e = A.alloc(&env_expo, (size_t)std::max<int64_t>(ne, 1));
    if (e == cudaSuccess) e = A.alloc(&redo, (size_t)std::max(g->p1.redo, g->p2.redo));
    if (e == cudaSuccess) e = A.alloc(&partial, (size_t)(std::max<int64_t>({g->p1.slots, g->p2.slots, 1}) * kDgSlotBytes));
    if (e == cudaSuccess) e = A.alloc(&g->d1.panel[0], (size_t)g->p1.bytes[0]);
    if (e == cudaSuccess) e = A.alloc(&g->d1.panel[1], (size_t)g->p1.bytes[1]);
    if (e == cudaSuccess) e = A.alloc(&g->d2.panel[0], (size_t)g->p2.bytes[0]);
    if (e == cudaSuccess) e = A.alloc(&g->d2.panel[1], (size_t)g->p2.bytes[1]);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      A.release();
      if (dg_release(h)) return dg_prepare(h, prec, use);   // another form's panels made way
      g->no_room = true;   // the CUDA-core kernels need none
      h->dg_form = 2;
      return MRD_OK;
    }
    if (e != cudaSuccess) return mrd_cuda_fail(ctx, e, "digit-split products: buffers");
    g->zero_bytes = (size_t)(DG_WORDS + nz) * 4;
    g->d1.expo[1] = g->words + DG_WORDS;
    g->d2.expo[0] = g->d1.expo[1] + g->p1.rows[1];
    dg_state(g->p1, g->d2.expo[0] + g->p2.rows[0], g->d1);
    dg_state(g->p2, g->d1.tickets + ns1, g->d2);
    g->d1.partial = g->d2.partial = partial;   // step 2 starts after step 1 has read its sums
    g->d1.redo = g->d2.redo = redo;            // (and its list)
    g->d1.expo[0] = env_expo;
    g->d2.expo[1] = env_expo + g->p1.rows[0];
    std::vector<uint8_t> host(std::max(b1, b2) + 16);
    dg_tables(g->p1, host.data(), tab, g->d1);   // pageable copies: consumed on return
    MRD_CUDA(ctx, cudaMemcpyAsync(tab, host.data(), b1, cudaMemcpyHostToDevice, s));
    dg_tables(g->p2, host.data(), tab + d1, g->d2);
    MRD_CUDA(ctx, cudaMemcpyAsync(tab + d1, host.data(), b2, cudaMemcpyHostToDevice, s));
    MRD_CUDA(ctx, dg_expand(g->d1, s));
    MRD_CUDA(ctx, dg_expand(g->d2, s));
    MRD_CUDA(ctx, cudaMemsetAsync(g->words, 0, g->zero_bytes, s));
    MRD_CUDA(ctx, dg_init());
    g->built = true;
    g->env_dirty = true;
    ++h->gen;
  }
  if (g->env_dirty || (h->env_captured && !h->in_lanczos)) {
    MRD_CUDA(ctx, cudaMemsetAsync(g->d1.expo[0], 0, (size_t)(g->p1.rows[0] + g->p2.rows[1]) * 4, s));
    MRD_CUDA(ctx, dg_pack(g->d1, 0, h->lw, beta, g->words, s));
    MRD_CUDA(ctx, dg_pack(g->d2, 1, h->wr, beta, g->words, s));
    g->env_dirty = cap;   // (packed by the replays, not now)
  }
  h->dg_form = 1;
  *use = true;
  return MRD_OK;
}

// Panels of all forms back to the cache (but not those that a caller's graph reads); the next application
// that needs them builds them again. Whether there were any.
bool dg_release(mrd_heff* h) {
  bool any = false;
  if (h->dg)
    for (auto& f : h->dg->forms) {
      if (!f->built || f->captured) continue;
      f->mem.release();
      f->built = false;
      any = true;
    }
  if (any) ++h->gen;   // captured Lanczos steps read them
  return any;
}

void dg_env_changed(mrd_heff* h) {
  if (h->dg)
    for (auto& f : h->dg->forms) {
      f->env_dirty = true;
      f->no_room = false;
    }
}

// theta_out = H_eff theta_in; ev: timing events (or null) before step 1, between the steps and
// after step 2. `out` has been cleared.
int dg_apply(mrd_heff* h, const double2* in, double2* out, const cudaEvent_t ev[3], bool cap) {
  mrd_ctx* ctx = h->ctx;
  cudaStream_t s = ctx->stream;
  DgForm* g = h->dg->cur;
  const int beta = g->beta;
  if (!h->in_lanczos && stream_capturing(s)) g->captured = true;
  // the error flag outlives a product; the exponents and the products' states do not
  MRD_CUDA(ctx, cudaMemsetAsync(g->words + DG_WORDS, 0, g->zero_bytes - DG_WORDS * 4, s));
  MRD_CUDA(ctx, dg_pack(g->d1, 1, in, beta, g->words, s));
  MRD_CUDA(ctx, record_event(ev[0], s, cap));
  auto product = [&](const DgPlan& p, const DgDev& d, double2* C) -> int {
    if (!h->per_task) {
      MRD_CUDA(ctx, dg_gemm(d, C, beta, g->words, h->n_sm, h->wait_ns, s));
      return MRD_OK;
    }
    for (size_t q = 0; q + 1 < p.item0.size(); ++q) {   // one launch per stacked block
      MRD_CUDA(ctx, cudaMemsetAsync(g->words + DG_CTR, 0, 4, s));
      MRD_CUDA(ctx, dg_gemm(d, C, beta, g->words, h->n_sm, h->wait_ns, s, (int)p.item0[q],
                            (int)(p.item0[q + 1] - p.item0[q])));
    }
    return MRD_OK;
  };
  int rc = product(g->p1, g->d1, h->z);
  if (rc != MRD_OK) return rc;
  MRD_CUDA(ctx, dg_redo(g->d1, h->lw, in, h->z, beta, g->words, h->n_sm, s));
  MRD_CUDA(ctx, record_event(ev[1], s, cap));
  MRD_CUDA(ctx, dg_pack(g->d2, 0, h->z, beta, g->words, s));
  if ((rc = product(g->p2, g->d2, out)) != MRD_OK) return rc;
  MRD_CUDA(ctx, dg_redo(g->d2, h->z, h->wr, out, beta, g->words, h->n_sm, s));
  MRD_CUDA(ctx, record_event(ev[2], s, cap));
  return MRD_OK;
}

// A wait of the digit-split products that gave up since the last check (MRD_E_TIMEOUT, then cleared).
int dg_status(mrd_heff* h) {
  if (!h->dg) return MRD_OK;
  int rc = MRD_OK;
  for (auto& f : h->dg->forms) {
    if (!f->built) continue;
    int herr = 0;
    MRD_CUDA(h->ctx, cudaMemcpyAsync(&herr, f->words + DG_ERR, 4, cudaMemcpyDeviceToHost, h->ctx->stream));
    MRD_CUDA(h->ctx, cudaStreamSynchronize(h->ctx->stream));
    if (!herr) continue;
    MRD_CUDA(h->ctx, cudaMemsetAsync(f->words + DG_ERR, 0, 4, h->ctx->stream));
    MRD_CUDA(h->ctx, cudaStreamSynchronize(h->ctx->stream));
    rc = mrd_fail(h->ctx, MRD_E_TIMEOUT, "digit-split GEMM: a bounded wait gave up (code " + std::to_string(herr) + ")");
  }
  return rc;
}
