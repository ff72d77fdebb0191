// Work list of the tensor-core FP64 grouped GEMM (f64_plan.h).
#include "f64_plan.h"

#include "core.h"

#include <algorithm>
#include <cmath>
#include <stdexcept>

namespace dmrg {

namespace {

inline uint64_t mix64(uint64_t h, uint64_t x) {
  h = (h ^ x) * 0x9E3779B97F4A7C15ull;
  return h ^ (h >> 29);
}

// ids of equal operand lists: open addressing over list hashes, lists compared in
// full against the first problem that has them
template <class Equal>
class ListIds {
 public:
  ListIds(size_t n, Equal eq) : eq_(eq) {
    size_t c = 16;
    while (c < 2 * n) c *= 2;
    slot_.assign(c, -1);
  }
  // the id of problem i's list (a new one when no earlier problem has it)
  int id(uint64_t h, int i) {
    const size_t m = slot_.size() - 1;
    for (size_t k = size_t(h) & m;; k = (k + 1) & m) {
      if (slot_[k] < 0) {
        slot_[k] = int(first_.size());
        first_.push_back(i);
        hash_.push_back(h);
        return slot_[k];
      }
      if (hash_[size_t(slot_[k])] == h && eq_(first_[size_t(slot_[k])], i)) return slot_[k];
    }
  }
  size_t size() const { return first_.size(); }

 private:
  Equal eq_;
  std::vector<int> slot_, first_;
  std::vector<uint64_t> hash_;
};

inline int up16(int x) { return (x + 15) & ~15; }

// n cut into equal tiles of at most `most`, a tile a multiple of `unit`
inline int tile_of(int64_t n, int most, int unit) {
  if (n <= most) return int(std::min<int64_t>(most, (n + unit - 1) / unit * unit));
  const int64_t t = (n + most - 1) / most;
  const int64_t w = (n + t - 1) / t;
  return int(std::min<int64_t>(most, (w + unit - 1) / unit * unit));
}

// long sums first, the longest at the front; prefix sums of the tiles' pieces
void order_tiles(F64PlanHost& out) {
  const auto mid = std::stable_partition(out.tiles.begin(), out.tiles.end(),
                                         [](const F64Unit& u) { return u.noct >= F64_LONG; });
  std::stable_sort(out.tiles.begin(), mid, [](const F64Unit& a, const F64Unit& b) { return a.noct > b.noct; });
  out.pieces.resize(out.tiles.size() + 1);
  out.pieces[0] = 0;
  for (size_t i = 0; i < out.tiles.size(); ++i)
    out.pieces[i + 1] = out.pieces[i] + (out.tiles[i].rows + F64_PR - 1) / F64_PR *
                                            ((out.tiles[i].nt + F64_PC - 1) / F64_PC);
}

}  // namespace

bool f64_small(const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s) {
  double mac = 0;
  for (const GemmProb& q : p) {
    int64_t len = 0, oct = 0;
    for (int k = q.s0; k < q.s1; ++k) {
      len += s[size_t(k)].K;
      oct += (s[size_t(k)].K + 7) / 8;
    }
    if (len > F64_SMALL_K) return false;
    mac += 8.0 * double(oct) * ((q.M + F64_PR - 1) / F64_PR * F64_PR) * ((q.N + F64_PC - 1) / F64_PC * F64_PC);
    if (mac > F64_SMALL_MAC) return false;
  }
  return true;
}

bool f64_run_plain(int forms, bool small, bool plain) {
  if (!(forms & (plain ? GEMM_PLAIN : GEMM_ANY))) throw std::logic_error("gemm_run: the plan was built without this form");
  return plain || small;
}

namespace {

// the plain form alone: every problem by itself, rows of A as rows; one pass
void build_plain(F64PlanHost& out, const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s) {
  out.rowref.resize(s.size());
  out.colref.resize(s.size());
  out.rows.resize(p.size());
  out.tiles.resize(p.size());
  out.pieces.resize(p.size() + 1);
  F64Ref *ra = out.rowref.data(), *rb = out.colref.data();
  F64Row* row = out.rows.data();
  F64Unit* tile = out.tiles.data();
  int* piece = out.pieces.data();
  int ns = 0, nt = 0, np = 0;
  bool any_long = false;
  for (const GemmProb& q : p) {
    if (q.M <= 0 || q.N <= 0) continue;
    const int cs = ns;
    int noct = 0;
    for (const GemmSeg *g = s.data() + q.s0, *e = s.data() + q.s1; g < e; ++g) {
      if (g->K <= 0) continue;
      ra[ns] = F64Ref{g->A, g->lda, 2 * g->K + (g->ta ? 1 : 0)};
      rb[ns] = F64Ref{g->B, g->ldb, 2 * g->K + (g->tb ? 0 : 1)};
      ++ns;
      noct += int(unsigned(g->K + 7) >> 3);
    }
    any_long = any_long || noct >= F64_LONG;
    row[nt] = F64Row{q.C, q.alpha, q.ldc, cs, 0, 2 * q.M + (q.accumulate ? 1 : 0)};
    tile[nt] = F64Unit{nt, 1, 0, q.M, 0, q.N, cs, ns - cs, 0, 0, noct, 0, -1};
    piece[nt] = np;
    np += int((unsigned(q.M) + F64_PR - 1) / F64_PR * ((unsigned(q.N) + F64_PC - 1) / F64_PC));
    ++nt;
  }
  piece[nt] = np;
  out.rowref.resize(size_t(ns));
  out.colref.resize(size_t(ns));
  out.rows.resize(size_t(nt));
  out.tiles.resize(size_t(nt));
  out.pieces.resize(nt ? size_t(nt) + 1 : 0);
  if (any_long) order_tiles(out);
}

}  // namespace

F64PlanHost f64_build_plan(const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s, int nsm, int what) {
  F64PlanHost out;
  f64_build_plan(out, p, s, nsm, what);
  return out;
}

void f64_build_plan(F64PlanHost& out, const std::vector<GemmProb>& p, const std::vector<GemmSeg>& s, int nsm, int what) {
  out.clear();
  if (!(what & F64_UNITS)) {
    build_plain(out, p, s);
    return;
  }
  const bool want_tiles = what & F64_TILES;
  const int np = int(p.size());
  // segments with K > 0, per problem (the caller's list itself when it holds nothing else)
  std::vector<int> f0(size_t(np) + 1, 0);
  std::vector<int> use;   // problems with an output
  use.reserve(size_t(np));
  bool whole = true;
  int at = 0;
  for (int i = 0; i < np && whole; ++i) {
    const GemmProb& q = p[size_t(i)];
    whole = q.M > 0 && q.N > 0 && q.s0 == at;
    for (int k = q.s0; k < q.s1; ++k) whole = whole && s[size_t(k)].K > 0;
    f0[size_t(i)] = at;
    at = q.s1;
  }
  std::vector<GemmSeg> kept;
  if (whole && at == int(s.size())) {
    f0[size_t(np)] = at;
    for (int i = 0; i < np; ++i) use.push_back(i);
  } else {
    kept.reserve(s.size());
    for (int i = 0; i < np; ++i) {
      f0[size_t(i)] = int(kept.size());
      if (p[size_t(i)].M > 0 && p[size_t(i)].N > 0) {
        use.push_back(i);
        for (int k = p[size_t(i)].s0; k < p[size_t(i)].s1; ++k)
          if (s[size_t(k)].K > 0) kept.push_back(s[size_t(k)]);
      }
    }
    f0[size_t(np)] = int(kept.size());
    whole = false;
  }
  const std::vector<GemmSeg>& seg = whole ? s : kept;
  if (use.empty()) return;

  // 1. lists shared on the B side (rows stacked) and on the A side (columns stacked)
  auto same_b = [&](int i, int j) {
    if (p[size_t(i)].N != p[size_t(j)].N || f0[size_t(i) + 1] - f0[size_t(i)] != f0[size_t(j) + 1] - f0[size_t(j)])
      return false;
    for (int a = f0[size_t(i)], b = f0[size_t(j)]; a < f0[size_t(i) + 1]; ++a, ++b) {
      const GemmSeg &x = seg[size_t(a)], &y = seg[size_t(b)];
      if (x.B != y.B || x.ldb != y.ldb || x.K != y.K || x.tb != y.tb) return false;
    }
    return true;
  };
  auto same_a = [&](int i, int j) {
    if (p[size_t(i)].M != p[size_t(j)].M || f0[size_t(i) + 1] - f0[size_t(i)] != f0[size_t(j) + 1] - f0[size_t(j)])
      return false;
    for (int a = f0[size_t(i)], b = f0[size_t(j)]; a < f0[size_t(i) + 1]; ++a, ++b) {
      const GemmSeg &x = seg[size_t(a)], &y = seg[size_t(b)];
      if (x.A != y.A || x.lda != y.lda || x.K != y.K || x.ta != y.ta) return false;
    }
    return true;
  };
  std::vector<int> kb(static_cast<size_t>(np), 0), ka(static_cast<size_t>(np), 0);
  std::vector<int64_t> sumM, sumN;
  std::vector<uint64_t> hashb(static_cast<size_t>(np)), hasha(static_cast<size_t>(np));
  const int nblk = int(use.size() / 4096) + 1;
  auto hash = [&](int i) {
    const GemmProb& q = p[size_t(i)];
    uint64_t hb = mix64(0x51ull, uint64_t(uint32_t(q.N))), ha = mix64(0xA7ull, uint64_t(uint32_t(q.M)));
    for (int k = f0[size_t(i)]; k < f0[size_t(i) + 1]; ++k) {
      const GemmSeg& g = seg[size_t(k)];
      hb = mix64(hb, uint64_t(reinterpret_cast<uintptr_t>(g.B)));
      hb = mix64(hb, (uint64_t(uint32_t(g.ldb)) << 32) | uint32_t(g.K * 2 + g.tb));
      ha = mix64(ha, uint64_t(reinterpret_cast<uintptr_t>(g.A)));
      ha = mix64(ha, (uint64_t(uint32_t(g.lda)) << 32) | uint32_t(g.K * 2 + g.ta));
    }
    hashb[size_t(i)] = hb;
    hasha[size_t(i)] = ha;
  };
  {
    const size_t work = use.size() + seg.size();
    if (work > 50000)
      host_parallel_for(nblk, [&](int b) {
        for (size_t k = use.size() * size_t(b) / size_t(nblk); k < use.size() * size_t(b + 1) / size_t(nblk); ++k)
          hash(use[k]);
      });
    else
      for (int i : use) hash(i);
    auto ids = [&](bool bside) {
      if (bside) {
        ListIds<decltype(same_b)> idb(use.size(), same_b);
        for (int i : use) {
          const int k = kb[size_t(i)] = idb.id(hashb[size_t(i)], i);
          if (size_t(k) == sumM.size()) sumM.push_back(0);
          sumM[size_t(k)] += p[size_t(i)].M;
        }
      } else {
        ListIds<decltype(same_a)> ida(use.size(), same_a);
        for (int i : use) {
          const int k = ka[size_t(i)] = ida.id(hasha[size_t(i)], i);
          if (size_t(k) == sumN.size()) sumN.push_back(0);
          sumN[size_t(k)] += p[size_t(i)].N;
        }
      }
    };
    if (work > 50000) host_parallel_for(2, [&](int b) { ids(b == 0); });
    else { ids(true); ids(false); }
  }
  // 2. orientation: the problem's share of its stack's 128-row tiles times the columns
  // (in the tensor core's steps of 16); equal shares keep the rows of A
  auto share = [](int rows, int64_t stack, int cols) {
    const double lanes = double((stack + F64_TM - 1) / F64_TM * F64_TM) / double(stack);
    return lanes * rows * double((cols + F64_TN - 1) / F64_TN) * tile_of(cols, F64_TN, 16);
  };
  const int nb = int(sumM.size());
  std::vector<int> grp(static_cast<size_t>(np), -1);
  std::vector<int> gcount(size_t(nb) + sumN.size(), 0);
  for (int i : use) {
    const GemmProb& q = p[size_t(i)];
    const bool tr = share(q.N, sumN[size_t(ka[size_t(i)])], q.M) < share(q.M, sumM[size_t(kb[size_t(i)])], q.N);
    grp[size_t(i)] = tr ? nb + ka[size_t(i)] : kb[size_t(i)];
    ++gcount[size_t(grp[size_t(i)])];
  }
  // 3. groups in the order of their first problem, members in problem order
  std::vector<int> gpos(gcount.size(), -1);
  std::vector<int> gorder;
  int npos = 0;
  for (int i : use) {
    const size_t g = size_t(grp[size_t(i)]);
    if (gpos[g] >= 0) continue;
    gpos[g] = npos;
    npos += gcount[g];
    gorder.push_back(int(g));
  }
  std::vector<int> member(static_cast<size_t>(npos));
  {
    std::vector<int> at = gpos;
    for (int i : use) member[size_t(at[size_t(grp[size_t(i)])]++)] = i;
  }
  out.rowref.resize(seg.size());
  out.colref.resize(seg.size());
  out.rows.resize(size_t(npos));
  for (int i : use) {
    const bool tr = grp[size_t(i)] >= nb;
    for (int k = f0[size_t(i)]; k < f0[size_t(i) + 1]; ++k) {
      const GemmSeg& g = seg[size_t(k)];
      const F64Ref a{g.A, g.lda, 2 * g.K + (g.ta ? 1 : 0)};
      const F64Ref b{g.B, g.ldb, 2 * g.K + (g.tb ? 0 : 1)};
      out.rowref[size_t(k)] = tr ? b : a;
      out.colref[size_t(k)] = tr ? a : b;
    }
  }
  // 4. tiles and their split over K.  Costs in SM clocks, roughly: a stage of 16 k
  // converts its rows and columns (a warp's 8 x 16 piece about 110 instructions, four
  // schedulers) while the tensor core runs its 36 products; a chunk adds its pass for
  // the exponents and its drain, a unit its fixed latencies
  struct Tile { int g, pos0, npos, row0, rows, n0, nt; };
  auto part_cost = [](int rows, int nt, int64_t oct) {
    const double stage = std::max(28.0 * ((rows + 7) / 8 + (nt + 7) / 8), 18.0 * up16(nt));
    return 0.5 * double(oct) * stage * 1.6 + double((oct + F64_CHUNK - 1) / F64_CHUNK) * 2500.0 + 3000.0;
  };
  std::vector<Tile> tiles;
  std::vector<int64_t> goct(gorder.size(), 0);
  double total = 0;
  for (size_t gi = 0; gi < gorder.size(); ++gi) {
    const size_t g = size_t(gorder[gi]);
    const int m0 = gpos[g], m1 = m0 + gcount[g];
    const bool tr = int(g) >= nb;
    int64_t R = 0;
    for (int m = m0; m < m1; ++m) {
      const GemmProb& q = p[size_t(member[size_t(m)])];
      F64Row& r = out.rows[size_t(m)];
      r.C = q.C;
      r.alpha = q.alpha;
      r.ldc = q.ldc;
      r.s0 = f0[size_t(member[size_t(m)])];
      r.pre = int(R);
      const int rows = tr ? q.N : q.M;
      r.m2 = 2 * rows + (q.accumulate ? 1 : 0);
      R += rows;
    }
    const int i0 = member[size_t(m0)];
    const int cols = tr ? p[size_t(i0)].M : p[size_t(i0)].N;
    int64_t oct = 0;
    for (int k = f0[size_t(i0)]; k < f0[size_t(i0) + 1]; ++k) oct += (seg[size_t(k)].K + 7) / 8;
    goct[gi] = oct;
    const int tm = tile_of(R, F64_TM, 8), tn = tile_of(cols, F64_TN, 16);
    int pos = m0;
    for (int64_t r0 = 0; r0 < R; r0 += tm) {
      const int rows = int(std::min<int64_t>(tm, R - r0));
      while (out.rows[size_t(pos)].pre + (out.rows[size_t(pos)].m2 >> 1) <= r0) ++pos;
      int last = pos;
      while (last + 1 < m1 && out.rows[size_t(last) + 1].pre < r0 + rows) ++last;
      for (int n0 = 0; n0 < cols; n0 += tn) {
        const int nt = std::min(tn, cols - n0);
        tiles.push_back(Tile{int(gi), pos, last - pos + 1, int(r0), rows, n0, nt});
        total += part_cost(rows, nt, oct);
      }
    }
  }
  const double target = total / (4.0 * std::max(1, nsm));
  std::vector<F64Unit> units;
  std::vector<int> keys;
  units.reserve(tiles.size());
  keys.reserve(tiles.size());
  if (want_tiles) out.tiles.reserve(tiles.size());
  for (const Tile& t : tiles) {
    const size_t g = size_t(gorder[size_t(t.g)]);
    const int m0 = gpos[g], i0 = member[size_t(m0)];
    const int cs = f0[size_t(i0)], nseg = f0[size_t(i0) + 1] - cs;
    const int64_t oct = goct[size_t(t.g)], nch = (oct + F64_CHUNK - 1) / F64_CHUNK;
    const double cc = part_cost(t.rows, t.nt, F64_CHUNK) - 3000.0;
    const int64_t per = std::max<int64_t>(1, std::min<int64_t>(nch, int64_t(std::max(1.0, (target - 3000.0) / cc))));
    const int64_t parts = nch ? (nch + per - 1) / per : 1;
    F64Unit u{};
    u.pos0 = t.pos0;
    u.npos = t.npos;
    u.row0 = t.row0;
    u.rows = t.rows;
    u.n0 = t.n0;
    u.nt = t.nt;
    u.cs = cs;
    u.nseg = nseg;
    u.trans = int(g) >= nb ? 1 : 0;
    u.part = -1;
    const int n16 = up16(t.nt);
    if (parts > 1) {
      out.reds.push_back(F64Red{t.pos0, t.row0, t.rows, t.n0, t.nt, u.trans, int(parts), n16, out.npart});
    }
    int sg = 0, k0 = 0;
    u.noct = int(oct);
    if (want_tiles) out.tiles.push_back(u);
    for (int64_t q = 0; q < parts; ++q) {
      // whole chunks, spread evenly
      const int64_t c0 = nch * q / parts, c1 = nch * (q + 1) / parts;
      u.sg = sg;
      u.k0 = k0;
      u.noct = int(std::min<int64_t>(c1 * F64_CHUNK, oct) - c0 * F64_CHUNK);
      if (parts > 1) {
        u.part = out.npart;
        out.npart += int64_t(F64_TM) * n16;
      }
      const double cost = part_cost(t.rows, t.nt, u.noct);
      units.push_back(u);
      keys.push_back(int(std::log2(cost) * 3.0));
      if (q + 1 < parts) {
        int left = u.noct;
        while (left > 0) {   // the octet after the unit's last one
          const int K = seg[size_t(cs + sg)].K, no = (K - k0 + 7) / 8;
          if (no > left) {
            k0 += 8 * left;
            left = 0;
          } else {
            left -= no;
            ++sg;
            k0 = 0;
          }
        }
      }
    }
  }
  // longest first; units of about the same cost keep their order, so that tiles that
  // read the same operands run at the same time (a counting sort: few distinct keys)
  {
    const int top = *std::max_element(keys.begin(), keys.end());
    std::vector<size_t> at(size_t(top) + 2, 0);
    for (int k : keys) ++at[size_t(top - k) + 1];
    for (size_t k = 1; k < at.size(); ++k) at[k] += at[k - 1];
    out.units.resize(units.size());
    for (size_t i = 0; i < units.size(); ++i) out.units[at[size_t(top - keys[i])]++] = units[i];
  }
  if (want_tiles) order_tiles(out);
}

}  // namespace dmrg
