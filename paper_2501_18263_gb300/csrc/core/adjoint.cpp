// Adjoint of the operator construction: the derivatives of
//     F = <lam| H_eff(t, v) |psi>
// with respect to the integrals t and v for a fixed MPS basis.  For lam = psi the
// normalised ground state, dF/dt_ij is the one-particle density matrix and dF/dv_ijkl
// half the two-particle one (the differentiation form; Sec. 2.2 needs these densities
// for the orbital rotations c~+ = U c+ of mode optimisation).
//
// F depends on the integrals only through the coefficients of the blocking steps
// (site matrices and integral-weighted sums of block operators, Sec. 2.3) and is
// linear in them.  Reverse mode:
//   1. at the bond, the adjoint of every fine block of every L' and R' operator from
//      the sigma terms (sigma_adjoint, sigma.cpp): for a term c op(O_L) (x) op(O_R)
//      and a psi block,  dF/dO_L = c s lam O_R psi^T  and  dF/dO_R = c s lam^T O_L psi
//      (s the Jordan-Wigner sign of the block);
//   2. down the left chain (B_b (x) site b, B_{b-1} (x) site b-1, ..., B_0 (x) site 0)
//      and up the right chain (site b+1 (x) C_{b+2}, ..., site L-1 (x) C_L): for each
//      blocking contribution E{rf, cf} += coef * op(src),
//        adj(src) += coef * op^T(adj E{rf, cf})      (a Kronecker accumulation)
//        dF/dcoef  = <adj E{rf, cf}, op(src)>        (a Frobenius product)
//      and dF/dcoef is spread over the integrals of coef (a linear form); then through
//      the renormalisation B' = U^T E U that made the block:
//        adj E{fr, fc} = U{fr rows} adj B'{r, c} U{fc rows}^T.
// The forward operators are the ones the engine already holds for the bond; the
// adjoint keeps one block's and one enlarged block's adjoints at a time, and cuts the
// sigma-term intermediates into chunks under mem_cap.
#include <algorithm>
#include <map>
#include <stdexcept>

#include "core.h"

namespace dmrg {

namespace {

using TargetMap = std::map<OpKey, std::map<std::pair<int, int>, int64_t>>;

TargetMap target_map(const AdjStep& s) {
  TargetMap m;
  for (const AdjTarget& t : s.tgt) m[s.keys[size_t(t.key)]][{t.rf, t.cf}] = t.off;
  return m;
}

// blocks of an operator set (ids 0 .. count - 1 in (operator, block) order)
int block_count(const OpSet& s) {
  int n = 0;
  for (auto& kv : s.ops) n += int(kv.second.blk.size());
  return n;
}

}  // namespace

void Engine::set_integrals(const std::vector<double>& t, const std::vector<double>& v) {
  const size_t L2 = size_t(P_.L) * P_.L;
  if (t.size() != L2 || v.size() != L2 * L2) throw std::runtime_error("set_integrals: wrong sizes");
  free_bond();
  P_.t = t;
  P_.v = v;
  for (int n = 1; n <= P_.L; ++n) {
    free_opset(lb_[n].ops);
    lb_[n].valid = false;
  }
  for (int m = 0; m < P_.L; ++m) {
    free_opset(rb_[m].ops);
    rb_[m].valid = false;
  }
}

void Engine::integral_gradient(const double* lam, const double* psi, std::vector<double>& raw) {
  if (bond_ < 0) throw std::runtime_error("integral_gradient: no bond prepared");
  const int L = P_.L, b = bond_;
  const int64_t L2 = int64_t(L) * L;
  raw.assign(size_t(L2 + L2 * L2), 0.0);
  if (!lb_[b].valid || !rb_[b + 2].valid) throw std::runtime_error("integral_gradient: blocks not built");

  // blocking step backwards: adjoint of the block operators (arena of blk.ops's
  // layout, allocated here) and the coefficient derivatives: Frobenius products of the
  // adjoints with the operators they multiply, spread over the integrals of each
  // coefficient (host, in a fixed order)
  auto back_blocking = [&](const AdjStep& st, const Block& blk, const double* adjE) -> double* {
    const int64_t nb = std::max<int64_t>(blk.ops.n_elem, 1);
    double* ob = static_cast<double*>(ex_->alloc(size_t(nb) * sizeof(double)));
    ex_->zero(ob, size_t(nb) * sizeof(double));
    // contributions dealt out to the source blocks (counting sort by block id, so that
    // each block sums its own in list order), and the products with a coefficient
    const int nblk = block_count(blk.ops);
    std::vector<const OpBlk*> blks(static_cast<size_t>(nblk));
    for (auto& kv : blk.ops.ops)
      for (auto& b : kv.second.blk) blks[size_t(b.id)] = &b;
    std::vector<int> first(size_t(nblk) + 1, 0);
    size_t nd = 0;
    for (const AdjTerm& x : st.terms) {
      if (x.src && x.val != 0.0) ++first[size_t(x.src->blk[size_t(x.src_blk)].id) + 1];
      nd += x.w1 > x.w0;
    }
    for (int i = 0; i < nblk; ++i) first[size_t(i) + 1] += first[size_t(i)];
    std::vector<KronTask> kt(static_cast<size_t>(first[size_t(nblk)]));
    std::vector<DotTask> dt;
    std::vector<const AdjTerm*> dl;
    dt.reserve(nd);
    dl.reserve(nd);
    {
      std::vector<int> at(first.begin(), first.end() - 1);
      for (const AdjTarget& tg : st.tgt) {
        const int rows = st.E.f_dim[tg.rf], cols = st.E.f_dim[tg.cf];
        const double* g = adjE + tg.off;
        for (int k = tg.t0; k < tg.t1; ++k) {
          const AdjTerm& x = st.terms[size_t(k)];
          const OpBlk* sb = x.src ? &x.src->blk[size_t(x.src_blk)] : nullptr;
          if (sb && x.val != 0.0) kt[size_t(at[size_t(sb->id)]++)] = KronTask{g, cols, x.trans, x.val};
          if (x.w1 > x.w0) {
            dt.push_back(sb ? DotTask{g, blk.ops.arena + sb->off, cols, sb->cols, rows, cols, x.trans}
                            : DotTask{g, nullptr, cols, 0, rows, cols, 2});
            dl.push_back(&x);
          }
        }
      }
    }
    std::vector<KronGroup> kg;
    for (int i = 0; i < nblk; ++i) {
      if (first[size_t(i)] == first[size_t(i) + 1]) continue;
      const OpBlk& sb = *blks[size_t(i)];
      kg.push_back(KronGroup{ob + sb.off, sb.cols, sb.rows, sb.cols, first[size_t(i)], first[size_t(i) + 1], 0});
    }
    if (!kg.empty()) ex_->kron(kg, kt);
    if (!dt.empty()) {
      double* d = static_cast<double*>(ex_->alloc(dt.size() * sizeof(double)));
      ex_->dots(dt, d);
      std::vector<double> h(dt.size());
      ex_->d2h(h.data(), d, h.size() * sizeof(double));
      ex_->release(d);
      for (size_t i = 0; i < h.size(); ++i)
        for (int k = dl[i]->w0; k < dl[i]->w1; ++k) raw[size_t(st.w[size_t(k)].first)] += st.w[size_t(k)].second * h[i];
    }
    return ob;
  };

  // renormalisation backwards: adjoint of the enlarged block of step `nx` (whose
  // isometry `iso` made block `B`) from the adjoint `ob` of B's operators
  auto back_renorm = [&](const AdjStep& nx, const Iso& iso, const Block& B, const double* ob) -> double* {
    const int64_t ne = std::max<int64_t>(nx.n, 1);
    double* ge = static_cast<double*>(ex_->alloc(size_t(ne) * sizeof(double)));
    ex_->zero(ge, size_t(ne) * sizeof(double));
    const Enlarged& E = nx.E;
    std::vector<int> c2s(E.coarse.q.size(), -1);
    for (size_t k = 0; k < iso.out.q.size(); ++k) {
      const int c = E.coarse.find(iso.out.q[k]);
      if (c < 0 || E.coarse.dim[c] != iso.rows[k]) throw std::runtime_error("adjoint: isometry and enlarged basis differ");
      c2s[c] = int(k);
    }
    // W(op, block) = adj B'{r <- c} U_c^T (dr x rows_c), then adj E{fr, fc} = U_r{fr rows} W{fc cols}:
    // the targets of every block operator's block, by block id
    std::vector<const Op*> kop(nx.keys.size(), nullptr);
    for (size_t k = 0; k < nx.keys.size(); ++k) {
      auto it = B.ops.ops.find(nx.keys[k]);
      if (it != B.ops.ops.end()) kop[k] = &it->second;
    }
    const int nblk = block_count(B.ops);
    std::vector<const OpBlk*> blks(size_t(nblk), nullptr);
    for (auto& kv : B.ops.ops)
      for (auto& b : kv.second.blk) blks[size_t(b.id)] = &b;
    // block of the operator at column sector c (one per column), -1 where it has none
    std::vector<int> tblk(nx.tgt.size(), -1), first(size_t(nblk) + 1, 0);
    {
      int key = -1;
      std::vector<int> bycol;
      for (size_t i = 0; i < nx.tgt.size(); ++i) {
        const AdjTarget& t = nx.tgt[i];
        const Op* bo = kop[size_t(t.key)];
        if (!bo) continue;
        if (t.key != key) {
          key = t.key;
          bycol.assign(iso.out.q.size(), -1);
          for (auto& b : bo->blk) bycol[size_t(b.c)] = b.id;
        }
        const int r = c2s[E.f_coarse[t.rf]], c = c2s[E.f_coarse[t.cf]];
        if (r < 0 || c < 0 || bycol[size_t(c)] < 0 || blks[size_t(bycol[size_t(c)])]->r != r) continue;
        tblk[i] = bycol[size_t(c)];
        ++first[size_t(tblk[i]) + 1];
      }
    }
    for (int i = 0; i < nblk; ++i) first[size_t(i) + 1] += first[size_t(i)];
    std::vector<int> order(static_cast<size_t>(first[size_t(nblk)]));
    {
      std::vector<int> at(first.begin(), first.end() - 1);
      for (size_t i = 0; i < nx.tgt.size(); ++i)
        if (tblk[i] >= 0) order[size_t(at[size_t(tblk[i])]++)] = int(i);
    }
    const int64_t cap = int64_t(1) << 27;
    double* W = nullptr;
    int64_t wcap = 0;
    std::vector<GemmProb> p1, p2;
    std::vector<GemmSeg> s1, s2;
    int64_t used = 0;
    auto flush = [&]() {
      if (!p1.empty()) ex_->gemm(p1, s1);
      if (!p2.empty()) ex_->gemm(p2, s2);
      p1.clear(); p2.clear(); s1.clear(); s2.clear();
      used = 0;
    };
    for (int bi = 0; bi < nblk; ++bi) {
      if (first[size_t(bi)] == first[size_t(bi) + 1]) continue;
      const OpBlk& bk = *blks[size_t(bi)];
      const int r = bk.r, c = bk.c;
      const int dr = iso.out.dim[r], dc = iso.out.dim[c], rows_c = iso.rows[c];
      const int64_t sz = int64_t(dr) * rows_c;
      if (used + sz > wcap) {
        flush();
        if (sz > wcap) {
          if (W) ex_->release(W);
          wcap = std::max(sz, std::min(cap, int64_t(1) << 22));
          W = static_cast<double*>(ex_->alloc(size_t(wcap) * sizeof(double)));
        }
      }
      double* w = W + used;
      used += sz;
      GemmProb q;
      q.C = w;
      q.ldc = rows_c;
      q.M = dr;
      q.N = rows_c;
      q.alpha = 1.0;
      q.accumulate = 0;
      q.s0 = int(s1.size());
      s1.push_back(GemmSeg{ob + bk.off, iso.mat[c], dc, dc, dc, 0, 1});
      q.s1 = int(s1.size());
      p1.push_back(q);
      for (int k = first[size_t(bi)]; k < first[size_t(bi) + 1]; ++k) {
        const AdjTarget& tg = nx.tgt[size_t(order[size_t(k)])];
        const int rf = tg.rf, cf = tg.cf;
        GemmProb q2;
        q2.C = ge + tg.off;
        q2.ldc = E.f_dim[cf];
        q2.M = E.f_dim[rf];
        q2.N = E.f_dim[cf];
        q2.alpha = 1.0;
        q2.accumulate = 0;
        q2.s0 = int(s2.size());
        s2.push_back(GemmSeg{iso.mat[r] + int64_t(E.f_row[rf]) * dr, w + E.f_row[cf], dr, rows_c, dr, 0, 0});
        q2.s1 = int(s2.size());
        p2.push_back(q2);
      }
    }
    flush();
    if (W) ex_->release(W);
    return ge;
  };

  // 1. the bond
  AdjStep SL = adjoint_step(true, lb_[b], b);
  AdjStep SR = adjoint_step(false, rb_[b + 2], b + 1);
  double* gl = static_cast<double*>(ex_->alloc(size_t(std::max<int64_t>(SL.n, 1)) * sizeof(double)));
  double* gr = static_cast<double*>(ex_->alloc(size_t(std::max<int64_t>(SR.n, 1)) * sizeof(double)));
  ex_->zero(gl, size_t(std::max<int64_t>(SL.n, 1)) * sizeof(double));
  ex_->zero(gr, size_t(std::max<int64_t>(SR.n, 1)) * sizeof(double));
  sigma_adjoint(lam, psi, target_map(SL), gl, target_map(SR), gr);

  // 2. left chain: step n enlarges B_n with site n; B_n came from step n-1
  {
    AdjStep cur = std::move(SL);
    double* adj = gl;
    for (int n = b; n >= 0; --n) {
      double* ob = back_blocking(cur, lb_[n], adj);
      ex_->release(adj);
      if (n == 0) {
        ex_->release(ob);
        break;
      }
      AdjStep nx = adjoint_step(true, lb_[n - 1], n - 1);
      adj = back_renorm(nx, liso_[n - 1], lb_[n], ob);
      ex_->release(ob);
      cur = std::move(nx);
    }
  }
  // right chain: step m enlarges C_{m+1} with site m; C_{m+1} came from step m+1
  {
    AdjStep cur = std::move(SR);
    double* adj = gr;
    for (int m = b + 1; m <= L - 1; ++m) {
      double* ob = back_blocking(cur, rb_[m + 1], adj);
      ex_->release(adj);
      if (m == L - 1) {
        ex_->release(ob);
        break;
      }
      AdjStep nx = adjoint_step(false, rb_[m + 2], m + 1);
      adj = back_renorm(nx, riso_[m + 1], rb_[m + 1], ob);
      ex_->release(ob);
      cur = std::move(nx);
    }
  }
  ex_->sync();
}

}  // namespace dmrg
