"""Performance cases of the two-site DMRG engine, through its public entry points.

Every case is one call (or the short sequence of calls) that a program using the
library makes: the sigma step at a prepared bond in both precisions, many problems
batched, the adjoint (density matrices), the truncation's eigensolver, a Davidson
solve with a bounded number of iterations, and a whole DMRG run.  Sizes are those of
the benchmark and the tests (L = 6 .. 32 orbitals, D = 16 .. 1024).  Inputs are the
package's seeded synthetic integrals and random isometric MPS bases.

`exact` restates the mathematics in numpy on the determinant basis (at most 12
orbitals, where it is small enough): the MPS basis states as explicit Fock-space
vectors, H on (alpha string) x (beta string) arrays.
"""
import math

import numpy as np
import torch

from paper_2501_18263_gb300 import binding, inputs

F64, BF16X = binding.PREC_FP64, binding.PREC_MIXED_BF16


def listed():
    return [
        # the smallest sigma of a real run: 8 orbitals at D = 64, where launches count
        {"name": "sigma_f64_L8_D64", "kind": "sigma", "prec": "f64", "L": 8, "na": 4, "nb": 4, "D": 64, "bond": 3},
        # FP64 sigma in the middle of a chain with unequal spins, left of the centre
        {"name": "sigma_f64_L20_D256", "kind": "sigma", "prec": "f64", "L": 20, "na": 11, "nb": 9, "D": 256, "bond": 7},
        # the FP64 arm of the benchmark's Davidson comparison (and the refinement sigma of the other)
        {"name": "sigma_f64_L32_D512", "kind": "sigma", "prec": "f64", "L": 32, "na": 16, "nb": 16, "D": 512, "bond": 15},
        # split-BF16 sigma of a small active space
        {"name": "sigma_bf16x_L12_D256", "kind": "sigma", "prec": "bf16x", "L": 12, "na": 6, "nb": 6, "D": 256, "bond": 5},
        # split-BF16 sigma, ordinary size, off the centre
        {"name": "sigma_bf16x_L24_D512", "kind": "sigma", "prec": "bf16x", "L": 24, "na": 13, "nb": 11, "D": 512, "bond": 9},
        # split-BF16 sigma at the metric's chain length
        {"name": "sigma_bf16x_L32_D1024", "kind": "sigma", "prec": "bf16x", "L": 32, "na": 16, "nb": 16, "D": 1024, "bond": 15},
        # many independent small problems in shared launches, replayed from a graph
        {"name": "batch_6_D256", "kind": "batch", "n": 6, "L_lo": 10, "L_hi": 13, "D": 256},
        # backward of the sigma step: one- and two-particle densities of a swept state
        {"name": "backward_L12_D128", "kind": "backward", "L": 12, "na": 6, "nb": 6, "D": 128, "bond": 5},
        {"name": "backward_L16_D256", "kind": "backward", "L": 16, "na": 8, "nb": 8, "D": 256, "bond": 7},
        # the truncation's eigensolver on the sector blocks of an enlarged block
        {"name": "eigh_L24_D1024", "kind": "eigh", "L": 24, "na": 12, "nb": 12, "D": 1024, "bond": 11},
        # one eigensolver step of a sweep, the iterations bounded as in early sweeps
        {"name": "davidson_f64_L16_D128", "kind": "davidson", "L": 16, "na": 8, "nb": 8, "D": 128, "bond": 7, "iters": 20},
        # a whole run: from the integrals to the energies of two sweeps with all states kept
        {"name": "dmrg_f64_L8_D256", "kind": "dmrg", "prec": "f64", "L": 8, "na": 4, "nb": 4, "D": 256, "sweeps": 2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sigma", "sigma", "sigma", "sigma", "batch", "backward", "eigh", "davidson", "dmrg"])
    if kind == "dmrg":
        L = rng.randint(5, 8)
        na = rng.randint(max(1, L // 2 - 1), L // 2 + 1)
        nb = rng.randint(max(1, L // 2 - 1), L // 2 + 1)
        return {"kind": kind, "prec": rng.choice(["f64", "bf16x"]), "L": L, "na": na, "nb": nb, "D": 4 ** (L // 2),
                "sweeps": rng.randint(1, 2)}
    if kind == "batch":
        lo = rng.randint(8, 12)
        return {"kind": kind, "n": rng.randint(2, 6), "L_lo": lo, "L_hi": lo + rng.randint(1, 2),
                "D": _log_int(rng, 48, 256)}
    L = rng.randint(6, 24)
    split = rng.randint(-1, 1)
    na, nb = L // 2 + split, L // 2 - split
    case = {"kind": kind, "L": L, "na": na, "nb": nb}
    if kind == "sigma":
        case["prec"] = rng.choice(["f64", "bf16x"])
        case["D"] = _log_int(rng, 16, 256 if case["prec"] == "f64" else 600)
    elif kind == "backward":
        case["L"], case["na"], case["nb"] = min(L, 14), min(L, 14) // 2, min(L, 14) // 2
        case["D"] = _log_int(rng, 16, 200)
    elif kind == "eigh":
        case["D"] = _log_int(rng, 64, 1024)
    else:
        case["D"] = _log_int(rng, 16, 128)
        case["iters"] = rng.randint(5, 25)
    L = case["L"]
    case["bond"] = rng.randint(max(0, L // 2 - 3), min(L - 2, L // 2 + 1))
    return case


# ---------------------------------------------------------------------------
# what a program has in hand before the call

def _prec(case):
    return BF16X if case.get("prec") == "bf16x" else F64


def _problem(case, seed):
    t, v = inputs.synthetic_integrals(case["L"], seed)
    bp = inputs.bond_problem(case["L"], case["na"], case["nb"], case["D"], case["bond"], seed + 1)
    return t, v, bp


def _handle(case, seed, prec, stream):
    t, v, bp = _problem(case, seed)
    d = binding.Dmrg(t, v, case["na"], case["nb"], D=case["D"], precision=prec, stream=stream.cuda_stream)
    d.load_bond_problem(bp)
    d.prepare(case["bond"])
    return d, bp


def _batch_cases(case):
    out = []
    for i in range(case["n"]):
        L = case["L_lo"] + i % (case["L_hi"] - case["L_lo"] + 1)
        na = (L + 1) // 2 + (1 if i % 3 == 2 else 0)
        out.append({"L": L, "na": na, "nb": L - na, "D": case["D"], "bond": L // 2 - 1})
    return out


def _eigh_orders(case):
    """Orders of the density matrix's sector blocks: L' sectors that psi occupies."""
    L, na, nb, D, b = (case[k] for k in ("L", "na", "nb", "D", "bond"))
    left = inputs.left_bond_sectors(L, na, nb, D, b)[b]
    right = inputs.right_bond_sectors(L, na, nb, D, b + 2)[b + 2]
    return [(r, c) for (_, _, r, c) in inputs.psi_block_shapes(left, right, na, nb)]


def _eigh_matrices(case, seed, device):
    """Density matrices A A^T of sector blocks with decaying column weights."""
    g = torch.Generator(device=device).manual_seed(seed)
    mats = []
    for r, c in _eigh_orders(case):
        m = max(c, r)
        A = torch.randn((r, m), dtype=torch.float64, device=device, generator=g)
        A *= torch.exp(-3.0 * torch.arange(m, dtype=torch.float64, device=device) / m)
        M = A @ A.T
        mats.append(0.5 * (M + M.T) / m)
    return mats


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    s = {"kind": kind, "case": case, "stream": torch.cuda.Stream()}
    if kind == "dmrg":
        s["t"], s["v"] = inputs.synthetic_integrals(case["L"], seed)
        s["seed"] = seed
    elif kind == "eigh":
        mats = _eigh_matrices(case, seed, dev)
        t, v = inputs.synthetic_integrals(2, seed)
        s["d"] = binding.Dmrg(t, v, 1, 1, D=4, stream=s["stream"].cuda_stream)
        s["n"] = [m.shape[0] for m in mats]
        s["A0"] = torch.cat([m.reshape(-1) for m in mats])
        s["A"], s["Z"] = torch.empty_like(s["A0"]), torch.empty_like(s["A0"])
        s["w"] = torch.empty(sum(s["n"]), dtype=torch.float64, device=dev)
    elif kind == "batch":
        s["d"], s["psi"], bonds = [], [], []
        for i, c in enumerate(_batch_cases(case)):
            d, bp = _handle(c, seed + 10 * i, BF16X, s["stream"])
            s["d"].append(d)
            s["psi"].append(torch.tensor(binding.pack_psi(bp.psi), dtype=torch.float64, device=dev))
            bonds.append(c["bond"])
        s["sigma"] = [torch.empty_like(p) for p in s["psi"]]
        s["batch"] = binding.Batch(s["d"], bonds)
    else:
        s["d"], bp = _handle(case, seed, _prec(case), s["stream"])
        s["psi"] = torch.tensor(binding.pack_psi(bp.psi), dtype=torch.float64, device=dev)
        s["x"] = torch.empty_like(s["psi"])
        if kind == "backward":
            L = case["L"]
            s["lam"] = torch.tensor(binding.pack_psi(inputs.random_psi_like(bp, seed + 2)), dtype=torch.float64,
                                    device=dev)
            s["g1"] = torch.empty((L, L), dtype=torch.float64, device=dev)
            s["g2"] = torch.empty((L, L, L, L), dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# one pass

def run(s):
    c, kind = s["case"], s["kind"]
    with torch.cuda.stream(s["stream"]):
        if kind == "sigma":
            s["d"].sigma(c["bond"], s["psi"].data_ptr(), s["x"].data_ptr())
            return s["x"]
        if kind == "batch":
            s["batch"].sigma([p.data_ptr() for p in s["psi"]], [x.data_ptr() for x in s["sigma"]], graph=True)
            return s["sigma"]
        if kind == "backward":
            s["g1"].zero_()
            s["g2"].zero_()
            s["d"].sigma_backward(c["bond"], s["psi"].data_ptr(), s["lam"].data_ptr(), s["g1"].data_ptr(),
                                  s["g2"].data_ptr())
            return {"g1": s["g1"], "g2": s["g2"]}
        if kind == "eigh":
            s["A"].copy_(s["A0"])
            s["d"].eigh_batch(s["n"], s["A"].data_ptr(), s["w"].data_ptr(), s["Z"].data_ptr())
            return {"w": s["w"], "Z": s["Z"]}
        if kind == "davidson":
            s["x"].copy_(s["psi"])
            e, _ = s["d"].davidson(c["bond"], s["x"].data_ptr(), tol=1e-11, max_iter=c["iters"], check=False)
            return {"energy": e, "psi": s["x"]}
        d = binding.Dmrg(s["t"], s["v"], c["na"], c["nb"], D=c["D"], seed=s["seed"], precision=_prec(c),
                         stream=s["stream"].cuda_stream)
        e = d.sweep(c["sweeps"], tol=1e-8, refine_all=True, max_iter=200)
        d.close()
        return {"energies": e}


# ---------------------------------------------------------------------------
# what a pass cannot do without

_Q = inputs.LOCAL_Q
# single-site operators by the charge they add: pairs (s' <- s) of local states
_SITE = {}
for _s, _q in enumerate(_Q):
    for _t, _p in enumerate(_Q):
        _SITE.setdefault((_p[0] - _q[0], _p[1] - _q[1]), []).append((_t, _s))


def _add(x, y, sign=1):
    return (x[0] + sign * y[0], x[1] + sign * y[1])


def _fines(layout, sec):
    """{coarse Q: {(s, sector): dim}} of an enlarged block."""
    return {Q: {(s, sec.q[k]): d for (s, k, d) in subs} for Q, subs in layout.items()}


def _term_counts(n_block, n_site):
    """Normal operators on block (x) site: {(block charge, site charge, spins): operators}, spins being the
    charges of the one or two elementary operators the term leaves to the other side."""
    up, dn = (1, 0), (0, 1)
    cnt = {"C": {}, "A": {}, "B": {}}

    def bump(k, cb, cs, spins, m):
        if m:
            key = (cb, cs, tuple(sorted(spins)))
            cnt[k][key] = cnt[k].get(key, 0) + m
    half = n_block // 2
    for a in (up, dn):
        bump("C", a, (0, 0), (a,), half)
        bump("C", (0, 0), a, (a,), n_site // 2)
        for b in (up, dn):
            mb = (-b[0], -b[1])
            bump("A", _add(a, b), (0, 0), (a, b), half * (half - 1) // 2 if a == b else half * half // 2)
            bump("A", a, b, (a, b), half)
            bump("B", _add(a, mb), (0, 0), (a, mb), half * half)
            bump("B", a, mb, (a, mb), half)
            bump("B", (-a[0], -a[1]), b, ((-a[0], -a[1]), b), half)
            bump("B", (0, 0), _add(a, mb), (a, mb), 1)
    bump("A", (0, 0), _add(up, dn), (up, dn), 1)
    return cnt


def _sigma_work(c):
    """(flops, operator bytes, psi elements) of one sigma step: the products of the
    charge-allowed sub-blocks of every term sum_nu O_L psi O_R^T, once each."""
    L, na, nb, D, b = (c[k] for k in ("L", "na", "nb", "D", "bond"))
    lsec = inputs.left_bond_sectors(L, na, nb, D, b)[b]
    rsec = inputs.right_bond_sectors(L, na, nb, D, b + 2)[b + 2]
    ef, ee = _fines(inputs.enlarged_layout(lsec), lsec), _fines(inputs.enlarged_layout(rsec), rsec)
    left = {Q: sum(f.values()) for Q, f in ef.items()}
    right = {Q: sum(f.values()) for Q, f in ee.items()}
    N = (na, nb)
    psi = {Q: (left[Q], right[_add(N, Q, -1)]) for Q in left if _add(N, Q, -1) in right}
    n_psi = sum(r * k for r, k in psi.values())
    flops, bytes_ = 0.0, 0.0

    def one_sided(fines, pair):
        """Elements and sum(rows * cols) of the sub-blocks that move (block, site) charge by pair, by source Q."""
        cb, cs = pair
        out = {}
        if cb == (0, 0):
            return out                      # identity on the block: a copy, no products
        for Q, f in fines.items():
            T = fines.get(_add(Q, _add(cb, cs)))
            if T is None:
                continue
            out[Q] = sum(f[(s, k)] * T[(t, _add(k, cb))] for (t, s) in _SITE[cs] for (u, k) in f
                         if u == s and (t, _add(k, cb)) in T)
        return out

    up, dn = (1, 0), (0, 1)
    nR = 2 * (L - b - 1)

    def complement(Q, T, spins):
        """Elements of a complementary operator's block (T <- Q) on site (x) block: the site takes none, one
        or both of a pair's elementary operators; three-index operators fill the whole block."""
        src, dst = ee[_add(N, Q, -1)], ee[_add(N, T, -1)]
        tot = _add(Q, T, -1)
        if len(spins) == 1:
            return sum(src.values()) * sum(dst.values())
        if tot == (0, 0):
            spins = (up, dn, (-1, 0), (0, -1))
        site = {(0, 0), tot} | {(-x[0], -x[1]) for x in spins}
        return sum(d * dst.get((t, _add(k, _add(tot, cs, -1))), 0) for cs in site for (t, s) in _SITE.get(cs, ())
                   for (u, k), d in src.items() if u == s)

    counts = _term_counts(2 * b, 2)
    for kind in ("C", "A", "B"):
        for (cb, cs, spins), m in counts[kind].items():
            blk = one_sided(ef, (cb, cs))
            tot = _add(cb, cs)
            both = 1 if kind == "B" else 2   # C and A act with their transposes as well
            for Q, (r, k) in psi.items():
                T = _add(Q, tot)
                if T not in psi:
                    continue
                e = complement(Q, T, spins)
                flops += both * m * 2.0 * (blk.get(Q, 0) * k + psi[T][0] * e)
                bytes_ += 8.0 * m * (blk.get(Q, 0) + e)
    for a in (up, dn):                       # S_q C_q^T and its transpose, q on the right
        for Q, (r, k) in psi.items():
            T = _add(Q, a)
            if T in psi:
                rT, kT = psi[T]
                site = sum(ee[_add(N, T, -1)].get((s, q), 0) * d for (s, q2), d in ee[_add(N, Q, -1)].items()
                           for q in (_add(q2, a, -1),))
                flops += 2.0 * (nR // 2) * 2.0 * (rT * r * k + rT * site)
                bytes_ += 8.0 * (nR // 2) * (rT * r + site)
    for r, k in psi.values():                # H_L' and H_R'
        flops += 2.0 * r * k * (r + k)
        bytes_ += 8.0 * (r * r + k * k)
    return flops, bytes_, n_psi


def work(case):
    kind = case["kind"]
    if kind == "eigh":
        n = [r for r, _ in _eigh_orders(case)]
        # tridiagonal form 4/3 n^3, eigenvectors back-transformed 2 n^3
        return {"bytes": 8.0 * sum(2 * x * x + x for x in n), "flops": sum(10.0 / 3.0 * x ** 3 for x in n)}
    if kind == "batch":
        w = [_sigma_work(c) for c in _batch_cases(case)]
        return {"bytes": sum(b + 16.0 * n for _, b, n in w), "flops": sum(f for f, _, _ in w)}
    if kind == "dmrg":
        # per step of a sweep at least a dozen sigma steps, full bond dimensions
        total_f = total_b = 0.0
        for b in range(case["L"] - 1):
            f, o, n = _sigma_work(dict(case, bond=b))
            total_f += 2 * 12 * f
            total_b += 2 * 12 * (o + 16.0 * n)
        return {"bytes": case["sweeps"] * total_b, "flops": case["sweeps"] * total_f}
    f, o, n = _sigma_work(case)
    if kind == "davidson":
        k = case["iters"] + 1
        # a sigma per iteration and the Gram-Schmidt passes over the growing subspace
        return {"bytes": k * (o + 16.0 * n) + 8.0 * n * k * k, "flops": k * f + 4.0 * n * k * k}
    if kind == "backward":
        return {"bytes": o + 16.0 * n + 8.0 * (case["L"] ** 2 + case["L"] ** 4), "flops": 2.0 * f}
    return {"bytes": o + 16.0 * n, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits on the determinant basis

def _strings(L, n):
    return np.array([s for s in range(1 << L) if bin(s).count("1") == n], dtype=np.int64)


def _excitations(L, n):
    """For every (k, l): targets, sources and signs of a+_k a_l on the sorted strings."""
    st = _strings(L, n)
    pos = np.full(1 << L, -1)
    pos[st] = np.arange(len(st))
    out = {}
    for k in range(L):
        for l in range(L):
            ok = (st >> l) & 1 == 1
            if k != l:
                ok &= (st >> k) & 1 == 0
            src = np.nonzero(ok)[0]
            s = st[src]
            lo, hi = min(k, l), max(k, l)
            between = (s >> (lo + 1)) & ((1 << max(hi - lo - 1, 0)) - 1)
            sign = 1.0 - 2.0 * (np.array([bin(x).count("1") for x in between]) & 1)
            out[k, l] = (pos[(s & ~(1 << l)) | (1 << k)], src, sign if k != l else np.ones(len(src)))
    return out


class _Fci:
    def __init__(self, L, na, nb):
        self.L, self.a, self.b = L, _excitations(L, na), _excitations(L, nb)
        self.shape = (math.comb(L, na), math.comb(L, nb))

    def E(self, k, l, x, out):
        t, s, g = self.a[k, l]
        out[t] += g[:, None] * x[s]
        t, s, g = self.b[k, l]
        out[:, t] += g[None, :] * x[:, s]

    def all_E(self, x, transposed=False):
        D = np.zeros((self.L * self.L,) + self.shape)
        for k in range(self.L):
            for l in range(self.L):
                self.E(*((l, k) if transposed else (k, l)), x, D[k * self.L + l])
        return D

    def H(self, t, v, x):
        L = self.L
        h = t - 0.5 * np.einsum("ijjl->il", v)
        G = 0.5 * (v.reshape(L * L, L * L) @ self.all_E(x).reshape(L * L, -1))
        y = np.zeros(self.shape)
        for i in range(L):
            for j in range(L):
                self.E(i, j, G[i * L + j].reshape(self.shape) + h[i, j] * x, y)
        return y


def _basis(sites, order):
    """Explicit vectors of an MPS block: {sector: (base-4 configuration codes, matrix)}."""
    vec = {(0, 0): (np.zeros(1, dtype=np.int64), np.ones((1, 1)))}
    for i in order:
        vec = {Q: (codes, M @ sites[i][Q]) for Q, (codes, M) in _enlarged(vec, i).items() if Q in sites[i]}
    return vec


def _enlarged(vec, site):
    out = {}
    for Q in sorted({_add(q, p) for q in vec for p in _Q}):
        parts = [(s, vec[_add(Q, p, -1)]) for s, p in enumerate(_Q) if _add(Q, p, -1) in vec]
        n = sum(M.shape[1] for _, (_, M) in parts)
        codes, rows, o = [], [], 0
        for s, (cd, M) in parts:
            codes.append(cd + s * 4 ** site)
            R = np.zeros((len(cd), n))
            R[:, o:o + M.shape[1]] = M
            rows.append(R)
            o += M.shape[1]
        out[Q] = (np.concatenate(codes), np.vstack(rows))
    return out


def _bits(codes, L):
    a = np.zeros(len(codes), dtype=np.int64)
    b = np.zeros(len(codes), dtype=np.int64)
    cross = np.zeros(len(codes), dtype=np.int64)   # (beta at i, alpha at j > i) pairs
    nb = np.zeros(len(codes), dtype=np.int64)
    for i in range(L):
        d = (codes // 4 ** i) % 4
        ai, bi = d >> 1, d & 1
        cross += nb * ai
        nb += bi
        a |= ai << i
        b |= bi << i
    return a, b, cross, nb


class _Embedding:
    """psi blocks <-> coefficients on (alpha string) x (beta string)."""

    def __init__(self, bp):
        L, k = bp.L, bp.bond
        self.bp = bp
        self.left = _enlarged(_basis(bp.left_sites, range(k)), k)
        self.right = _enlarged(_basis(bp.right_sites, range(L - 1, k + 1, -1)), k + 1)
        pa, pb = np.full(1 << L, -1), np.full(1 << L, -1)
        sa, sb = _strings(L, bp.na), _strings(L, bp.nb)
        pa[sa], pb[sb] = np.arange(len(sa)), np.arange(len(sb))
        self.shape = (len(sa), len(sb))
        self.where = []
        for QL, QR, _ in bp.psi:
            (cl, _), (cr, _) = self.left[QL], self.right[QR]
            al, bl, xl, nl = _bits(cl, L)
            ar, br, xr, _ = _bits(cr, L)
            na_r = np.array([bin(x).count("1") for x in ar])
            sign = 1.0 - 2.0 * ((xl[:, None] + xr[None, :] + nl[:, None] * na_r[None, :]) & 1)
            self.where.append((pa[al[:, None] | ar[None, :]], pb[bl[:, None] | br[None, :]], sign))

    def up(self, blocks):
        x = np.zeros(self.shape)
        for (QL, QR, m), (ia, ib, sign) in zip(blocks, self.where):
            x[ia, ib] += sign * (self.left[QL][1] @ m @ self.right[QR][1].T)
        return x

    def down(self, y):
        return np.concatenate([(self.left[QL][1].T @ (sign * y[ia, ib]) @ self.right[QR][1]).ravel()
                               for (QL, QR, _), (ia, ib, sign) in zip(self.bp.psi, self.where)])


def _exact_sigma(case, seed):
    t, v, bp = _problem(case, seed)
    emb = _Embedding(bp)
    return emb.down(_Fci(bp.L, bp.na, bp.nb).H(t, v, emb.up(bp.psi)))


def _sym8(g):
    g = 0.5 * (g + g.transpose(1, 0, 2, 3))
    g = 0.5 * (g + g.transpose(0, 1, 3, 2))
    return 0.5 * (g + g.transpose(2, 3, 0, 1))


def exact(case, seed):
    kind = case["kind"]
    if kind == "eigh":   # eigenvectors are defined up to their sign: no value
        w = [np.linalg.eigvalsh(m.cpu().numpy()) for m in _eigh_matrices(case, seed, torch.device("cuda"))]
        return {"w": np.concatenate(w), "Z": None}
    if kind == "batch":
        return [_exact_sigma(c, seed + 10 * i) if c["L"] <= 10 else None for i, c in enumerate(_batch_cases(case))]
    if kind == "davidson" or case["L"] > 12:
        return None
    if kind == "sigma":
        return _exact_sigma(case, seed)
    if kind == "backward":
        t, v, bp = _problem(case, seed)
        emb, fci, L = _Embedding(bp), _Fci(case["L"], case["na"], case["nb"]), case["L"]
        psi, lam = emb.up(bp.psi), emb.up(inputs.random_psi_like(bp, seed + 2))
        D = fci.all_E(psi).reshape(L * L, -1)
        g1 = (D @ lam.reshape(-1)).reshape(L, L)
        g2 = (fci.all_E(lam, transposed=True).reshape(L * L, -1) @ D.T).reshape(L, L, L, L)
        g2 -= np.einsum("jk,il->ijkl", np.eye(L), g1)
        return {"g1": 0.5 * (g1 + g1.T), "g2": _sym8(g2)}
    # whole run with all states kept: the lowest eigenvalue, by Lanczos with full reorthogonalisation
    t, v = inputs.synthetic_integrals(case["L"], seed)
    fci = _Fci(case["L"], case["na"], case["nb"])
    n = fci.shape[0] * fci.shape[1]
    q = np.random.default_rng(0).standard_normal(n)
    V, a, b = [q / np.linalg.norm(q)], [], []
    for k in range(min(n, 140)):
        w = fci.H(t, v, V[-1].reshape(fci.shape)).reshape(-1)
        a.append(float(w @ V[-1]))
        for _ in range(2):
            B = np.array(V)
            w = w - B.T @ (B @ w)
        b.append(float(np.linalg.norm(w)))
        if b[-1] < 1e-9:
            break
        V.append(w / b[-1])
    m = len(a)
    T = np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1)
    return {"energies": np.full(case["sweeps"], np.linalg.eigvalsh(T)[0])}
