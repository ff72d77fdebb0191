"""FP64 sigma with operators and a wave function whose elements span twenty orders of
magnitude, element by element: every element of sigma is held against the sum of the
magnitudes of its own terms, not against the norm.  The basis is the
occupation basis (complete, unit vectors), where a row of an operator holds elements as
different as the integrals are.

Bound: a product of the digit form is within (578 k + 2^14) 2^-54 < 2^-37 of the sum of its
terms' magnitudes (k <= 192 of a chunk; smaller results are computed plainly), and sigma
is two such products: 2^-36."""
import numpy as np
import pytest

import oracle as O
from paper_2501_18263_gb300 import binding as B
from paper_2501_18263_gb300 import inputs as I
from gpu_util import stream, to_dev

pytestmark = pytest.mark.gpu


def _graded_integrals(L, rng):
    def mag(shape):
        return 2.0 ** -rng.uniform(0, 60, shape)
    t = mag((L, L))
    t = np.triu(t) + np.triu(t, 1).T
    v = np.zeros((L,) * 4)
    p = [(i, j) for i in range(L) for j in range(i + 1)]
    w = mag((len(p), len(p)))
    for a, (i, j) in enumerate(p):
        for b, (k, l) in enumerate(p[:a + 1]):
            for x in {(i, j, k, l), (j, i, k, l), (i, j, l, k), (j, i, l, k)}:
                v[x] = v[x[2], x[3], x[0], x[1]] = w[a, b]
    return t, v


def _terms(t, v, n, x):
    """sum over the terms of H of |term| |x|: determinants as (alpha string, beta string)."""
    L = t.shape[0]

    def annihilate(k):   # |a_p| from k to k - 1 particles, by p
        src, dst = O.strings(L, k), {m: i for i, m in enumerate(O.strings(L, k - 1))}
        A = np.zeros((L, len(dst), len(src)))
        for j, m in enumerate(src):
            for p in range(L):
                if m >> p & 1:
                    A[p, dst[m ^ (1 << p)], j] = 1.0
        return A
    A, A2 = annihilate(n), annihilate(n - 1)
    E = np.einsum("pxi,qxj->pqij", A, A)                       # |a+_p a_q|
    P = np.einsum("sxy,qyj->sqxj", A2, A)                      # |a_s a_q|
    one = np.einsum("pq,pqij->ij", t, E)
    one += 0.5 * np.einsum("rpxi,prxj->ij", P, np.einsum("pqrs,sqxj->prxj", v, P, optimize=True), optimize=True)
    x = x.reshape(one.shape)
    y = one @ x + x @ one.T
    return (y + np.einsum("pqij,pqkj->ik", E, np.einsum("pqrs,rskl,jl->pqkj", v, E, x, optimize=True),
                          optimize=True)).ravel()


@pytest.mark.parametrize("bond, spread, filled", [(3, 0, 1.0), (3, 70, 1.0), (3, 0, 0.01), (2, 40, 0.05), (4, 20, 0.002)])
def test_graded_sigma_by_element(bond, spread, filled):
    """filled: part of psi that is not zero, so that a row's large elements meet zeros."""
    L, na, nb = 8, 4, 4
    rng = np.random.default_rng(10 * bond + spread)
    t, v = _graded_integrals(L, rng)
    bp = I.bond_problem(L, na, nb, 4 ** (L // 2), bond, seed=3, kind="select")
    psi = [(a, b, x * 2.0 ** -rng.uniform(0, spread, x.shape) * (rng.random(x.shape) < filled)) for a, b, x in bp.psi]
    ref, parts = O.projected_sigma(t, v, na, nb, bp, psi, return_parts=True)
    x = np.abs(parts["x"])
    assert sum(p.size for _, _, p in psi) == O.fci_dim(L, na, nb)   # the whole space
    cfg = O.config_index(L, na, nb)
    full = np.zeros(4 ** L)
    full[cfg] = _terms(t, v, na, x)
    U, V = parts["U"], parts["V"]
    S = np.einsum("ca,cstd,db->astb", U, full.reshape(U.shape[0], 4, 4, V.shape[0]), V, optimize=True)
    scale = np.abs(B.pack_psi(O.dense_to_psi(S, bp.left_bonds[bond].as_array(), bp.right_bonds[bond + 2].as_array(),
                                             na, nb)))
    d = B.Dmrg(t, v, na, nb, D=4 ** (L // 2), stream=stream())
    d.load_bond_problem(bp)
    d.prepare(bond)
    a = to_dev(B.pack_psi(psi))
    out = to_dev(np.zeros(a.numel()))
    d.sigma(bond, a.data_ptr(), out.data_ptr())
    err = np.abs(out.cpu().numpy() - B.pack_psi(ref))
    assert np.all(err <= 2.0 ** -36 * scale), float(np.max(err / np.where(scale > 0, scale, 1.0)))
    d.close()
