"""FP64 products on both sides of their dispatch (plain multiply-adds for small launches,
digit products on the tensor cores above) and the eigensolver's reduction around the
orders where it goes from one CTA to a cluster.

Scaling psi by a power of two scales every operand row's exponent and nothing else, so
sigma scales exactly in either form; an infinity or NaN of the input reaches the output.
Eigensolver bounds: 64 n eps, relative to the matrix norm."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2501_18263_gb300 import binding as B
from paper_2501_18263_gb300 import inputs as I
from gpu_util import assert_blocks, rel, stream, to_dev

pytestmark = pytest.mark.gpu


def _handle(L, na, nb, D, bond, seed):
    t, v = I.synthetic_integrals(L, seed)
    bp = I.bond_problem(L, na, nb, D, bond, seed=seed + 100)
    d = B.Dmrg(t, v, na, nb, D=D, stream=stream())
    d.load_bond_problem(bp)
    d.prepare(bond)
    return t, v, bp, d


@pytest.mark.parametrize("L, na, nb, D, bond", [(4, 2, 2, 6, 1), (6, 2, 3, 24, 2), (9, 4, 5, 60, 0), (10, 5, 5, 130, 6),
                                                (11, 6, 4, 200, 4)])
def test_sigma_matches_the_oracle_and_scales_exactly(L, na, nb, D, bond):
    t, v, bp, d = _handle(L, na, nb, D, bond, 40 + L)
    lay, n = d.layout(bond)
    psi = to_dev(B.pack_psi(bp.psi))
    out = [torch.empty_like(psi) for _ in range(3)]
    ref = B.pack_psi(O.projected_sigma(t, v, na, nb, bp, bp.psi))
    d.sigma(bond, psi.data_ptr(), out[0].data_ptr())
    assert rel(out[0].cpu().numpy(), ref) < 1e-13
    assert_blocks(out[0].cpu().numpy(), ref, lay, 1e-10)
    for i, e in ((1, 300), (2, -300)):
        x = psi * 2.0 ** e
        d.sigma(bond, x.data_ptr(), out[i].data_ptr())
        assert torch.equal(out[i] * 2.0 ** -e, out[0])
    for bad in (float("nan"), float("inf")):
        x = psi.clone()
        x[n // 2] = bad
        d.sigma(bond, x.data_ptr(), out[1].data_ptr())
        assert not bool(torch.isfinite(out[1][n // 2]))
        d.sigma(bond, psi.data_ptr(), out[2].data_ptr())    # and leaves nothing behind
        assert torch.equal(out[2], out[0])
    d.close()


@pytest.mark.parametrize("orders", [(62, 63, 64, 65), (78, 79, 80, 81, 82, 87, 88, 89, 96), (127, 128, 129, 255, 256, 257)])
def test_eigensolver_around_the_cluster_threshold(orders):
    t, v = I.synthetic_integrals(2, 5)
    d = B.Dmrg(t, v, 1, 1, D=4, stream=stream())
    rng = np.random.default_rng(sum(orders))
    mats = []
    for n in orders:
        P = rng.standard_normal((n, n)) * np.exp(-np.arange(n) / 25.0)[None, :]
        mats.append(P @ P.T)
    A = torch.tensor(np.concatenate([M.ravel() for M in mats]), device="cuda")
    Z, w = torch.empty_like(A), torch.empty(sum(orders), dtype=torch.float64, device="cuda")
    d.eigh_batch(list(orders), A.data_ptr(), w.data_ptr(), Z.data_ptr())
    zs, ws = Z.cpu().numpy(), w.cpu().numpy()
    zo = wo = 0
    for n, M in zip(orders, mats):
        z, x = zs[zo:zo + n * n].reshape(n, n), ws[wo:wo + n]
        zo, wo = zo + n * n, wo + n
        eps, nrm = np.finfo(float).eps, np.linalg.norm(M, 2)
        assert np.max(np.abs(x - np.linalg.eigvalsh(M))) <= 64 * n * eps * nrm
        assert np.linalg.norm(M @ z - z * x[None, :]) <= 64 * n * eps * nrm
        assert np.max(np.abs(z.T @ z - np.eye(n))) <= 64 * n * eps
    d.close()
