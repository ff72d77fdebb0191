"""Merges of the divide-and-conquer eigensolver where its root finder, its deflation and
its leaves can go wrong: sizes around one and two leaves and one warp of roots, clustered,
repeated, graded and widely scaled spectra, couplings of zero between blocks.

Bounds: 64 n eps relative to the matrix norm (residual, orthogonality, eigenvalues)."""
import numpy as np
import pytest
import torch

from paper_2501_18263_gb300 import binding as B
from paper_2501_18263_gb300 import inputs as I
from gpu_util import stream

pytestmark = pytest.mark.gpu


def _spectra(n, rng):
    j = np.arange(n)
    one = 2.0 * np.eye(n) - np.diag(np.ones(n - 1), 1) - np.diag(np.ones(n - 1), -1)
    split = one.copy()
    for b in (n // 2, n // 3):
        if 0 < b < n:
            split[b - 1, b] = split[b, b - 1] = 0.0
    wilkinson = np.diag(np.abs(j - n // 2).astype(float)) + np.diag(np.ones(n - 1), 1) + np.diag(np.ones(n - 1), -1)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    lams = [1.0 + 1e-13 * rng.standard_normal(n),                  # one cluster
            np.where(j < n // 2, 1.0, -1.0) * np.ones(n),           # two eigenvalues
            2.0 ** -(j * 300.0 / n),                                # graded over 90 orders
            np.concatenate([np.zeros(n - n // 4), rng.random(n // 4)])]
    dense = [(Q * lam) @ Q.T for lam in lams]
    return [one, split, wilkinson, 1e140 * wilkinson, 1e-130 * wilkinson] + [0.5 * (M + M.T) for M in dense]


@pytest.mark.parametrize("n", [2, 31, 33, 34, 63, 64, 65, 66, 97, 129, 193, 260])
def test_spectra(n):
    t, v = I.synthetic_integrals(2, 5)
    d = B.Dmrg(t, v, 1, 1, D=4, stream=stream())
    mats = _spectra(n, np.random.default_rng(n))
    A = torch.tensor(np.stack(mats), device="cuda")
    Z, w = torch.empty_like(A), torch.empty(len(mats) * n, dtype=torch.float64, device="cuda")
    d.eigh_batch([n] * len(mats), A.data_ptr(), w.data_ptr(), Z.data_ptr())
    zs, ws = Z.cpu().numpy(), w.cpu().numpy().reshape(len(mats), n)
    eps = np.finfo(float).eps
    for M, z, x in zip(mats, zs, ws):
        nrm = np.linalg.norm(M, 2) or 1.0
        assert np.all(np.diff(x) >= 0)
        assert np.max(np.abs(x - np.linalg.eigvalsh(M))) <= 64 * n * eps * nrm
        assert np.linalg.norm((M / nrm) @ z - z * (x / nrm)[None, :]) <= 64 * n * eps
        assert np.max(np.abs(z.T @ z - np.eye(n))) <= 64 * n * eps
    d.close()
