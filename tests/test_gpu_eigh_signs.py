"""Eigenvectors of dmrg_eigh_batch come out with the signs of the QL iteration of
hypot-and-quotient rotations: the last bits of a rotation decide now and then whether a
coupling is negligible one iteration earlier, and every iteration turns signs around.

Matrices are Gram matrices of integers (exact in FP64 whatever the order of the sums);
bit c of an expected mask: the largest component of eigenvector c is negative, recorded
from that iteration.  Each of these turned when rotations were formed from a reciprocal
square root instead."""
import numpy as np
import pytest
import torch

from paper_2501_18263_gb300 import binding as B
from paper_2501_18263_gb300 import inputs as I
from gpu_util import stream

pytestmark = pytest.mark.gpu

SIGNS = [(852, 17, 0x632f), (2151, 14, 0x1f6b), (2510, 32, 0x9d3c4d80), (2664, 31, 0x7d8f8f58), (4223, 9, 0x1e4),
         (5307, 8, 0xdc), (6576, 6, 0x1b), (8159, 8, 0xa4), (9261, 25, 0x18d45a1), (9816, 22, 0x12bd97),
         (10601, 32, 0x5bdd51d7), (12510, 19, 0x30c17), (13763, 32, 0x2be11a6), (15624, 2, 0x0), (18636, 7, 0x1c)]


def _gram(seed, n):
    r = np.random.default_rng([seed, n])
    decay = 2.0 ** -np.floor(np.arange(n) * r.integers(0, 16) / 8.0)
    P = np.floor((r.random((n, n)) - 0.5) * 2 ** 22 * decay[None, :])
    return (P @ P.T) * 2.0 ** -44


def test_eigenvector_signs():
    t, v = I.synthetic_integrals(2, 5)
    d = B.Dmrg(t, v, 1, 1, D=4, stream=stream())
    n = [m for _, m, _ in SIGNS]
    A = torch.tensor(np.concatenate([_gram(s, m).ravel() for s, m, _ in SIGNS]), device="cuda")
    Z, w = torch.empty_like(A), torch.empty(sum(n), dtype=torch.float64, device="cuda")
    d.eigh_batch(n, A.data_ptr(), w.data_ptr(), Z.data_ptr())
    z, o = Z.cpu().numpy(), 0
    for seed, m, mask in SIGNS:
        Q = z[o:o + m * m].reshape(m, m)
        o += m * m
        top = Q[np.argmax(np.abs(Q), 0), np.arange(m)]
        assert sum(1 << c for c in range(m) if top[c] < 0) == mask, seed
    d.close()
