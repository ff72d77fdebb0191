"""Orders that the density-matrix eigensolver takes: up to 14506, as long as two vectors and
the scalars fit in an SM's shared memory; three of them are kept there up to 9670."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_18263_gb300", "csrc")


@pytest.mark.parametrize("n, vectors", [(1, 3), (2, 3), (352, 3), (6000, 3), (9670, 3), (9671, 2), (14506, 2),
                                        (14507, -1), (32767, -1)])
def test_orders(tmp_path, n, vectors):
    so = str(tmp_path / "syev.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, os.path.join(HERE, "syev_shared_emulate.cpp"),
                    "-o", so], check=True)
    bytes_ = ctypes.c_long()
    assert ctypes.CDLL(so).syev_vectors(n, ctypes.byref(bytes_)) == vectors
    if vectors > 0:
        assert 8 * (vectors * (n + 2) + 40) <= bytes_.value <= 227 * 1024
