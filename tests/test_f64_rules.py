"""Rules of the FP64 digit form on the CPU, with the kernel's own arithmetic.

Chunk sums: rows graded one way against columns graded the other, where the largest
elements meet small ones, held against the sum of their terms' magnitudes.  Bound: a sum
kept in digits is at least 2^54 in units in which it is off by at most 578 k + 2^14; one
computed again rounds k times."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_18263_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("f64") / "rules.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I" + CSRC,
                    os.path.join(HERE, "f64_rules_emulate.cpp"), os.path.join(CSRC, "core", "f64_plan.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def _chunk(lib, a, b):
    P = ctypes.POINTER(ctypes.c_double)
    out = ctypes.c_double()
    again = lib.f64_chunk(a.ctypes.data_as(P), b.ctypes.data_as(P), len(a), ctypes.byref(out))
    terms = [Fraction(x) * Fraction(y) for x, y in zip(a.tolist(), b.tolist())]
    scale = sum(abs(x) for x in terms)
    return again, float(abs(Fraction(out.value) - sum(terms)) / scale) if scale else abs(out.value)


@pytest.mark.parametrize("K", [1, 2, 8, 64, 192])
@pytest.mark.parametrize("spread", [0, 8, 12, 20, 30, 40, 60, 200])
def test_chunk_sums_keep_small_terms(lib, K, spread):
    rng = np.random.default_rng(1000 * K + spread)
    bound = (578 * K + 2 ** 14) * 2.0 ** -54 + K * 2.0 ** -52
    ramp = 2.0 ** -(spread * np.arange(K) / max(1, K - 1))
    for signs in (0, 1):
        for _ in range(20):
            a, b = rng.uniform(0.5, 1.0, K) * ramp, rng.uniform(0.5, 1.0, K) * ramp[::-1]
            if signs:
                a *= rng.choice([-1.0, 1.0], K)
            assert _chunk(lib, a, b)[1] <= bound
    a, b = np.zeros(K), np.zeros(K)    # a large element against a zero
    a[0], b[-1] = 1.0, 1.0
    a[-1] = b[0] = 2.0 ** -spread / 3 if K > 1 else 1.0
    assert _chunk(lib, a, b)[1] <= bound
    b[0] = 0.0 if K > 1 else 1.0
    assert _chunk(lib, a, b)[1] <= bound


@pytest.mark.parametrize("K", [8, 64, 192])
def test_few_ordinary_sums_are_computed_again(lib, K):
    rng = np.random.default_rng(K)
    again = [_chunk(lib, rng.standard_normal(K), rng.standard_normal(K))[0] for _ in range(4000)]
    assert np.mean(again) < 2e-3


ANY, PLAIN = 1, 2


@pytest.mark.parametrize("forms, small, plain, route", [
    (ANY, 0, 0, 0), (ANY, 1, 0, 1), (PLAIN, 0, 1, 1), (PLAIN, 1, 1, 1), (ANY | PLAIN, 0, 0, 0), (ANY | PLAIN, 0, 1, 1),
    (ANY | PLAIN, 1, 0, 1), (ANY, 0, 1, -1), (ANY, 1, 1, -1), (PLAIN, 0, 0, -1), (PLAIN, 1, 0, -1), (0, 0, 0, -1)])
def test_a_plan_runs_only_in_a_form_it_was_built_for(lib, forms, small, plain, route):
    assert lib.f64_route(forms, small, plain) == route


@pytest.mark.parametrize("seed", range(8))
def test_lists_of_an_earlier_plan_leave_nothing(lib, seed):
    assert lib.f64_reused_lists(seed) == 0
