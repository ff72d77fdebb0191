"""Work list of the tensor-core FP64 GEMM (csrc/core/f64_plan.h) on the CPU: a host
interpreter walks its units with the kernel's digit arithmetic, every access checked
against the operands' arena, and each C = alpha sum_seg op(A) op(B) (+ C) is compared
with the plain product in extended precision.  Forms: both orders of either operand,
strides above the extents, stacked problems (a shared B list, a shared A list), K lists
of one to many ragged segments, split sums, empty lists, accumulation.

Bound: inputs are truncated at 2^-62 of their row's (column's) largest element and the
digit weights above 7 dropped, 2^-58 of the largest products per k in all; each chunk's
sum, its factor alpha and each of the adds of at most `adds` partial sums round once."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2501_18263_gb300", "csrc")


class Prob(ctypes.Structure):
    _fields_ = [("C", ctypes.c_void_p), ("ldc", ctypes.c_int), ("M", ctypes.c_int), ("N", ctypes.c_int),
                ("s0", ctypes.c_int), ("s1", ctypes.c_int), ("alpha", ctypes.c_double), ("acc", ctypes.c_int)]


class Seg(ctypes.Structure):
    _fields_ = [("A", ctypes.c_void_p), ("B", ctypes.c_void_p), ("lda", ctypes.c_int), ("ldb", ctypes.c_int),
                ("K", ctypes.c_int), ("ta", ctypes.c_int), ("tb", ctypes.c_int)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("f64") / "emulate.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I" + CSRC,
                    os.path.join(HERE, "f64_plan_emulate.cpp"), os.path.join(CSRC, "core", "f64_plan.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


class Arena:
    def __init__(self, rng, n, wide):
        self.a = rng.standard_normal(n)
        if wide:   # magnitudes over many orders, zeros, tiny numbers
            self.a *= 2.0 ** rng.integers(-60, 60, n)
            self.a[rng.random(n) < 0.05] = 0.0
            self.a[rng.random(n) < 0.02] = 5e-324
        self.at = 0

    def take(self, rows, cols, ld):
        o = self.at
        self.at += rows * ld
        assert self.at <= self.a.size
        return o

    def addr(self, o):
        return self.a.ctypes.data + 8 * o


def _operand(ar, rng, rows, k, trans):
    """(offset, ld, matrix rows x k); trans: stored k x rows."""
    r, c = (k, rows) if trans else (rows, k)
    ld = c + int(rng.integers(0, 4))
    o = ar.take(r, c, ld)
    m = ar.a[o:o + r * ld].reshape(r, ld)[:, :c]
    return o, ld, (m.T if trans else m)


def _run(lib, ar, probs, out, nsm):
    """probs: (coff, ldc, M, N, alpha, acc, [(A, B)]), operands as _operand gives them + trans flags."""
    P = (Prob * len(probs))()
    segs = []
    refs = []
    for i, (co, ldc, M, N, alpha, acc, sl) in enumerate(probs):
        P[i] = Prob(out.ctypes.data + 8 * co, ldc, M, N, len(segs), len(segs) + len(sl), alpha, acc)
        ref = np.zeros((M, N), dtype=np.longdouble)
        mag = np.zeros((M, N))
        ra, cb, K = np.zeros(M), np.zeros(N), 0
        for (a, ta), (b, tb) in sl:
            segs.append(Seg(ar.addr(a[0]), ar.addr(b[0]), a[1], b[1], a[2].shape[1], ta, tb))
            A, B = a[2], b[2]
            if A.shape[1] and M and N:
                ref += A.astype(np.longdouble) @ B.T.astype(np.longdouble)
                mag += np.abs(A) @ np.abs(B).T
                ra, cb = np.maximum(ra, np.abs(A).max(1)), np.maximum(cb, np.abs(B).max(1))
                K += A.shape[1]
        old = out[co:co + M * ldc].reshape(M, ldc)[:, :N].copy() if M and N else np.zeros((M, N))
        ref = alpha * ref + (old if acc else 0)
        adds = K / 8 + len(sl) + 4
        bound = abs(alpha) * (adds * 2.0 ** -52 * mag + K * 2.0 ** -57 * np.outer(ra, cb)) + \
            (2.0 ** -52 * np.abs(old) if acc else 0) + 1e-300
        refs.append((co, ldc, M, N, ref, bound))
    S = (Seg * max(1, len(segs)))(*segs)
    # the plain form, alone and with the other's stacking: the same bits
    for what in (2, 3):
        plain = out.copy()
        Q = (Prob * len(probs))()
        for i in range(len(probs)):
            ctypes.memmove(ctypes.byref(Q[i]), ctypes.byref(P[i]), ctypes.sizeof(Prob))
            Q[i].C = plain.ctypes.data + 8 * probs[i][0]
        assert lib.f64_emulate_plain(Q, len(probs), S, len(segs), ctypes.c_void_p(ar.addr(0)),
                                     ctypes.c_void_p(ar.addr(ar.a.size)), what) == 0
        if what == 2:
            first = plain
        for co, ldc, M, N, ref, bound in refs:
            if M and N:
                got = plain[co:co + M * ldc].reshape(M, ldc)[:, :N]
                assert np.all(np.abs(got - ref) <= bound)
    assert np.array_equal(first, plain)
    stat = (ctypes.c_double * 3)()
    rc = lib.f64_emulate(P, len(probs), S, len(segs), nsm, ctypes.c_void_p(ar.addr(0)),
                         ctypes.c_void_p(ar.addr(ar.a.size)), stat)
    assert rc == 0
    assert stat[2] <= 24.0
    for co, ldc, M, N, ref, bound in refs:
        if M and N:
            got = out[co:co + M * ldc].reshape(M, ldc)[:, :N]
            assert np.all(np.abs(got - ref) <= bound)
    return stat


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("case", range(8))
def test_units_reproduce_the_products(lib, case, wide):
    rng = np.random.default_rng(100 * wide + case)
    ar = Arena(rng, 400000, wide)
    out = rng.standard_normal(200000)
    co = [0]

    def place(M, N):
        ldc = N + int(rng.integers(0, 3))
        o = co[0]
        co[0] += M * ldc
        return o, ldc
    probs = []
    nsm = 4
    if case < 4:       # one problem alone in each storage order; ragged sizes and K lists
        ta, tb = case & 1, case >> 1
        for (M, N, Ks) in [(1, 1, [1]), (7, 3, [9]), (130, 17, [5, 8, 1]), (128, 64, [16]), (33, 65, [24] * 9),
                           (16, 129, [193]), (3, 2, [40] * 12), (20, 5, [])]:
            sl = [((_operand(ar, rng, M, K, ta), ta), (_operand(ar, rng, N, K, not tb), tb)) for K in Ks]
            probs.append((*place(M, N), M, N, 1.0, 0, sl))
    elif case < 6:     # stacks: problems that share their B (case 4) or A list (case 5)
        K = [12, 7]
        shared = [_operand(ar, rng, 35, k, i) for i, k in enumerate(K)]
        for j in range(23):
            n = 1 + j % 13
            own = [_operand(ar, rng, n, k, (i + j) & 1) for i, k in enumerate(K)]
            alpha = -1.0 if j & 1 else 0.75
            if case == 4:
                sl = [((own[i], (i + j) & 1), (shared[i], 1 - i)) for i in range(2)]
                probs.append((*place(n, 35), n, 35, alpha, j % 3 == 0, sl))
            else:
                sl = [((shared[i], i), (own[i], 1 - ((i + j) & 1))) for i in range(2)]
                probs.append((*place(35, n), 35, n, alpha, j % 3 == 0, sl))
    elif case == 6:    # a long list split over units, accumulated; many SMs
        Ks = [int(k) for k in rng.integers(1, 41, 150)]
        sl = [((_operand(ar, rng, 40, K, 0), 0), (_operand(ar, rng, 21, K, 0), 1)) for K in Ks]
        probs.append((*place(40, 21), 40, 21, -1.0, 1, sl))
        nsm = 152
    else:              # segments without elements, empty outputs, segments of one k
        one = [((_operand(ar, rng, 9, 1, 0), 0), (_operand(ar, rng, 9, 1, 0), 1)) for _ in range(70)]
        nul = [((_operand(ar, rng, 9, 0, 0), 0), (_operand(ar, rng, 9, 0, 0), 1))]
        probs.append((*place(9, 9), 9, 9, 1.0, 0, one[:35] + nul + one[35:]))
        probs.append((*place(9, 9), 9, 9, 1.0, 1, nul))
        probs.append((*place(0, 9), 0, 9, 1.0, 0, one))
        probs.append((*place(9, 0), 9, 0, 1.0, 0, one))
    stat = _run(lib, ar, probs, out, nsm)
    if case == 6:
        assert stat[1] > 0   # the split was exercised


def test_infinities_and_nan_propagate(lib):
    rng = np.random.default_rng(9)
    ar = Arena(rng, 4000, 0)
    a, b = _operand(ar, rng, 6, 10, 0), _operand(ar, rng, 5, 10, 0)
    a[2][1, 3], a[2][2, 0], b[2][4, 2] = np.inf, np.nan, -np.inf
    out = np.zeros(30)
    P = (Prob * 1)(Prob(out.ctypes.data, 5, 6, 5, 0, 1, 1.0, 0))
    S = (Seg * 1)(Seg(ar.addr(a[0]), ar.addr(b[0]), a[1], b[1], 10, 0, 1))
    stat = (ctypes.c_double * 3)()
    assert lib.f64_emulate(P, 1, S, 1, 4, ctypes.c_void_p(ar.addr(0)), ctypes.c_void_p(ar.addr(4000)), stat) == 0
    with np.errstate(invalid="ignore"):
        ref = a[2] @ b[2].T
    got = out.reshape(6, 5)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    fine = np.isfinite(ref)
    assert np.allclose(got[fine], ref[fine], rtol=1e-13)


@pytest.mark.parametrize("M, N, nseg, K, small", [
    ([1], [1], [1], [512], 1),                       # the longest sum one warp keeps
    ([1], [1], [1], [513], 0),
    ([1, 1], [1, 1], [1, 2], [4, 256, 257], 0),      # over two segments
    ([8] * 2, [4] * 2, [1, 0], [512], 1),            # an empty list
    ([], [], [], [], 1),
    ([8] * 366, [4] * 366, [1] * 366, [256] * 366, 1),    # 2 998 272 counted
    ([8] * 367, [4] * 367, [1] * 367, [256] * 367, 0),    # 3 006 464
    ([1] * 367, [1] * 367, [1] * 367, [249] * 367, 0),    # the same pieces and octets, ragged
])
def test_small_launches_are_plain(lib, M, N, nseg, K, small):
    ints = [(ctypes.c_int * max(1, len(x)))(*x) for x in (M, N, nseg, K)]
    assert lib.f64_emulate_small(len(M), ints[0], ints[1], ints[2], len(K), ints[3]) == small
