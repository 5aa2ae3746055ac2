"""The FP64 cell's source (csrc/cell.cuh, built for the CPU by host_cell.cpp)
against exact rational arithmetic: every path's error bound, and the range of
the group sums that the emulated paths take, on fields of one and both signs."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

WEIGHTS = {1: (0.164, 0.164, 0.164), 2: (0.0412, 0.164, 0.164), 3: (0.164, 0.0412, 0.09)}


@pytest.fixture(scope="module")
def cells(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host_cell") / "host_cell.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + os.path.join(CUDA, "include"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_2211_15716_gb300", "csrc"),
                    os.path.join(HERE, "host_cell.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).host_cells

    def run(t, ci, w):
        t, ci, w = (np.ascontiguousarray(a, dtype=np.float64) for a in (t, ci, w))
        out, path = np.empty(len(t)), np.empty(len(t), dtype=np.int32)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        ng = fn(ctypes.c_int(len(t)), p(t), p(ci), p(w), p(out), p(path))
        return out, path, ng

    return run


def _stencils(kind, rng, n):
    """[n, 7] centre, x-, x+, y-, y+, z-, z+."""
    if kind == "smooth":
        return rng.uniform(1.2, 2.7, (n, 1)) * (1 + 1e-4 * rng.standard_normal((n, 7)))
    if kind == "negative":
        return -_stencils("smooth", rng, n)
    if kind == "wide":  # one binade, group sums around 2^45 to 2^48 ulps
        return 3.0 * (1 + 0.01 * rng.uniform(-2, 2, (n, 7)))
    if kind == "across zero":
        return 1e-3 * rng.uniform(-1, 1, (n, 1)) + 1e-5 * rng.standard_normal((n, 7))
    if kind == "across two":
        return 2.0 + 1e-4 * rng.standard_normal((n, 7))
    if kind == "uniform":
        return rng.uniform(-1, 1, (n, 7))
    if kind == "positive":
        return rng.uniform(0, 1, (n, 7))
    if kind == "signs":  # group sums near multiples of 2^54 ulps
        return rng.choice([-1.0, 1.0], (n, 7)) * rng.uniform(0.999, 1.0, (n, 7))
    # group sums within 2^48 ulps of +-2^55 and +-2^56: centre c, the six
    # neighbours near -c / 3 (equal weights: the sum is -8 c)
    c = rng.choice([-1.0, 1.0], (n, 1)) * rng.uniform(0.99, 1.01, (n, 1))
    t = np.repeat(c, 7, axis=1) * np.array([1.0] + [-1.0 / 3.0] * 6)
    return t * (1 + 2.0 ** -9 * rng.uniform(-1, 1, (n, 7)))


KINDS = ["smooth", "negative", "wide", "across zero", "across two", "uniform", "positive", "signs",
         "thirds"]


def _group_sums(t, u, ng):
    """The exact group sums of the second differences in units of u."""
    d = [(Fr(t[1 + 2 * k]) + Fr(t[2 + 2 * k]) - 2 * Fr(t[0])) / u for k in range(3)]
    return {1: [d[0] + d[1] + d[2]], 2: [d[0], d[1] + d[2]], 3: d}[ng]


@pytest.mark.parametrize("ng", [1, 2, 3])
@pytest.mark.parametrize("kind", KINDS)
def test_error_and_range(cells, kind, ng):
    rng = np.random.default_rng(23)
    n = 1500
    t, ci = _stencils(kind, rng, n), rng.uniform(0.4, 0.667, n)
    w = WEIGHTS[ng]
    out, path, groups = cells(t, ci, w)
    assert groups == ng
    wr = [Fr(v) for v in w]
    for i in range(n):
        s = [float(v) for v in t[i]]
        u = Fr(2) ** (int(np.frexp(max(map(abs, s)))[1]) - 53)  # ulp of the largest value
        d2 = [Fr(s[1 + 2 * k]) + Fr(s[2 + 2 * k]) - 2 * Fr(s[0]) for k in range(3)]
        c = Fr(float(ci[i]))
        exact = Fr(s[0]) + c * sum(a * b for a, b in zip(wr, d2))
        # the values' rounding to u (6 Ci w < 1), two roundings of the result,
        # half an ulp of the weights' roundings; 2^-44 of Ci sum |w d2|
        bound = Fr(7, 2) * u + Fr(2) ** -44 * c * sum(a * abs(b) for a, b in zip(wr, d2))
        assert abs(Fr(float(out[i])) - exact) <= bound, (i, path[i], s)
        if path[i] == 0:
            # the correction's Ci of 24 bits costs an eighth of an ulp at 2^45
            assert max(abs(g) for g in _group_sums(s, u, ng)) <= 2 ** 45 + 2 ** 22, (i, s)
        elif path[i] == 1:  # (the rounded values' sum is within 6 of the exact one)
            assert max(abs(g) for g in _group_sums(s, u, ng)) <= 2 ** 47 + 2 ** 22 + 6, (i, path[i], s)
