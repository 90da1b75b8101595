"""Every graph's window tables fit in shared memory: the passes of dense graphs whose lists, coupling by coupling, do
not fit take lists that carry the bond, and a pass for which those do not fit either is done in two."""
import ctypes
import os
import subprocess
from math import comb

import numpy as np
import pytest

from paper_2505_02901_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2505_02901_gb300", "csrc")
F64, F32, F32X8 = range(3)


@pytest.fixture(scope="module")
def fit(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fit") / "libfit.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                           os.path.join(HERE, "host_window_fit_shim.cpp")])
    lib = ctypes.CDLL(so)

    def call(N, nup, bonds, J):
        b = np.ascontiguousarray(bonds, dtype=np.int32)
        j = np.ascontiguousarray(J, dtype=np.float64)
        f, listed = np.zeros(3, np.int32), np.zeros(2, np.int32)
        p = lambda a, t: a.ctypes.data_as(ctypes.POINTER(t))
        n = lib.window_fit(N, nup, p(b, ctypes.c_int32), len(b), p(j, ctypes.c_double), p(f, ctypes.c_int32),
                           p(listed, ctypes.c_int32))
        return n, f, listed
    return call


def _shells(lx, ly, n):
    """The bonds of the n shortest distances of a periodic lattice, and their shells."""
    by = {}
    for a in range(lx * ly):
        for b in range(a):
            dx, dy = abs(a % lx - b % lx), abs(a // lx - b // lx)
            by.setdefault(min(dx, lx - dx) ** 2 + min(dy, ly - dy) ** 2, []).append((a, b))
    bonds = [(b, s) for s, d in enumerate(sorted(by)[:n]) for b in by[d]]
    return np.array([b for b, _ in bonds], dtype=np.int32), np.array([s for _, s in bonds])


def _graph(name, N):
    rng = np.random.default_rng(N)
    if name == "complete":
        return np.array([(i, j) for i in range(N) for j in range(i)], dtype=np.int32), None
    if name == "long_range":  # a ring with bonds up to four sites away, coupling by distance
        bonds = [(i, (i + d) % N) for d in (1, 2, 3, 4) for i in range(N)]
        return np.array(bonds, dtype=np.int32), np.repeat(np.arange(4), N)
    nb = int(rng.integers(6 * N, N * (N - 1) // 2))
    return W.random_bonds(N, nb, N), None


@pytest.mark.parametrize("name", ["complete", "long_range", "random"])
@pytest.mark.parametrize("N,nup", [(24, 12), (25, 6), (26, 13), (28, 14), (30, 15), (32, 16), (32, 7), (35, 17), (36, 18), (40, 10)])
def test_tables_fit(fit, name, N, nup):
    bonds, shell = _graph(name, N)
    nb, wide = len(bonds), comb(N, nup) >= 2 ** 32 - 1
    rng = np.random.default_rng(7)
    four = rng.integers(0, 4, nb) if shell is None else shell
    for J in (np.ones(nb), np.array([1.0, 0.5, 0.25, 0.75])[four], rng.standard_normal(nb)):
        n, f, _ = fit(N, nup, bonds, J)
        assert n > 0
        assert f[F64]
        if not wide:  # beside 64-bit row offsets FP32 may be left without
            assert f[F32] and f[F32X8]


@pytest.mark.parametrize("lx,ly,shells", [(5, 6, 4), (4, 8, 4), (4, 6, 5), (5, 5, 4), (6, 6, 4), (6, 6, 6)])
def test_lattices_with_many_shells(fit, lx, ly, shells):
    """Lattices whose lists coupling by coupling do not fit take others in some of their passes only."""
    bonds, shell = _shells(lx, ly, shells)
    n, f, listed = fit(lx * ly, lx * ly // 2, bonds, 2.0 ** -shell)
    assert n > 0 and f[F64] and (f.all() or lx * ly == 36)
    if shells == 4 and lx * ly < 36:
        assert listed[0] > 0 and listed[1] > 0
