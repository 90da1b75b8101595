"""The window product's tables on the CPU: the tiles of every pass visit every row once, every index stays
inside what it indexes, the two rows of a pair read rows of opposite parity (no bank conflicts), and the
passes add up to the oracle's product."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2505_02901_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2505_02901_gb300", "csrc")


@pytest.fixture(scope="module")
def win(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("win") / "libwin.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                           os.path.join(HERE, "host_window_shim.cpp")])
    return ctypes.CDLL(so)


def _ptr(a, t):
    return a.ctypes.data_as(ctypes.POINTER(t))


def _case(name):
    if name == "chain13":
        return 13, 5, W.chain(13), None
    if name == "chain17_nup0":
        return 17, 0, W.chain(17), None
    if name == "chain16_nup2":
        return 16, 2, W.chain(16), None
    if name == "ladder16":
        return 16, 8, W.ladder(8, 2), "random"
    if name == "square4x4":
        return 16, 8, *W.square_j1j2(4, 4)
    if name == "square3x5":
        return 15, 7, *W.square_j1j2(3, 5)
    if name == "triangular4":
        return 16, 7, *W.triangular(4)
    if name == "square5x3_random":
        return 15, 6, W.square_j1j2(5, 3)[0], "random"
    if name == "square4x5":
        return 20, 7, *W.square_j1j2(4, 5)
    if name == "random17":
        return 17, 8, W.random_bonds(17, 60, 5), "random"
    if name == "complete14":
        return 14, 7, np.array([(i, j) for i in range(14) for j in range(i)], dtype=np.int32), None
    return 14, 13, np.array([(0, 13)], dtype=np.int32), None  # one bond across the word


CASES = ["chain13", "chain17_nup0", "chain16_nup2", "ladder16", "square4x4", "square3x5", "triangular4",
         "square5x3_random", "square4x5", "random17", "complete14", "one_bond"]


# ctas: 152 share few tiles each (one run by cost), 1 and 2 have many (a run of every popcount)
@pytest.mark.parametrize("value_bytes,nv,bond,ctas", [(8, 1, 0, 152), (8, 1, 1, 2), (8, 1, 0, 1), (4, 1, 0, 2), (4, 1, 1, 1),
                                                      (4, 8, 0, 1), (8, 2, 0, 3), (8, 8, 1, 2)])
@pytest.mark.parametrize("name", CASES)
def test_passes_reproduce_the_product(win, orc, name, value_bytes, nv, bond, ctas):
    N, nup, bonds, J = _case(name)
    if J is None:
        J = np.ones(len(bonds))
    elif isinstance(J, str):
        J = W.uniform_couplings(len(bonds), 7)
    bonds = np.ascontiguousarray(bonds, dtype=np.int32)
    J = np.ascontiguousarray(J, dtype=np.float64)
    states = orc.enumerate_states(N, nup)
    rng = np.random.default_rng(1)
    x = rng.standard_normal((states.size, nv))
    y = np.zeros_like(x)
    rc = win.window_product(N, nup, _ptr(bonds, ctypes.c_int32), len(bonds), _ptr(J, ctypes.c_double), value_bytes, nv,
                            bond, ctas, _ptr(x, ctypes.c_double), _ptr(y, ctypes.c_double))
    assert rc == 0
    for v in range(nv):
        ref = orc.apply_u1(N, states, bonds, J, np.ascontiguousarray(x[:, v]))
        # a row adds at most 2 nb + 1 terms, each rounded once: far inside 1e-12 of its magnitude
        assert np.abs(y[:, v] - ref).max() <= 1e-12 * max(1.0, np.abs(J).sum()) * np.abs(x).max()


@pytest.mark.parametrize("name,N,most", [("chain", 24, 3), ("chain", 28, 3), ("ladder", 28, 3), ("square4x6", 24, 3),
                                         ("square4x8", 32, 4), ("square6x6", 36, 6), ("chain", 40, 4)])
def test_windows_of_the_lattices(win, name, N, most):
    """The lattices' windows hold every bond in as few passes as their geometry allows (rows of a window times
    the sites of a row at most 12); the lowest four sites are in a window together or not at all."""
    if name == "chain":
        bonds = W.chain(N)
    elif name == "ladder":
        bonds = W.ladder(N // 2, 2)
    else:
        bonds = W.square_j1j2(int(name[6]), int(name[8]))[0]
    bonds = np.ascontiguousarray(bonds, dtype=np.int32)
    out = np.zeros((16, 13), dtype=np.int32)
    n = win.window_sites(N, N // 2, _ptr(bonds, ctypes.c_int32), len(bonds), _ptr(out, ctypes.c_int32), 16)
    assert n <= most
    sets = [set(int(v) for v in row[1:] if v >= 0) for row in out[:n]]
    assert all(len(s) <= 12 and len(s & {0, 1, 2, 3}) in (0, 4) for s in sets)
    assert all(bool(row[0]) == (0 in s) for row, s in zip(out[:n], sets))
    assert all(any({int(i), int(j)} <= s for s in sets) for i, j in bonds)
