"""The representative search of rings (chains with rotations and reflections) against every image, on the CPU."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2505_02901_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ring") / "libring.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", so,
                           os.path.join(HERE, "host_ring_shim.cpp")])
    return ctypes.CDLL(so)


def _images(N, dih, s):
    """[elements][words]: T_n s moves bit i + n to i, R_n s moves bit n - i to i (mod N)."""
    out = []
    for refl in range(dih + 1):
        for n in range(N):
            w = np.zeros_like(s)
            for i in range(N):
                j = (n - i) % N if refl else (i + n) % N
                w |= ((s >> np.uint64(j)) & np.uint64(1)) << np.uint64(i)
            out.append(w)
    return np.array(out)


@pytest.mark.parametrize("dih", [0, 1])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 9, 12, 31, 32, 33, 36, 63, 64])
def test_every_image(shim, N, dih):
    rng = np.random.default_rng(N)
    if N <= 12:
        s = np.arange(1 << N, dtype=np.uint64)
    else:
        mask = np.uint64((1 << N) - 1)
        full = rng.integers(0, 1 << 63, size=(4, 500), dtype=np.uint64) * np.uint64(2) + rng.integers(0, 2, 500, dtype=np.uint64)
        per = [sum(((int(v) & ((1 << p) - 1)) << k) for k in range(0, 64, p)) & ((1 << 64) - 1)
               for p in range(1, 33) for v in full[0, :6]]  # periodic words: stabilisers
        few = [(1 << int(a)) | (1 << int(b)) for a, b in rng.integers(0, N, size=(100, 2))]
        s = np.concatenate([full[0], full[1] & full[2], full[1] & full[2] & full[3], full[1] | full[2],
                            np.array(per + few, dtype=np.uint64), np.array([0, (1 << N) - 1], dtype=np.uint64)]) & mask
    rep, cand, cnt = np.zeros_like(s), np.zeros(s.size, np.int32), np.zeros(s.size, np.int32)
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (s, rep, cand, cnt)]
    shim.shim_ring_orbit(N, dih, ctypes.c_int64(s.size), *p)
    im = _images(N, dih, s)
    assert (rep == im.min(0)).all()
    assert (cnt == (im == rep).sum(0)).all()
    assert (im[cand, np.arange(s.size)] == rep).all()
