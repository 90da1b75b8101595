"""exp(-i t T) e_1 through the QR eigenpairs of a tridiagonal: whole, split, graded and degenerate ones."""
import numpy as np
import pytest

from test_host_tridiag import _d, _p, _T, lib  # noqa: F401  (the fixture)


@pytest.mark.parametrize("t", [0.05, 2.0, -7.0])
@pytest.mark.parametrize("kind", ["random", "split", "graded", "constant", "diagonal"])
@pytest.mark.parametrize("m", [1, 2, 3, 40, 120])
def test_real_time(lib, m, kind, t):
    rng = np.random.default_rng(m)
    a, b = rng.standard_normal(m) - 1.0, rng.uniform(0.1, 3.0, m)
    if kind == "split":
        b[m // 2] = 0.0
    elif kind == "graded":
        a, b = a * 10.0 ** (-np.arange(m) / 3.0), b * 10.0 ** (-np.arange(m) / 3.0)
    elif kind == "constant":
        a[:], b[:] = 0.0, 1.0
    elif kind == "diagonal":
        b[:] = 0.0
    a, b = _d(a), _d(b)
    cr, ci = _d(np.zeros(m)), _d(np.zeros(m))
    lib.shim_expm_e1(m, _p(a), _p(b), 0.0, t, _p(cr), _p(ci))
    w, V = np.linalg.eigh(_T(a, b[: m - 1] if len(b) > m - 1 else b))
    want = V @ (np.exp(-1j * t * w) * V[0])
    # two backward stable eigensolvers: each some 2^-53 m |T| off, times t in the phases
    assert np.abs(cr + 1j * ci - want).max() <= 1e-15 * m * (1.0 + abs(t) * np.abs(w).max())
