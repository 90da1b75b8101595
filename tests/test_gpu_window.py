"""The window passes on the GPU at the edges of their range: blocks of few up or few down spins (tiles of one
row, units of one word), graphs with many windows and with lists that carry their bond, vectors that are not
16-byte aligned, eight vectors, and both FP64 arithmetics."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _graph(name):
    if name == "ladder24":
        return 24, W.ladder(12, 2)
    if name == "square4x6":
        return 24, W.square_j1j2(4, 6)[0]
    if name == "triangular5":
        return 25, W.triangular(5)[0]
    if name == "random26":
        return 26, W.random_bonds(26, 70, 11)
    return 24, np.array([(i, j) for i in range(24) for j in range(i)], dtype=np.int32)  # complete24


CASES = [("square4x6", 1), ("square4x6", 2), ("square4x6", 23), ("square4x6", 12), ("ladder24", 9), ("triangular5", 12),
         ("random26", 5), ("random26", 21), ("complete24", 6)]


@pytest.mark.parametrize("couplings", ["uniform", "random"])
@pytest.mark.parametrize("name,nup", CASES)
def test_products_match_oracle(orc, name, nup, couplings):
    A = api()
    N, bonds = _graph(name)
    nb = len(bonds)
    J = np.where(np.arange(nb) % 3 == 0, 0.5, 1.0) if couplings == "uniform" else W.uniform_couplings(nb, 5, -1.0, 1.5)
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    X = np.random.default_rng(7).standard_normal((st.size, 8))
    Y = np.stack([orc.apply_u1(N, st, bonds, J, np.ascontiguousarray(X[:, k])) for k in range(8)], 1)
    nan = float("nan")
    y = torch.full((st.size,), nan, dtype=torch.float64, device="cuda")
    ham.apply(torch.from_numpy(np.ascontiguousarray(X[:, 0])).cuda(), out=y)
    assert rel_l2(y.cpu().numpy(), Y[:, 0]) <= 1e-12
    # FP32: inputs rounded to FP32 (relative 2^-25 on average) and at most a few hundred rounded additions per
    # row, each within 2^-24 of its partial sum: far inside 1e-6 in the 2-norm
    X32 = X.astype(np.float32)
    buf = torch.full((st.size + 1,), nan, dtype=torch.float32, device="cuda")
    buf[1:] = torch.from_numpy(np.ascontiguousarray(X32[:, 0]))
    y32 = torch.full((st.size + 1,), nan, dtype=torch.float32, device="cuda")
    ham.apply(buf[1:], out=y32[1:])  # four bytes past a 16-byte boundary
    assert rel_l2(y32[1:].cpu().numpy(), Y[:, 0]) <= 1e-6
    for shift in (0, 1):  # eight vectors, aligned and not
        b8 = torch.full((st.size * 8 + shift,), nan, dtype=torch.float32, device="cuda")
        b8[shift:] = torch.from_numpy(X32).reshape(-1).cuda()
        y8 = torch.full_like(b8, nan)
        ham.apply(b8[shift:].view(st.size, 8), out=y8[shift:].view(st.size, 8))
        assert rel_l2(y8[shift:].view(st.size, 8).cpu().numpy(), Y) <= 1e-6


def test_new_couplings_change_the_lists(orc):
    """Couplings of another pattern of equal values (lists coupling by coupling, then with the bond, then back)."""
    A = api()
    N, bonds = _graph("square4x6")
    st = orc.enumerate_states(N, 5)
    ham = A.Hamiltonian(A.Basis(N, 5, bonds), np.ones(len(bonds)))
    x = np.random.default_rng(8).standard_normal(st.size)
    xd = torch.from_numpy(x).cuda()
    for J in (W.square_j1j2(4, 6)[1], W.uniform_couplings(len(bonds), 9), W.uniform_couplings(len(bonds), 10),
              np.full(len(bonds), -0.25), np.arange(len(bonds)) * 0.125):
        ham.set_couplings(J)
        assert rel_l2(ham.apply(xd).cpu().numpy(), orc.apply_u1(N, st, bonds, J, x)) <= 1e-12
