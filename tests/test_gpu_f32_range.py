"""FP32 products of entries near the top of the range: finite where J/2 times an entry, and the row's sum, are."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nvec", [1, 8])
@pytest.mark.parametrize("name", ["square4x6", "ladder24", "square4x5"])
def test_large_entries_do_not_overflow(orc, name, nvec):
    """Entries of 0.5e38 to 1e38 and J = 0.05: with F of the at most 96 bonds flipping a row is at most (0.025 F +
    0.0125 |96 - 2 F|) 1e38 <= 2.4e38, while a sum of a few entries exceeds the largest FP32 number, 3.4e38."""
    A = api()
    N, nup, bonds = {"square4x6": (24, 8, W.square_j1j2(4, 6)[0]), "ladder24": (24, 9, W.ladder(12, 2)),
                     "square4x5": (20, 10, W.square_j1j2(4, 5)[0])}[name]
    J = np.full(len(bonds), 0.05)
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    X = (np.random.default_rng(5).uniform(0.5, 1.0, (st.size, nvec)) * 1e38).astype(np.float32)
    y = ham.apply(torch.from_numpy(X).cuda().squeeze(1) if nvec == 1 else torch.from_numpy(X).cuda()).cpu().numpy()
    assert np.isfinite(y).all()
    Y = np.stack([orc.apply_u1(N, st, bonds, J, X[:, k].astype(np.float64)) for k in range(nvec)], 1).reshape(y.shape)
    # at most a hundred or so rounded operations per row, each within 2^-24 of its partial sum, all of one sign but
    # the diagonal: inside 1e-5
    assert rel_l2(y.astype(np.float64) / 1e38, Y / 1e38) <= 1e-5
