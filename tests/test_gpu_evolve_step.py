"""The fused step of the evolution's second pass at the edges of its grid: one element, less and more than a CTA."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t,tau", [(0.7, 0.0), (0.0, 0.4), (0.5, 0.2)])
@pytest.mark.parametrize("N,nup", [(3, 0), (2, 1), (7, 3), (10, 5), (11, 5)])
def test_against_dense(orc, N, nup, t, tau):
    A = api()
    bonds = W.chain(N) if N > 2 else np.array([(0, 1)], dtype=np.int32)
    J = W.uniform_couplings(len(bonds), 3)
    st = orc.enumerate_states(N, nup)
    w, V = np.linalg.eigh(orc.dense_u1(N, st, bonds, J))
    psi = orc.rng_normal(5, 0, st.size) + 1j * orc.rng_normal(6, 0, st.size)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    got, _ = ham.evolve(torch.from_numpy(psi).cuda(), t=t, tau=tau, max_iter=100, tol=1e-13)
    want = V @ (np.exp(-(tau + 1j * t) * w) * (V.T @ psi))
    assert rel_l2(got.cpu().numpy(), want) <= 1e-11  # the estimate stops at 1e-13; its rounding is far below 1e-11
