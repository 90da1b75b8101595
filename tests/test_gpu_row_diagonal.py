"""The row loop's FP32 diagonal: products with random couplings are as exact as those with uniform ones."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e34])
@pytest.mark.parametrize("N,nup,nb", [(23, 11, 103), (21, 5, 60), (16, 8, 40), (22, 3, 200)])
def test_random_couplings(orc, N, nup, nb, scale):
    """sum J/4 and the sum of J/2 over the flipping bonds are some tens of J and their difference a few: in FP32 sums
    the diagonal misses 3e-6 J and the product 5e-7.  In units of 2^-30 of the sum it misses 2e-8 J; what is left is
    the rounding of x, of J/2 and of some fifty additions, half of 2^-24 each: 2e-7 in the 2-norm at the most."""
    A = api()
    bonds = W.random_bonds(N, nb, 5)
    J = W.uniform_couplings(nb, 3) * scale
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    X = np.random.default_rng(4).standard_normal((st.size, 8)).astype(np.float32)
    Y = np.stack([orc.apply_u1(N, st, bonds, J, X[:, k].astype(np.float64)) for k in range(8)], 1)
    for nvec in (1, 2, 4, 8):
        x = torch.from_numpy(np.ascontiguousarray(X[:, :nvec])).cuda()
        y = ham.apply(x.squeeze(1) if nvec == 1 else x).cpu().numpy().reshape(-1, nvec)
        assert rel_l2(y.astype(np.float64) / scale, Y[:, :nvec] / scale) <= 2.5e-7
    x = torch.from_numpy(X).cuda()
    y = torch.empty_like(x)
    A.batch_apply([ham], [x], [y])
    assert rel_l2(y.cpu().numpy().astype(np.float64) / scale, Y / scale) <= 2.5e-7
