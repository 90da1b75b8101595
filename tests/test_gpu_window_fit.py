"""Dense graphs on the GPU whose window tables, listed coupling by coupling, do not fit in shared memory."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _dense25():
    """290 bonds on 25 sites, four coupling values: the lists of one pass take 232 to 254 KB in every value type."""
    bonds = W.random_bonds(25, 290, 20)
    return bonds, np.array([1.0, 0.5, 0.25, 0.75])[np.random.default_rng(20).integers(0, 4, len(bonds))]


def test_dense_graph_in_a_batch_and_alone(orc):
    """The product in FP64, in FP32 and on eight FP32 vectors, alone and in a batch beside a chain."""
    A = api()
    bonds, J = _dense25()
    st = orc.enumerate_states(25, 8)
    ham = A.Hamiltonian(A.Basis(25, 8, bonds), J)
    chain = A.Hamiltonian(A.Basis(18, 9, W.chain(18)), np.ones(18))
    st2 = orc.enumerate_states(18, 9)
    rng = np.random.default_rng(3)
    X, X2 = rng.standard_normal((st.size, 8)), rng.standard_normal((st2.size, 8))
    Y = np.stack([orc.apply_u1(25, st, bonds, J, np.ascontiguousarray(X[:, k])) for k in range(8)], 1)
    Y2 = np.stack([orc.apply_u1(18, st2, W.chain(18), np.ones(18), np.ascontiguousarray(X2[:, k])) for k in range(8)], 1)
    assert rel_l2(ham.apply(torch.from_numpy(np.ascontiguousarray(X[:, 0])).cuda()).cpu().numpy(), Y[:, 0]) <= 1e-12
    # FP32: inputs rounded to FP32 (relative 2^-25 on average) and at most a few hundred rounded additions per
    # row, each within 2^-24 of its partial sum: far inside 1e-6 in the 2-norm
    x = torch.from_numpy(X.astype(np.float32)).cuda()
    assert rel_l2(ham.apply(x[:, 0].contiguous()).cpu().numpy(), Y[:, 0]) <= 1e-6
    assert rel_l2(ham.apply(x).cpu().numpy(), Y) <= 1e-6
    x2 = torch.from_numpy(X2.astype(np.float32)).cuda()
    y, y2 = torch.full_like(x, float("nan")), torch.full_like(x2, float("nan"))
    A.batch_apply([ham, chain], [x, x2], [y, y2])
    assert rel_l2(y.cpu().numpy(), Y) <= 1e-6
    assert rel_l2(y2.cpu().numpy(), Y2) <= 1e-6
