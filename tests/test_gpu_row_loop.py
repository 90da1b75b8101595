"""FP64 products of the row loop: flips walked as set bits (32 bonds at a time) and the diagonal in integers, at the
edges of both: bond counts around 32, more bonds than the integer table holds, couplings without a unit."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", ["one", "spread", "tiny"])
@pytest.mark.parametrize("N,nup,nb", [(2, 1, 1), (9, 4, 31), (11, 5, 32), (11, 5, 33), (13, 6, 65), (16, 8, 40), (23, 3, 60),
                                      (10, 5, 2100)])
def test_fp64_products(orc, N, nup, nb, scale):
    A = api()
    pairs = W.random_bonds(N, min(nb, N * (N - 1) // 2), 3) if N > 2 else np.array([(0, 1)], dtype=np.int32)
    bonds = np.ascontiguousarray(pairs[np.arange(nb) % len(pairs)])  # repeated pairs beyond the distinct ones
    J = W.uniform_couplings(nb, 4, -1.0, 1.5)
    if scale == "spread":
        J = J * 10.0 ** -(np.arange(nb) % 25)
    elif scale == "tiny":
        J = J * 2.0 ** -1000
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    X = np.random.default_rng(2).standard_normal((st.size, 8))
    for nv in (1, 2, 4, 8):
        x = np.ascontiguousarray(X[:, :nv] if nv > 1 else X[:, 0])
        got = ham.apply(torch.from_numpy(x).cuda()).cpu().numpy().reshape(st.size, nv)
        want = np.stack([orc.apply_u1(N, st, bonds, J, np.ascontiguousarray(X[:, k])) for k in range(nv)], 1)
        # nb rounded terms of one row, each within 2^-53 of sum |J| |x|, which cancellation takes down to no less
        # than about 1/100 of it for random signs: 100 sqrt(2100) 2^-53 < 1e-12
        f = 2.0 ** 1000 if scale == "tiny" else 1.0
        assert rel_l2(got * f, want * f) <= 1e-12
