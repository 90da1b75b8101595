"""New couplings on a handle in use: a failed allocation changes nothing, and products in flight keep their tables."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import _lib, workloads as W

pytestmark = pytest.mark.gpu


def test_failed_allocation_leaves_the_handle(orc):
    A = api()
    bonds = W.square_j1j2(4, 6)[0]
    nb = len(bonds)
    st = orc.enumerate_states(24, 8)
    ham = A.Hamiltonian(A.Basis(24, 8, bonds), np.ones(nb))
    x = np.random.default_rng(1).standard_normal(st.size)
    xd = torch.from_numpy(x).cuda()
    x32 = xd.float()
    ones = orc.apply_u1(24, st, bonds, np.ones(nb), x)
    assert rel_l2(ham.apply(xd).cpu().numpy(), ones) <= 1e-12  # allocates the workspace
    J = W.uniform_couplings(nb, 3)  # another pattern of equal couplings: other lists
    _lib.lib().xd_debug_fail_alloc(0)
    try:
        with pytest.raises(_lib.XDError):
            ham.set_couplings(J)
    finally:
        _lib.lib().xd_debug_fail_alloc(-1)
    assert rel_l2(ham.apply(xd).cpu().numpy(), ones) <= 1e-12
    # FP32: a few dozen rounded additions per row, each within 2^-24 of its partial sum
    assert rel_l2(ham.apply(x32).cpu().numpy(), ones) <= 1e-6
    ham.set_couplings(J)
    assert rel_l2(ham.apply(xd).cpu().numpy(), orc.apply_u1(24, st, bonds, J, x)) <= 1e-12


def test_products_in_flight_keep_their_tables(orc):
    """Products on another stream, still running when the couplings change, are those of the couplings before."""
    A = api()
    bonds = W.square_j1j2(4, 6)[0]
    nb = len(bonds)
    ham = A.Hamiltonian(A.Basis(24, 12, bonds), np.ones(nb))
    x = torch.randn(ham.dim, dtype=torch.float64, device="cuda")
    want = ham.apply(x).clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    ys = [torch.empty_like(x) for _ in range(40)]
    with torch.cuda.stream(side):
        for y in ys:
            ham.apply(x, out=y)
    ham.set_couplings(W.uniform_couplings(nb, 3))
    torch.cuda.synchronize()
    assert all(torch.equal(y, want) for y in ys)
