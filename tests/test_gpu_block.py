"""The block kernel where it is taken: FP32 on dense graphs of 20 to 23 sites, and FP64 from 24 sites on when the
window passes' workspace cannot be had."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import _lib, workloads as W

pytestmark = pytest.mark.gpu


def _complete(n):
    return np.array([(i, j) for i in range(n) for j in range(i)], dtype=np.int32)


# on both sides of the lines: long prefix blocks with 76 bonds and more, few rows with 80 and more
@pytest.mark.parametrize("N,nup,nb", [(23, 11, 75), (23, 12, 77), (23, 11, 253), (21, 10, 210), (22, 3, 79), (22, 3, 81),
                                      (20, 1, 120), (20, 18, 190), (23, 22, 253), (20, 10, 190)])
def test_fp32_below_24_sites(orc, N, nup, nb):
    A = api()
    bonds = _complete(N) if nb == N * (N - 1) // 2 else W.random_bonds(N, nb, 7)
    J = W.uniform_couplings(nb, 3, -1.0, 1.5)
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    x = np.random.default_rng(1).standard_normal(st.size)
    y = orc.apply_u1(N, st, bonds, J, x)
    # FP32: inputs rounded to FP32 and at most 254 rounded additions per row, each within 2^-24 of its partial sum,
    # couplings of both signs summed in FP32 on the diagonal: inside 1e-5 in the 2-norm
    assert rel_l2(ham.apply(torch.from_numpy(x).cuda().float()).cpu().numpy(), y) <= 1e-5
    assert rel_l2(ham.apply(torch.from_numpy(x).cuda()).cpu().numpy(), y) <= 1e-12
    e32 = ham.lanczos(max_iter=40, seed=3, storage=torch.float32)["evals"]
    e64 = ham.lanczos(max_iter=40, seed=3)["evals"]
    assert abs(e32[0] - e64[0]) <= 1e-4 * np.abs(J).sum()


@pytest.mark.parametrize("name", ["square4x6", "chain24"])
def test_fp64_without_the_workspace(orc, name):
    A = api()
    bonds = W.square_j1j2(4, 6)[0] if name == "square4x6" else W.chain(24)
    J = W.uniform_couplings(len(bonds), 3)
    st = orc.enumerate_states(24, 8)
    ham = A.Hamiltonian(A.Basis(24, 8, bonds), J)
    x = np.random.default_rng(2).standard_normal(st.size)
    xd = torch.from_numpy(x).cuda()
    y = orc.apply_u1(24, st, bonds, J, x)
    out = torch.full_like(xd, float("nan"))
    if name == "chain24":  # prefix passes: their tables first, on the first product
        ham.apply(xd, out=out)
        ham = A.Hamiltonian(ham.basis, J)
    _lib.lib().xd_debug_fail_alloc(0)
    try:
        ham.apply(xd, out=out)
    finally:
        _lib.lib().xd_debug_fail_alloc(-1)
    assert rel_l2(out.cpu().numpy(), y) <= 1e-12
    out.fill_(float("nan"))
    ham.apply(xd, out=out)  # the next product takes the workspace
    assert rel_l2(out.cpu().numpy(), y) <= 1e-12
