"""Per-bond bilinear forms at the edges of the kernel's tiles (512 rows), of its launches (64 bonds) and of the range in
which the diagonal sums run in integers."""
import numpy as np
import pytest
import torch

from gpu_common import api
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0, 500, -500, -540])  # p near 1, 2^1000, 2^-1000 and 2^-1080 (subnormal)
@pytest.mark.parametrize("N,nup,nb", [(2, 1, 1), (12, 4, 15), (12, 4, 16), (13, 4, 17), (23, 2, 63), (12, 6, 64), (17, 5, 65),
                                      (18, 9, 129)])
def test_edges(orc, N, nup, nb, scale):
    A = api()
    bonds = W.random_bonds(N, nb, 3) if nb > 1 else np.array([(0, 1)], dtype=np.int32)
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), np.ones(nb))
    g, x = orc.rng_normal(1, 0, st.size), orc.rng_normal(2, 0, st.size)
    g[st.size // 2:] *= 2.0 ** -30  # a tile's largest product far above the others
    ref = orc.bond_forms(N, st, bonds, g, x)
    f = 2.0 ** scale  # exact
    dJ = ham.bilinear(torch.from_numpy(g * f).cuda(), torch.from_numpy(x * f).cuda()).cpu().numpy()
    # sums of dim products, each within a few 2^-53 of sum |g||x|; subnormal products: dim roundings of 2^-1075 each
    bound = 1e-14 * np.abs(g).sum() * np.abs(x).max()
    if scale == -540:
        bound += st.size * 2.0 ** (1080 - 1074)
    assert np.abs(dJ / f / f - ref).max() <= bound


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_not_finite_stays_so(bad):
    A = api()
    bonds = W.chain(12)
    ham = A.Hamiltonian(A.Basis(12, 6, bonds), np.ones(12))
    x = torch.ones(924, dtype=torch.float64, device="cuda")
    g = torch.ones_like(x)
    x[700] = bad
    assert not torch.isfinite(ham.bilinear(g, x)).any()
    x[:] = 0.0
    x[900] = 2.0  # the first tile has no product
    assert torch.isfinite(ham.bilinear(g, x)).all()
