"""The cooperative Lanczos passes of small blocks: one tile and several, a last tile that is nearly empty, the flips
of a row kept in shared memory and (too many bonds, too many rows) looked up at each step."""
import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _block(name):
    if name == "complete17":  # 136 bonds: the flips of 256 rows do not fit
        return 17, 8, np.array([(i, j) for i in range(17) for j in range(i)], dtype=np.int32)
    if name == "square4x5":  # 722 tiles: more than fit with their flips
        return 20, 10, W.square_j1j2(4, 5)[0]
    N, nup = {"rows3": (3, 1), "rows252": (10, 5), "rows462": (11, 5), "rows924": (12, 6), "rows1287": (13, 5),
              "rows7315": (22, 4)}[name]
    return N, nup, W.chain(N)


@pytest.mark.parametrize("storage", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", ["rows3", "rows252", "rows462", "rows924", "rows1287", "rows7315", "square4x5", "complete17"])
def test_second_pass_rebuilds_the_first(orc, name, storage):
    A = api()
    N, nup, bonds = _block(name)
    J = W.uniform_couplings(len(bonds), 9, 0.3, 1.2)
    st = orc.enumerate_states(N, nup)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    m = min(8, st.size - 1)
    _, psi, info = ham.ground_state(max_iter=m, seed=4, storage=storage)
    a, b = np.asarray(info["alpha"]), np.asarray(info["beta"])
    m = len(a)
    c = np.linalg.eigh(np.diag(a) + np.diag(b[:m - 1], 1) + np.diag(b[:m - 1], -1))[1][:, 0]
    v = orc.rng_normal(4, 0, st.size)
    v, vp, ref = v / np.linalg.norm(v), np.zeros(st.size), np.zeros(st.size)
    for k in range(m):
        ref += c[k] * v
        if k < m - 1:
            w = orc.apply_u1(N, st, bonds, J, v) - a[k] * v - (b[k - 1] * vp if k else 0.0)
            vp, v = v, w / b[k]
    p = psi.double().cpu().numpy()
    # m <= 8 steps of the same recurrence: a step's rounding (2^-53 or 2^-24 relative) is carried on with a factor of
    # order |H| / beta < 10 a step, at most 10^7 for the first; a wrong flip or coefficient shows at 0.1 or more
    assert rel_l2(p * np.sign(p @ ref), ref) <= (1e-9 if storage == torch.float64 else 1e-2)
