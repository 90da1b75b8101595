"""Blocks of 24 sites and more on both sides of the row count from which the window and block kernels take them."""
import itertools

import numpy as np
import pytest
import torch

from gpu_common import api, rel_l2
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _graph(name, N):
    return {"chain": W.chain(N), "ladder": W.ladder(N // 2, 2), "random": W.random_bonds(N, 3 * N, 4)}[name]


def _dense(N, nup, bonds, J):
    """The matrix of a block of few rows, words ascending (Eq. 1)."""
    words = sorted(sum(1 << i for i in c) for c in itertools.combinations(range(N), nup))
    at = {w: k for k, w in enumerate(words)}
    H = np.zeros((len(words), len(words)))
    for k, w in enumerate(words):
        for (i, j), v in zip(bonds, J):
            if ((w >> i) ^ (w >> j)) & 1:
                H[k, k] -= 0.25 * v
                H[k, at[w ^ (1 << int(i)) ^ (1 << int(j))]] += 0.5 * v
            else:
                H[k, k] += 0.25 * v
    return H


@pytest.mark.parametrize("name", ["chain", "ladder", "random"])
@pytest.mark.parametrize("N,nup", [(24, 1), (28, 2), (40, 1), (40, 2), (40, 0), (24, 24), (30, 28)])
def test_few_rows(name, N, nup):
    """Every width and type against the matrix, and the lowest eigenvalue."""
    A = api()
    bonds = _graph(name, N)
    J = W.uniform_couplings(len(bonds), 5, -1.0, 1.5)
    H = _dense(N, nup, bonds.tolist(), J)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    X = np.random.default_rng(2).standard_normal((len(H), 8))
    x = torch.from_numpy(X).cuda()
    for nvec in (1, 2, 8):
        xs = x[:, 0].contiguous() if nvec == 1 else x[:, :nvec].contiguous()
        want = H @ (X[:, 0] if nvec == 1 else X[:, :nvec])
        # a row adds at most nb + 1 terms: each rounded once, far inside 1e-13 (FP64) and 1e-5 (FP32) in the 2-norm
        assert rel_l2(ham.apply(xs).cpu().numpy(), want) <= 1e-13
        assert rel_l2(ham.apply(xs.float()).cpu().numpy(), want) <= 1e-5
    y = torch.empty_like(x, dtype=torch.float32)
    A.batch_apply([ham], [x.float()], [y])
    assert rel_l2(y.cpu().numpy(), H @ X) <= 1e-5
    evals = np.atleast_1d(ham.lanczos(max_iter=min(200, len(H)), seed=3)["evals"])
    assert abs(evals[0] - np.linalg.eigvalsh(H)[0]) <= 1e-9 * max(1.0, np.abs(J).sum())


@pytest.mark.parametrize("couplings", ["uniform", "random"])
@pytest.mark.parametrize("name,N,nup", [("chain", 30, 6), ("ladder", 30, 24), ("random", 30, 6), ("chain", 40, 5),
                                        ("random", 40, 35), ("ladder", 40, 5)])
def test_windows_of_few_up_or_down_spins(name, N, nup, couplings):
    """Just above the line (593,775 and 658,008 rows): tiles of few rows and units of one word, against the row loop,
    which two FP64 vectors take at every size."""
    A = api()
    bonds = _graph(name, N)
    J = np.ones(len(bonds)) if couplings == "uniform" else W.uniform_couplings(len(bonds), 6, -1.0, 1.5)
    ham = A.Hamiltonian(A.Basis(N, nup, bonds), J)
    x = torch.randn(ham.dim, 8, dtype=torch.float64, device="cuda")
    want = torch.cat([ham.apply(x[:, k:k + 2].contiguous()) for k in range(0, 8, 2)], 1)
    # FP64: both within a few hundred roundings of 2^-45 of the terms; FP32: inputs and sums rounded to 2^-24
    y = ham.apply(x[:, 0].contiguous())
    assert float((y - want[:, 0]).norm() / want[:, 0].norm()) <= 1e-12
    y = ham.apply(x[:, 0].float().contiguous()).double()
    assert float((y - want[:, 0]).norm() / want[:, 0].norm()) <= 1e-6
    y = ham.apply(x.float()).double()
    assert float((y - want).norm() / want.norm()) <= 1e-6
