"""Two threads with blocks of different sizes: launches of one kernel with different amounts of shared memory."""
import threading

import numpy as np
import pytest
import torch

from gpu_common import api
from paper_2505_02901_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _hams(A, kind):
    if kind == "symmetric":  # translations of rings of 12 and of 16 sites
        out = []
        for n in (12, 16):
            perms = np.array([[(i + r) % n for i in range(n)] for r in range(n)], dtype=np.int32)
            out.append(A.Hamiltonian(A.Basis(n, n // 2, W.chain(n), (perms, np.ones(n))), np.ones(n)))
        return out
    # 24 sites, sparse graphs: prefix passes in FP64, the batched layout in FP32, with tables of 24 and of 30 bonds
    return [A.Hamiltonian(A.Basis(24, 12, b), np.ones(len(b))) for b in (W.chain(24), W.random_bonds(24, 30, 1))]


@pytest.mark.parametrize("kind,dtype", [("sparse24", torch.float64), ("sparse24", torch.float32), ("symmetric", torch.float64)])
def test_products_in_two_threads(kind, dtype):
    A = api()
    hams = _hams(A, kind)
    xs = [torch.randn(h.dim, dtype=dtype, device="cuda") for h in hams]
    want = [h.apply(x).clone() for h, x in zip(hams, xs)]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(2)

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                y = torch.empty_like(xs[k])
                start.wait()
                for _ in range(4000):
                    hams[k].apply(xs[k], out=y)
                torch.cuda.current_stream().synchronize()
                if not torch.equal(y, want[k]):
                    errors.append("thread %d: another result" % k)
        except Exception as e:  # noqa: BLE001
            errors.append("thread %d: %s" % (k, e))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors
