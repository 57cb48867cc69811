"""The other ways through a solve on a cluster of blocks (wide sizes): every one of them against the
same instances in a batch that runs on one block each."""
import numpy as np
import pytest
import torch

from paper_1703_00443_gb300 import inputs, qp_backward, qp_forward
from tests.helpers import oracle_solve_and_grad, rel_err

DEV = "cuda:0"
pytestmark = pytest.mark.gpu
# batches that take clusters of 8, 4 and 2 blocks, and one block each (152 SMs)
BATCHES = (1, 20, 40, 80)


def _run(data, g, B, options=None, backward=True):
    """(status, iterations, z, λ, ν, gradients) of the last of B copies."""
    T = [torch.from_numpy(np.ascontiguousarray(np.repeat(x[None], B, 0))).to(DEV) for x in data]
    f = qp_forward(*T, options=options)
    out = [f.status, f.iters, f.z, f.lam, f.nu]
    if backward:
        out += list(qp_backward(f, torch.from_numpy(np.repeat(g[None], B, 0)).to(DEV)))
    torch.cuda.synchronize()
    return [t[-1].cpu() for t in out]


def _same(a, b):
    return all(torch.equal(torch.nan_to_num(x.double(), nan=7e77), torch.nan_to_num(y.double(), nan=7e77))
               for x, y in zip(a, b))


def _plain(n, p, m, dtype=np.float32):
    batch = inputs.random_batch(1, n, p, m, workload=inputs.WL_PLAIN, dtype=dtype)
    g = inputs.upstream_grad(1, n, workload=inputs.WL_PLAIN, dtype=dtype)
    return batch, g


@pytest.mark.parametrize("n,m", [(352, 0), (400, 60)])
def test_equality_constrained(n, m):
    """No inequality: the first block finishes alone after the setup."""
    batch, g = _plain(n, 0, m)
    data = [x[0] for x in (batch.Q, batch.q, batch.G, batch.h, batch.A, batch.b)]
    outs = [_run(data, g[0], B) for B in BATCHES]
    assert int(outs[0][0]) == 0 and all(_same(outs[0], o) for o in outs[1:])
    sols, refs = oracle_solve_and_grad(batch, g, [0])
    assert rel_err(outs[0][2].double().numpy()[None], [sols[0]["z"]]).max() <= 1e-5
    assert rel_err(outs[0][6].double().numpy()[None], [refs[0]["dq"]],
                   1e-3 * np.linalg.norm(g, axis=1)).max() <= 1e-4


@pytest.mark.parametrize("n,p,m,dtype", [
    (352, 120, 4, np.float32),       # register-tile Cholesky, one slot a thread
    (356, 170, 9, np.float32),       # two slots
    (480, 160, 40, np.float64),      # blocked Cholesky and sweep in FP64, the sweep's panels in global memory
    (352, 40, 4, np.float64),        # register-tile Cholesky in FP64
])
def test_factorisations(n, p, m, dtype):
    batch, g = _plain(n, p, m, dtype)
    data = [x[0] for x in (batch.Q, batch.q, batch.G, batch.h, batch.A, batch.b)]
    outs = [_run(data, g[0], B) for B in BATCHES]
    assert int(outs[0][0]) == 0 and all(_same(outs[0], o) for o in outs[1:])
    sols, refs = oracle_solve_and_grad(batch, g, [0])
    ztol, gtol = (1e-5, 1e-4) if dtype == np.float32 else (1e-9, 1e-8)
    assert rel_err(outs[0][2].double().numpy()[None], [sols[0]["z"]]).max() <= ztol
    assert rel_err(outs[0][6].double().numpy()[None], [refs[0]["dq"]],
                   1e-3 * np.linalg.norm(g, axis=1)).max() <= gtol
