"""Wide sizes of the global-memory path (n + neq >= 352 after padding): an instance is shared by a
cluster of blocks whose number follows the batch, and its results must not depend on it."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1703_00443_gb300 import _lib, inputs, qp_backward, qp_forward
from paper_1703_00443_gb300.packed import PackedBatch
from tests.helpers import oracle_solve_and_grad, rel_err

DEV = "cuda:0"
# first wide size, odd inequality counts (unaligned rows of the Schur complement), the blocked
# Cholesky (more than 176 inequalities) with a remainder block
SIZES = [(352, 24, 0), (345, 21, 7), (340, 205, 13)]


def _solve(idx, n, p, m):
    batch = inputs.random_batch(2, n, p, m, workload=inputs.WL_PLAIN)
    g = inputs.upstream_grad(2, n, workload=inputs.WL_PLAIN)
    T = [torch.from_numpy(np.ascontiguousarray(x[idx])).to(DEV)
         for x in (batch.Q, batch.q, batch.G, batch.h, batch.A, batch.b)]
    f = qp_forward(*T)
    grads = qp_backward(f, torch.from_numpy(np.ascontiguousarray(g[idx])).to(DEV))
    torch.cuda.synchronize()
    return batch, g, f, grads


@pytest.mark.gpu
@pytest.mark.parametrize("n,p,m", SIZES)
def test_results_do_not_depend_on_the_cluster_size(n, p, m):
    """Batches of 1, 20, 40 and 80 take clusters of 8, 4, 2 and 1 blocks; bit-identical results,
    and z* and dq of the single instance within the FP32 path's tolerances of the oracle."""
    batch, g, f1, g1 = _solve([0], n, p, m)
    assert (f1.status == 0).all()
    sols, refs = oracle_solve_and_grad(batch, g, [0])
    assert rel_err(f1.z.double().cpu().numpy(), [sols[0]["z"]]).max() <= 1e-5
    assert rel_err(g1[1].double().cpu().numpy(), [refs[0]["dq"]],
                   1e-3 * np.linalg.norm(g[:1], axis=1)).max() <= 1e-4
    for B in (20, 40, 80):
        _, _, f, gr = _solve([i % 2 for i in range(B)], n, p, m)
        for a, b in zip((f1.z, f1.lam, f1.nu, f1.iters, *g1), (f.z, f.lam, f.nu, f.iters, *gr)):
            assert torch.equal(a[0], b[0]) and (B < 40 or torch.equal(a[0], b[38])), B


@pytest.mark.gpu
def test_packed_wide_instances_equal_alone():
    """A packed batch with shared wide instances, unshared ones and both other paths."""
    sizes = [(400, 120, 20)] + [(352, 20, 0)] * 2 + [(140, 200, 30)] * 3 + [(20, 30, 5)] * 4
    inst = [inputs.random_qp(*s, workload=inputs.WL_UNEVEN, index=i) for i, s in enumerate(sizes)]

    def run(sz, ins):
        pb = PackedBatch(sz, device=DEV)
        out = pb.forward(*pb.pack([tuple(np.float32(x) for x in t) for t in ins]))
        torch.cuda.synchronize()
        return pb, pb.unpack(out.z, "q"), pb.unpack(out.lam, "h"), out.status
    pb, z, lam, st = run(sizes, inst)
    assert (st[:len(sizes)] == 0).all() and pb.sizes.reserved >> 8 == 3
    for i, (s, t) in enumerate(zip(sizes, inst)):
        _, za, la, _ = run([s], [t])
        assert torch.equal(z[i], za[0]) and torch.equal(lam[i], la[0]), i


def test_plan_puts_wide_instances_first_and_shares_the_longest():
    lib = _lib.load()
    sizes = [(20, 30, 5), (140, 200, 30), (352, 20, 0), (500, 500, 125), (100, 60, 20)]
    dims = np.ascontiguousarray(np.array(sizes, dtype=np.int32))
    desc, S, o = (_lib.QPInstanceDesc * 5)(), _lib.QPPackedSizes(), _lib.QPOptions()
    lib.qp_default_options(0, ctypes.byref(o))
    rc = lib.qp_packed_plan(ctypes.byref(o), 0, 5, dims.ctypes.data_as(ctypes.c_void_p), desc,
                            ctypes.byref(S))
    assert rc == 0 and S.n_global == 3
    assert [desc[k].id for k in range(3)] == [3, 2, 1]          # wide by cost, then the other
    assert S.reserved >> 8 == 2 and 1 <= S.reserved & 255 <= 2  # wide, shared
