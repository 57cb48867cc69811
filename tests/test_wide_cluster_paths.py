"""The other ways through a solve on a cluster of blocks (wide sizes): every one of them against the
same instances in a batch that runs on one block each."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1703_00443_gb300 import _lib, default_options, inputs, qp_backward, qp_forward
from paper_1703_00443_gb300.packed import PackedBatch
from tests import test_cluster_emulation_cpu as cases
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


def _options(**kw):
    o = default_options(torch.float32)
    for k, v in kw.items():
        setattr(o, k, v)
    return o


@pytest.mark.parametrize("name,make,options,status", [
    ("singular Q", cases._singular, {}, 0),
    # (whether the Newton system or the certificate comes first depends on rounding: as on one block,
    # in every kernel of every size)
    ("infeasible, no certificate", cases._infeasible, {}, 2),
    ("infeasible", lambda: cases._infeasible(seed=3), {}, 5),
    ("max_iter", lambda: cases._data(352, 24, 0, np.float32), {"max_iter": 2}, 1),
    ("time limit", lambda: cases._data(352, 24, 0, np.float32), {"time_limit_us": 1}, 6),
    ("NaN in q", lambda: cases._poisoned(1), {}, 3),
    ("NaN in Q", lambda: cases._poisoned(0), {}, 3),
    ("indefinite Q", cases._indefinite, {}, 2),
])
def test_statuses(name, make, options, status):
    data = make()
    outs = [_run(data[:6], data[6], B, _options(**options)) for B in BATCHES]
    assert int(outs[0][0]) == status
    for B, o in zip(BATCHES[1:], outs[1:]):
        assert _same(outs[0], o), B


@pytest.mark.parametrize("sms,blocks", [(60, [1, 11, 0, 0]), (28, [0, 1, 10, 1]), (0, [0, 0, 0, 12])])
def test_packed_levels_equal_alone(sms, blocks):
    """Clusters of eight, four and two blocks and unshared instances side by side with both other paths."""
    lib = _lib.load()
    sizes = [(352, 20, 0)] * 9 + [(400, 120, 20)] + [(352, 20, 0)] * 2 + [(200, 200, 50)] * 2 + \
        [(20, 30, 5)] * 3
    inst = [tuple(np.float32(x) for x in inputs.random_qp(*s, workload=inputs.WL_UNEVEN, index=i))
            for i, s in enumerate(sizes)]
    pb = PackedBatch(sizes, device=DEV, sms=sms)
    counts = (ctypes.c_int32 * 4)()
    assert lib.qp_packed_blocks(ctypes.byref(pb.sizes), counts) == 0 and list(counts) == blocks
    out = pb.forward(*pb.pack(inst))
    torch.cuda.synchronize()
    z, lam = pb.unpack(out.z, "q"), pb.unpack(out.lam, "h")
    assert (out.status[:len(sizes)] == 0).all()
    for i, (s, t) in enumerate(zip(sizes, inst)):
        one = PackedBatch([s], device=DEV)
        o = one.forward(*one.pack([t]))
        assert torch.equal(z[i], one.unpack(o.z, "q")[0]), i
        assert torch.equal(lam[i], one.unpack(o.lam, "h")[0]), i


def test_the_batches_above_take_the_clusters_they_are_meant_for():
    lib = _lib.load()
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("counts for 152 SMs")
    assert [lib.qp_blocks_per_instance(None, 0, B, 352, 24, 0) for B in BATCHES] == [8, 4, 2, 1]


def test_a_streams_first_packed_call_may_be_captured():
    """The side streams come with the call, under capture too."""
    sizes = [(352, 20, 0), (400, 120, 20), (200, 200, 50), (20, 30, 5)]
    inst = [tuple(np.float32(x) for x in inputs.random_qp(*s, workload=inputs.WL_UNEVEN, index=i))
            for i, s in enumerate(sizes)]
    pb = PackedBatch(sizes, device=DEV)
    P = pb.pack(inst)
    ref = pb.forward(*P).z.clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        out = pb.forward(*P)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out.z, ref)


def test_a_plan_that_shares_what_cannot_be_shared():
    """`reserved` of another origin: 700 inequalities have their panels in global memory, where the
    blocks of a cluster would exchange.  One block takes the instance; a size below the wide line runs
    on a cluster as well."""
    for size in ((700, 700, 0), (200, 200, 50)):
        t = tuple(np.float32(x) for x in inputs.random_qp(*size, workload=inputs.WL_UNEVEN, index=3))
        z = []
        for reserved in (1 << 8, 1 << 8 | 1):
            pb = PackedBatch([size], device=DEV)
            pb.sizes.reserved = reserved
            out = pb.forward(*pb.pack([t]))
            torch.cuda.synchronize()
            assert int(out.status[0]) == 0
            z.append(out.z.clone())
        assert torch.equal(*z), size
