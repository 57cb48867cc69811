"""Wide sizes (n + neq >= 352 after padding) in full batches, one block per instance: the products'
copies ahead at the edges of their batches, on one block as on eight, and no slower than the kernel
of the other sizes."""
import os
import re

import numpy as np
import pytest
import torch

from paper_1703_00443_gb300 import _lib, inputs, qp_backward, qp_forward
from paper_1703_00443_gb300.packed import PackedBatch
from tests.helpers import oracle_solve_and_grad, rel_err

DEV = "cuda:0"


def test_wide_kernels_hold_no_spilled_views_over_their_calls():
    """The wide kernels took 2656 bytes of spill loads in an iteration's body; that traffic goes to L2.
    A quarter of it is the bound (the compiler's own report, kept by the build)."""
    log = os.path.join(_lib.BUILD, "fwd_f32_wide.ptxas.log")
    if not os.path.exists(log):
        pytest.skip("the library was not built here")
    found = re.findall(r"Function properties for \S*qp_fwd_(?:packed_)?large_kernelIfL[ib]([12])E\S*\n"
                       r".*?(\d+) bytes spill loads", open(log).read())
    assert found and all(int(loads) <= 2656 // 4 for _, loads in found), found


def test_packed_kernels_carry_no_tensor_core_routine():
    """They never call it (by the compiler's report, kept by the build)."""
    logs = [os.path.join(_lib.BUILD, f"fwd_f32_{k}.ptxas.log") for k in ("large", "wide")]
    if not all(os.path.exists(log) for log in logs):
        pytest.skip("the library was not built here")
    kernels = [k for log in logs for k in open(log).read().split("Compiling entry function")[1:]]
    packed = [k for k in kernels if "qp_fwd_packed_large_kernel" in k.split("\n")[0]]
    assert len(packed) == 3 and not any("tc_sweep_superblocks" in k for k in packed)
    assert sum("tc_sweep_superblocks" in k for k in kernels) == 3      # the fixed-size ones do


# rows of one lane group and one more, two rows per group with a partial batch, rows off 16-byte
# boundaries, FP64 (a quad is two copies) with and without equalities
@pytest.mark.gpu
@pytest.mark.parametrize("n,p,m,dtype", [(352, 65, 0, np.float32), (360, 132, 9, np.float32),
                                         (353, 20, 0, np.float32), (352, 30, 4, np.float64),
                                         (354, 66, 0, np.float64)])
def test_copies_ahead_at_the_edges(n, p, m, dtype):
    """One instance (eight blocks) against the oracle, within the tolerances of its type, and bit for bit
    against the same instance in a batch of 80 (one block each)."""
    batch = inputs.random_batch(1, n, p, m, workload=inputs.WL_PLAIN, dtype=dtype)
    g = inputs.upstream_grad(1, n, workload=inputs.WL_PLAIN, dtype=dtype)
    out = []
    for B in (1, 80):
        T = [torch.from_numpy(np.ascontiguousarray(np.repeat(x, B, 0))).to(DEV)
             for x in (batch.Q, batch.q, batch.G, batch.h, batch.A, batch.b)]
        f = qp_forward(*T)
        gr = qp_backward(f, torch.from_numpy(np.repeat(g, B, 0)).to(DEV))
        out.append([t[-1].cpu() for t in (f.status, f.iters, f.z, f.lam, f.nu, *gr)])
    assert int(out[0][0]) == 0
    for a, b in zip(*out):
        assert torch.equal(a, b)
    sols, refs = oracle_solve_and_grad(batch, g, [0])
    ztol, gtol = (1e-5, 1e-4) if dtype == np.float32 else (1e-9, 1e-8)
    assert rel_err(out[0][2].double().numpy()[None], [sols[0]["z"]]).max() <= ztol
    assert rel_err(out[0][6].double().numpy()[None], [refs[0]["dq"]],
                   1e-3 * np.linalg.norm(g, axis=1)).max() <= gtol


@pytest.mark.gpu
@pytest.mark.parametrize("n,p,m", [(500, 20, 0), (352, 176, 0)])
def test_a_full_batch_is_not_slower_than_on_the_other_sizes_kernel(n, p, m):
    """A packed plan whose `reserved` is 0 runs its instances on the kernel of the sizes below the line, one
    block each; it was up to 1.25 times as fast.  Best of eight, 5% for the spread."""
    sizes = [(n, p, m)] * 128
    base = [inputs.random_qp(n, p, m, workload=inputs.WL_UNEVEN, index=i) for i in range(4)]
    inst = [tuple(np.float32(x) for x in base[i % 4]) for i in range(128)]
    best = []
    for wide in (True, False):
        pb = PackedBatch(sizes, device=DEV)
        assert pb.sizes.reserved >> 8 == 128 and pb.sizes.reserved & 255 == 0
        if not wide:
            pb.sizes.reserved = 0
        P = pb.pack(inst)
        out = pb.forward(*P)
        ms = []
        for _ in range(8):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            pb.forward(*P, out=out)
            e1.record()
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        assert (out.status == 0).all()
        best.append(min(ms))
    assert best[0] <= 1.05 * best[1], best
