"""CPU check of the cluster kernels (wide sizes, several blocks per instance) from their source, under
AddressSanitizer: the blocks of a cluster run side by side, and a barrier that one of them does not
reach deadlocks (the run times out).  Every way through a solve, against the same instance on one
block, bit for bit; converged ones against the oracle too.  A device of few SMs is made believe, so
that the planner takes two blocks (or four, or one)."""
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

import oracle
from tests.test_kernel_emulation_cpu import BUILD, _objects, driver, pytestmark  # noqa: F401

SMS = {1: "1", 2: "3", 4: "6"}    # SMs for which a batch of one takes that many blocks


def _data(n, p, m, dtype, seed=0):
    """A feasible QP with Q positive definite: z0 strictly inside G z ≤ h, A z0 = b."""
    r = np.random.default_rng([71, seed, n, p, m])
    L = r.standard_normal((n, n)) / np.sqrt(n)
    G, A, z0 = r.standard_normal((p, n)), r.standard_normal((m, n)), r.standard_normal(n)
    x = [L @ L.T + np.eye(n), r.standard_normal(n), G, G @ z0 + r.uniform(0.2, 1.0, p), A, A @ z0,
         r.standard_normal(n)]
    return [np.ascontiguousarray(v, dtype=dtype) for v in x]


def _singular(n=352, p=20, k=4):
    """Q of rank n − k, its null space fixed by k equalities: the setup is repeated with Q + δI."""
    d = _data(n, p, k, np.float32, seed=1)
    d[0][n - k:] = 0
    d[0][:, n - k:] = 0
    d[4][:] = 0
    d[4][np.arange(k), n - k + np.arange(k)] = 1
    d[2][:, n - k:] = 0      # (so that the inequalities stay feasible whatever b is)
    return d


def _infeasible(n=352, p=8, seed=2):
    d = _data(n, p, 0, np.float32, seed=seed)
    d[2][:2] = 0
    d[2][0, 0], d[2][1, 0] = 1, -1
    d[3][:2] = -1            # z_0 ≤ −1 and z_0 ≥ 1
    return d


def _poisoned(which):
    d = _data(352, 8, 0, np.float32, seed=3)
    d[which].flat[5] = np.nan
    return d


def _indefinite():
    d = _data(352, 8, 0, np.float32, seed=4)
    d[0][200, 200] = -3      # fails with and without δI
    return d


# name: data, environment, forward status, whether the oracle's solution is expected
CASES = {
    "fp32": (_data(352, 24, 0, np.float32), {}, 0, True),
    "fp32_rows_off_16_bytes": (_data(345, 21, 7, np.float32), {}, 0, True),
    # (three factorisations: the emulation takes 15 s for each on two blocks)
    "fp32_blocked_cholesky": (_data(340, 177, 13, np.float32), {"EMU_MAX_ITER": "1"}, 1, False),
    "fp64": (_data(352, 20, 0, np.float64), {}, 0, True),
    "no_inequality": (_data(352, 0, 12, np.float32), {}, 0, True),
    "singular_q": (_singular(), {}, 0, True),
    "infeasible": (_infeasible(), {}, 5, False),
    "max_iter": (_data(352, 24, 0, np.float32), {"EMU_MAX_ITER": "2"}, 1, False),
    "time_limit": (_data(352, 24, 0, np.float32), {"EMU_TIME_LIMIT_US": "1"}, 6, False),
    "nan_in_q": (_poisoned(1), {}, 3, False),
    "nan_in_the_matrix": (_poisoned(0), {}, 3, False),
    "failed_pivot": (_indefinite(), {}, 2, False),
    # a tensor-core wait that runs out in the last block only: the setup is repeated as for a singular Q
    "late_tensor_core": (_data(352, 24, 0, np.float32), {"EMU_LATE_BLOCK": "last"}, 0, True),
}


def _solve(exe, name, blocks):
    data, env, _, _ = CASES[name]
    n, p, m, dt = data[0].shape[0], data[2].shape[0], data[4].shape[0], data[0].dtype
    fin, fout = (os.path.join(BUILD, f"cl_{k}_{name}_{blocks}.bin") for k in ("in", "out"))
    with open(fin, "wb") as f:
        f.write(np.array([1, n, p, m, 0 if dt == np.float32 else 1, 0], np.int32).tobytes())
        for a in data:
            f.write(a.tobytes())
    env = {k: str(blocks - 1) if v == "last" else v for k, v in env.items()}
    r = subprocess.run([exe, fin, fout], capture_output=True, text=True, timeout=900,
                       env=dict(os.environ, ASAN_OPTIONS="detect_leaks=0:abort_on_error=1",
                                EMU_SMS=SMS[blocks], **env))
    assert r.returncode == 0, (name, blocks, r.stderr[-3000:])
    o = np.fromfile(fout, dtype=np.uint8)
    st, bst = np.frombuffer(o[-8:].tobytes(), dtype=np.int32)
    vals = np.frombuffer(o[:-8].tobytes(), dtype=dt)
    return int(st), int(bst), vals


@pytest.fixture(scope="module")
def runs(driver):  # noqa: F811
    jobs = [(name, b) for name in CASES for b in (2, 1)] + [("max_iter", 4)]
    with ThreadPoolExecutor(3) as ex:
        return dict(zip(jobs, ex.map(lambda j: _solve(driver, *j), jobs)))


@pytest.mark.parametrize("name", list(CASES))
def test_a_cluster_takes_every_path_as_one_block_does(runs, name):
    data, _, status, solved = CASES[name]
    st, bst, vals = runs[name, 2]
    assert st == status and (bst & 0xff) == status, (st, bst)
    assert bool(bst & 0x200) == (name in ("singular_q", "late_tensor_core"))
    for blocks in (1, 4):
        if (name, blocks) in runs:
            assert runs[name, blocks][:2] == (st, bst)
            assert np.array_equal(runs[name, blocks][2], vals, equal_nan=True), blocks
    if solved:
        Q, q, G, h, A, b, g = (np.float64(x) for x in data)
        sol = oracle.solve(Q, q, G, h, A, b)
        gr = oracle.backward(Q, G, h, A, sol, g)
        n, p, m = len(q), len(h), len(b)
        ztol, gtol = (1e-5, 1e-4) if data[0].dtype == np.float32 else (1e-9, 1e-8)
        z, dq = vals[:n], vals[n + p + m + n * n:][:n]
        assert np.abs(z - sol["z"]).max() <= ztol * max(1.0, np.abs(sol["z"]).max())
        assert np.abs(dq - gr["dq"]).max() <= gtol * max(np.linalg.norm(g), np.abs(gr["dq"]).max())


def test_the_planner_takes_the_blocks_that_are_meant():
    """(of the device the tests assume: 152 SMs, also where none is visible)"""
    from paper_1703_00443_gb300 import _lib
    lib = _lib.load()
    f = lambda B, n, p, m, dt=0: lib.qp_blocks_per_instance(None, dt, B, n, p, m)  # noqa: E731
    assert [f(B, 352, 24, 0) for B in (1, 14, 15, 34, 35, 68, 69, 128)] == [8, 8, 4, 4, 2, 2, 1, 1]
    assert f(1, 351, 20, 0) == 8 and f(1, 336, 20, 0) == 1 and f(1, 100, 100, 50) == 1
    assert f(1, 700, 700, 0) == 1              # its panels are in global memory: no room to exchange
    assert f(1, 352, 20, 0, 1) == 8 and f(-1, 352, 20, 0) == -1
