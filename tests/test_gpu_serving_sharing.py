"""The server shares large instances among thread blocks where SMs stand idle, not under load."""
import numpy as np
import pytest

from paper_1703_00443_gb300 import inputs
from paper_1703_00443_gb300.serving import QPServer

pytestmark = pytest.mark.gpu


def test_sharing_follows_the_load():
    data = tuple(np.float32(x) for x in inputs.random_qp(360, 360, 90, workload=inputs.WL_SERVE, index=0))
    g = np.float32(inputs.upstream_grad(1, 360, workload=inputs.WL_SERVE)[0])
    server = QPServer(device="cuda:0", max_batch=64)
    try:
        alone = server.submit(*data, g).result(timeout=120)
        assert alone["status"] == 0 and server.stats()["shared_instances"] == 1
        futs = [server.submit(*data, g) for _ in range(600)]
        results = [f.result(timeout=300) for f in futs]
        st = server.stats()
    finally:
        server.close()
    # the first of the burst may still find idle SMs; planned as if alone, all but a few were shared
    assert st["shared_instances"] - 1 <= 150, st
    for r in results:
        for k in ("z", "lam", "nu", "dQ"):
            assert np.array_equal(r[k], alone[k]), k
    assert server.sms.held == 0
