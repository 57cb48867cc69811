"""The plan's choice of the wide instances that several blocks share (host logic, no GPU needed; the
counts hold for 152 SMs, which the planner takes where no device is visible)."""
import ctypes

import numpy as np
import pytest

from paper_1703_00443_gb300 import _lib


def _plan(sizes, cost=None, sms=-1):
    """(execution order, instances on 8, 4, 2 and 1 blocks) of a packed plan."""
    lib = _lib.load()
    B = len(sizes)
    dims = np.ascontiguousarray(np.array(sizes, dtype=np.int32))
    desc, S, o = (_lib.QPInstanceDesc * B)(), _lib.QPPackedSizes(), _lib.QPOptions()
    lib.qp_default_options(0, ctypes.byref(o))
    c = None if cost is None else np.ascontiguousarray(cost, dtype=np.float32)
    assert lib.qp_packed_plan_sms(ctypes.byref(o), 0, B, dims.ctypes.data_as(ctypes.c_void_p), None,
                                  None if c is None else c.ctypes.data_as(ctypes.c_void_p), sms,
                                  desc, ctypes.byref(S)) == 0
    counts = (ctypes.c_int32 * 4)()
    assert lib.qp_packed_blocks(ctypes.byref(S), counts) == 0
    return [desc[k].id for k in range(B)], list(counts)


@pytest.mark.parametrize("count", [1, 14, 18, 28, 29, 30, 33, 34, 35, 36, 60, 68])
def test_equal_large_instances_are_all_shared(count):
    """One left on a single block would take twice as long as the others (34 of n = 500, 28 of them
    shared: 23 ms against 14)."""
    _, (n8, n4, n2, n1) = _plan([(500, 500, 125)] * count)
    assert n8 + n4 + n2 == count and n1 == 0
    assert 8 * n8 + 4 * n4 + 2 * n2 <= 152 * 9 // 10


def test_more_equal_instances_than_pairs_of_sms_are_not_shared():
    """69 clusters of two would not be resident at once; the rest would wait for them."""
    for count in (100, 152, 400):
        assert _plan([(500, 500, 125)] * count)[1] == [0, 0, 0, count]


@pytest.mark.parametrize("cost", [[0.0] * 5, [1.0, 2.0, 3.0, 4.0, 5.0], [1e-3] * 4 + [9e-3],
                                  [float("inf")] * 5])
def test_costs_order_the_instances_and_do_not_choose_the_shared_ones(cost):
    """Costs that are all equal, ranks, or no times at all: the four large instances are shared, in the
    order of the costs; the fifth is not worth it and cannot be (the panels of 600 inequalities are in
    global memory), so it comes after them."""
    order, counts = _plan([(512, 512, 128)] * 4 + [(352, 600, 0)], cost)
    assert order == (sorted(range(4), key=lambda i: -cost[i]) + [4])
    assert counts == [4, 0, 0, 1]


@pytest.mark.parametrize("sizes", [[(500, 500, 125)] * 20, [(512, 512, 128)] + [(400, 400, 100)] * 9,
                                   [(500, 500, 125)] * 3 + [(20, 20, 5)] * 60])
def test_a_plan_for_part_of_the_device_takes_no_more(sizes):
    last = 10 ** 9
    for sms in (152, 120, 76, 40, 20, 8, 1, 0):
        _, (n8, n4, n2, n1) = _plan(sizes, sms=sms)
        blocks = 8 * n8 + 4 * n4 + 2 * n2
        assert blocks <= sms and n8 + n4 + n2 + n1 == sum(n + m >= 352 for n, _, m in sizes)
        assert blocks <= last     # never more of a smaller part
        last = blocks
    assert _plan(sizes, sms=152) == _plan(sizes) == _plan(sizes, sms=10 ** 6)


def test_server_plans_for_the_sms_that_stand_idle():
    from paper_1703_00443_gb300.serving import SMShare
    s = SMShare(152)
    assert s.free(0) == 152                       # alone: the whole device
    a = s.take(2 + 7 * 2)                         # two requests on eight blocks each
    assert (a, s.free(0), s.free(30)) == (16, 136, 106)
    b = s.take(400)                               # a batch larger than the device holds all of it
    assert b == 152 and s.free(0) == 0
    s.release(a)
    assert s.free(0) == 0
    s.release(b)
    assert s.free(0) == 152 and s.free(200) == 0  # a queue that will fill it
