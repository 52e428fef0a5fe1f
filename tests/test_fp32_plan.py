"""How the FP32 path spreads a network's tiles over the SMs: panda_fp32_plan is
host code, so these run on the CPU."""
from __future__ import annotations

import pytest


@pytest.fixture(scope="module", autouse=True)
def library():
    from paper_1507_07039_gb300 import build
    build.build()


def plan(*args):
    from paper_1507_07039_gb300 import panda
    return panda.panda_fp32_plan(*args)


@pytest.mark.parametrize("T,G", [(1, 1), (125, 125), (60, 300), (250, 600), (250, 2100), (500, 1000), (1000, 3000),
                                 (1024, 2048), (1000, 17000)])
def test_no_cta_without_work(T, G):
    """An SM holds one CTA of these kernels, so one without an item takes it from
    another network of a set."""
    p = plan(T, G)
    for q in range(2):
        assert 1 <= p["ctas"][q] <= 152
        assert p["ctas"][q] <= p["items"][q] * (2 if p["pair"] else 1), p


def test_bad_arguments_are_refused():
    from paper_1507_07039_gb300 import panda
    for args in ((0, 10, 152), (10, 0, 152), (46001, 10, 152), (10, 10, 1)):
        with pytest.raises(panda.PandaError):
            panda.panda_fp32_plan(*args)


def test_planning_is_a_small_part_of_a_create():
    """A create of 1000 x 17000 from host arrays takes about 9 ms and plans on the
    host; the plan took 1.6 to 3.9 ms of it, 0.2 now.  The best of twenty runs."""
    import time
    best = 1.0
    for _ in range(20):
        t0 = time.perf_counter()
        plan(1000, 17000)
        best = min(best, time.perf_counter() - t0)
    assert best < 1e-3
