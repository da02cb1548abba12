"""Bounded device-side waits: a warp gives up together."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    from paper_2103_00438_gb300 import wfq
    wfq.load()
    return wfq


@pytest.fixture(scope="module")
def ctx(W):
    c = W.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("limit_us", [50, 1000])
def test_a_wait_that_runs_out_ends_for_the_whole_warp(ctx, limit_us):
    for _ in range(5):
        alone, together, code = ctx.selftest_wait(limit_us)
        assert 0 <= alone < 32          # lane 0 gave up; the others may have seen success
        assert together == 0            # none goes on to a warp-wide instruction without lane 0
        assert code == 9
