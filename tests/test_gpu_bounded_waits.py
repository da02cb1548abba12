"""Bounded device-side waits: a warp gives up together, and an apply whose wait gave up says so
(the failure injected on the host)."""
import numpy as np
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


CALLS = [("fp64", "fp64", 2), ("fp64", "fp64", 6), ("fp64", "df", 6), ("pairs", "df", 1), ("pairs", "df", 6),
         ("sym", "df", 2), ("bf16", "mixed", 5), ("none", "mixed", 3)]


@pytest.fixture(scope="module")
def geometry(W, ctx, S):
    stores = {"fp64": W.STORE_FP64, "pairs": W.STORE_F32X2, "sym": W.STORE_F32X2_SYM, "bf16": W.STORE_BF16X2, "none": 0}
    xyz = S.random_cluster(200, seed=3)
    return {k: W.Geometry(ctx, xyz, S.carbon_params(1.51), store=v) for k, v in stores.items()}


@pytest.mark.parametrize("store,prec,ncplx", CALLS)
def test_an_apply_whose_wait_gave_up_reports_it(W, ctx, geometry, S, store, prec, ncplx):
    import torch
    g, pr = geometry[store], {"fp64": W.PREC_FP64, "df": W.PREC_DF, "mixed": W.PREC_MIXED}[prec]
    dt = np.complex64 if prec == "mixed" else np.complex128
    om = np.linspace(0.01, 0.1, ncplx)
    x = S.random_complex((200, ncplx), seed=1).astype(dt)
    want, y = np.empty_like(x), np.empty_like(x)
    g.apply(om, x, want, prec=pr)
    ctx.selftest_fail_next_apply()
    with pytest.raises(W.WfqError) as e:
        g.apply(om, x, y, prec=pr)
    assert e.value.code == -6 and np.isnan(y.view(y.real.dtype)).all()
    # device memory: the call returns before its kernels have run, so y alone can tell
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    ctx.selftest_fail_next_apply()
    g.apply(om, xd, yd, prec=pr)
    assert torch.isnan(torch.view_as_real(yd)).all()
    # and nothing is left for the next calls
    g.apply(om, x, y, prec=pr)
    assert np.array_equal(y, want)


def test_a_solve_after_a_failed_apply_is_not_failed(W, ctx, geometry, S):
    import torch
    g = geometry["pairs"]
    x = torch.from_numpy(S.random_complex((200, 6), seed=1)).cuda()
    ctx.selftest_fail_next_apply()
    g.apply(np.linspace(0.01, 0.1, 6), x, torch.empty_like(x), prec=W.PREC_DF)
    _, _, status = g.solve_gmres_shifted(S.ev([0.5]), np.eye(3)[:1], rel_tol=1e-8)
    assert status == "WFQ_OK"
