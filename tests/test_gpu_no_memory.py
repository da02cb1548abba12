"""Applies that take digit slices need more workspace than the plain sums; without memory for it the
plain sums serve the call (failures injected on the host)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store,prec,n,ncplx,allocs", [("fp64", "fp64", 300, 6, 2), ("fp64", "fp64", 4100, 2, 2),
                                                       ("fp64", "df", 300, 6, 2), ("pairs", "df", 300, 6, 2),
                                                       ("sym", "df", 700, 2, 7), ("pairs", "fp64", 3100, 1, 6)])
def test_an_apply_without_memory_for_the_digits(S, store, prec, n, ncplx, allocs):
    """The call's own two allocations come first; every later one that the digits make may fail."""
    import torch
    from paper_2103_00438_gb300 import wfq as W
    ctx = W.Context(0)
    flag = {"fp64": W.STORE_FP64, "pairs": W.STORE_F32X2, "sym": W.STORE_F32X2_SYM}[store]
    g = W.Geometry(ctx, S.random_cluster(n, seed=2), S.carbon_params(1.51), store=flag)
    om = np.linspace(0.01, 0.1, ncplx)
    x = torch.from_numpy(S.random_complex((n, ncplx), seed=1)).cuda()
    want, y = torch.empty_like(x), torch.empty_like(x)
    pr = W.PREC_FP64 if prec == "fp64" else W.PREC_DF
    g.apply(om, x, want, prec=pr)
    for nth in range(3, 3 + allocs):
        y.zero_()
        ctx.selftest_fail_alloc(nth)
        g.apply(om, x, y, prec=pr)
        ctx.selftest_fail_alloc(0)
        # both sums' bounds: n 2^-53 and n 2^-48 of the terms, the largest of which bound y
        tol = n * 2.0 ** (-50 if prec == "fp64" and store == "fp64" else -45) * want.abs().max()
        assert float((y - want).abs().max()) <= float(tol), nth
    ctx.selftest_fail_alloc(1)
    with pytest.raises(W.WfqError) as e:
        g.apply(om, x, y, prec=pr)
    assert e.value.code == -3
    g.close()
    ctx.close()
