"""Admission counts what a solve allocates: the smallest budget at which a server takes a request holds
the structure and the pool's high-water mark of the same solve alone."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _smallest_budget(W, ctx, g, om, dirs, m):
    """By bisection over servers that are only asked, the accepted requests served."""
    lo, hi = 1, 1 << 33
    while hi - lo > 65536:
        mid = (lo + hi) // 2
        sv = W.Server(ctx, nworkers=1, budget_bytes=mid, max_columns=64)
        try:
            sv.poll(sv.submit(g, om, dirs, m=m, rel_tol=1e-2), wait=True)
            hi = mid
        except W.WfqError:
            lo = mid
        sv.close()
    return hi


@pytest.mark.parametrize("store", ["sym", "pairs", "fp64"])
def test_a_request_is_admitted_with_what_its_solve_allocates(S, store):
    from paper_2103_00438_gb300 import wfq as W
    ctx = W.Context(0)
    flag = {"sym": W.STORE_F32X2_SYM | W.STORE_BF16X2, "pairs": W.STORE_F32X2 | W.STORE_BF16X2,
            "fp64": W.STORE_FP64 | W.STORE_BF16X2}[store]
    g = W.Geometry(ctx, S.nanotube(10, 10, 40), S.carbon_params(1.04), store=flag)
    om, dirs, m = S.ev(np.linspace(0.5, 1.5, 8)), np.eye(3), 2
    if store == "sym":   # tiles only: the server solves by mixed block GMRES
        g.solve_gmres(om, dirs, m=m, rel_tol=1e-2, max_iter=400, prec=W.PREC_MIXED)
    else:
        g.solve_gmres_shifted(om, dirs, rel_tol=1e-2)
    high = ctx.memory_stats()["pool_used_high"]
    budget = _smallest_budget(W, ctx, g, om, dirs, m)
    print(store, "high-water", high, "counted", budget - g.info()["device_bytes"])
    assert budget - g.info()["device_bytes"] >= high
    g.close()
    ctx.close()
