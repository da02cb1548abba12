"""bench.py names the D product that the library runs (CPU), and the bytes it divides by are those
that product reads (GPU)."""
import numpy as np
import pytest


def test_the_product_follows_the_storage():
    import bench
    from paper_2103_00438_gb300 import wfq as W
    name = lambda n, store: bench.shifted_product(n, store, W)[0].split()[0]
    assert name(20000, W.STORE_F32X2) == name(3072, W.STORE_F32X2 | W.STORE_FP64) == "k_gemv_digits"
    assert name(1000, W.STORE_F32X2_SYM | W.STORE_BF16X2) == "k_gemv_digits"
    assert name(3071, W.STORE_F32X2) == name(20000, W.STORE_FP64) == "k_dgemv_df"
    assert name(20000, 0) == "k_dotf_dfv"
    assert "double-float" in bench.shifted_product(1000, W.STORE_F32X2, W)[1]


@pytest.mark.gpu
@pytest.mark.parametrize("store,n,rule", [("pairs", 3160, "triangle"), ("pairs", 1000, "full"), ("sym", 1000, "triangle"),
                                          ("fp64", 1000, "full"), ("none", 400, "nothing")])
def test_bytes_of_the_shifted_solvers_product(S, store, n, rule):
    from paper_2103_00438_gb300 import wfq as W
    ctx = W.Context(0)
    flag = {"pairs": W.STORE_F32X2, "sym": W.STORE_F32X2_SYM, "fp64": W.STORE_FP64, "none": 0}[store]
    g = W.Geometry(ctx, S.nanotube(10, 10, n // 40), S.carbon_params(1.04), store=flag)
    n = g.n
    ctx.profile(True)
    g.solve_gmres_shifted(S.ev([0.5, 1.0]), np.eye(3), rel_tol=1e-8)
    launches, _, work = ctx.profile_read(W.KT_DGEMV_DF)
    ctx.profile(False)
    tiles = -(-n // 64)
    want = {"triangle": tiles * (tiles + 1) / 2 * 64 * 64 * 8, "full": 8.0 * n * n, "nothing": 0.0}[rule]
    assert launches > 0 and work == launches * want
    g.close()
    ctx.close()
