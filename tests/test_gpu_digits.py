"""GPU parity of the digit-slice products.  csrc/gemm_digits.cu: FP64 and double-float applies
of more than 4 complex columns on stored planes, at the edges of their tiles (128 atoms, 32 and
64 real columns), odd sizes, and columns that are not finite.  csrc/gemv_digits.cu (below): few
columns from the stored float pairs, at the edges of its 64-atom tiles and 128-row blocks.

Bound per element, with s = |D| |x| and B_c = max_i sqrt(2) eta_i * 2 max_j |x_jc| (the bounds'
product, each at most twice too large by rounding up to a power of two):
    |dy_i| <= tau (sum_p Kbar_ip (s_i + s_j) + |z| |x_i|) + 4 P_i N 2^(-t) B_c,
tau = (nnz_i + 8) 2^-53 for the sparse term's FP64 sums, and the digits left out: products with
a + b >= S and the digits past the S-th add at most 2^-49 (S = 7) and 2^-57 (S = 8) of B_c per
entry (7 products below 2^14 at weight 2^(-8S), against 2^12 for the bounds' product).
"""
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


@pytest.mark.parametrize("n", [1, 97, 128, 129, 600])
@pytest.mark.parametrize("ncplx", [5, 16, 17, 32, 33])
@pytest.mark.parametrize("store,prec", [("fp64", "fp64"), ("fp64", "df"), ("pairs", "df")])
def test_apply_many_columns_within_digit_bound(W, ctx, orc, S, n, ncplx, store, prec):
    xyz = S.random_cluster(n, seed=n + 5)
    p = S.carbon_params(1.51)
    p["r0"] = 2.7
    eta = np.random.default_rng(n).uniform(0.3, 1.3, n)
    D = orc.d_matrix(xyz, eta)
    rowptr, col, val = orc.kbar_csr(xyz, p, cutoff_eps=p["cutoff_eps"])
    g = W.Geometry(ctx, xyz, p, eta=eta, store=W.STORE_FP64 if store == "fp64" else W.STORE_F32X2)
    om = np.linspace(0.01, 0.1, ncplx)
    z = np.array([orc.z_of_omega(w, p) for w in om])
    x = S.random_complex((n, ncplx), seed=3) * 10.0 ** np.linspace(-8, 8, ncplx)
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_FP64 if prec == "fp64" else W.PREC_DF)
    K = np.zeros((n, n))
    for i in range(n):
        K[i, col[rowptr[i]:rowptr[i + 1]]] = val[rowptr[i]:rowptr[i + 1]]
    P = K.sum(axis=1)
    Dl, xl = D.astype(np.longdouble), x.astype(np.clongdouble)
    u = Dl @ xl
    ref = np.empty_like(xl)
    for i in range(n):
        ref[i] = (K[i][:, None] * (u - u[i])).sum(axis=0) - z * xl[i]
    s = np.abs(D) @ np.abs(x)
    scale = K @ s + P[:, None] * s + np.abs(z) * np.abs(x)
    nnz = np.diff(rowptr)[:, None]
    B = np.sqrt(2.0) * eta.max() * 2.0 * np.maximum(np.abs(x.real).max(axis=0), np.abs(x.imag).max(axis=0))
    t = 57 if prec == "fp64" else 49
    bound = (nnz + 8) * 2.0 ** -53 * scale + 4.0 * P[:, None] * n * 2.0 ** -t * B + 1e-300
    assert np.all(np.abs(y - ref) <= bound)


@pytest.mark.parametrize("store,prec", [("fp64", "fp64"), ("pairs", "df")])
def test_columns_that_are_not_finite_stay_apart(W, ctx, S, store, prec):
    n, ncplx = 300, 20
    xyz = S.random_cluster(n, seed=9)
    g = W.Geometry(ctx, xyz, S.carbon_params(1.51), store=W.STORE_FP64 if store == "fp64" else W.STORE_F32X2)
    pr = W.PREC_FP64 if prec == "fp64" else W.PREC_DF
    om = np.linspace(0.01, 0.1, ncplx)
    x = S.random_complex((n, ncplx), seed=4)
    want, got = np.empty_like(x), np.empty_like(x)
    g.apply(om, x, want, prec=pr)
    bad = x.copy()
    bad[17, 3] = np.inf
    bad[5, 11] = np.nan
    g.apply(om, bad, got, prec=pr)
    ok = [c for c in range(ncplx) if c not in (3, 11)]
    # FP64: such a block takes plain FP64 for all its columns (chain rounding: n 2^-53 per term)
    scale = np.abs(want[:, ok]).max()
    assert np.all(np.abs(got[:, ok] - want[:, ok]) <= (n * 2.0 ** -50 * scale if prec == "fp64" else 0.0))
    assert not np.isfinite(got[:, 3].real).any() and not np.isfinite(got[:, 11].real).any()


def _pairs_bound(orc, xyz, eta, p, om, x):
    """Exact y (long double), and the bound of a product from float pairs by digit slices."""
    n = len(xyz)
    D = orc.d_matrix(xyz, eta)
    rowptr, col, val = orc.kbar_csr(xyz, p, cutoff_eps=p["cutoff_eps"])
    z = np.array([orc.z_of_omega(w, p) for w in om])
    u = (D @ x.real.astype(np.longdouble)) + 1j * (D @ x.imag.astype(np.longdouble))
    s = np.abs(D) @ np.abs(x)
    ref, scale = np.empty_like(u), np.empty_like(s)
    P = np.empty((n, 1))
    for i in range(n):
        q, k = col[rowptr[i]:rowptr[i + 1]], val[rowptr[i]:rowptr[i + 1]][:, None]
        ref[i] = (k * (u[q] - u[i])).sum(axis=0) - z * x[i]
        scale[i] = (k * (s[q] + s[i])).sum(axis=0) + np.abs(z) * np.abs(x[i])
        P[i] = k.sum()
    B = np.sqrt(2.0) * np.max(eta) * 2.0 * np.maximum(np.abs(x.real).max(axis=0), np.abs(x.imag).max(axis=0))
    nnz = np.diff(rowptr)[:, None]
    # pairs: 2^-48 of each entry; digits: 2^-54 of the bounds' product per entry and what is left out
    return ref, (2.0 ** -48 + (nnz + 8) * 2.0 ** -53) * scale + 4.0 * P * n * 2.0 ** -53 * B + 1e-300


@pytest.mark.parametrize("n", [1, 63, 64, 65, 129, 200, 513])
@pytest.mark.parametrize("ncplx", [1, 2, 3, 5])
def test_few_columns_from_symmetric_tiles_within_digit_bound(W, ctx, orc, S, n, ncplx):
    xyz = S.random_cluster(n, seed=n + 11)
    p = S.carbon_params(1.51)
    p["r0"] = 2.7
    eta = np.random.default_rng(n).uniform(0.3, 1.3, n)
    g = W.Geometry(ctx, xyz, p, eta=eta, store=W.STORE_F32X2_SYM)
    om = np.linspace(0.01, 0.1, ncplx)
    x = S.random_complex((n, ncplx), seed=6) * 10.0 ** np.linspace(-6, 6, ncplx)
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_DF)
    ref, bound = _pairs_bound(orc, xyz, eta, p, om, x)
    assert np.all(np.abs(y - ref) <= bound)


@pytest.mark.parametrize("n", [3072, 3135])
def test_few_columns_from_planes_within_digit_bound(W, ctx, orc, S, n):
    xyz = S.random_cluster(n, seed=n)
    p = S.carbon_params(1.51)
    p["r0"] = 2.7
    eta = np.full(n, p["eta"])
    g = W.Geometry(ctx, xyz, p, store=W.STORE_F32X2)
    om = np.linspace(0.01, 0.1, 3)
    x = S.random_complex((n, 3), seed=6)
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_FP64)   # up to 4 columns without a stored FP64 D
    ref, bound = _pairs_bound(orc, xyz, eta, p, om, x)
    assert np.all(np.abs(y - ref) <= bound)


def test_hardnesses_far_apart_keep_the_double_float_product(W, ctx, orc, S):
    n = 200
    xyz = S.random_cluster(n, seed=5)
    p = S.carbon_params(1.51)
    p["r0"] = 2.7
    eta = 10.0 ** np.random.default_rng(5).uniform(-2, 1, n)   # row bounds 2^10 apart
    g = W.Geometry(ctx, xyz, p, eta=eta, store=W.STORE_F32X2_SYM)
    x = S.random_complex((n, 2), seed=6)
    y = np.empty_like(x)
    om = np.array([0.02, 0.05])
    g.apply(om, x, y, prec=W.PREC_DF)
    D = orc.d_matrix(xyz, eta)
    ref, _ = _pairs_bound(orc, xyz, eta, p, om, x)
    rowptr, col, val = orc.kbar_csr(xyz, p, cutoff_eps=p["cutoff_eps"])
    s = np.abs(D) @ np.abs(x)
    tau = 8 * 2.0 ** -48 * np.sqrt(n)   # the double-float bound
    for i in range(n):
        q, k = col[rowptr[i]:rowptr[i + 1]], val[rowptr[i]:rowptr[i + 1]][:, None]
        z = np.array([orc.z_of_omega(w, p) for w in om])
        assert np.all(np.abs(y[i] - ref[i]) <= tau * ((k * (s[q] + s[i])).sum(axis=0) + np.abs(z) * np.abs(x[i])))


@pytest.mark.parametrize("ncplx", [5, 8, 9, 16, 17, 32])
def test_sparse_term_columns_do_not_depend_on_their_block(W, ctx, S, ncplx):
    """The digit products are exact per column, so an FP64 block of 33 columns and its first
    ncplx agree to the last bit if the neighbour term's lane layouts (8, 16, 32 columns per row,
    chunks) do."""
    n = 341
    xyz = S.random_cluster(n, seed=21)
    g = W.Geometry(ctx, xyz, S.sodium_params(), store=W.STORE_FP64)
    om = np.linspace(0.01, 0.1, 33)
    x = S.random_complex((n, 33), seed=2)
    full, part = np.empty_like(x), np.empty((n, ncplx), dtype=complex)
    g.apply(om, x, full, prec=W.PREC_FP64)
    g.apply(om[:ncplx], np.ascontiguousarray(x[:, :ncplx]), part, prec=W.PREC_FP64)
    assert np.array_equal(part, full[:, :ncplx])
