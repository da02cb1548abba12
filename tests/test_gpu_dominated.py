"""Applies to columns that a few entries dominate, where an error relative to the column's largest
entry is not small beside the result: y is held to the bounds of the plain FP64 and double-float
sums, entry by entry.

With s = |D| |x| and m nonzero entries in the column, an FP64 sum is within (m + 16) 2^-53 s (16 for
the entries of D, whose square roots, quotients and erf round differently here and in the oracle),
a double-float one within 8 2^-48 sqrt(m) s (the bound of the other tests; it supposes signs that
vary, so double-float sums take it here for few entries only)."""
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


def _column(kind, n, rng):
    """One column: one entry, five entries, or magnitudes over 14 decades."""
    x = np.zeros(n, dtype=complex)
    if kind == "spread":
        x[:] = (rng.uniform(0.5, 1, n) + 1j * rng.uniform(0.5, 1, n)) * 10.0 ** rng.uniform(-14, 0, n)
        x[rng.integers(n)] = 0.7 + 0.6j
    else:   # "mixed": five entries, beside another kind of column
        k = rng.choice(n, 1 if kind == "one" else 5, replace=False)
        x[k] = rng.uniform(0.5, 1, len(k)) + 1j * rng.uniform(0.5, 1, len(k))
    return x


def _tau(prec, m):
    return (m + 16) * 2.0 ** -53 if prec == "fp64" else 8 * 2.0 ** -48 * np.sqrt(m) + 16 * 2.0 ** -53


@pytest.mark.parametrize("prec,planes,ncplx,kind",
                         [("fp64", False, c, k) for c in (3, 6) for k in ("one", "five", "spread")]
                         + [("df", pl, 6, k) for pl in (False, True) for k in ("one", "five")])
def test_bem_columns(W, ctx, S, prec, planes, ncplx, kind):
    from oracle import bem
    n = 1501
    surf = S.spheroid_surface(n, 60.0, 30.0)
    A = bem.a_matrix(surf["xyz"], surf["normal"], surf["area"], surf["curvature"])
    # bound of an entry: the normal's dot product cancels
    d = np.abs(surf["xyz"][:, None] - surf["xyz"][None])
    r = np.sqrt((d ** 2).sum(-1)) + np.eye(n)
    B = surf["area"][:, None] * (np.abs(surf["normal"])[:, None] * d).sum(-1) / r ** 3
    B[np.arange(n), np.arange(n)] = np.abs(np.diag(A))
    g = W.BemGeometry(ctx, surf["xyz"], surf["normal"], surf["area"], surf["curvature"], S.drude_metal_params(),
                      store=W.STORE_FP64 | (W.STORE_F32X2 if planes else 0))
    rng = np.random.default_rng(ncplx)
    x = np.stack([_column(kind, n, rng) for _ in range(ncplx)], axis=1)
    om = S.ev(np.linspace(2.0, 4.5, ncplx))
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_FP64 if prec == "fp64" else W.PREC_DF)
    z = np.array([bem.z_of_omega(w, S.drude_metal_params()) for w in om])
    m = np.count_nonzero(x[:, 0])
    ref = A.astype(np.longdouble) @ x.astype(np.clongdouble) - z * x
    bound = _tau(prec, m) * (B @ (np.abs(x.real) + np.abs(x.imag)) + np.abs(z) * np.abs(x))
    assert np.all(np.abs(y - ref) <= bound)


def _far_pair(S, n, distance):
    """Two clusters a distance apart: at 1e5 bohr the entries of D between them are 2^-17 of its largest."""
    a = S.random_cluster(n - n // 3, seed=n)
    b = S.random_cluster(n // 3, seed=n + 1)
    return np.concatenate([a, b + np.array([distance, 0.0, 0.0])])


def _check(W, ctx, orc, S, n, ncplx, store, prec, kind, zero_imag=False, distance=1e5):
    """As for BEM, through the neighbour term; a double-float sum of m entries within (m + 8) 2^-48 s
    (a rounding of at most 2^-48 s in each step)."""
    xyz = _far_pair(S, n, distance)
    p = S.carbon_params(1.51)
    p["r0"] = 2.7
    D = orc.d_matrix(xyz, np.full(n, p["eta"]))
    rowptr, col, val = orc.kbar_csr(xyz, p, cutoff_eps=p["cutoff_eps"])
    flag = {"fp64": W.STORE_FP64, "pairs": W.STORE_F32X2, "sym": W.STORE_F32X2_SYM}[store]
    g = W.Geometry(ctx, xyz, p, store=flag)
    rng = np.random.default_rng(n + ncplx)
    x = np.stack([_column(kind, n, rng) for _ in range(ncplx)], axis=1)
    if kind == "random":
        x = S.random_complex((n, ncplx), seed=2)
    if kind == "mixed":
        x[:, 0] = S.random_complex((n, 1), seed=2)[:, 0]   # a column for the digits beside the others
    if zero_imag:
        x = x.real + 0j
    om = np.linspace(0.01, 0.1, ncplx)
    z = np.array([orc.z_of_omega(w, p) for w in om])
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_FP64 if prec == "fp64" else W.PREC_DF)
    u = (D @ x.real.astype(np.longdouble)) + 1j * (D @ x.imag.astype(np.longdouble))
    s = D @ (np.abs(x.real) + np.abs(x.imag))
    m = np.count_nonzero(x, axis=0)
    tau = (m + 16) * 2.0 ** -53 if prec == "fp64" else (m + 8) * 2.0 ** -48 + 16 * 2.0 ** -53
    for i in range(n):
        q, k = col[rowptr[i]:rowptr[i + 1]], val[rowptr[i]:rowptr[i + 1]][:, None]
        ref = (k * (u[q] - u[i])).sum(axis=0) - z * x[i]
        scale = (k * (s[q] + s[i])).sum(axis=0) + np.abs(z) * (np.abs(x[i].real) + np.abs(x[i].imag))
        assert np.all(np.abs(y[i] - ref) <= (tau + (len(q) + 8) * 2.0 ** -53) * scale), i


@pytest.mark.parametrize("kind", ["one", "five", "spread", "mixed"])
@pytest.mark.parametrize("store,prec", [("fp64", "fp64"), ("fp64", "df"), ("pairs", "df")])
def test_blocks_of_columns(W, ctx, orc, S, store, prec, kind):
    _check(W, ctx, orc, S, 451, 6, store, prec, kind)


@pytest.mark.parametrize("store,prec", [("fp64", "fp64"), ("pairs", "df")])
def test_a_block_without_a_column_for_the_digits(W, ctx, orc, S, store, prec):
    _check(W, ctx, orc, S, 300, 33, store, prec, "one", zero_imag=True)


@pytest.mark.parametrize("kind", ["random", "mixed", "spread"])
@pytest.mark.parametrize("store", ["fp64", "pairs"])
@pytest.mark.parametrize("n,ncplx", [(451, 5), (300, 33), (97, 6)])
def test_double_float_blocks_that_need_eight_digits(W, ctx, orc, S, n, ncplx, store, kind):
    """3000 bohr apart, random columns pass the test of eight digits and not that of seven."""
    _check(W, ctx, orc, S, n, ncplx, store, "df", kind, distance=3e3)


@pytest.mark.parametrize("kind", ["one", "spread", "mixed"])
@pytest.mark.parametrize("ncplx", [2, 3, 4])
def test_few_columns_of_a_stored_fp64_operator(W, ctx, orc, S, ncplx, kind):
    _check(W, ctx, orc, S, 4100, ncplx, "fp64", "fp64", kind)


@pytest.mark.parametrize("kind", ["one", "five", "spread", "mixed"])
@pytest.mark.parametrize("n,ncplx,store", [(451, 1, "sym"), (451, 2, "sym"), (700, 3, "sym"), (700, 19, "sym"),
                                           (3100, 1, "pairs"), (3100, 3, "pairs")])
def test_few_columns_from_float_pairs(W, ctx, orc, S, n, ncplx, store, kind):
    _check(W, ctx, orc, S, n, ncplx, store, "df", kind)


@pytest.mark.parametrize("store", ["sym", "pairs"])
def test_a_zero_imaginary_part_needs_no_other_sums(W, ctx, orc, S, store):
    _check(W, ctx, orc, S, 3100 if store == "pairs" else 451, 2, store, "df", "mixed", zero_imag=True)


@pytest.mark.parametrize("store", ["sym", "pairs"])
@pytest.mark.parametrize("ndir", [1, 3, 6])
def test_a_solve_from_localised_start_vectors(W, ctx, orc, S, store, ndir):
    """A flake's right-hand side is zero but at its edge: the first Arnoldi vectors may go to the
    double-float sums, later ones to the digits.
    q against LU within 1e-7, as for the other solves to 1e-10."""
    xyz = S.honeycomb_flake(23 if store == "pairs" else 9)   # 3174 and 486 atoms
    p = S.carbon_params(1.51)
    g = W.Geometry(ctx, xyz, p, store=W.STORE_F32X2 if store == "pairs" else W.STORE_F32X2_SYM)
    rng = np.random.default_rng(ndir)
    dirs = rng.standard_normal((ndir, 3))
    dirs[:, 2] = 0.0
    om = S.ev([0.8])
    q, _, status = g.solve_gmres_shifted(om, dirs, rel_tol=1e-10, max_iter=2000, prec=W.PREC_FP64)
    assert status == "WFQ_OK"
    D = orc.d_matrix(xyz, np.full(len(xyz), p["eta"]))
    rowptr, col, val = orc.kbar_csr(xyz, p, cutoff_eps=p["cutoff_eps"])
    K = np.zeros_like(D)
    for i in range(len(xyz)):
        K[i, col[rowptr[i]:rowptr[i + 1]]] = val[rowptr[i]:rowptr[i + 1]]
    A = K @ D - K.sum(axis=1)[:, None] * D
    A = A.astype(complex)
    A[np.arange(len(xyz)), np.arange(len(xyz))] -= orc.z_of_omega(om[0], p)
    ref = np.linalg.solve(A, g.rhs(dirs, E0=1.0).astype(complex))
    assert np.linalg.norm(q - ref) <= 1e-7 * np.linalg.norm(ref)
