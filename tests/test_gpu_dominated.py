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
    else:
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
