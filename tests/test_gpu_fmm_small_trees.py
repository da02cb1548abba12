"""FMM products of structures with few leaves or many atoms a leaf: the M2L by box and by octant, the
near field's groups of targets and of columns.  All of them add the same terms in the same order, so a
column's result does not depend on the block it is in, and none of them may be slow."""
import numpy as np
import pytest

from test_gpu_fmm import TAU_FMM, _reference

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


def _structure(S, name):
    if name == "sphere":
        return S.fcc_sphere(4.23, S.fcc_sphere_radius_for(5000, 4.23), 0.05, seed=1), S.sodium_params()   # octree, 64 leaves
    if name == "tube":
        return S.nanotube(5, 5, 50), S.carbon_params(1.04)
    if name == "disk":
        return S.graphene_disk(20.0, vacancy_frac=0.01, seed=1), S.carbon_params(1.84)
    return S.honeycomb_flake(9), S.carbon_params(1.51)   # quadtree, 486 atoms


@pytest.mark.parametrize("name,order", [("flake", 2), ("flake", 3), ("flake", 5), ("flake", 9), ("flake", 16),
                                        ("disk", 6), ("tube", 3), ("tube", 6), ("sphere", 4), ("sphere", 5)])
def test_a_column_does_not_depend_on_its_block(W, ctx, S, name, order):
    xyz, p = _structure(S, name)
    g = W.Geometry(ctx, xyz, p, store=0)
    g.fmm_build(order)
    n, full = len(xyz), 70
    om = np.linspace(0.01, 0.1, full)
    x = S.random_complex((n, full), seed=4).astype(np.complex64)
    want, got = np.empty_like(x), np.empty_like(x)
    g.apply(om, x, want, prec=W.PREC_FMM)
    for c in (1, 2, 3, 8, 9, 16, 17, 35):
        part = np.empty((n, c), np.complex64)
        g.apply(om[:c], np.ascontiguousarray(x[:, :c]), part, prec=W.PREC_FMM)
        # the neighbour term of up to 4 columns adds over lanes: 2^-20 of the largest y there
        tol = 2.0 ** -20 * np.abs(want[:, :c]).max() if c <= 4 else 0.0
        assert np.abs(part - want[:, :c]).max() <= tol, c
    g.close()


@pytest.mark.parametrize("order", [5, 9, 16])
def test_orders_with_other_numbers_of_nodes(W, ctx, orc, S, order):
    from oracle import fmm
    xyz, p = _structure(S, "flake")
    g = W.Geometry(ctx, xyz, p, store=0)
    g.fmm_build(order)
    om = S.ev([0.3, 0.9, 1.6])
    x = S.random_complex((len(xyz), 3), seed=31)
    y = g.apply(om, x.astype(np.complex64), np.empty((len(xyz), 3), np.complex64), prec=W.PREC_FMM)
    y_f, _, scale = _reference(orc, fmm, xyz, p, om, x.astype(np.complex64).astype(complex), order)
    assert (np.abs(y - y_f) / scale).max() <= TAU_FMM
    g.close()


def test_many_atoms_a_leaf_are_spread_over_the_sms(W, ctx, S):
    """A 15k-atom sphere has 64 leaves of 230 atoms.  16 columns take 2.3 ms; with a leaf to a warp they
    took 116 ms.  12 ms leaves room for a slow clock."""
    import torch
    xyz = S.fcc_sphere(4.23, S.fcc_sphere_radius_for(15000, 4.23), 0.05, seed=1)
    g = W.Geometry(ctx, xyz, S.sodium_params(), store=0)
    g.fmm_build(4)
    x = torch.randn((g.n, 16), dtype=torch.complex64, device="cuda")
    y, om, st = torch.empty_like(x), np.linspace(0.01, 0.1, 16), torch.cuda.current_stream()
    times = []
    for _ in range(4):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.apply(om, x, y, prec=W.PREC_FMM, stream=st)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b))
    g.close()
    assert min(times) <= 12.0
