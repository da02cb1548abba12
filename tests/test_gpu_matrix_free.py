"""The matrix-free tensor-core product at the edges of its work split: groups of generator warps that
get no stage, a last stage of padding, blocks with too few pipeline stages for the groups."""
import numpy as np
import pytest

from test_gpu_parity import TAU_MIXED, _carbon, _mixed_bound, _oracle_apply

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


@pytest.mark.parametrize("n,ncplx", [(2, 1), (100, 96), (129, 60), (700, 127), (257, 129), (300, 190), (260, 250)])
def test_product_at_the_edges_of_the_stage_groups(W, ctx, orc, S, n, ncplx):
    xyz = S.random_cluster(n, seed=n)
    n = len(xyz)
    p = _carbon(S, r0=2.7)
    g = W.Geometry(ctx, xyz, p, store=0)
    sysm = orc.System(xyz, p)
    om = S.ev(np.linspace(0.3, 1.5, ncplx))
    x = S.random_complex((n, ncplx), seed=3).astype(np.complex64)
    y = np.empty_like(x)
    g.apply(om, x, y, prec=W.PREC_MIXED)
    for c in sorted({0, ncplx // 2, ncplx - 1}):
        z, xc = sysm.z(om[c]), x[:, c].astype(np.complex128)
        ref = _oracle_apply(orc, sysm, z, xc)
        assert np.max(np.abs(y[:, c] - ref) / _mixed_bound(sysm, z, xc)) <= TAU_MIXED


@pytest.mark.parametrize("ncplx", [48, 64, 80, 96])   # 7, 6, 6 and 5 stages fit
def test_many_stages_where_the_ring_is_cut_to_whole_groups(W, ctx, orc, S, ncplx):
    xyz = S.random_cluster(2300, seed=8)
    p = _carbon(S, r0=2.7)
    g = W.Geometry(ctx, xyz, p, store=0)
    sysm = orc.System(xyz, p)
    om = S.ev(np.linspace(0.3, 1.5, ncplx))
    x = S.random_complex((len(xyz), ncplx), seed=3).astype(np.complex64)
    y = np.empty_like(x)
    for _ in range(3):
        g.apply(om, x, y, prec=W.PREC_MIXED)
    for c in (0, ncplx // 2, ncplx - 1):
        z, xc = sysm.z(om[c]), x[:, c].astype(np.complex128)
        ref = _oracle_apply(orc, sysm, z, xc)
        assert np.max(np.abs(y[:, c] - ref) / _mixed_bound(sysm, z, xc)) <= TAU_MIXED
