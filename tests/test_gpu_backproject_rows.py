"""The backprojector where detector rows are far apart along z: every launch
configuration against the FP64 oracle (rel-L2 <= 1e-5, the bound of every FP32
operator test here) and against the projector as its transpose, over spans of
more than 256 voxels, along which a rounded row position would drift."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import cuda, host, rel_l2

pytestmark = pytest.mark.gpu

VZ = 0.05


def _geom(spacing, nx=10, ny=9, nz=260, views=5):
    """Rows `spacing` voxels apart at the axis (1/1.03 to 1.03 of it in the volume)."""
    dv = spacing * VZ * 700.0 / 400.0
    return synth.Geometry(nx=nx, ny=ny, nz=nz, vx=1.0, vy=1.0, vz=VZ, n_views=views, sod=400.0, sdd=700.0,
                          nu=int(2.2 * max(nx, ny) / 1.7) + 3, nv=int(1.75 * VZ * nz / dv) + 4, du=1.7, dv=dv)


def _check(G, g, rng):
    import paper_2605_12085_gb300 as fbl
    views = list(range(g.n_views))
    y = rng.standard_normal((len(views), g.nv, g.nu)).astype(np.float32)
    got = host(fbl.backproject(G, cuda(y), views))
    assert rel_l2(got, oracle.backproject(g, y.astype(np.float64), views)) <= 1e-5
    x = rng.uniform(0, 1, g.vol_shape).astype(np.float32)
    ax = host(fbl.project(G, cuda(x), views))
    lhs, rhs = float((ax * y).sum()), float((x * got).sum())
    assert abs(lhs - rhs) <= 1e-5 * np.linalg.norm(ax) * np.linalg.norm(y)


@pytest.mark.parametrize("vpl", [2, 4, 16, 28])
@pytest.mark.parametrize("spacing", [1.9, 2.1, 4, 9, 16, 40, 100, 119, 121, 200, 500])
def test_rows_far_apart_match_oracle(spacing, vpl):
    import paper_2605_12085_gb300 as fbl
    g = _geom(spacing)
    G = fbl.geometry_create(g)
    fbl.geometry_set_launch(G, 8, 1, vpl)
    _check(G, g, np.random.default_rng(vpl))


@pytest.mark.parametrize("spacing", [1.5, 12, 40])
def test_default_configuration_of_a_volume_that_fills_the_gpu(spacing):
    import paper_2605_12085_gb300 as fbl
    g = _geom(spacing, nx=56, ny=56, views=3)
    _check(fbl.geometry_create(g), g, np.random.default_rng(1))


@pytest.mark.parametrize("spacing", [20, 200])
def test_batch_with_rows_far_apart_equals_single_solvers(spacing):
    # the volume asks for strips and runs in columns, beside one that runs in strips
    import paper_2605_12085_gb300 as fbl
    gs = [_geom(spacing, nx=12, ny=11, nz=70, views=8), _geom(1.2, nx=9, ny=14, nz=40, views=6)]
    rng = np.random.default_rng(5)
    Gs, bs, ps = [], [], []
    for q, g in enumerate(gs):
        G = fbl.geometry_create(g)
        fbl.geometry_set_launch(G, 4, 0, 28)
        Gs.append(G)
        bs.append(fbl.project(G, cuda(rng.uniform(0, 1, g.vol_shape).astype(np.float32)), range(g.n_views)))
        ps.append(fbl.params_default(N0=3, alpha0=1e-2, mu=0.1, seed=q))
    xs = [cuda(np.zeros(g.vol_shape, np.float32)) for g in gs]
    B = fbl.fblisa_batch_create(Gs, ps)
    for _ in range(3):
        B.step(xs, bs)
    for g, G, p, b, xb in zip(gs, Gs, ps, bs, xs):
        S, x = fbl.fblisa_create(G, p), cuda(np.zeros(g.vol_shape, np.float32))
        for _ in range(3):
            S.step(x, b)
        assert np.array_equal(host(x), host(xb))


@pytest.mark.parametrize("vpl", [16, 28])
@pytest.mark.parametrize("spacing", [0.8, 1.2, 1.5, 1.7, 1.9])
def test_strips_are_no_further_off_than_columns(spacing, vpl):
    # one view at a time, so that the weights' error is not lost in the sums' rounding: strips
    # hold a position to half of 2^-23 rows (up to 2 voxels), columns to a few 2^-24 voxels
    import paper_2605_12085_gb300 as fbl
    g = _geom(spacing, nx=16, ny=15, views=7)
    G = fbl.geometry_create(g)
    rng = np.random.default_rng(2)
    err = {vpl: 0.0, 4: 0.0}
    for v in range(g.n_views):
        y = rng.standard_normal((1, g.nv, g.nu)).astype(np.float32)
        ref = oracle.backproject(g, y.astype(np.float64), [v])
        for form in err:
            fbl.geometry_set_launch(G, 8, 1, form)
            err[form] += rel_l2(host(fbl.backproject(G, cuda(y), [v])), ref) ** 2
    assert err[vpl] <= err[4]
