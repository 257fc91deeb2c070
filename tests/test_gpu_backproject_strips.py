"""The backprojector's strips at the sizes where they can go wrong: every kind
of z-profile (rows per voxel below 1, in [1, 3/2], in (3/2, 2), above), detectors
that end inside the volume (clamped rows), volumes a voxel past a patch or a
z-span, and more views than one list of profiles or one ballot holds -- each
launch configuration against the FP64 oracle (rel-L2 <= 1e-5, the bound of every
FP32 operator test here)."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import cuda, host, rel_l2

pytestmark = pytest.mark.gpu


def _geom(n, dv, nv, views, du=1.7):
    return synth.Geometry(nx=n[0], ny=n[1], nz=n[2], vx=1.0, vy=1.0, vz=1.0, n_views=views, sod=400.0, sdd=700.0,
                          nu=int(2.2 * max(n[0], n[1]) / du) + 3, nv=nv, du=du, dv=dv)


CASES = {
    "two_rows": _geom((9, 17, 33), 2.6, 24, 70),
    "three_rows": _geom((17, 8, 65), 1.5, 84, 9),
    "four_rows": _geom((8, 9, 40), 1.0, 77, 33),
    "many_rows": _geom((10, 7, 20), 0.5, 71, 12),
    "span_256": _geom((9, 9, 257), 1.8, 260, 5),
    "span_192": _geom((7, 12, 193), 1.7, 120, 4),   # detector ends inside the volume
    "fine_columns": _geom((20, 20, 24), 1.7, 30, 40, du=0.5),
    "one_voxel": _geom((1, 1, 1), 1.7, 3, 3),
}


@pytest.mark.parametrize("vpl", [2, 4, 16, 28])
@pytest.mark.parametrize("name", sorted(CASES))
def test_strip_backprojection_matches_oracle(name, vpl):
    import paper_2605_12085_gb300 as fbl
    g = CASES[name]
    G = fbl.geometry_create(g)
    fbl.geometry_set_launch(G, 8, 1, vpl)
    rng = np.random.default_rng(len(name))
    views = [int(v) for v in rng.permutation(g.n_views)]
    y = rng.standard_normal((len(views), g.nv, g.nu)).astype(np.float32)
    ref = oracle.backproject(g, y.astype(np.float64), views)
    assert rel_l2(host(fbl.backproject(G, cuda(y), views)), ref) <= 1e-5


def test_batch_of_columns_and_strips_equals_single_solvers():
    # a batch whose volumes take both forms of the backprojector runs them in two
    # launches over one tile list; each volume equals its own solver bit for bit
    import paper_2605_12085_gb300 as fbl
    gs = [_geom((9, 9, 33), 1.7, 60, 8), _geom((12, 10, 40), 1.7, 70, 6), _geom((8, 17, 20), 1.7, 40, 10)]
    vpls = [2, 28, 16]
    Gs, bs = [fbl.geometry_create(g) for g in gs], []
    rng = np.random.default_rng(3)
    for g, G, v in zip(gs, Gs, vpls):
        fbl.geometry_set_launch(G, 8, 1, v)
        x = rng.uniform(0, 1, g.vol_shape).astype(np.float32)
        bs.append(fbl.project(G, cuda(x), range(g.n_views)))
    ps = [fbl.params_default(N0=3, alpha0=1e-2, mu=0.1, seed=v) for v in vpls]
    xs = [cuda(np.zeros(g.vol_shape, np.float32)) for g in gs]
    B = fbl.fblisa_batch_create(Gs, ps)
    for _ in range(3):
        B.step(xs, bs)
    for g, G, p, b, xb in zip(gs, Gs, ps, bs, xs):
        S, x = fbl.fblisa_create(G, p), cuda(np.zeros(g.vol_shape, np.float32))
        for _ in range(3):
            S.step(x, b)
        assert np.array_equal(host(x), host(xb))


def test_views_beyond_one_launch_are_added():
    # more than 512 MiB of residual rows run in several launches: the same sums as
    # two calls of one launch each (FP32 sums in another order: 1e-6)
    import torch
    import paper_2605_12085_gb300 as fbl
    g = synth.Geometry(nx=40, ny=33, nz=70, vx=1.0, vy=1.0, vz=1.0, n_views=720, sod=400.0, sdd=700.0, nu=520, nv=400,
                       du=0.25, dv=0.5)
    G = fbl.geometry_create(g)
    fbl.geometry_set_launch(G, 8, 1, 28)
    gen = torch.Generator("cuda").manual_seed(2)
    y = torch.rand((720, 400, 520), device="cuda", generator=gen)
    views = list(range(720))
    x = fbl.backproject(G, y, views)
    two = fbl.backproject(G, y[:300].contiguous(), views[:300])
    fbl.backproject(G, y[300:].contiguous(), views[300:], x=two, accumulate=True)
    assert rel_l2(host(x), host(two)) <= 1e-6
