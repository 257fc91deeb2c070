"""Infinite and NaN pixels in the backprojection: exactly the voxels that their
rays touch are infinite or NaN, whatever the launch configuration.  Every kind of z-profile
(rows per voxel below 1, in [1, 3/2], in (3/2, 2), above); an even number of
rows and views off the axes, so that no ray crosses a plane at a voxel's centre."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import cuda, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vpl", [4, 16, 28])
@pytest.mark.parametrize("dv,nv", [(2.6, 46), (1.5, 80), (1.0, 120), (0.5, 240)])
def test_nonfinite_pixels_reach_the_voxels_of_their_rays(dv, nv, vpl):
    import paper_2605_12085_gb300 as fbl
    g = synth.Geometry(nx=19, ny=12, nz=66, vx=1.0, vy=1.0, vz=1.0, n_views=4, sod=400.0, sdd=700.0, nu=26, nv=nv,
                       du=1.7, dv=dv, angles=(0.3, 1.9, 3.4, 5.1))
    G = fbl.geometry_create(g)
    fbl.geometry_set_launch(G, 8, 1, vpl)
    rng = np.random.default_rng(3)
    y = rng.standard_normal((4, nv, 26)).astype(np.float32)
    bad = {np.inf: [(0, nv // 2, 12), (2, 5, 20)], -np.inf: [(1, nv // 3, 9)], np.nan: [(3, 2 * nv // 3, 15), (0, 0, 11)]}
    t, clean = np.zeros(y.shape), y.copy()
    for value, pixels in bad.items():
        for p in pixels:
            t[p], y[p], clean[p] = 1.0, value, 0.0
    got = host(fbl.backproject(G, cuda(y), range(4)))
    weight = oracle.backproject(g, t, range(4))
    assert not np.isfinite(got[weight > 1e-6]).any()
    free = weight == 0
    assert np.isfinite(got[free]).all()
    assert rel_l2(got[free], oracle.backproject(g, clean.astype(np.float64), range(4))[free]) <= 1e-5


@pytest.mark.parametrize("n", [1, 2047, 2048, 2600])
def test_view_lists_of_any_length(n):
    # the word that notes such pixels stands behind the view list: in one copy with it below
    # 2048 views, cleared by itself above; repeated views (sums of n FP32 terms: 1e-5)
    import paper_2605_12085_gb300 as fbl
    g = synth.Geometry(nx=9, ny=8, nz=12, vx=1.0, vy=1.0, vz=1.0, n_views=5, sod=400.0, sdd=700.0, nu=12, nv=16, du=1.7, dv=1.5)
    G = fbl.geometry_create(g)
    fbl.geometry_set_launch(G, 4, 0, 28)
    rng = np.random.default_rng(n)
    views = [int(v) for v in rng.integers(0, 5, n)]
    y = rng.standard_normal((n, 16, 12)).astype(np.float32)
    ref = oracle.backproject(g, y.astype(np.float64), views)
    assert rel_l2(host(fbl.backproject(G, cuda(y), views)), ref) <= 1e-5
    y[n - 1, 8, 6] = np.nan
    hit = np.zeros(y.shape)
    hit[n - 1, 8, 6] = 1.0
    weight = oracle.backproject(g, hit, views)
    got = host(fbl.backproject(G, cuda(y), views))
    assert np.isnan(got[weight > 1e-6]).all() and np.isfinite(got[weight == 0]).all()
    assert rel_l2(host(fbl.backproject(G, cuda(np.nan_to_num(y)), views))[weight == 0], ref[weight == 0]) <= 1e-5
