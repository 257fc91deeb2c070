"""A batched volume whose residual rows exceed 512 MiB: its views run in the same
parts as in its single-volume launches, so its iterates are the single-volume
solver's bit for bit here too."""
import numpy as np
import pytest

import synth
from gpu_common import host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vpl", [16, 28])
def test_views_beyond_one_launch_in_a_batch(vpl):
    import torch
    import paper_2605_12085_gb300 as fbl
    g = synth.Geometry(nx=40, ny=33, nz=70, vx=1.0, vy=1.0, vz=1.0, n_views=720, sod=400.0, sdd=700.0, nu=520, nv=400,
                       du=0.25, dv=0.7)
    small = synth.small_geometry(nx=12, ny=10, nz=40, n_views=9, nu=30, nv=70)
    p = [fbl.params_default(N0=720, alpha0=1e-4, mu=0.1), fbl.params_default(N0=9, alpha0=1e-3, mu=0.1)]
    G = [fbl.geometry_create(g), fbl.geometry_create(small)]
    gen = torch.Generator("cuda").manual_seed(3)
    bs = []
    for q in G:
        fbl.geometry_set_launch(q, 4, 0, vpl)
    for q, h in zip(G, (g, small)):
        bs.append(fbl.project(q, torch.rand(h.vol_shape, device="cuda", generator=gen), range(h.n_views)))
    xs = [torch.zeros(h.vol_shape, device="cuda") for h in (g, small)]
    B = fbl.fblisa_batch_create(G, p)
    rec = [B.step(xs, bs) for _ in range(2)]
    for v, h in enumerate((g, small)):
        S, x = fbl.fblisa_create(G[v], p[v]), torch.zeros(h.vol_shape, device="cuda")
        for it in range(2):
            st = S.step(x, bs[v])
            assert st["grad_norm2"] == rec[it][v]["grad_norm2"]
        assert np.array_equal(host(x), host(xs[v]))
