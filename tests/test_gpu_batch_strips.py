"""Batched volumes whose backprojector runs in strips: iterates, steps and ||g||^2
(an input of the learned first step) equal the single-volume solver's bit for
bit, in every storage type, with the plain and the learned first step; sizes a
voxel past a patch and a z-span, all three heights of a strip."""
import numpy as np
import pytest

import synth
from gpu_common import host

pytestmark = pytest.mark.gpu

SIZES = [((17, 24, 40), 28), ((9, 16, 193), 16), ((24, 9, 257), 28), ((8, 8, 33), 16), ((30, 7, 20), 2)]


@pytest.mark.parametrize("learned", [False, True])
@pytest.mark.parametrize("dtype", ["float32", "bfloat16", "float16"])
def test_batched_strips_equal_single_solvers(dtype, learned):
    import torch
    import paper_2605_12085_gb300 as fbl
    from paper_2605_12085_gb300 import proposal
    td = getattr(torch, dtype)
    code = {"float32": fbl.F32, "bfloat16": fbl.BF16, "float16": fbl.F16}[dtype]
    net = proposal.load()[0] if learned else None
    Gs, ps, bs, shapes = [], [], [], []
    gen = torch.Generator("cuda").manual_seed(4)
    for q, (n, vpl) in enumerate(SIZES):
        g = synth.small_geometry(nx=n[0], ny=n[1], nz=n[2], n_views=12 + q, nu=int(1.6 * max(n[:2])) + 3, nv=n[2] + 9)
        G = fbl.geometry_create(g)
        fbl.geometry_set_launch(G, 4, 0, vpl)
        x = torch.rand(g.vol_shape, device="cuda", generator=gen).to(td)
        Gs.append(G)
        shapes.append(g.vol_shape)
        bs.append(fbl.project(G, x, range(g.n_views), y_dtype=code))
        ps.append(fbl.params_default(N0=4 + q % 2, alpha0=1e-2, mu=0.05, seed=q, x_dtype=code, b_dtype=code))
    xs = [torch.zeros(s, device="cuda", dtype=td) for s in shapes]
    B = fbl.fblisa_batch_create(Gs, ps)
    if learned:
        B.set_proposal(net)
    recs = [B.step(xs, bs) for _ in range(4)]
    for v, shape in enumerate(shapes):
        S, x = fbl.fblisa_create(Gs[v], ps[v]), torch.zeros(shape, device="cuda", dtype=td)
        if learned:
            S.set_proposal(net)
        for rec in recs:
            st = S.step(x, bs[v])
            for key in ("alpha", "f_x", "f_xbar", "grad_norm2", "j_start"):
                assert st[key] == rec[v][key], (v, key)
        assert np.array_equal(host(x), host(xs[v]))
