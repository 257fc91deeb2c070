"""A rejected trial's objective may end early; what the line search reports may not
change.  The accepted step, its objective and, where no step passes, the last
trial's objective are compared with the complete objectives of the trial points,
formed one by one with the library's stateless calls (the operators' parity with
the oracle is tested elsewhere).  The detector and the batch give several waves
of blocks, so that blocks of a rejected trial do leave."""
import numpy as np
import pytest

import synth
from gpu_common import cuda, host, rel_l2

pytestmark = pytest.mark.gpu

G16 = synth.small_geometry(nx=72, ny=64, nz=60, n_views=24, nu=196, nv=170, du=0.8, dv=0.8)


def _problem(fbl):
    import torch
    G = fbl.geometry_create(G16)
    xt = cuda(synth.phantom(G16, 6, 77).astype(np.float32))
    b = fbl.project(G, xt, range(G16.n_views))
    b += 0.01 * b.max() * torch.randn(b.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    return G, xt, b


def _trials(fbl, G, x, b, views, p, n):
    """(x_bar, f, rhs) of the first n trials, every objective complete."""
    scale = G16.n_views / len(views)
    r = fbl.project(G, x, views) - b[list(views)]
    f = 0.5 * scale * fbl.residual_norm(G, x, views, b)
    g = fbl.backproject(G, r, views) * scale
    out, alpha = [], p.alpha0
    for _ in range(n):
        xb, (gd, dd, _l1) = fbl.prox_reduce(x, g, alpha, p.mu)
        out.append((xb, 0.5 * scale * fbl.residual_norm(G, xb, views, b), f + gd + dd / (2 * alpha)))
        alpha *= p.beta
    return out


@pytest.mark.parametrize("graph", [0, 1, "batch"])
@pytest.mark.parametrize("cols", [4, 8])
def test_accepted_step_and_objective_are_those_of_complete_trials(graph, cols):
    import paper_2605_12085_gb300 as fbl
    G, xt, b = _problem(fbl)
    fbl.geometry_set_launch(G, cols, 1, 28)
    p = fbl.params_default(N0=16, alpha0=1.0, mu=0.2, seed=9, use_graph=int(graph == 1))
    S = fbl.fblisa_batch_create([G], [p]) if graph == "batch" else fbl.fblisa_create(G, p)
    x = 0.7 * xt
    for _ in range(3):
        x0 = x.clone()
        st = S.step([x], [b])[0] if graph == "batch" else S.step(x, b)
        views = S.last_batch(0) if graph == "batch" else S.last_batch()
        tr = _trials(fbl, G, x0, b, views, p, st["backtracks"] + 1)
        assert st["backtracks"] >= 3
        assert all(f > rhs for _, f, rhs in tr[:-1]) and tr[-1][1] <= tr[-1][2]
        assert abs(st["f_xbar"] - tr[-1][1]) <= 1e-5 * tr[-1][1]
        assert rel_l2(host(x), host(tr[-1][0])) <= 1e-5


@pytest.mark.parametrize("graph", [0, 1])
def test_last_trial_of_a_failed_search_is_complete(graph):
    import paper_2605_12085_gb300 as fbl
    G, xt, b = _problem(fbl)
    p = fbl.params_default(N0=16, alpha0=1.0, mu=0.2, seed=9, max_backtracks=2, use_graph=graph)
    S = fbl.fblisa_create(G, p)
    x = 0.7 * xt
    x0 = x.clone()
    rc, st = S.step_raw(x, b)
    assert fbl.STATUS[rc] == "FBL_E_LINESEARCH" and np.array_equal(host(x), host(x0))
    last = _trials(fbl, G, x0, b, S.last_batch(), p, 3)[-1]
    assert abs(st["f_xbar"] - last[1]) <= 1e-5 * last[1]
    assert abs(st["margin"] - (last[2] - last[1])) <= 1e-5 * last[1]


@pytest.mark.parametrize("cols", [4, 8])
def test_a_batch_large_enough_to_stop_its_trials_early(cols):
    """Four volumes: more than eight waves of blocks, the batch's line for the limit
    (a batch of one, above, lies below it)."""
    import paper_2605_12085_gb300 as fbl
    G, xt, b = _problem(fbl)
    Gs = [G] + [fbl.geometry_create(G16) for _ in range(3)]
    for q in Gs:
        fbl.geometry_set_launch(q, cols, 1, 28)
    ps = [fbl.params_default(N0=16, alpha0=1.0, mu=0.2, seed=9 + v) for v in range(4)]
    S = fbl.fblisa_batch_create(Gs, ps)
    xs = [(0.7 + 0.05 * v) * xt for v in range(4)]
    for _ in range(2):
        x0 = [x.clone() for x in xs]
        for v, st in enumerate(S.step(xs, [b] * 4)):
            tr = _trials(fbl, G, x0[v], b, S.last_batch(v), ps[v], st["backtracks"] + 1)
            assert st["backtracks"] >= 3
            assert all(f > rhs for _, f, rhs in tr[:-1]) and tr[-1][1] <= tr[-1][2]
            assert abs(st["f_xbar"] - tr[-1][1]) <= 1e-5 * tr[-1][1]
            assert rel_l2(host(xs[v]), host(tr[-1][0])) <= 1e-5
