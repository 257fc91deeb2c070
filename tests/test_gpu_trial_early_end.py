"""A rejected trial's objective does end early, and a trial whose objective is not
finite is reported all the same, in the host loop, the graph and the batch.

The early end is seen in the time of a further trial: searches of which every trial
is rejected (the test hook force_reject), once with steps whose objective passes the
limit in the first wave of blocks and once with steps so small that it never does.
The detector gives eleven waves of blocks (the batch twice as many), most of a
trial's time; the time per trial has to differ by a factor of two."""
import numpy as np
import pytest

import synth
from gpu_common import host

pytestmark = pytest.mark.gpu

GEOM = synth.small_geometry(nx=128, ny=128, nz=64, n_views=96, nu=220, nv=120, du=0.9, dv=0.9)
NONFINITE, LINESEARCH = 6, 5


def _solver(fbl, mode, alpha0, **kw):
    import torch
    Gs = [fbl.geometry_create(GEOM) for _ in range(2 if mode == "batch" else 1)]
    ps = [fbl.params_default(N0=96, alpha0=alpha0, mu=0.1, use_graph=int(mode == "graph"), **kw) for _ in Gs]
    gen = torch.Generator("cuda").manual_seed(1)
    # data well above the projections of x: the gradient is negative, a long step goes far up
    bs = [5.0 + torch.rand((96, 120, 220), device="cuda", generator=gen) for _ in Gs]
    xs = [0.01 * torch.rand(GEOM.vol_shape, device="cuda", generator=gen) for _ in Gs]
    S = fbl.fblisa_batch_create(Gs, ps) if mode == "batch" else fbl.fblisa_create(Gs[0], ps[0])
    step = (lambda x, b: S.step_raw(x, b)) if mode == "batch" else (lambda x, b: S.step_raw(x[0], b[0]))
    return step, xs, bs


def _trial_ms(fbl, mode, alpha0):
    import torch
    ms = []
    for trials in (20, 60):
        step, xs, bs = _solver(fbl, mode, alpha0, beta=0.95, max_backtracks=trials, force_reject=1)
        times = []
        for _ in range(4):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record()
            rc, _ = step(xs, bs)
            e1.record()
            torch.cuda.synchronize()
            assert rc == LINESEARCH
            times.append(e0.elapsed_time(e1))
        ms.append(min(times[1:]))
    return (ms[1] - ms[0]) / 40


@pytest.mark.parametrize("mode", ["host", "graph", "batch"])
def test_rejected_trials_end_early(mode):
    import paper_2605_12085_gb300 as fbl
    early, full = _trial_ms(fbl, mode, 1.0), _trial_ms(fbl, mode, 1e-12)
    assert early <= 0.5 * full, (early, full)


@pytest.mark.parametrize("mode", ["host", "graph", "batch"])
@pytest.mark.parametrize("data,alpha0", [(1e17, 1.0), (1.0, 1e25)])
def test_nonfinite_trials_are_reported(mode, data, alpha0):
    # data: squares up to 1e37, finite in FP32, and a first trial point far beyond; alpha0: an
    # ordinary residual, and a step that takes the trial point there
    import paper_2605_12085_gb300 as fbl
    step, xs, bs = _solver(fbl, mode, alpha0)
    for b in bs:
        b.mul_(data)
    before = [host(x) for x in xs]
    rc, st = step(xs, bs)
    assert rc == NONFINITE, (rc, st)
    assert all(np.array_equal(host(x), x0) for x, x0 in zip(xs, before))
