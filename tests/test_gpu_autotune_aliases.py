"""Launch configurations that are the same kernel are timed once: their times in the
autotuner's report are one number, and the first of them is the one chosen."""
import pytest

import synth

pytestmark = pytest.mark.gpu

ORDER = [4, 2, 8, 16, 24, 28]  # of the report's times


@pytest.mark.parametrize("dv,wide", [(1.5, False), (6.0, True)])
def test_equal_launches_share_a_time(dv, wide):
    import paper_2605_12085_gb300 as fbl
    g = synth.Geometry(nx=40, ny=36, nz=64, vx=1.0, vy=1.0, vz=1.0, n_views=12, sod=400.0, sdd=700.0, nu=90, nv=90, du=1.5, dv=dv)
    rep = fbl.geometry_autotune(fbl.geometry_create(g), n_sel=6)
    ms = dict(zip(ORDER, rep["k2_ms"]))
    assert all(t > 0 for t in ms.values())
    assert ms[24] == ms[4] and ms[28] == ms[8]
    if wide:  # rows more than 2 voxels apart: strips run as 4
        assert ms[8] == ms[16] == ms[4]
    assert rep["k2_vpl"] in ([2, 4] if wide else [2, 4, 8, 16])
    assert ms[rep["k2_vpl"]] == min(ms.values())
