"""prox_tv started from a dual that holds infinities: the first step takes the dual
as it is.  One step, compared with the FP64 oracle where that is finite (the
infinite component's own voxels become NaN there); tolerance of the other TV tests."""
import numpy as np
import pytest

from oracle import tv as otv
from gpu_common import cuda, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.inf, -np.inf])
@pytest.mark.parametrize("component", [0, 1, 2])
def test_infinite_start_dual(component, value):
    import paper_2605_12085_gb300 as fbl
    rng = np.random.default_rng(4)
    shape = (9, 31, 40)
    v = rng.uniform(0.2, 0.8, shape).astype(np.float32)
    q0 = (0.3 * rng.standard_normal((3,) + shape)).astype(np.float32)
    q0[component, 4, 14, 29] = value
    q = cuda(q0)
    x = host(fbl.prox_tv(cuda(v), 0.08, 1, x_max=0.9, q=q, q_in=True))
    with np.errstate(invalid="ignore"):
        xr, qr = otv.prox_tv(v, 0.08, 1, x_max=0.9, q0=q0)
    ok = np.isfinite(xr)
    assert 0 < (~ok).sum() <= 2
    assert rel_l2(x[ok], xr[ok]) <= 1e-5
    okq = np.isfinite(qr)
    assert rel_l2(host(q)[okq], qr[okq]) <= 1e-4
