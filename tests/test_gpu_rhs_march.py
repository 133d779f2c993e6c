"""The FAS right-hand side of the FP32 correction form as a column march (coarse sides above 64), and its
residual and restriction on fine sides that the march's tiles do not divide (112 and above)."""
import numpy as np
import pytest

import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


# fine sides: last tiles of 8 .. 16 columns and 0 .. 8 rows; coarse sides 60 (not marched), 72, 88, 104, 128
@pytest.mark.parametrize("n", [120, 144, 176, 208, 256])
def test_mixed_solve_with_the_marches(n):
    """The mixed solve reaches its tolerance and the FP64 solve's field: the residual is 1e-8 of the
    source; if all of it lay in the lowest mode, which holds at least 1e-3 of the source's norm,
    phi would be off by 1e-5."""
    import paper_1511_08200_gb300 as mg
    ctx = ctx_fixture()
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 71))
    phi, _, info = ctx.solve_fifth_force(d, mg.default_params(alpha=alpha, s=s, h=h, tol=1e-8, precision="mixed"))
    ref, _, _ = ctx.solve_fifth_force(d, mg.default_params(alpha=alpha, s=s, h=h, tol=1e-11))
    ctx.close()
    assert info.status in (0, 1)
    a, b = host(phi), host(ref)
    assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
