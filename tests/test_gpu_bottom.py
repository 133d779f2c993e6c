"""The bottom of the FP32 V-cycles in one CTA: every hierarchy that ends in it, odd sweep counts (the
arrays change places at every sweep), a capped and a converged coarsest grid."""
import numpy as np
import pytest

import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


# 16: 8, 4; 24: 12, 6; 32 and 64: 16, 8, 4; 48: 24 by launches, 12, 6
@pytest.mark.parametrize("n", [16, 24, 32, 48, 64])
@pytest.mark.parametrize("nu", [(2, 2, 500), (1, 2, 500), (3, 1, 4), (2, 1, 7)])
def test_mixed_solve_through_the_bottom(n, nu):
    """The mixed solve reaches its tolerance and the FP64 solve's field.  The residual is 1e-8 of the
    source; if all of it lay in the lowest mode, which holds at least 1e-3 of the source's norm,
    phi would be off by 1e-5."""
    import paper_1511_08200_gb300 as mg
    ctx = ctx_fixture()
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 61))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-8, precision="mixed")
    p.nu1, p.nu2, p.nu_coarse = nu
    phi, _, info = ctx.solve_fifth_force(d, p)
    q = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-11)
    ref, _, _ = ctx.solve_fifth_force(d, q)
    ctx.close()
    assert info.status in (0, 1)
    a, b = host(phi), host(ref)
    assert np.abs(a - b).max() <= 1e-5 * np.abs(b).max()
