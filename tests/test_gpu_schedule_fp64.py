"""FP64 sides of 48 and more have one sweep kernel: no schedule changes a solve there."""
import numpy as np
import pytest

import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [48, 64, 96])
def test_no_schedule_changes_the_values(n):
    import paper_1511_08200_gb300 as mg
    ctx = ctx_fixture()
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 31))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-10)
    mg.tune_clear()
    ref = host(ctx.solve_fifth_force(d, p)[0])
    for sch in [dict(form=mg.SWEEP_TWO_PASS, block=b) for b in (32, 512)] + \
               [dict(form=mg.SWEEP_FUSED, chunk=c) for c in (0, 8)] + [dict(form=mg.SWEEP_MARCH, chunk=0)]:
        mg.tune_clear()
        for m in (n, n // 2):
            if m >= 48:
                mg.schedule_set(0, "fp64", m, **sch)
        assert np.array_equal(host(ctx.solve_fifth_force(d, p)[0]), ref), sch
    mg.tune_clear()
    ctx.autotune(n, "fp64")   # one candidate, the default
    got, tuned = mg.schedule_get(0, "fp64", n)
    mg.tune_clear()
    default, _ = mg.schedule_get(0, "fp64", n)
    ctx.close()
    assert tuned and got.ms > 0 and (got.form, got.block, got.chunk) == (default.form, default.block, default.chunk)
