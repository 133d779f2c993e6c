"""The FP32 column march on sides that its 16 x 32 tiles do not divide (the automatic chunk of the
fused form), and in the short chunks of small grids."""
import numpy as np
import pytest

import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


# last tiles of 4 .. 28 columns and 4 .. 12 rows
@pytest.mark.parametrize("n", [32, 36, 40, 48, 52, 56, 60, 64, 72, 88, 104, 120, 176])
def test_ragged_march_solve_is_bit_identical(n):
    """The same update of the same operands in the same order as the fused gather kernel, which a
    set chunk of planes selects: a mixed solve is equal to the bit."""
    import paper_1511_08200_gb300 as mg
    ctx = ctx_fixture()
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.5, 51))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-8, precision="mixed")
    sides = [m for m in (n >> q for q in range(8)) if m >= 32 and m % 4 == 0]
    out = []
    for chunk in (16, 0):
        mg.tune_clear()
        if chunk:
            for m in sides:
                mg.schedule_set(0, "mixed", m, form=mg.SWEEP_FUSED, chunk=chunk)
        phi, _, info = ctx.solve_fifth_force(d, p)
        out.append((host(phi), info.cycles))
    mg.tune_clear()
    ctx.close()
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][0], out[1][0]), np.argwhere(out[0][0] != out[1][0])[:8].tolist()
