"""The FP64 coarse visits that start over because a value outgrows its unit (a first attempt without
headroom forces it), and those that give up."""
import numpy as np
import pytest

import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    c.close()


def _counts(i):
    return i.status, i.cycles, i.coarse_sweeps, i.disc_clamped


# The start is solved to 1e-4, so the unit comes from the field's values, which do not fit it without
# headroom: 1, 2 and 3 attempts fail, and the next has the default's unit.
@pytest.mark.parametrize("bits", [-6, -14, -22])
@pytest.mark.parametrize("n", [16, 24, 32, 48])
def test_a_repeated_visit_is_the_same(ctx, n, bits):
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 41))
    start, _, _ = ctx.solve_fifth_force(d, mg.default_params(alpha=alpha, s=s, h=h, tol=1e-4))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12)
    out = []
    for b in (2, bits):
        ctx.set_visit_headroom(b)
        phi, _, info = ctx.solve_fifth_force(d, p, phi=start.clone(), warm=True)
        out.append((host(phi), _counts(info)))
    ctx.set_visit_headroom()
    assert out[0][1] == out[1][1] and out[0][1][0] == 0
    assert np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("bits", [-6, -22])
@pytest.mark.parametrize("pf", [(16, 16, 16), (24, 20, 36), (48, 40, 24), (16, 48, 40)])
def test_a_repeated_patch_visit_is_the_same(ctx, pf, bits):
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    m = max(pf)
    d = dev(np.ascontiguousarray(workload.lognormal_delta(m + m % 2, 1.0, 42)[:pf[0], :pf[1], :pf[2]]))
    box = dev(0.1 * s * h * h * np.random.default_rng(4).standard_normal([q + 2 for q in pf]))
    ctx.relax_patch(d, mg.default_params(alpha=alpha, s=s, h=h, tol=1e-4), 0.01 * s, box)
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12)
    out = []
    for b in (2, bits):
        ctx.set_visit_headroom(b)
        got, info = ctx.relax_patch(d, p, 0.01 * s, box.clone())
        out.append((host(got), _counts(info)))
    ctx.set_visit_headroom()
    assert out[0][1] == out[1][1] and out[0][1][0] == 0
    assert np.array_equal(out[0][0], out[1][0])


@pytest.mark.parametrize("n", [16, 32])
def test_a_visit_that_gives_up_leaves_no_correction(ctx, n):
    """Seven attempts from -62 bits end at -14: the sweeps of the finest grid remain, which do not make
    the field worse, and nothing that is not finite gets into it."""
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 43))
    start, _, i0 = ctx.solve_fifth_force(d, mg.default_params(alpha=alpha, s=s, h=h, tol=1e-4))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12, max_cycles=3)
    ctx.set_visit_headroom(-62)
    phi, _, info = ctx.solve_fifth_force(d, p, phi=start.clone(), warm=True, raise_on_status=False)
    ctx.set_visit_headroom()
    assert info.status == mg.E_NOT_CONVERGED
    assert np.isfinite(host(phi)).all() and info.rel_residual <= i0.rel_residual


def test_headroom_is_checked(ctx):
    import paper_1511_08200_gb300 as mg
    for bits in (3, -65):
        with pytest.raises(mg.MG5Error):
            ctx.set_visit_headroom(bits)
