"""The coarse visits in one cluster (k_visit.cu): solves whose coarse grids take every distribution
(CTA 0 alone, one plane a CTA, two planes a CTA, a shorter last CTA; even, odd and ragged sides),
against the oracle.  Solves to 1e-12 agree with the oracle's to 1e-10 (residual over error, as in the
other parity tests)."""
import numpy as np
import pytest

import oracle
import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    c.close()


def _mg():
    import paper_1511_08200_gb300 as mg
    return mg


@pytest.mark.parametrize("n,kw", [(8, {}), (16, {}), (24, {}), (32, {}), (48, {}), (64, dict(nu1=3, nu2=1)),
                                  (32, dict(nu1=1, nu2=1)), (32, dict(nu1=1, nu2=2)), (48, dict(nu_coarse=3))])
def test_periodic(ctx, n, kw):
    alpha, s, h = nominal()
    d = workload.lognormal_delta(n, 1.0, n)
    p = _mg().default_params(alpha=alpha, s=s, h=h, tol=1e-12, **kw)
    phi, _, info = ctx.solve_fifth_force(dev(d), p)
    ref, _ = oracle.solve(d, alpha, s, h, tol=1e-13)
    assert info.status == 0
    assert rel_l2(host(phi), ref) <= 1e-10


@pytest.mark.parametrize("fmg", [False, True])
@pytest.mark.parametrize("unit", [1e-20, 1.0, 1e15])
def test_any_unit_and_a_cold_start(ctx, unit, fmg):
    """phi and its source in any unit (the visit's exponent is its own); linear (alpha = 0) too."""
    alpha, s, h = nominal()
    n = 32
    d = workload.lognormal_delta(n, 1.0, 2)
    for a in (alpha / unit, 0.0):
        p = _mg().default_params(alpha=a, s=s * unit, h=h, tol=1e-12)
        phi, _, info = ctx.solve_fifth_force(dev(d), p, fmg=fmg)
        ref, _ = oracle.solve(d, a * unit, s, h, tol=1e-13)
        assert info.status == 0
        assert rel_l2(host(phi) / unit, ref) <= 1e-10


@pytest.mark.parametrize("pf", [(8, 8, 8), (16, 16, 16), (24, 20, 36), (20, 24, 12), (36, 18, 20), (48, 40, 24),
                                (14, 12, 10)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 2)])
def test_patch(ctx, pf, nu):
    alpha, s, h = nominal()
    m = max(pf)
    d = np.ascontiguousarray(workload.lognormal_delta(m + m % 2, 1.0, 1)[:pf[0], :pf[1], :pf[2]])
    rng = np.random.Generator(np.random.PCG64(4))
    box = 0.1 * s * h * h * rng.standard_normal([p + 2 for p in pf])
    p = _mg().default_params(alpha=alpha, s=s, h=h, tol=1e-12, nu1=nu[0], nu2=nu[1])
    got, info = ctx.relax_patch(dev(d), p, 0.01 * s, dev(box))
    ref, _, _ = oracle.relax_patch(d, box, alpha, s, h, 0.01 * s, tol=1e-12)
    assert info.status == 0
    assert rel_l2(host(got), ref) <= 1e-10
    # the ghosts are the caller's
    g = host(got)
    for a in range(3):
        for e in (0, -1):
            assert np.array_equal(np.take(g, e, a), np.take(box, e, a))


def test_not_finite_input_is_reported(ctx):
    mg = _mg()
    alpha, s, h = nominal()
    d = workload.lognormal_delta(32, 1.0, 2)
    d[3, 4, 5] = np.nan
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-10)
    _, _, info = ctx.solve_fifth_force(dev(d), p, raise_on_status=False)
    assert info.status == mg.E_NONFINITE
