"""The split-arithmetic FP64 kernels (mg5_split.cuh) at the edges of their tiles and of their
range, against the oracle.

Tolerances: a sweep's change of a cell is good to ~2^-44 of itself and the sum is rounded in FP64:
1e-13 of the field's largest value.  A residual is good to ~2^-46 of its largest term plus the FP64
oracle's own rounding of the face sum, 2^-53 * 12 |phi| / h^2: both derived below per case."""
import numpy as np
import pytest

import oracle
import workload
from tests.gpu_common import ctx_fixture, dev, host, nominal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    c.close()


def _fields(n, seed, amp=1.0, eps=1.0):
    """A smooth field plus 1% noise whose nonlinear terms are of the order of eps of the linear ones."""
    alpha, s, h = nominal()
    rng = np.random.Generator(np.random.PCG64(seed))
    x = 2 * np.pi * np.arange(n) / n
    phi = (np.sin(x)[:, None, None] * np.cos(2 * x)[None, :, None] + 0.5 * np.sin(x)[None, None, :]
           + 0.01 * rng.standard_normal((n, n, n)))
    lap = sum(np.roll(phi, d, a) for a in range(3) for d in (1, -1)) - 6 * phi
    phi *= eps * h * h / (alpha * np.abs(lap).max())
    f = oracle.operator(phi, h, alpha) * (1 + 0.3 * rng.standard_normal((n, n, n)))
    return phi * amp, f * amp, h, alpha / amp


def _tols(phi, f, c, h, alpha):
    lap = (sum(np.roll(phi, d, a) for a in range(3) for d in (1, -1)) - 6 * phi) / h**2
    terms = np.abs(f).max() + abs(c) + np.abs(lap).max() + 4 * alpha * np.abs(lap).max()**2
    return 1e-13 * np.abs(phi).max(), 2.0**-44 * terms + 2.0**-53 * 12 * np.abs(phi).max() / h**2


@pytest.mark.parametrize("n", [48, 50, 62, 64, 66, 72, 94, 98, 130, 160])
def test_sweep_and_residual_match_oracle(ctx, n):
    phi, f, h, alpha = _fields(n, n)
    c = 0.01 * np.abs(f).max()
    ts, tr = _tols(phi, f, c, h, alpha)
    got = host(ctx.step_sweep(dev(phi), dev(f), c, h, alpha))
    assert np.abs(got - oracle.sweep(phi, f, c, h, alpha)).max() <= ts
    got = host(ctx.step_residual(dev(phi), dev(f), c, h, alpha))
    assert np.abs(got - oracle.residual(phi, f, c, h, alpha)).max() <= tr


@pytest.mark.parametrize("amp", [1e-25, 1e12, 1e40])
def test_any_unit_of_length(ctx, amp):
    """Tiles whose exponent leaves the FP32 range are computed in FP64: the result scales."""
    n = 64
    phi, f, h, alpha = _fields(n, 3, amp)
    ts, tr = _tols(phi, f, 0.0, h, alpha)
    got = host(ctx.step_sweep(dev(phi), dev(f), 0.0, h, alpha))
    assert np.abs(got - oracle.sweep(phi, f, 0.0, h, alpha)).max() <= ts
    got = host(ctx.step_residual(dev(phi), dev(f), 0.0, h, alpha))
    assert np.abs(got - oracle.residual(phi, f, 0.0, h, alpha)).max() <= tr


def test_strongly_nonlinear_cells(ctx):
    """Discriminants on both sides of 0.25, and clamped ones, take the FP64 root."""
    n = 64
    phi, f, h, alpha = _fields(n, 5, eps=6.0)
    got = host(ctx.step_sweep(dev(phi), dev(f), 0.0, h, alpha))
    ref = oracle.sweep(phi, f, 0.0, h, alpha)
    # a cell at the double root moves by the square root of a rounding of its discriminant
    assert np.abs(got - ref).max() <= 1e-9 * np.abs(ref).max()


def test_zero_field_is_exact(ctx):
    n = 64
    _, f, h, alpha = _fields(n, 7)
    got = host(ctx.step_residual(dev(np.zeros_like(f)), dev(f), 0.25, h, alpha))
    assert np.array_equal(got, f + 0.25)


def test_non_finite_cells_stay_local(ctx):
    """A NaN source reaches its own cell's residual, a NaN value its stencil; the other cells are
    the FP64 values."""
    n = 64
    phi, f, h, alpha = _fields(n, 9)
    _, tr = _tols(phi, f, 0.0, h, alpha)
    f2 = f.copy()
    f2[5, 6, 7] = np.nan
    got = host(ctx.step_residual(dev(phi), dev(f2), 0.0, h, alpha))
    ref = oracle.residual(phi, f, 0.0, h, alpha)
    bad = np.isnan(got)
    assert bad.sum() == 1 and bad[5, 6, 7]
    assert np.abs(got - ref)[~bad].max() <= tr
    p2 = phi.copy()
    p2[9, 8, 31] = np.inf
    got = host(ctx.step_residual(dev(p2), dev(f), 0.0, h, alpha))
    bad = ~np.isfinite(got)
    assert bad.sum() == 19
    assert np.abs(got - ref)[~bad].max() <= tr


def test_residual_over_its_source(ctx):
    n = 64
    phi, f, h, alpha = _fields(n, 11)
    want = host(ctx.step_residual(dev(phi), dev(f), 0.0, h, alpha))
    g = dev(f)
    ctx.step_residual(dev(phi), g, 0.0, h, alpha, out=g)
    assert np.array_equal(host(g), want)


@pytest.mark.parametrize("pf", [(48, 40, 72), (42, 40, 62), (66, 34, 34)])
def test_patch_matches_oracle(ctx, pf):
    """Ragged refinements whose finest grid takes the split kernels."""
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    m = max(pf)
    d = np.ascontiguousarray(workload.lognormal_delta(m + m % 2, 1.0, 1)[:pf[0], :pf[1], :pf[2]])
    box = np.zeros([p + 2 for p in pf])
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12)
    got, info = ctx.relax_patch(dev(d), p, 0.0, dev(box))
    r = oracle.patch_residual(host(got), s * d, 0.0, h, alpha)
    assert info.status == 0
    assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(s * d)
