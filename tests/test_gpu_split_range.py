"""The split-arithmetic FP64 kernels where a tile's values are tiny beside its source: residuals whose
squares leave the FP32 range, tiles of zeros, and sources that a tile's unit would round away."""
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


def _guess(kind, n, unit):
    """A warm start in units of h^2 s (the size of h^2 times the source), tiny in most tiles or in all:
    a Gaussian that falls to 1e-17 at the corners, noise of 1e-16 (both far above 2^-90), noise of 1
    in half of the grid and 1e-7 in the other (a thread's tiles then differ by 2^23)."""
    rng = np.random.default_rng(n)
    if kind == "gaussian":
        x = np.arange(n) - n / 2 + 0.5
        g = np.exp(-x**2 / (2 * (0.098 * n) ** 2))
        return unit * g[:, None, None] * g[None, :, None] * g[None, None, :]
    u = unit * rng.standard_normal((n,) * 3)
    if kind == "noise":
        return 1e-16 * u
    u[n // 2:] *= 1e-7
    return 1e-9 * u


@pytest.mark.parametrize("n", [64, 128, 144])
@pytest.mark.parametrize("kind", ["gaussian", "noise", "halves"])
def test_warm_start_from_a_tiny_guess(ctx, n, kind):
    """Reaches its tolerance and the cold solve's field.  Each residual is 1e-12 of the source; if all
    of both lay in the lowest mode, which holds at least 1e-3 of the source's norm, the fields would
    differ by 2e-9."""
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 81))
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12)
    cold, _, _ = ctx.solve_fifth_force(d, p)
    phi = dev(_guess(kind, n, h * h * s))
    phi, _, info = ctx.solve_fifth_force(d, p, phi=phi, warm=True)
    assert info.status == 0 and info.rel_residual <= 1e-12
    assert rel_l2(host(phi), host(cold)) <= 2e-9


def test_patch_from_a_tiny_guess_without_presmoothing(ctx):
    """The finest grid's restriction sees the guess itself."""
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    pf = (48, 40, 72)
    d = np.ascontiguousarray(workload.lognormal_delta(72, 1.0, 1)[:pf[0], :pf[1], :pf[2]])
    box = 1e-16 * h * h * s * np.random.default_rng(5).standard_normal([q + 2 for q in pf])
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-12, nu1=0, nu2=4)
    got, info = ctx.relax_patch(dev(d), p, 0.0, dev(box))
    r = oracle.patch_residual(host(got), s * d, 0.0, h, alpha)
    assert info.status == 0
    assert np.linalg.norm(r) <= 2e-12 * np.linalg.norm(s * d)


@pytest.mark.parametrize("n", [64, 66])
def test_large_and_small_residuals_over_their_source(ctx, n):
    """Residuals of 2^33 .. 2^68 of a tile's unit, in place: each is the source to the rounding of the sum
    (2^-47 where it is a pair)."""
    alpha, s, h = nominal()
    rng = np.random.default_rng(n)
    phi = rng.standard_normal((n,) * 3)
    f = 2.0 ** rng.uniform(15.0, 50.0, (n,) * 3) / h**2
    for out in (False, True):
        g = dev(f)
        got = host(ctx.step_residual(dev(phi), g, 0.0, h, 1e-12, out=g if out else None))
        ref = oracle.residual(phi, f, 0.0, h, 1e-12)
        assert np.all(np.abs(got - ref) <= 2.0**-46 * np.abs(ref) + 2.0**-46 * 24 * np.abs(phi).max() / h**2)


@pytest.mark.parametrize("n", [64, 66])
@pytest.mark.parametrize("where", ["everywhere", "a block"])
@pytest.mark.parametrize("size", [1e-30, 1e-24, 1.0, 1e20])
def test_sweep_of_zeros(ctx, n, where, size):
    """The half-sweep of a tile of zeros, with h^2 f of any size (alpha f stays what it is): a change is
    good to 2^-44 of itself, in a tile's unit to 2^-60 of the largest."""
    alpha, s, h = nominal()
    rng = np.random.default_rng(n)
    f = rng.standard_normal((n,) * 3)
    f[:, :, n // 2:] = 0.0
    phi = np.zeros_like(f)
    scale = size / h**2
    if where == "a block":
        phi[n // 2:] = 0.1 * h * h * rng.standard_normal((n - n // 2, n, n))
    a = 0.01 / scale
    got = host(ctx.step_sweep(dev(phi * scale), dev(f * scale), 0.0, h, a))
    ref = oracle.sweep(phi * scale, f * scale, 0.0, h, a)
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
    quiet = np.s_[2:n // 2 - 2, :, n // 2 + 2:-2]   # no source and no value around
    assert np.array_equal(got[quiet], np.zeros_like(got[quiet]))


@pytest.mark.parametrize("n", [64, 128])
@pytest.mark.parametrize("nu", [(2, 2), (0, 3)])
def test_a_solve_scales_by_powers_of_two(ctx, n, nu):
    """The linear equation in units 2^-70 apart (h^2 f is 1e-9 and 1e-30): no smoothing is lost, so the
    cycles are the same, and the fields to what two residuals of 1e-11 leave if all of both lay in the
    lowest mode (at least 1e-3 of the source's norm)."""
    import paper_1511_08200_gb300 as mg
    _, s, h = nominal()
    d = dev(workload.lognormal_delta(n, 1.0, 82))
    out = []
    for u in (1.0, 2.0**-70):
        p = mg.default_params(alpha=0.0, s=s * u, h=h, tol=1e-11, nu1=nu[0], nu2=nu[1])
        phi, _, info = ctx.solve_fifth_force(d, p)
        out.append((host(phi) / u, info.cycles, info.status))
    assert out[0][1:] == out[1][1:] and out[0][2] == 0
    assert rel_l2(out[0][0], out[1][0]) <= 2e-8
