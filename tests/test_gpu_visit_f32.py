"""A coarse visit of the FP32 V-cycles as the solves run it (marched sweeps, right-hand side and
restriction, tiled prolongation, the bottom in one CTA) against the kernels that gather, a launch a step."""
import numpy as np
import pytest

import workload
from tests import _pins
from tests.gpu_common import ctx_fixture, host, nominal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = ctx_fixture()
    yield c
    c.close()


def _f32(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _visit(ctx, n, nu):
    import paper_1511_08200_gb300 as mg
    alpha, s, h = nominal()
    p = mg.default_params(alpha=alpha, s=s, h=h, tol=1e-8, precision="mixed")
    p.nu1, p.nu2, p.nu_coarse = nu
    B = _pins.fft_poisson(s * workload.lognormal_delta(n, 1.0, 91), h)   # the linear field
    e = 1e-2 * B * (1.0 + 0.1 * workload.lognormal_delta(n, 1.0, 92))
    f = 1e-2 * s * (workload.lognormal_delta(n, 1.0, 93) + 0.1)
    args = (_f32(e), _f32(f), _f32(B), 1e-3 * s, p)
    (a, ca), (b, cb) = ctx.step_visit_f32(*args, plain=True), ctx.step_visit_f32(*args)
    return host(a), ca, host(b), cb


# Marches: rhs above 64, restriction from 112 on sides that are no multiple of 32 and from 32 on those that are;
# sweeps on ragged sides; last tiles of 4 .. 24 columns and 4 .. 12 rows.  12, 24, 48, 96: the bottom of 12^3.
@pytest.mark.parametrize("n", [12, 20, 24, 36, 48, 60, 72, 80, 88, 104, 112, 120, 144, 176, 208, 240])
@pytest.mark.parametrize("nu", [(2, 2, 500), (1, 2, 4), (3, 0, 7)])
def test_visit_is_bit_identical(ctx, n, nu):
    """No statistics but in the gather kernels' order: equal to the bit."""
    a, ca, b, cb = _visit(ctx, n, nu)
    assert ca == cb
    assert np.array_equal(a, b), np.argwhere(a != b)[:8].tolist()


@pytest.mark.parametrize("n", [8, 16, 32, 64, 96, 128, 160])
@pytest.mark.parametrize("nu", [(2, 2, 4), (1, 2, 4), (3, 1, 7)])
def test_visit_with_other_sums(ctx, n, nu):
    """Multiples of 32 (the march's own statistics) and the bottom of 8^3 and 16^3: a mean that is rounded
    otherwise moves c by a few 2^-24 of the residual, and the fields by some of their roundings: 2^-17 of
    the largest value (the coarsest grid's sweeps are capped, so that no stopping test turns)."""
    a, ca, b, cb = _visit(ctx, n, nu)
    top = np.abs(a).max()
    assert np.abs(a - b).max() <= 2.0**-17 * top
    _, s, _ = nominal()
    assert abs(ca - cb) <= 2.0**-17 * 1e-2 * s
