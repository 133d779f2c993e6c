"""Interpolation to a refinement of values near the largest double: no intermediate result may leave the range."""
import numpy as np
import pytest

import oracle
from tests.gpu_common import ctx_fixture, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [1.0, 1e306, 1.7e308])
@pytest.mark.parametrize("n", [16, 24])
def test_values_near_the_largest_double(n, top):
    """Weighted means of eight values: within four roundings of the largest of them; as finite as they are."""
    ctx = ctx_fixture()
    c = np.random.default_rng(n).uniform(-1.0, 1.0, (n,) * 3)
    c[2, 3, 4], c[2, 3, 5] = 1.0, -1.0
    c *= top
    o, p = (n - 3, 1, 2), (6, 8, 10)
    got = host(ctx.refine_interpolate(dev(c), o, p, 1))
    ref = oracle.refine_interpolate(c / top, o, p, 1)
    assert np.isfinite(got).all()
    assert np.abs(got / top - ref).max() <= 1e-15
    c[5, 5, 5], c[2, 3, 4] = np.inf, np.nan
    got = host(ctx.refine_interpolate(dev(c), (0, 0, 0), (n // 2,) * 3, 1))
    ref = oracle.refine_interpolate(c, (0, 0, 0), (n // 2,) * 3, 1)
    ctx.close()
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    ok = np.isfinite(ref)
    assert np.abs((got[ok] - ref[ok]) / top).max() <= 1e-15


@pytest.mark.parametrize("top", [1e306, 1.7e308])
def test_boxes_too(top):
    ctx = ctx_fixture()
    box = np.random.default_rng(3).uniform(-1.0, 1.0, (12, 14, 16)) * top
    got = host(ctx.refine_interpolate_box(dev(box), 1, (1, 2, 3), (4, 6, 8), 1))
    ref = host(ctx.refine_interpolate_box(dev(box / top), 1, (1, 2, 3), (4, 6, 8), 1))
    ctx.close()
    assert np.isfinite(got).all() and np.abs(got / top - ref).max() <= 1e-15
