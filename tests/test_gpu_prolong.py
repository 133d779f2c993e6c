"""The tiled prolongation (coarse sides above 32): part-filled tiles, values over many binary orders in
one tile, tiles that are zero, tiny or not finite."""
import numpy as np
import pytest

import oracle
from tests.gpu_common import ctx_fixture, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [32, 34, 40, 50, 64, 96, 100])
@pytest.mark.parametrize("kind", ["even", "wide", "holes", "tiny", "huge"])
def test_prolong_tiles_match_oracle(nc, kind):
    """Off by at most 1e-15 of the largest coarse value (the fixed-point parts 1.3e-16, the oracle's
    multiply-adds three roundings) and the rounding of the sum."""
    ctx = ctx_fixture()
    rng = np.random.default_rng(nc)
    c = rng.standard_normal((nc,) * 3)
    if kind == "wide":
        c *= 2.0 ** rng.integers(-60, 1, size=c.shape)
    elif kind == "holes":
        c[nc // 4: 3 * nc // 4] = 0.0
    elif kind == "tiny":
        c *= 1e-290
    elif kind == "huge":
        c *= 1e300
    f = rng.standard_normal((2 * nc,) * 3) * np.abs(c).max()
    got = host(ctx.step_prolong_add(dev(c), dev(f)))
    ref = oracle.prolong_add(c, f)
    ctx.close()
    assert np.all(np.abs(got - ref) <= 1e-15 * np.abs(c).max() + 2.3e-16 * np.abs(ref))


def test_prolong_tiles_keep_what_is_not_finite():
    """A coarse Inf or NaN reaches the fine cells that read it and no others."""
    ctx = ctx_fixture()
    nc = 40
    c = np.random.default_rng(1).standard_normal((nc,) * 3)
    c[3, 5, 7], c[20, 39, 0] = np.inf, np.nan
    f = np.zeros((2 * nc,) * 3)
    got = host(ctx.step_prolong_add(dev(c), dev(f)))
    ref = oracle.prolong_add(c, f)
    ctx.close()
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    ok = np.isfinite(ref)
    assert np.all(np.abs(got[ok] - ref[ok]) <= 1e-15 * 6.0)
