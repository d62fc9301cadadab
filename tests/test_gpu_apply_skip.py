"""The FP64 apply over a whole grid copies tiles (3D: layers of a unit) that
hold no active unknown.  Against the oracle's matrix on geometries with large inactive regions,
at sizes around the tiles; and infinities, NaN and values near the overflow
limit must spread as the full arithmetic spreads them (0 times infinity is NaN),
which the FP32 apply, without such a shortcut, shows."""
import numpy as np
import pytest

from gpu_common import abs_matvec, gpu_apply_fields, gpu_context, oracle_system, require_gpu
from paper_1010_2832_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {
    "bumps2d": lambda: W.bumps_2d(97, seed=4),
    "disk2d": lambda: W.disk_in_box(70, radius=0.12),
    "rand2d": lambda: W.random_small((33, 17), seed=5),
    "rand3d": lambda: W.random_small((37, 19, 23), seed=6, dim=3),
    "col3d": lambda: W.column_3d(24),
    "tall3d": lambda: W.random_small((20, 9, 61), seed=9, dim=3),
}
_c = {}


def _setup(name):
    require_gpu()
    if name not in _c:
        wl = CASES[name]()
        _c[name] = (wl, oracle_system(wl), gpu_context(wl)[0])
    return _c[name]


@pytest.mark.parametrize("name", list(CASES))
def test_fp64_apply_matches_the_matrix(name):
    wl, S, ctx = _setup(name)
    x = np.random.default_rng(1).normal(size=S.A.shape[0])
    y = gpu_apply_fields(ctx, x, 0)
    # each entry sums at most about thirty products, each rounded a few times
    assert np.all(np.abs(y - S.A @ x) <= 1e-13 * abs_matvec(S.A, x) + 1e-300)
    # scaled by 2^905 every tile that holds a value takes the full arithmetic,
    # and a power of two changes no rounding
    big = gpu_apply_fields(ctx, x * 2.0 ** 905, 0)
    assert np.all(np.isfinite(big))
    assert np.array_equal(big * 2.0 ** -905, y)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("name", list(CASES))
def test_non_finite_values_spread_alike(name, value):
    wl, S, ctx = _setup(name)
    rng = np.random.default_rng(2)
    n = S.A.shape[0]
    for k in rng.integers(0, n, 6):
        x = rng.normal(size=n)
        x[k] = value
        y64 = gpu_apply_fields(ctx, x, 0)
        y32 = gpu_apply_fields(ctx, x, 1)
        assert np.array_equal(np.isnan(y64), np.isnan(y32))
        assert np.array_equal(np.isinf(y64), np.isinf(y32))
