"""The sampling tables of environments with black texels: running sums in order,
so that no entry is below the one before it and a black texel or row has no width
(a sample that fell on one would have a density of an ulp over the total)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev  # noqa: E402


def tables(env):
    E = irgs.EnvMap(dev(env))
    m = E.export()
    E.close()
    return m["row_cdf"], m["col_cdf"]


def black_stretches(h, w, seed):
    """Random rows with a black stretch each, and black rows."""
    rng = np.random.default_rng(seed)
    env = np.exp(rng.normal(size=(h, w, 3))).astype(np.float32)
    for r in range(h):
        a, b = np.sort(rng.integers(0, w + 1, 2))
        env[r, a:b] = 0.0
    env[rng.random(h) < 0.3] = 0.0
    return env


def equal_lights(h, w, seed):
    """A few equal lights on black."""
    rng = np.random.default_rng(seed)
    env = np.zeros((h, w, 3), np.float32)
    for r in range(0, h, 2):
        env[r, rng.choice(w, min(w, 2 + r % 5), replace=False)] = 0.1 + rng.random(3)
    return env


@pytest.mark.parametrize("make", [black_stretches, equal_lights])
@pytest.mark.parametrize("h,w", [(1, 1), (3, 31), (33, 32), (200, 65), (64, 512), (257, 1000)])
def test_never_decrease_and_flat_over_black(make, h, w):
    env = make(h, w, h * w)
    row, col = tables(env)
    lum = (env.astype(np.float64) @ np.array([0.2126, 0.7152, 0.0722]))
    d = np.diff(col, axis=1)
    assert np.all(d >= 0) and np.all(d[lum == 0] == 0)
    d = np.diff(row)
    assert np.all(d >= 0) and np.all(d[lum.sum(1) == 0] == 0)


@pytest.mark.parametrize("w", [1, 31, 32, 33, 512, 1001])
def test_running_sums_bit_for_bit(w):
    """One row: sin(theta) is 1, so the table is NumPy's sequential sum of the luminances."""
    for make in (black_stretches, equal_lights):
        for seed in range(8):
            env = make(1, w, seed)
            e = env[0].astype(np.float64)
            lum = 0.2126 * e[:, 0] + 0.7152 * e[:, 1] + 0.0722 * e[:, 2]
            row, col = tables(env)
            want = np.concatenate([[0.0], np.cumsum(lum)])
            assert np.array_equal(col[0], want)
            assert row[0] == 0.0 and row[1] == want[-1]


def test_samples_never_land_on_black():
    """Every sample's density is that of a lit texel: luminance over its mean on the sphere."""
    h, w = 64, 256
    env = equal_lights(h, w, 5)
    lum = env.astype(np.float64) @ np.array([0.2126, 0.7152, 0.0722])
    total = (lum * np.sin((np.arange(h) + 0.5) * np.pi / h)[:, None]).sum()
    E = irgs.EnvMap(dev(env))
    _, pdf, valid = irgs.relight_sample_rays(E, 1 << 16, 16, 7)
    E.close()
    assert bool((valid == 1).all())
    # inside a texel sin(theta) moves by up to half a texel around its centre's: a factor of 2 at the poles, less elsewhere
    assert float(pdf.min()) > 0.45 * lum[lum > 0].min() / total * w * h / (2 * np.pi ** 2)
