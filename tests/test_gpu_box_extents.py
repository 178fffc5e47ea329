"""Support boxes of discs of any size: they hold the disc's extent in 64 bits and
are at most the padding (1e-5 of the extent and 1e-6 of the coordinates, plus
rounding) larger, also where its square leaves FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev  # noqa: E402
from tests.helpers import frame_of, scene  # noqa: E402


@pytest.mark.parametrize("su,sv", [(1e-30, 1e-30), (1e-25, 1e-2), (1e-3, 0.5), (1.0, 1e25), (1e19, 1e19), (3e20, 7e30), (1e36, 2e-9)])
def test_boxes_hold_the_discs(su, sv):
    rng = np.random.default_rng(int(abs(np.log(su) + 3 * np.log(sv))))
    n = 64
    quats = rng.normal(size=(n, 4))
    quats[:8] = [[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 1, 0], [0, 0, 0, 1], [1, 1, 0, 0], [1, 0, 1, 0], [1, 0, 0, 1], [1, 1, 1, 1]]
    sc = scene(rng.uniform(-1, 1, (n, 3)), quats, np.tile([su, sv], (n, 1)), rng.uniform(0.004, 0.9, n), np.zeros((n, 1)))
    S = irgs.Scene(*(dev(a) for a in sc.arrays()))
    perm, _, _, boxes = S.export()
    assert S.status() == 0
    mu, q, s, o = (a.astype(np.float64)[perm] for a in (sc.means, sc.quats, sc.scales, sc.opacity))
    rc = np.sqrt(np.clip(2 * np.log(o / np.float64(np.float32(1 / 255))), 0, 9))
    for j in range(n):
        tu, tv, _ = frame_of(q[j])
        e = rc[j] * np.hypot(s[j, 0] * tu, s[j, 1] * tv)
        pad = 3e-5 * e + 3e-6
        lo, hi = boxes[j, :3].astype(np.float64), boxes[j, 3:].astype(np.float64)
        assert np.all(lo <= mu[j] - e) and np.all(hi >= mu[j] + e)
        assert np.all(lo >= mu[j] - e - pad) and np.all(hi <= mu[j] + e + pad)
