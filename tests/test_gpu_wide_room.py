"""The room for wide nodes: two thirds of the surfels, reached exactly by full
binary trees of 2^(2 k + 1) leaves, and what a resident scene takes in all."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev  # noqa: E402
from tests.helpers import scene  # noqa: E402


def grid(n, scale=0.01):
    """One surfel per Morton cell, so that the radix tree is full."""
    m = np.arange(n)
    p = np.zeros((n, 3))
    for b in range(12):
        p[:, 2 - b % 3] += ((m >> b) & 1) << (b // 3)
    return scene(p, np.tile([1.0, 0.2, 0.1, 0.3], (n, 1)), np.full((n, 2), scale), np.full(n, 0.5), np.ones((n, 1)))


@pytest.mark.parametrize("hierarchy", ["radix", "clustered"])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 8, 32, 512, 2048])
@pytest.mark.parametrize("scale", [0.01, 3.4e38])   # boxes beyond FP32: areas that are not numbers
def test_full_trees_fit(n, hierarchy, scale):
    sc = grid(n, scale)
    S = irgs.Scene(*(dev(a) for a in sc.arrays()), hierarchy=hierarchy)
    W = S.export_wide()
    assert S.status() == 0
    kids = W[:, 24:28].view(np.int32)
    there = kids != np.iinfo(np.int32).min
    assert len(W) <= max((2 * n - 1) // 3, 1)
    if hierarchy == "radix" and scale < 1 and n in (8, 32, 512, 2048):
        assert len(W) == (2 * n - 1) // 3
    assert np.all(there.all(1) | ~((kids >= 0).any(1)))     # four children, or leaves alone
    assert np.array_equal(np.sort(~kids[there & (kids < 0)]), np.arange(n))
    S.refit(means=S.means + 0.25)
    assert S.status() == 0 and len(S.export_wide()) <= max((2 * n - 1) // 3, 1)


def test_bytes_per_surfel():
    sc = synth.object_scene(n=100_000, seed=2)
    S = irgs.Scene(*(dev(a) for a in sc.arrays()))
    assert sc.features.shape[1] == 10 and S.device_bytes() <= 515 * 100_000
