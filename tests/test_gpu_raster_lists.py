"""Tile lists of the rasteriser: lengths around the runs that are sorted by a
block (2,048) and merged, rectangles around the 32 tiles that a thread hands
out itself, equal depths, discs seen from the side and close to the camera.
Bars as in test_gpu_raster."""
import numpy as np
import pytest

import oracle
import synth
from tests.helpers import scene
from tests.test_gpu_raster import compare, ocam, opar

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from paper_2412_15867_gb300 import serve  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402


def cloud(n, seed, spread, size, tilt, opacity, layers=None):
    rng = np.random.default_rng(seed)
    means = rng.uniform(-spread, spread, (n, 3)).astype(np.float32)
    if layers:   # depths without rounding, many of them equal: their order is the user's
        means[:, 2] = (rng.integers(0, layers, n) / 16384).astype(np.float32)
    quats = np.c_[np.ones(n), rng.uniform(-tilt, tilt, (n, 3))].astype(np.float32)
    return scene(means, quats, (size * rng.uniform(0.5, 1.5, (n, 2))).astype(np.float32),
                 rng.uniform(*opacity, n).astype(np.float32), rng.uniform(size=(n, 3)).astype(np.float32))


def check(sc, cam, p, frac=0.999):
    S = make_scene(irgs, sc)
    out = irgs.rasterize(S, cam, p)
    assert S.status() == 0
    ref = oracle.rasterize(sc, ocam(cam), opar(p))
    print(compare(out, ref, frac=frac))
    return out


@pytest.mark.parametrize("n", [1, 31, 33, 255, 257, 2047, 2048, 2049, 4096, 4097, 6200])
@pytest.mark.parametrize("layers", [6000, 7])
def test_list_lengths(n, layers):
    sc = cloud(n, 3 * n + 1, 0.2, 0.3, 0.2, (0.01, 0.03), layers)
    cam = serve.make_camera((0, 0, 5.0), 13, 11, target=(0, 0, 0), fov_deg=4.0)
    out = check(sc, cam, irgs.TraceParams(k=16, feat_count=3, t_min=0.1, T_min=0.0))
    assert int(out["n_hits"].max()) > 0.9 * n


@pytest.mark.parametrize("w,h", [(16, 512), (512, 17), (97, 81), (113, 80), (300, 200)])
def test_rectangles_of_many_tiles(w, h):
    """Discs of a few pixels and of the whole image, in one warp."""
    a, b = cloud(150, w, 1.0, 0.02, 1.0, (0.3, 0.9)), cloud(150, h, 1.0, 1.5, 1.0, (0.05, 0.3))
    mix = np.random.default_rng(w + h).permutation(300)
    sc = scene(*(np.concatenate([x, y])[mix] for x, y in zip(a.arrays(), b.arrays())))
    cam = serve.make_camera((0, 0, 4.0), w, h, target=(0, 0, 0), fov_deg=40.0)
    check(sc, cam, irgs.TraceParams(k=16, feat_count=3, t_min=0.1))


@pytest.mark.parametrize("eye", [(0.0, 0.0, 4.0), (0.9, 0.1, 0.2), (0.0, 0.2, 0.0)])
def test_oblique_discs_and_cameras_among_them(eye):
    """Long thin discs, seen from outside and from between them. A hit's depth is
    off by 3e-7 tau / |n.d|: above 1e-4 for |n.d| < 3e-3 tau, which a few in 1e5
    of the hits of randomly turned discs are, twenty to a pixel."""
    rng = np.random.default_rng(17)
    sc = cloud(800, 18, 1.0, 0.1, 3.0, (0.1, 0.95))
    arr = list(sc.arrays())
    arr[2] = (arr[2] * np.c_[rng.uniform(0.01, 0.1, 800), rng.uniform(1, 4, 800)]).astype(np.float32)
    cam = serve.make_camera(eye, 120, 90, target=(0.3, 0.2, -0.5), fov_deg=60.0)
    check(scene(*arr), cam, irgs.TraceParams(k=16, feat_count=3, t_min=0.01), frac=0.99)
