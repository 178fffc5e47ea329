"""Work cut into pieces: environments of fewer and more texels than a slice
holds or the slices can be, and served tiles that are no multiple of a unit's
128 rays."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from paper_2412_15867_gb300 import serve  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402


@pytest.mark.parametrize("h,w", [(1, 1), (1, 7), (3, 5), (31, 66), (32, 64), (401, 353)])
def test_constant_environment(h, w):
    """Prefiltering a constant gives it back, and the sampling tables count texels
    (sums of up to 141,553 FP32 terms in slices: 1e-5 relative)."""
    L = np.array([1.5, 0.25, 3.0], np.float32)
    E = irgs.EnvMap(dev(np.broadcast_to(L, (h, w, 3)).copy()))
    m = E.export()
    E.close()
    seen = m["pref"].any(-1)          # a coarse environment may have no texel centre in front of a direction
    assert seen.mean() > 0.4 and np.all(np.abs(m["pref"][seen] - L) <= 1e-5 * L)
    lum = 0.2126 * float(L[0]) + 0.7152 * float(L[1]) + 0.0722 * float(L[2])
    s = np.sin((np.arange(h) + 0.5) * np.pi / h)
    np.testing.assert_allclose(m["col_cdf"], lum * s[:, None] * np.arange(w + 1)[None], rtol=1e-12, atol=1e-300)
    np.testing.assert_allclose(m["row_cdf"], np.concatenate([[0], np.cumsum(lum * s * w)]), rtol=1e-12, atol=1e-300)
    if h >= 31:                       # the cosine integral over texel centres converges with the texel size
        assert np.all(np.abs(m["irr"] - L) <= 8.0 / h ** 2 * L)


def test_non_finite_texels_stay_on_their_side():
    """A texel enters only the sums of directions that face it."""
    env = np.ones((16, 32, 3), np.float32)
    env[0, :] = np.inf                # around +z
    m = irgs.EnvMap(dev(env)).export()
    assert np.isfinite(m["irr"][-4:]).all() and not np.isfinite(m["irr"][:4]).any()
    assert np.isfinite(m["pref"][:, -8:]).all()


@pytest.mark.parametrize("tile_px", [1, 127, 128, 129, 1000])
def test_served_tiles(tile_px):
    S = make_scene(irgs, synth.object_scene(n=4000, seed=71))
    srv = serve.Server([S], tile_px=tile_px, max_tiles=4096, step_rays=1 << 20)
    eye = (2.5, -2.0, 1.5)
    h = srv.submit(serve.RenderRequest(scene=0, eye=eye, width=40, height=24))
    g = srv.submit(serve.RelightRequest(scene=0, eye=eye, width=24, height=16, spp=3, env=dev(synth.env_map(seed=3, height=16, width=32)), seed=4))
    srv.run_until_idle()
    assert S.status() == 0
    o, d = serve.camera_rays(serve.make_camera(eye, 40, 24))
    ref = irgs.trace_forward(S, o, d, srv.render_p)
    for k in ("feat", "depth", "opacity"):
        assert torch.equal(h.out[k], ref[k]), k
    assert torch.isfinite(g.out["rgb"]).all()
    srv.close()
