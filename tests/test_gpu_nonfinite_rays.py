"""Rays that are not finite (masked pixels, points without a normal) hit nothing
and cost next to nothing, whichever way their batch is walked, and their
neighbours stay together. The bars are 20 times above what the calls take and
as far below what a walk of the whole hierarchy per ray takes."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402

P = irgs.TraceParams(k=16, feat_count=10)


@pytest.fixture(scope="module")
def scene():
    return make_scene(irgs, synth.object_scene(n=300_000, seed=5))


def ms(fn, reps=5):
    fn()
    best = float("inf")
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("what,value", [("d", np.nan), ("d", np.inf), ("o", np.nan), ("o", -np.inf)])
@pytest.mark.parametrize("axes", [(0, 1, 2), (1,)])
def test_rays_that_hit_nothing(scene, what, value, axes):
    ro, rd = synth.random_rays_through_scene(30_000, seed=3, box=1.0, radius=3.0)
    (rd if what == "d" else ro)[:, list(axes)] = value
    ro, rd = dev(ro), dev(rd)
    for flags in (0, irgs.FLAG_WARP, irgs.FLAG_PER_THREAD):
        p = P.with_(flags=flags)
        out = irgs.trace_forward(scene, ro, rd, p, max_hit_ids=4)
        assert scene.status() == 0
        for k in ("feat", "depth", "opacity", "n_hits"):
            assert not out[k].any(), k
        assert (out["hit_ids"] == -1).all()
        g = irgs.trace_backward(scene, ro, rd, p, {k: v for k, v in out.items() if k != "hit_ids"},
                                torch.ones(30_000, 10, device="cuda"))
        assert not any(v.any() for v in g.values())
        assert ms(lambda: irgs.trace_forward(scene, ro, rd, p)) < 1.5


@pytest.mark.parametrize("w,h", [(200, 200), (800, 800), (1100, 960)])
@pytest.mark.parametrize("share", [0.01, 0.1])
def test_neighbours_stay_together(scene, w, h, share):
    """A view with masked pixels: by a warp per ray, as packets, in compacted rounds."""
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=9), w, h)
    bad = np.random.default_rng(w).random(w * h) < share
    bad[[0, 1, w - 1, w]] = False          # by these the batch's rows are told
    masked = rd.copy()
    masked[bad] = np.nan
    ro, rd, masked, bad = dev(ro), dev(rd), dev(masked), dev(bad)
    a, b = irgs.trace_forward(scene, ro, rd, P, max_hit_ids=8), irgs.trace_forward(scene, ro, masked, P, max_hit_ids=8)
    assert scene.status() == 0
    for k in a:
        assert torch.equal(a[k][~bad], b[k][~bad]), k
    for k in ("feat", "depth", "opacity", "n_hits"):
        assert not b[k][bad].any(), k
    assert ms(lambda: irgs.trace_forward(scene, ro, masked, P)) < 1.5 * ms(lambda: irgs.trace_forward(scene, ro, rd, P))


def test_points_without_a_normal(scene):
    gb = [dev(a) for a in synth.gbuffer_points(4096, seed=2)]
    gb[1][::2] = float("nan")
    env = dev(synth.env_map(seed=8, height=16, width=32))
    p = irgs.TraceParams(k=16, feat_count=3, t_min=1e-3)
    rgb = irgs.shade_mc(scene, *gb, env, 32, 32, 9, p)["rgb"]
    assert scene.status() == 0 and torch.isfinite(rgb[1::2]).all()
    assert ms(lambda: irgs.shade_mc(scene, *gb, env, 32, 32, 9, p)) < 10.0


def test_points_without_a_position(scene):
    """Their rays meet nothing: everything is seen, nothing is lit indirectly, and
    fused and regrouped estimates see the same (their colours round differently)."""
    gb = [dev(a) for a in synth.gbuffer_points(4096, seed=3)]
    gb[0][::2, 1] = float("nan")
    env = dev(synth.env_map(seed=8, height=16, width=32))
    E = irgs.EnvMap(env)
    p = irgs.TraceParams(k=16, feat_count=3, t_min=1e-3)
    q = irgs.TraceParams(k=16, feat_count=7, feat_offset=3, t_min=1e-3)
    calls = [lambda r: irgs.shade_mc(scene, *gb, env, 16, 16, 9, p.with_(flags=r), want_aux=True),
             lambda r: irgs.relight(scene, E, *gb, 32, 9, q.with_(flags=r), want_aux=True)]
    for call in calls:
        a, b = call(0), call(irgs.FLAG_PER_THREAD)
        assert scene.status() == 0
        assert not a["ind"][::2].any() and torch.equal(a["vis"][::2], a["vis"][::2].round()) and a["ind"][1::2].any()
        assert torch.equal(a["vis"], b["vis"])
        assert ms(lambda: call(0)) < 10.0
    E.close()
