"""The packet walk and the regrouping of pixel rows against the per-ray walk,
bit for bit: image widths that leave columns or rows over, rows whose strips
cross the axes' signs, warps that hold rays of two cameras, batches that mix
packets with rays that do not run together, rays that are not finite, and
cut-offs that the buffer's early closing depends on."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402


@pytest.fixture(scope="module")
def scenes():
    return {"object": make_scene(irgs, synth.object_scene(n=20_000, seed=61)),
            "cloud": make_scene(irgs, synth.tiny_scene(seed=62, n=1500, n_feat=10))}


def same(S, ro, rd, p, rows=slice(None)):
    a = irgs.trace_forward(S, dev(ro), dev(rd), p, max_hit_ids=48)
    b = irgs.trace_forward(S, dev(ro), dev(rd), p.with_(flags=irgs.FLAG_PER_THREAD), max_hit_ids=48)
    torch.cuda.synchronize()
    assert S.status() == 0
    for k in a:
        assert torch.equal(a[k][rows], b[k][rows]), k
    return a


@pytest.mark.parametrize("which", ["object", "cloud"])
@pytest.mark.parametrize("w,h,cams", [(64, 64, 1), (33, 40, 1), (35, 17, 2), (37, 9, 3), (512, 3, 1), (100, 8, 2), (31, 33, 2)])
def test_image_sizes(scenes, which, w, h, cams):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(cams, seed=w), w, h)
    a = same(scenes[which], ro, rd, irgs.TraceParams(k=16, feat_count=10))
    assert (a["n_hits"] > 0).any()


@pytest.mark.parametrize("eye", [(0.0, 0.0, 4.0), (4.0, 0.0, 0.02), (0.0, -3.0, 0.3), (2.0, 2.0, 0.01)])
def test_axis_directions_and_grazing_views(scenes, eye):
    ro, rd = synth.look_at_rays(eye, (0, 0, 0), 48, 48)
    same(scenes["object"], ro, rd, irgs.TraceParams(k=16, feat_count=10))


@pytest.mark.parametrize("T_min,alpha_max,t_min,t_max", [(0.0, 0.99, 0.0, np.inf), (0.5, 0.99, 0.0, np.inf),
                                                         (1e-4, 1.0, 3.2, 4.1), (1e-30, 0.99, 0.0, 5.0)])
def test_cutoffs(scenes, T_min, alpha_max, t_min, t_max):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=5), 48, 40)
    p = irgs.TraceParams(k=8, feat_count=3, T_min=T_min, alpha_max=alpha_max, t_min=t_min, t_max=t_max)
    for S in scenes.values():
        same(S, ro, rd, p)


def test_mixed_batch_with_non_finite_rays(scenes):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=6), 64, 40)
    ri, di = synth.random_rays_through_scene(ro.shape[0], seed=7, box=2.0, radius=4.0)
    pick = np.random.default_rng(8).random(ro.shape[0]) < 0.1
    ro[pick], rd[pick] = ri[pick], di[pick]
    bad = np.arange(5, ro.shape[0], 97)
    rd[bad[0::3]] = np.nan
    rd[bad[1::3], 1] = np.inf
    ro[bad[2::3], 0] = np.nan
    ok = np.ones(ro.shape[0], bool)
    ok[bad] = False
    p = irgs.TraceParams(k=16, feat_count=10)
    a = same(scenes["object"], ro, rd, p, rows=torch.from_numpy(ok).cuda())
    # the neighbours of a non-finite ray are not touched by it
    keep = np.nonzero(ok)[0]
    b = irgs.trace_forward(scenes["object"], dev(ro[keep]), dev(rd[keep]), p)
    for k in b:
        assert torch.equal(a[k][torch.from_numpy(keep).cuda()], b[k]), k


def test_replayed_backward_of_rows(scenes):
    """No hit lists, pixel rows: the backward replays the packets' march."""
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(2, seed=9), 41, 27)
    p = irgs.TraceParams(k=16, feat_count=10)
    gf, gd, go = synth.upstream_grads(ro.shape[0], 10, seed=10)
    got = []
    for q in (p, p.with_(flags=irgs.FLAG_PER_THREAD)):
        fwd = irgs.trace_forward(scenes["object"], dev(ro), dev(rd), q)
        got.append(irgs.trace_backward(scenes["object"], dev(ro), dev(rd), q, fwd, dev(gf), dev(gd), dev(go)))
    for k in got[0]:   # the same terms, added in another order
        scale = got[1][k].abs().max()
        assert (got[0][k] - got[1][k]).abs().max() <= 1e-5 * scale, k
