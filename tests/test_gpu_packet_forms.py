"""Batches as packets (FLAG_WARP, whatever their size) against the per-ray walk,
bit for bit: image widths that leave columns or rows over, rows whose strips
cross the axes' signs, warps that hold rays of two cameras, packets mixed with
rays that do not run together or are not finite, cut-offs, replays; and pixel
rows in compacted rounds, whose lists and states go by slot and whose rays by
pixel."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402

W, T = irgs.FLAG_WARP, irgs.FLAG_PER_THREAD


@pytest.fixture(scope="module")
def scenes():
    return {"object": make_scene(irgs, synth.object_scene(n=20_000, seed=61)),
            "cloud": make_scene(irgs, synth.tiny_scene(seed=62, n=1500, n_feat=10))}


def same(S, ro, rd, p, ids=48):
    a = irgs.trace_forward(S, dev(ro), dev(rd), p.with_(flags=W), max_hit_ids=ids)
    b = irgs.trace_forward(S, dev(ro), dev(rd), p.with_(flags=T), max_hit_ids=ids)
    assert S.status() == 0
    for k in a:
        assert torch.equal(a[k], b[k]), k
    return a


@pytest.mark.parametrize("which", ["object", "cloud"])
@pytest.mark.parametrize("w,h,cams", [(64, 64, 1), (33, 40, 1), (35, 31, 2), (37, 9, 4), (512, 3, 1), (100, 8, 2), (31, 34, 2), (333, 20, 1), (130, 67, 2)])
def test_image_sizes(scenes, which, w, h, cams):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(cams, seed=w), w, h)
    a = same(scenes[which], ro, rd, irgs.TraceParams(k=16, feat_count=10))
    assert (a["n_hits"] > 0).any()


@pytest.mark.parametrize("eye", [(0.0, 0.0, 4.0), (4.0, 0.0, 0.02), (0.0, -3.0, 0.3), (2.0, 2.0, 0.01), (-1.1, 0.0, 1.0)])
@pytest.mark.parametrize("fc", [1, 3, 10])
def test_axis_directions_and_grazing_views(scenes, eye, fc):
    ro, rd = synth.look_at_rays(eye, (0, 0, 0), 48, 48)
    same(scenes["object"], ro, rd, irgs.TraceParams(k=16, feat_count=fc))


@pytest.mark.parametrize("T_min,alpha_max,t_min,t_max", [(0.0, 0.99, 0.0, np.inf), (0.5, 0.99, 0.0, np.inf),
                                                         (1e-4, 1.0, 3.2, 4.1), (1e-30, 0.99, 0.0, 5.0)])
def test_cutoffs(scenes, T_min, alpha_max, t_min, t_max):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=5), 48, 40)
    p = irgs.TraceParams(k=8, feat_count=3, T_min=T_min, alpha_max=alpha_max, t_min=t_min, t_max=t_max)
    for S in scenes.values():
        same(S, ro, rd, p)


@pytest.mark.parametrize("share", [0.02, 0.1, 0.5])
def test_mixed_batches(scenes, share):
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=6), 64, 40)
    ri, di = synth.random_rays_through_scene(ro.shape[0], seed=7, box=2.0, radius=4.0)
    pick = np.random.default_rng(8).random(ro.shape[0]) < share
    ro[pick], rd[pick] = ri[pick], di[pick]
    bad = np.arange(5, ro.shape[0], 97)
    rd[bad[0::3]] = np.nan
    rd[bad[1::3], 1] = np.inf
    ro[bad[2::3], 0] = np.nan
    a = same(scenes["object"], ro, rd, irgs.TraceParams(k=16, feat_count=10))
    assert not a["n_hits"][torch.from_numpy(bad).cuda()].any()
    # and the neighbours of a non-finite ray are not touched by it
    keep = np.setdiff1d(np.arange(ro.shape[0]), bad)
    b = irgs.trace_forward(scenes["object"], dev(ro[keep]), dev(rd[keep]), irgs.TraceParams(k=16, feat_count=10, flags=W), max_hit_ids=48)
    for k in b:
        assert torch.equal(a[k][torch.from_numpy(keep).cuda()], b[k]), k


@pytest.mark.parametrize("w,h", [(41, 27), (130, 67), (1000, 301)])
def test_replays(scenes, w, h):
    """No hit lists, and lists that most rays overflow: the backward replays the packets' march."""
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(2, seed=9), w, h)
    p = irgs.TraceParams(k=16, feat_count=10)
    gf, gd, go = (dev(a) for a in synth.upstream_grads(ro.shape[0], 10, seed=10))
    ro, rd = dev(ro), dev(rd)
    want = None
    for flags, ids in ((T, 0), (W, 0), (W, 2)):
        q = p.with_(flags=flags)
        fwd = irgs.trace_forward(scenes["object"], ro, rd, q, max_hit_ids=ids)
        g = irgs.trace_backward(scenes["object"], ro, rd, q, fwd, gf, gd, go)
        want = g if want is None else want
        for k in g:   # the same terms, added in another order
            assert (g[k] - want[k]).abs().max() <= 1e-5 * want[k].abs().max(), k
    assert scenes["object"].status() == 0


@pytest.mark.parametrize("w,h,cams", [(1027, 1029, 1), (701, 503, 3)])
def test_rows_in_compacted_rounds(w, h, cams):
    """2^20 rays and more, rows by rows, with columns and rows left over."""
    S = make_scene(irgs, synth.object_scene(n=300_000, seed=1001))
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(cams, seed=17), w, h)
    assert ro.shape[0] >= 1 << 20 and w % 4 and h % 8
    for p in (irgs.TraceParams(k=16, feat_count=10), irgs.TraceParams(k=8, feat_count=3)):
        a = irgs.trace_forward(S, dev(ro), dev(rd), p, max_hit_ids=40)
        b = irgs.trace_forward(S, dev(ro), dev(rd), p.with_(flags=T), max_hit_ids=40)
        assert S.status() == 0
        assert float((a["n_hits"] > 32).float().mean()) > 0.05      # these go on in the second launch
        for k in a:
            assert torch.equal(a[k], b[k]), k
