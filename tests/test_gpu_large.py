"""Sizes beyond which a part changes its form: more surfels than the build sorts
itself (2^22), than leave a byte of a k-buffer entry free (2^24), more image
tiles than are ordered by length (2^16). Surfels that are never hit fill the
scenes up, so the results are those of the scene without them."""
import numpy as np
import pytest

import oracle
import synth
from tests.test_gpu_raster import compare, ocam, opar

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from paper_2412_15867_gb300 import serve  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402
from tests.helpers import scene as surfels  # noqa: E402


def filled(sc, n, seed):
    """sc's surfels, in order, at random places among n; where each went."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    at = torch.randperm(n, generator=g, device="cuda")[:sc.n].sort().values
    arr = []
    for a in sc.arrays():
        a = dev(a)
        full = torch.rand((n,) + a.shape[1:], generator=g, device="cuda")
        if a.dim() == 1:
            full.zero_()      # no opacity: never hit
        elif a.shape[1] == 3:
            full = full * 5 - 2.5
        full[at] = a
        arr.append(full)
    return irgs.Scene(*arr), at


@pytest.mark.parametrize("n", [(1 << 22) + 1, (1 << 24) + 1])
@pytest.mark.parametrize("hierarchy_rebuilt", [False, True])
def test_many_surfels(n, hierarchy_rebuilt):
    sc = synth.object_scene(n=30_000, seed=91)
    few = make_scene(irgs, sc)
    many, at = filled(sc, n, 92)
    if hierarchy_rebuilt:
        many.update()
        many.refit()
    assert many.status() == 0
    p = irgs.TraceParams(k=16, feat_count=10)
    ro, rd = (dev(a) for a in synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=3), 201, 150))
    a = irgs.trace_forward(few, ro, rd, p, max_hit_ids=64)
    want = torch.where(a["hit_ids"] >= 0, at.int()[a["hit_ids"].clamp(min=0).long()], a["hit_ids"])
    for flags in (0, irgs.FLAG_WARP, irgs.FLAG_PER_THREAD):
        b = irgs.trace_forward(many, ro, rd, p.with_(flags=flags), max_hit_ids=64)
        assert many.status() == 0
        for k in ("feat", "depth", "opacity", "n_hits"):
            assert torch.equal(a[k], b[k]), (k, flags)
        assert torch.equal(want, b["hit_ids"]), flags
    gf, gd, go = (dev(x) for x in synth.upstream_grads(ro.shape[0], 10, seed=10))
    small = irgs.trace_backward(few, ro, rd, p, a, gf, gd, go)
    for fwd in (b, {k: v for k, v in b.items() if k != "hit_ids"}):
        large = irgs.trace_backward(many, ro, rd, p, fwd, gf, gd, go)
        for k in small:
            assert (large[k][at] - small[k]).abs().max() <= 1e-5 * small[k].abs().max(), k
    env = dev(synth.env_map(seed=8, height=16, width=32))
    q = irgs.TraceParams(k=16, feat_count=3, t_min=1e-3)
    for points in (2000, (1 << 17) + 1):     # a warp per ray, and pools of rays
        gb = [dev(x) for x in synth.gbuffer_points(points, seed=4)]
        assert torch.equal(irgs.shade_mc(few, *gb, env, 32, 32, 5, q)["rgb"], irgs.shade_mc(many, *gb, env, 32, 32, 5, q)["rgb"])
    assert many.status() == 0


@pytest.mark.parametrize("w,h", [(4097, 4090), (16, 16 * 65600)])
def test_many_tiles(w, h):
    rng = np.random.default_rng(3)
    n = 24
    sc = surfels(rng.uniform(-1, 1, (n, 3)), rng.normal(size=(n, 4)), rng.uniform(0.02, 0.3, (n, 2)),
                 rng.uniform(0.2, 0.9, n), rng.uniform(size=(n, 3)))
    S = make_scene(irgs, sc)
    cam = serve.make_camera((0.4, 3.0, 1.0), w, h, target=(0, 0, 0), fov_deg=40.0)
    p = irgs.TraceParams(k=16, feat_count=3, t_min=0.1)
    out = irgs.rasterize(S, cam, p)
    assert S.status() == 0
    print(compare(out, oracle.rasterize(sc, ocam(cam), opar(p))))
