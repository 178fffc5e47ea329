"""Batches traced with a warp per ray against packets and per-ray walks, bit
for bit, at the batch sizes where the library changes between them."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402


@pytest.fixture(scope="module")
def scenes():
    return {"object": make_scene(irgs, synth.object_scene(n=20_000, seed=81)),
            "cloud": make_scene(irgs, synth.tiny_scene(seed=82, n=1500, n_feat=10))}


def equal(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k


def grads_close(a, b):
    """The same terms, added in another order."""
    for k in a:
        assert float((a[k] - b[k]).abs().max()) <= 1e-5 * float(b[k].abs().max()), k


@pytest.mark.parametrize("R", [1, 3, 4, 5, 31, 33, 1000])
@pytest.mark.parametrize("fc", [1, 3, 10, 16])
def test_small_batches(scenes, R, fc):
    """A few rays, each a warp: channels up to the list's 16, hit lists that end early."""
    S = make_scene(irgs, synth.tiny_scene(seed=83, n=700, n_feat=16))
    ro, rd = (dev(a) for a in synth.random_rays_through_scene(R, seed=R, box=1.0, radius=3.0))
    p = irgs.TraceParams(k=16, feat_count=fc)
    for ids in (0, 1, 32, 80):
        a = irgs.trace_forward(S, ro, rd, p, max_hit_ids=ids)
        for flag in (irgs.FLAG_WARP, irgs.FLAG_PER_THREAD):
            equal(a, irgs.trace_forward(S, ro, rd, p.with_(flags=flag), max_hit_ids=ids))


@pytest.mark.parametrize("which", ["object", "cloud"])
@pytest.mark.parametrize("T_min,alpha_max,t_min,t_max", [(0.0, 0.99, 0.0, np.inf), (0.5, 0.99, 0.0, np.inf),
                                                         (1e-4, 1.0, 3.2, 4.1), (1e-30, 0.99, 0.0, 5.0)])
def test_cutoffs_with_packets(scenes, which, T_min, alpha_max, t_min, t_max):
    ro, rd = (dev(a) for a in synth.camera_batch_rays(synth.hemisphere_cameras(2, seed=5), 48, 41))
    p = irgs.TraceParams(k=8, feat_count=3, T_min=T_min, alpha_max=alpha_max, t_min=t_min, t_max=t_max)
    a = irgs.trace_forward(scenes[which], ro, rd, p, max_hit_ids=48)
    equal(a, irgs.trace_forward(scenes[which], ro, rd, p.with_(flags=irgs.FLAG_WARP), max_hit_ids=48))


@pytest.mark.parametrize("rays", ["view", "random"])
def test_around_the_line_to_packets(scenes, rays):
    """2^18 rays and one more; backward with lists (few rays are longer, many
    are, all are) and without."""
    S, n = scenes["object"], (1 << 18) + 1
    if rays == "view":
        ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(2, seed=3), 512, 257)
    else:
        ro, rd = synth.random_rays_through_scene(n, seed=4, box=1.0, radius=3.0)
    ro, rd = dev(ro[:n]), dev(rd[:n])
    p = irgs.TraceParams(k=16, feat_count=10)
    ref = irgs.trace_forward(S, ro, rd, p.with_(flags=irgs.FLAG_PER_THREAD), max_hit_ids=64)
    gf, gd, go = (dev(a) for a in synth.upstream_grads(n, 10, seed=6))
    for R in (n - 1, n):
        a = irgs.trace_forward(S, ro[:R], rd[:R], p, max_hit_ids=64)
        equal(a, {k: v[:R] for k, v in ref.items()})
        want = irgs.trace_backward(S, ro[:R], rd[:R], p.with_(flags=irgs.FLAG_PER_THREAD), a, gf[:R], gd[:R], go[:R])
        for ids in (0, 1, 4, 32):
            f = irgs.trace_forward(S, ro[:R], rd[:R], p, max_hit_ids=ids)
            grads_close(irgs.trace_backward(S, ro[:R], rd[:R], p, f, gf[:R], gd[:R], go[:R]), want)
    assert S.status() == 0


def points(n, seed):
    return tuple(dev(a) for a in synth.gbuffer_points(n, seed=seed))


@pytest.mark.parametrize("log_rays,spp", [(19, 64), (23, 256)])
def test_sampled_batches_around_their_lines(scenes, log_rays, spp):
    """Shading and relighting of one point more than a line's rays: the points
    before it are the same bit for bit, their gradients to the order of sums."""
    S = scenes["object"]
    n = (1 << log_rays) // spp
    gb = points(n + 1, seed=7)
    env = dev(synth.env_map(seed=8, height=16, width=32))
    E = irgs.EnvMap(env)
    p = irgs.TraceParams(k=16, feat_count=3, t_min=1e-3)
    q = irgs.TraceParams(k=16, feat_count=7, feat_offset=3, t_min=1e-3)
    less = tuple(a[:n] for a in gb)
    a = irgs.shade_mc(S, *less, env, spp // 2, spp // 2, 9, p, want_aux=True)
    more = irgs.shade_mc(S, *gb, env, spp // 2, spp // 2, 9, p, want_aux=True)
    equal(a, {k: v[:n] for k, v in more.items()})
    a = irgs.relight(S, E, *less, spp, 10, q, want_aux=True)
    equal(a, {k: v[:n] for k, v in irgs.relight(S, E, *gb, spp, 10, q, want_aux=True).items()})
    g = torch.zeros((n + 1, 3), device="cuda")
    g[:n] = torch.from_numpy(np.random.default_rng(11).normal(size=(n, 3)).astype(np.float32)).cuda()
    a = irgs.shade_mc_backward(S, *less, env, spp // 2, spp // 2, 9, p, g[:n])
    b = irgs.shade_mc_backward(S, *gb, env, spp // 2, spp // 2, 9, p, g)
    grads_close({k: v[:n] if k in ("albedo", "rough") else v for k, v in b.items()}, a)
    E.close()
    assert S.status() == 0
