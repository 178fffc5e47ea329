"""Rounding of the pre-integrated maps against the same sums in 64 bits.

An addition to a partial sum S rounds with an rms error of about 2.5e-8 S, a
chain of L like terms by sqrt(L / 3) of that. Over groups of 32 texels (8e-8
each), the groups of a slice and the slices (errors carried) that leaves under
2e-8 of the total, and the last few roundings of a value 4.5e-8: about 5e-8. The
bar is twice that; one accumulator per slice and plain sums of 63 and 217 slices
come to 1.4e-7 and more. Level 1 weighs a few texels by a peak of width 0.04,
whose argument carries the directions' rounding: 2e-7."""
import math

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev  # noqa: E402

D = torch.float64


def dirs(h, w):
    th = (torch.arange(h, device="cuda", dtype=D) + 0.5) / h * math.pi
    ph = (torch.arange(w, device="cuda", dtype=D) + 0.5) / w * 2 * math.pi - math.pi
    return torch.stack([th.sin()[:, None] * ph.cos(), th.sin()[:, None] * ph.sin(), th.cos()[:, None].expand(h, w)], -1).reshape(-1, 3)


def exact(env):
    h, w = env.shape[:2]
    d, e = dirs(h, w), env.double().reshape(-1, 3)
    edge = torch.cos(torch.arange(h + 1, device="cuda", dtype=D) / h * math.pi)
    omega = ((edge[:-1] - edge[1:]) * 2 * math.pi / w)[:, None].expand(h, w).reshape(-1)
    N, R = dirs(32, 64), dirs(64, 128)
    irr = torch.zeros(2048, 3, device="cuda", dtype=D)
    num, den = torch.zeros(5, 8192, 3, device="cuda", dtype=D), torch.zeros(5, 8192, device="cuda", dtype=D)
    for a in range(0, d.shape[0], 1 << 13):
        db, eb, ob = (t[a:a + (1 << 13)] for t in (d, e, omega))
        irr += (N @ db.T).clamp(min=0) @ (eb * ob[:, None])
        c = R @ db.T
        x2 = (1 - c) / 2
        for l in range(5):
            g = c.clamp(min=0) * ob / ((1 - x2) * ((l + 1) / 5) ** 4 + x2) ** 2
            num[l] += g @ eb
            den[l] += g.sum(1)
    return irr / math.pi, num / den[..., None]


@pytest.mark.parametrize("h,w", [(16, 32), (61, 127), (64, 128), (256, 512), (300, 600)])
def test_rounding_of_the_maps(h, w):
    env = dev(synth.env_map(seed=1, height=h, width=w))
    irr, pref = exact(env)
    E = irgs.EnvMap(env)
    m = E.export()
    E.close()
    rms = lambda a, b: float((((torch.from_numpy(a).cuda().double().reshape(b.shape) - b) / b) ** 2).mean().sqrt())
    assert rms(m["irr"], irr) <= 1e-7
    for l in range(5):
        assert rms(m["pref"][l], pref[l]) <= (2e-7 if l == 0 else 1e-7), l
