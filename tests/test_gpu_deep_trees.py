"""A hierarchy whose walk holds as many deferred siblings as its stack takes: at
every level the nearest child leads on and three inner ones stay behind. All
boxes hold the rays' origin, so nothing is dropped on the way."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev  # noqa: E402


def comb(levels):
    """Morton codes: level i is the subtree whose first set bit is bit i, with the
    given number of leaves (8: three inner children stay behind, 4: one); two
    leaves at the end. Discs shrink by a quarter per level, slower than their
    distance from the end, so that the larger subtree of a level is opened first."""
    codes, size = [], []
    for i, leaves in enumerate(levels):
        for k in range(leaves):
            sub = k << (3 if leaves == 8 else 2)
            codes.append(1 << (29 - i) | k << (29 - i - (3 if leaves == 8 else 2)))
            size.append(8.0 * 2.0 ** (-i / 3))
    codes[7] = (1 << 30) - 1          # the far corner of the bounds
    codes += [0, 1]
    size += [8.0 * 2.0 ** (-len(levels) / 3)] * 2
    codes = np.array(codes, np.int64)
    q = np.zeros((len(codes), 3))
    for b in range(10):
        for a in range(3):
            q[:, a] += ((codes >> (29 - 3 * b - a)) & 1) << (9 - b)
    n = len(codes)
    half = np.array(size)
    rng = np.random.default_rng(5)
    nrm = np.ones(3) / np.sqrt(3.0)
    axis = np.cross([0, 0, 1.0], nrm)
    quat = np.concatenate([[1 + nrm[2]], axis])
    quat /= np.linalg.norm(quat)
    opacity = rng.uniform(0.01, 0.02, n)
    rc = np.sqrt(2 * np.log(opacity * 255))
    scale = half / (rc * np.sqrt(2.0 / 3.0))
    feats = rng.uniform(size=(n, 3))
    return synth.Surfels(*(np.ascontiguousarray(a, dtype=np.float32)
                           for a in (q / 1023, np.tile(quat, (n, 1)), np.tile(scale[:, None], (1, 2)), opacity, feats)))


@pytest.mark.parametrize("levels", [[8] * 21, [8] * 22, [8] * 22 + [4], [8] * 22 + [4, 4], [8] * 20 + [4] * 7])
def test_stacks_hold_them(levels):
    sc = comb(levels)
    S = irgs.Scene(*(dev(a) for a in sc.arrays()), hierarchy="radix")
    # as many wide nodes deep as there are levels
    W = S.export_wide()
    kids = W[:, 24:28].view(np.int32)
    w, depth = 0, 0
    while True:
        inner = kids[w][kids[w] >= 0]
        if len(inner) == 0:
            break
        assert kids[w][0] == inner[0]
        w, depth = inner[0], depth + 1
    assert depth >= len(levels)
    rng = np.random.default_rng(1)
    rd = rng.normal(size=(64, 3)).astype(np.float32)
    rd /= np.linalg.norm(rd, axis=1, keepdims=True)
    ro = np.full((64, 3), 1e-3, np.float32)
    p = irgs.TraceParams(k=16, feat_count=3, T_min=0.0)
    ref = irgs.trace_forward(S, dev(ro), dev(rd), p)
    assert S.status() == 0
    for flags in (irgs.FLAG_PER_THREAD, irgs.FLAG_WARP):
        out = irgs.trace_forward(S, dev(ro), dev(rd), p.with_(flags=flags))
        assert S.status() == 0
        for k in ref:
            assert torch.equal(ref[k], out[k]), k
    assert int(ref["n_hits"].max()) > 150
