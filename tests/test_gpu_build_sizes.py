"""The cooperative build at the sizes where its pieces change: one cluster per
tile and block more or less, the number of threads that share a cluster, the
switch to one block, a sort piece of one key more. Order, hierarchy and traces
are compared with NumPy's stable sort, with the definition of a hierarchy, and
with the radix tree over the same surfels (bitwise: traces do not depend on the
hierarchy)."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2412_15867_gb300 as irgs  # noqa: E402
from tests.gpu_util import dev, make_scene  # noqa: E402

SIZES = [2, 33, 991, 992, 993, 1024, 1025, 4864, 4865, 14592, 14593, 34049, 150784, 150785]


@pytest.mark.parametrize("n", SIZES)
def test_order_hierarchy_and_traces(n):
    sc = synth.object_scene(n=max(n, 64), seed=n).subset(np.arange(n))
    S = make_scene(irgs, sc)
    perm, keys, nodes, boxes = S.export()
    assert S.status() == 0
    assert np.array_equal(np.sort(perm), np.arange(n))
    order = np.lexsort((perm, keys))                      # sorted, ties in user order
    assert np.array_equal(order, np.arange(n))
    child = nodes[:, 12:14].view(np.int32)
    leaves = ~child[child < 0]
    inner = child[child >= 0]
    assert np.array_equal(np.sort(leaves), np.arange(n)) and np.array_equal(np.sort(inner), np.arange(1, n - 1))
    lo = np.stack([nodes[:, 0:3], nodes[:, 6:9]], 1)
    hi = np.stack([nodes[:, 3:6], nodes[:, 9:12]], 1)
    of_leaf = child < 0
    assert np.array_equal(lo[of_leaf], boxes[~child[of_leaf], :3]) and np.array_equal(hi[of_leaf], boxes[~child[of_leaf], 3:])
    assert np.array_equal(lo[~of_leaf], lo[child[~of_leaf]].min(1)) and np.array_equal(hi[~of_leaf], hi[child[~of_leaf]].max(1))
    S.update()
    again = S.export()
    for a, b in zip((perm, keys, nodes, boxes), again):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    R = irgs.Scene(*(dev(a) for a in sc.arrays()), alpha_min=1 / 255, hierarchy="radix")
    ro, rd = synth.camera_batch_rays(synth.hemisphere_cameras(1, seed=3), 40, 24)
    p = irgs.TraceParams(k=16, feat_count=10)
    a, b = irgs.trace_forward(S, dev(ro), dev(rd), p), irgs.trace_forward(R, dev(ro), dev(rd), p)
    for k in a:
        assert torch.equal(a[k], b[k]), k


def test_update_and_refit_replay_from_a_graph():
    sc = synth.object_scene(n=5000, seed=9)
    S = make_scene(irgs, sc)
    before = S.export()
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            S.update()
            S.refit()
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert S.status() == 0
    for a, b in zip(before, S.export()):
        assert np.array_equal(a.view(np.uint8), b.view(np.uint8))
