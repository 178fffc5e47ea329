"""A build whose grid barrier runs out: each of the three cooperative kernels
leaves an error bit, and what it could not make is replaced by something that
every later step can use without leaving its arrays. The control words are
set so that the first wait of one kernel finds the barrier given up."""
import ctypes as C
import subprocess

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2412_15867_gb300 import _build, _lib  # noqa: E402
from tests.gpu_util import dev  # noqa: E402

HARNESS = r"""
#include "scene.cu"
namespace irgs { void count_launches(uint64_t) {} }
using namespace irgs;
// which: control words of the kernel whose barrier is given up (8 order, 10 clustering, 12 collapse)
extern "C" int broken_build(const irgs_surfels* s, int which, uint32_t* status, int32_t* perm, uint32_t* keys,
                            float* nodes, float* boxes, float* wide, uint32_t* n_wide) {
    irgs_scene sc = nullptr;
    if (build_scene_impl(s, 1.f / 255.f, 0u, 0, &sc) != IRGS_OK) return 1;
    const int64_t n = sc->n;
    const uint32_t words[2] = {0xC0000000u, 1u};   // the count stays below every target; somebody gave up
    cudaMemset(sc->perm, 0x7f, 4 * n);
    cudaMemset(sc->keys, 0xa5, 4 * n);
    cudaMemset(sc->nodes, 0, sizeof(Node) * (n - 1));
    cudaMemset(sc->refit_flag, 0, 4 * (n - 1));
    cudaError_t e = enqueue_control(sc, 0);
    if (e == cudaSuccess) e = cudaMemcpy(sc->bounds + which, words, sizeof(words), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = enqueue_order(sc, s, 0);
    if (e == cudaSuccess) e = enqueue_pack(sc, s, 0);
    if (e == cudaSuccess) e = enqueue_ploc(sc, 0);
    const uint32_t* gate = sc->bounds + kCtlFallback;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    k_karras<<<blocks, 256>>>(sc->keys, n, sc->nodes, sc->leaf_parent, sc->node_parent, gate);
    k_refit<<<blocks, 256>>>(n, sc->leaf_box, sc->leaf_parent, sc->node_parent, sc->nodes, sc->refit_flag, sc->status, gate);
    if (e == cudaSuccess) e = enqueue_wide(sc, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    auto get = [&](void* to, const void* from, size_t b) { if (e == cudaSuccess) e = cudaMemcpy(to, from, b, cudaMemcpyDeviceToHost); };
    get(status, sc->status, 4);
    get(perm, sc->perm, 4 * n);
    get(keys, sc->keys, 4 * n);
    get(nodes, sc->nodes, sizeof(Node) * (n - 1));
    get(boxes, sc->leaf_box, 24 * n);
    get(wide, sc->wide, sizeof(WideNode));
    get(n_wide, sc->wide_counters + kWideLevels, 4);
    free_scene(sc);
    return e == cudaSuccess ? 0 : 2;
}
"""
BAD_TREE = 2


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("barrier")
    src, so = d / "harness.cu", d / "harness.so"
    src.write_text(HARNESS)
    r = subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return C.CDLL(str(so))


@pytest.mark.parametrize("which", ["none", "order", "clustering", "collapse"])
def test_given_up_barrier(harness, which):
    n = 5000
    sc = synth.object_scene(n=n, seed=3)
    t = [dev(a) for a in sc.arrays()]
    s = _lib.Surfels(*(x.data_ptr() for x in t), n, sc.features.shape[1])
    status, n_wide = np.zeros(1, np.uint32), np.zeros(1, np.uint32)
    perm, keys = np.zeros(n, np.int32), np.zeros(n, np.uint32)
    nodes, boxes, wide = np.zeros((n - 1, 16), np.float32), np.zeros((n, 6), np.float32), np.zeros(32, np.float32)
    # "none": the fallback flag and the unused word behind it, so that the radix tree replaces the clustering's
    words = {"none": 14, "order": 8, "clustering": 10, "collapse": 12}[which]
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    assert harness.broken_build(C.byref(s), words, p(status), p(perm), p(keys), p(nodes), p(boxes), p(wide), p(n_wide)) == 0
    assert status[0] == (0 if which == "none" else BAD_TREE)
    # a permutation in the order of the keys, and a hierarchy over all of its leaves, whatever gave up
    assert np.array_equal(np.sort(perm), np.arange(n)) and np.all(np.diff(keys.astype(np.int64)) >= 0)
    if which == "order":
        assert np.array_equal(perm, np.arange(n))
    child = nodes[:, 12:14].view(np.int32)
    assert np.array_equal(np.sort(~child[child < 0]), np.arange(n))
    assert np.array_equal(np.sort(child[child >= 0]), np.arange(1, n - 1))
    leaf = child < 0
    assert np.array_equal(np.stack([nodes[:, 0:3], nodes[:, 6:9]], 1)[leaf], boxes[~child[leaf], :3])
    kids = wide[24:28].view(np.int32)
    if which == "collapse":   # nothing below the root was made: nothing may be walked into
        assert n_wide[0] == 1 and np.all(kids == np.iinfo(np.int32).min)
    else:
        assert n_wide[0] > n // 4 and np.all(kids != np.iinfo(np.int32).min)
