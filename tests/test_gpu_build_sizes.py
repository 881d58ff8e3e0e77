"""The tree build at the sizes where its kernels change shape: one to a few
triangles, one sorting block against two (256), the clustering that ends in
one block (1024) against the one that starts with launches over the chip, and
several of its blocks and launch batches.  Codes, order, radix tree and boxes
equal the oracle's bit for bit; the clustered tree is valid and the same on a
repeat."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs
from gpu_util import ctx, need_cuda
from test_gpu_ploc import _check_tree, _upload

pytestmark = pytest.mark.gpu


def _soup(T, flat):
    """T random small triangles; flat: all in one plane, with repeated codes."""
    rng = np.random.default_rng(T)
    c = rng.random((T, 1, 3)) * 8.0 - 4.0
    if flat:
        c[..., 2] = -2.5
        c = np.round(c * 4.0) / 4.0
    v = (c + rng.normal(size=(T, 3, 3)) * 0.05).reshape(-1, 3).astype(np.float32)
    return v, np.arange(3 * T, dtype=np.int32).reshape(T, 3), rng.random((3 * T, 2)).astype(np.float32)


@pytest.mark.parametrize("T", [1, 2, 3, 31, 33, 255, 256, 257, 512, 1023, 1024, 1025, 1026, 1153, 2049, 33025])
@pytest.mark.parametrize("flat", [False, True])
def test_build_at_block_edges(orc, T, flat):
    need_cuda()
    verts, tris, uv = _soup(T, flat)
    c = ctx()
    hs = [_upload(c, b, verts, tris, uv) for b in (dpcs.DPCS_BVH_LBVH, dpcs.DPCS_BVH_PLOC, dpcs.DPCS_BVH_PLOC)]
    try:
        (codes, order, child, box), p, q = [c.export(h, T) for h in hs]
    finally:
        for h in hs:
            c.free(h)
    rc, ro, rch, rb = orc.lbvh(verts, tris)
    np.testing.assert_array_equal(codes, rc)
    np.testing.assert_array_equal(order, ro)
    np.testing.assert_array_equal(child, rch)
    np.testing.assert_array_equal(box.view(np.uint32), rb.view(np.uint32))
    for x, y in zip(p, q):
        np.testing.assert_array_equal(x.view(np.uint32), y.view(np.uint32))
    np.testing.assert_array_equal(p[1], order)
    if T > 2:
        depth, _ = _check_tree(verts, tris, p[1], p[2], p[3])
        assert depth <= 64
