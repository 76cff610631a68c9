"""Depth order of the Gaussian-views (csrc/sort.cu) through the tile lists.

Every list must be in (float32 depth, id) order and hold each Gaussian-view at
most once, and all lists together every instance: sizes at and past the
one-CTA sort (4096 keys), around the 2048-key tiles, past the switch to 4096-key
tiles, equal depths (ids decide), and more than 16 views (64-bit keys).
"""
import numpy as np
import pytest

from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n,V,flat", [(1, 1, False), (4096, 1, False), (4097, 1, False), (2048 * 5, 1, True),
                                      (2048 * 7 + 1, 2, False), (100, 17, True), (3001, 18, False),
                                      (2_600_003, 1, False)])
def test_lists_are_in_depth_order(n, V, flat):
    import torch
    g = scenes.plain_gaussians(n % 97, n, 0, scale_lo=0.001, scale_hi=0.004)
    if flat:  # a few depths only
        g["mean"][:, 2] = 2.0 + 0.25 * (np.arange(n) % 5)
    T = [np.eye(4) for _ in range(V)]
    for v in range(V):
        T[v][0, 3] = 0.01 * v
    cams = [scenes.Camera(40.0, 40.0, 24.0, 18.0, 48, 36, t) for t in T]
    R = B.Renderer(n_feat=0, k=1, list_cap=-1)
    R.forward(B.to_set(g), cams)
    torch.cuda.synchronize()
    st = R.stats()
    gv, keys = R.copy_buffer(0).astype(np.int64), R.copy_buffer(1)
    assert len(gv) == st["n_listed"] == st["n_instances"] and st["n_visible"] == len(np.unique(gv))
    z = R.copy_buffer(3).reshape(-1, 4)[gv, 2].view(np.uint32)
    assert np.array_equal(np.lexsort((gv, z, keys)), np.arange(len(gv)))
    assert len(np.unique(keys.astype(np.int64) * (n * V) + gv)) == len(gv)
    R.close()
