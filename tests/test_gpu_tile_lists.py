"""Row-wise tile lists (csrc/bin.cu) against the general path.

The allocation-free forward (csrc/noalloc.cu) writes every (tile, Gaussian)
instance and sorts it; the context forward builds its lists row by row.  Same
projection, same blend kernel, so equal lists give equal images bit for bit,
the list positions in n_contrib included.  Scenes at the edges of the row-wise
form: one Gaussian, runs of 128 plus one, one-tile-wide and one-tile-high
views, rows of more than 255 columns and Gaussians of more than 22 rows (kept
as rectangles), steps of more entries than the queue, lists cut and rebuilt.
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


def cam(W, H, f, T=np.eye(4)):
    return scenes.Camera(f, f, W / 2.0, H / 2.0, W, H, np.asarray(T))


POSES = scenes.arc_poses(5, 3)
CASES = {
    "one": (1, [cam(64, 48, 60.0)], 0.05, 0.1),
    "run_edges": (129, [cam(50, 37, 60.0)], 0.005, 0.05),
    "column_view": (1500, [cam(9, 2005, 900.0)], 0.02, 0.2),
    "row_view": (1500, [cam(2005, 9, 900.0)], 0.02, 0.2),
    "wide_rows": (300, [cam(4230, 37, 900.0)], 0.5, 3.0),
    "tall": (300, [cam(70, 1003, 900.0)], 0.3, 2.0),
    "ragged_views": (5000, [cam(333, 217, 300.0, POSES[0]), cam(70, 129, 90.0, POSES[1]), cam(17, 16, 20.0, POSES[2])],
                     0.005, 0.06),
    "dense": (60_000, [cam(160, 120, 150.0)], 0.005, 0.03),
}


@pytest.mark.parametrize("cap", [0, -1, 3])
@pytest.mark.parametrize("name", sorted(CASES))
def test_rowwise_lists_equal_the_instance_sort(name, cap):
    import torch
    n, cams, lo, hi = CASES[name]
    gs = B.to_set(scenes.plain_gaussians(21, n, 0, scale_lo=lo, scale_hi=hi))
    R = B.Renderer(n_feat=0, k=1, list_cap=cap)
    img = R.forward(gs, cams)
    ref = B.render_forward_static(gs, cams, R.alloc_images(cams), 0)
    torch.cuda.synchronize()
    for k in ("n_contrib", "T", "color", "depth"):
        assert torch.equal(img[k], ref[k]), k
    st = R.stats()
    gv, keys = R.copy_buffer(0).astype(np.int64), R.copy_buffer(1)
    ranges = R.copy_buffer(2).reshape(-1, 2).astype(np.int64)
    assert len(gv) == st["n_listed"] and (cap != -1 or len(gv) == st["n_instances"])
    # (tile, depth, id) order, each Gaussian-view at most once a tile
    z = R.copy_buffer(3).reshape(-1, 4)[gv, 2].view(np.uint32)
    assert np.array_equal(np.lexsort((gv, z, keys)), np.arange(len(gv)))
    assert len(np.unique(keys.astype(np.int64) * (n * len(cams)) + gv)) == len(gv)
    assert np.array_equal(np.bincount(keys, minlength=len(ranges)), ranges[:, 1] - ranges[:, 0])
    R.close()
