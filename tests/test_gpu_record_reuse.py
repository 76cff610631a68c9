"""Gradient records kept by a context between backward calls.

The blend backward lists the Gaussian-views it stages and the next backward
clears only those records, so a context that has seen other scenes, sizes and
masks must give what a fresh one gives.  Sums of atomic adds in FP32: equal up
to their order (1e-5 relative, as between two runs of one scene).
"""
import numpy as np
import pytest

from gpu_cases import rel_l2
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu
NF = 16


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def one(R, seed, n, V, per_view, mask, scale_grad):
    import torch
    cams = scenes.cameras(seed, V, 130, 75, 110.0)
    g = scenes.plain_gaussians(seed, n, NF)
    gs = B.to_set([g] * V if per_view else g, per_view=per_view)
    img = R.forward(gs, cams)
    _, dimg = R.loss(img, B.targets_to_device(scenes.targets(seed + 1, cams, NF, weighted=True)))
    for _ in range(2):  # a second backward of the same forward starts from the first's records
        grad, pose = R.backward(dimg, mask, scale_grad=scale_grad)
    torch.cuda.synchronize()
    out = dict(rec=R.copy_buffer(6))
    if grad is not None:
        out.update({k: getattr(grad, k).cpu().numpy() for k in ("mean_opacity", "scale", "quat", "color", "feat")})
    if pose is not None:
        out["pose"] = pose.cpu().numpy()
    return out


def test_reused_context_equals_a_fresh_one():
    both, gauss, pose = B.GRAD_POSE | B.GRAD_GAUSS, B.GRAD_GAUSS, B.GRAD_POSE
    R = B.Renderer(n_feat=NF, k=1)
    for step in [(1, 5000, 1, False, both, 0.0), (2, 700, 2, True, both, 1e-4), (3, 9001, 3, True, pose, 0.0),
                 (4, 33, 1, False, gauss, 1e-3), (5, 2500, 2, False, both, 1e-4), (6, 9001, 3, True, gauss, 0.0)]:
        a = one(R, *step)
        F = B.Renderer(n_feat=NF, k=1)
        b = one(F, *step)
        F.close()
        assert set(a) == set(b)
        for k in a:
            assert a[k].shape == b[k].shape and rel_l2(a[k], b[k]) < 1e-5, (step, k)
            assert np.array_equal(a[k] == 0, b[k] == 0), (step, k)
    R.close()
