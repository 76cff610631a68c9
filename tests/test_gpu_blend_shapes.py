"""Shapes of the blend kernels (csrc/composite.cu) by the number of tiles: one
tile, the last frame with two tiles per SM and the first beyond, and one whose
tiles fit the GPU at once only with eight CTAs per SM.  A view alone and the
same view in a batch of many take different shapes: the forward's arithmetic per
pixel is the same in all (bit-equal images), the gradients are sums of FP32
atomics in another order (1e-4 of the largest, 200 blended values a pixel).
"""
import pytest

from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def step(g, cams, nf, seed):
    import torch
    R = B.Renderer(n_feat=nf)
    img = R.forward(g, cams)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = cams[0].width * cams[0].height
    one = {k: torch.randn(c * n, generator=gen, device="cuda") for k, c in (("color", 3), ("depth", 1), ("feat", nf))}
    d = {k: torch.zeros_like(img[k]) for k in one}
    for k in one:
        d[k].reshape(-1)[:one[k].numel()] = one[k]  # only the first view has a gradient
    grad, pose = R.backward(d, B.GRAD_POSE | B.GRAD_GAUSS)
    torch.cuda.synchronize()
    out = [img[k].reshape(-1)[:c * n].clone() for k, c in (("color", 3), ("depth", 1), ("feat", nf), ("T", 1))]
    gr = [getattr(grad, k).clone() for k in ("mean_opacity", "scale", "quat", "color", "feat")] + [pose[0].clone()]
    R.close()
    return out, gr


@pytest.mark.parametrize("W,H,nf,views", [(16, 16, 0, 2), (15, 13, 32, 2), (304, 256, 16, 2), (305, 256, 16, 4),
                                          (160, 120, 0, 12), (160, 120, 16, 13), (160, 120, 32, 12), (640, 480, 16, 2)])
def test_alone_equals_in_a_batch(W, H, nf, views):
    import torch
    g = B.to_set(scenes.plain_gaussians(W + nf, 400, nf))
    cams = scenes.cameras(3, views, W, H, 1.0 * W)
    a, da = step(g, cams[:1], nf, 5)
    b, db = step(g, cams, nf, 5)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    for x, y in zip(da, db):
        if x.numel():
            assert (x - y).abs().max() <= 1e-4 * x.abs().max()
