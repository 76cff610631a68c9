"""Tile lists of views with many tiles: both sides of the sizes where csrc/bin.cu fills
a view's lists in bands of its rows (8191 tiles a view) and where a batch goes to the
general path that writes every instance (16384 tiles a view).

A batch with one view above 16384 tiles takes the general path whole.  The views under
test (a large one and a small one) are rendered with and without such a view: same
projection and blend kernel, so equal lists give equal images bit for bit, the list
positions in n_contrib included.
"""
import numpy as np
import pytest

from gpu_cases import rel_l2
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu

N = 400


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def cam(W, H):
    f = 0.7 * min(W, H) + 300.0
    return scenes.Camera(f, f, W / 2.0, H / 2.0, W, H, np.eye(4))


def general(gs, cams):
    """cams through the general path: images, tile and Gaussian of every list entry (of cams)."""
    R = B.Renderer(n_feat=0, k=1, list_cap=-1)
    img = R.forward(gs, list(cams) + [cam(2064, 2048)])  # 129 x 128 tiles
    keys, gv = R.copy_buffer(1), R.copy_buffer(0)
    R.close()
    mine = keys < sum(tiles(c) for c in cams)
    return img, keys[mine], gv[mine]


def assert_images(img, ref, cams):
    import torch
    P = sum(c.width * c.height for c in cams)
    for k in ("color", "depth", "T", "n_contrib"):
        n = P * (3 if k == "color" else 1)
        assert torch.equal(img[k].reshape(-1)[:n], ref[k].reshape(-1)[:n]), k


def tiles(c):
    return -(-c.width // 16) * -(-c.height // 16)


# 8064, 8320, 16384 tiles; one of 1024 tiles each way
SIZES = [(2048, 1008), (2033, 1029), (2048, 2048), (16384, 250), (241, 16384)]


@pytest.mark.parametrize("W,H", SIZES)
def test_lists_equal_the_general_path(W, H):
    import torch
    cams = [cam(W, H), cam(70, 129)]
    gs = B.to_set(scenes.plain_gaussians(3, N, 0, scale_lo=0.005, scale_hi=0.3))
    ref, keys, gvs = general(gs, cams)
    for cap in (-1, 0, 3):
        R = B.Renderer(n_feat=0, k=1, list_cap=cap)
        img = R.forward(gs, cams)
        torch.cuda.synchronize()
        assert_images(img, ref, cams)
        # cut after three entries, pixels are open: the lists are made again whole
        assert R.stats()["list_refills"] == (1 if cap == 3 else 0)
        assert np.array_equal(R.copy_buffer(1), keys) and np.array_equal(R.copy_buffer(0), gvs)
        R.close()


@pytest.mark.parametrize("W,H", SIZES)
def test_cut_lists(W, H):
    # every Gaussian covers the frame, nearly opaque: three stop a pixel, lists of eight are
    # cut in every tile and never made again
    import torch
    cams = [cam(W, H), cam(70, 129)]
    g = scenes.plain_gaussians(4, N, 0, scale_lo=400.0, scale_hi=800.0)
    g["opacity"][:] = 0.999
    gs = B.to_set(g)
    ref, keys, gvs = general(gs, cams)
    R = B.Renderer(n_feat=0, k=1, list_cap=8)
    img = R.forward(gs, cams)
    torch.cuda.synchronize()
    assert_images(img, ref, cams)
    st = R.stats()
    assert st["list_refills"] == 0 and st["n_listed"] == 8 * st["n_tiles"] and st["n_instances"] > st["n_listed"]
    first = np.searchsorted(keys, np.arange(st["n_tiles"]))
    assert np.array_equal(R.copy_buffer(0).reshape(-1, 8), gvs[first[:, None] + np.arange(8)])
    R.close()


def test_one_context_over_all_paths():
    # sums of atomic adds in FP32: equal up to their order
    import torch
    NF = 16
    g = scenes.plain_gaussians(5, N, NF, scale_lo=0.005, scale_hi=0.1)
    gs = B.to_set(g)

    def step(R, cams):
        img = R.forward(gs, cams)
        _, dimg = R.loss(img, B.targets_to_device(scenes.targets(6, cams, NF, weighted=True)))
        grad, pose = R.backward(dimg, B.GRAD_POSE | B.GRAD_GAUSS)
        torch.cuda.synchronize()
        out = {k: getattr(grad, k).cpu().numpy() for k in ("mean_opacity", "scale", "quat", "color", "feat")}
        return dict(out, pose=pose.cpu().numpy(), color=img["color"].cpu().numpy())

    R = B.Renderer(n_feat=NF, k=1)
    for cams in ([cam(130, 75)], [cam(2033, 1029), cam(70, 129)], [cam(2064, 2048)], [cam(2048, 1008)],
                 [cam(70, 129), cam(2048, 1040)], [cam(2064, 2048), cam(130, 75)], [cam(130, 75)]):
        a = step(R, cams)
        F = B.Renderer(n_feat=NF, k=1)
        b = step(F, cams)
        F.close()
        assert np.array_equal(a["color"], b["color"])
        for k in a:
            assert rel_l2(a[k], b[k]) < 1e-5, (k, [(c.width, c.height) for c in cams])
    R.close()
