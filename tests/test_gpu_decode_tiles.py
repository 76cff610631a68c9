"""Tiles of the FP32 decode (csrc/decode.cu): row counts around the 64-row tile,
odd and even K (records stored singly or in pairs), output arrays that are only
16-byte aligned, calls large enough that a warp takes whole tiles.

Rows are independent and every element has one summation order, so a call must
equal the same rows decoded in other calls bit for bit; against the oracle (FP64)
an output is a chain of 38 and 32 FMAs (70 roundings, u = 6e-8) of values of a few
units: 2e-5 absolute plus relative.
"""
import numpy as np
import pytest

import oracle
from gpu_cases import round_cams, round_dict
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu
FIELDS = ("mean_opacity", "scale", "quat", "color", "feat")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def setup(A, K, nf, V):
    anc = round_dict(scenes.anchors(A, A, K))
    mlp = round_dict(scenes.mlp_weights(K, K, nf, bias_sigma=0.1))
    cams = round_cams(scenes.cameras(A + 1, V, 64, 48, 60.0))
    return anc, mlp, cams, B.Renderer(n_feat=nf, k=K)


@pytest.mark.parametrize("A,K,nf,V", [(1, 1, 16, 1), (63, 7, 16, 1), (64, 10, 0, 1), (65, 4, 32, 2), (43, 16, 16, 3),
                                      (200, 3, 32, 1)])
def test_tile_edges_match_the_oracle(A, K, nf, V):
    import torch
    anc, mlp, cams, R = setup(A, K, nf, V)
    ad, md = B.anchors_to_device(anc, mlp)
    g = R.decode(ad, md, cams)
    # the same into arrays 16 bytes past a 32-byte boundary
    shift = lambda t: torch.zeros(t.numel() + 4, device="cuda")[4:].view(t.shape)
    o = B.GaussianSet(*(shift(getattr(g, k)) for k in FIELDS), True)
    R.decode(ad, md, cams, out=o)
    torch.cuda.synchronize()
    for k in FIELDS:
        assert torch.equal(getattr(g, k), getattr(o, k)), k
    for v, cam in enumerate(cams):
        ref = oracle.decode(anc, mlp, cam, K, nf)
        mo = np.concatenate([ref["mean"], ref["opacity"].reshape(-1, 1)], 1)
        for k, r in (("mean_opacity", mo), ("scale", ref["scale"]), ("quat", ref["quat"]), ("color", ref["color"]),
                     ("feat", ref["feat"])):
            a = getattr(g, k)[v].cpu().numpy()[:, :r.shape[1]]
            assert np.allclose(a, r, rtol=2e-5, atol=2e-5), (k, v, np.abs(a - r).max())
    R.close()


def test_whole_tile_calls_equal_split_ones():
    import torch
    A, K = 640_007, 1
    anc, mlp, cams, R = setup(3, K, 0, 1)
    _, md = B.anchors_to_device(anc, mlp)
    gen = torch.Generator(device="cuda").manual_seed(1)
    u = lambda *s: torch.rand(*s, generator=gen, device="cuda")
    ad = dict(pos=u(A, 3) + 1.5, feat=u(A, 32) - 0.5, offsets=u(A, K, 3) * 0.1, scaling=u(A, 3) * 0.1 + 0.01)
    g = R.decode(ad, md, cams)
    for lo, hi in ((0, 5000), (300_001, 310_000), (A - 77, A)):
        part = R.decode({k: v[lo:hi].contiguous() for k, v in ad.items()}, md, cams)
        for k in FIELDS[:4]:
            assert torch.equal(getattr(g, k)[:, lo * K:hi * K], getattr(part, k)), (k, lo)
    R.close()
