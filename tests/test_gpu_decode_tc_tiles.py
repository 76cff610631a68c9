"""Tiles of the BF16 tensor-core decode (csrc/decode_tc.cu): row counts around the
128-row tile and the warps' 32 rows, 1 to 16 Gaussians an anchor, feature chunks
of 64 columns with and without a remainder; nothing is written past the outputs.

Reference: the same MLPs in FP64 with the operands (x, W1, hidden values, W2)
rounded to BF16.  The FP32 sums can round a hidden value the other way, 2^-8 of it
times a weight (values up to about 4, weights up to 0.43): 1e-2 on an output, and
1e-4 on average, since few are that close.
"""
import math

import numpy as np
import pytest

from gpu_cases import round_cams, round_dict
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu
FIELDS = ("mean_opacity", "scale", "quat", "color", "feat")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def reference(anc, mlp, cam, K, nf):
    import torch
    r16 = lambda a: torch.tensor(a, dtype=torch.float32).bfloat16().double()
    T = np.asarray(cam.T_cw, np.float64)
    r = anc["pos"] + T[:3, :3].T @ T[:3, 3]
    d = np.linalg.norm(r, axis=1, keepdims=True)
    e = np.tile([math.sin(math.pi * cam.t_norm), math.cos(math.pi * cam.t_norm)], (len(r), 1))
    z = r16(np.concatenate([anc["feat"], r / d, d, e], 1)) @ r16(mlp["w1"]).T + torch.tensor(mlp["b1"])
    h = [torch.relu(z[:, :32]), torch.relu(z[:, 32:64]), torch.relu(z[:, 64:96]), torch.nn.functional.softplus(z[:, 96:])]
    lo = [0, K, 8 * K, 11 * K, K * (11 + nf)]
    y = [r16(h[i].numpy()) @ r16(mlp["w2"][lo[i]:lo[i + 1]]).T + torch.tensor(mlp["b2"][lo[i]:lo[i + 1]])
         for i in range(4)]
    A = len(r)
    cov = y[1].reshape(A, K, 7)
    zero = torch.zeros(A, K, 1, dtype=torch.float64)
    out = dict(mean_opacity=torch.cat([torch.tensor(anc["pos"][:, None] + anc["offsets"]),
                                       torch.sigmoid(y[0]).reshape(A, K, 1)], 2),
               scale=torch.cat([torch.tensor(anc["scaling"])[:, None] * torch.sigmoid(cov[..., :3]), zero], 2),
               quat=cov[..., 3:], color=torch.cat([torch.sigmoid(y[2]).reshape(A, K, 3), zero], 2),
               feat=y[3].reshape(A, K, nf))
    return {k: v.reshape(A * K, -1).numpy() for k, v in out.items()}


@pytest.mark.parametrize("A,K,nf,V", [(1, 1, 16, 1), (127, 10, 16, 1), (129, 10, 32, 1), (43, 3, 16, 3), (100, 7, 32, 2),
                                      (64, 8, 32, 2), (321, 16, 16, 1), (65, 9, 0, 2)])
def test_tiles_match_rounded_mlps(A, K, nf, V):
    import torch
    anc = round_dict(scenes.anchors(A, A, K))
    mlp = round_dict(scenes.mlp_weights(K, K, nf, bias_sigma=0.1))
    cams = round_cams(scenes.cameras(A + 1, V, 64, 48, 60.0))
    R = B.Renderer(n_feat=nf, k=K, decode_bf16=1)
    ad, md = B.anchors_to_device(anc, mlp)
    empty = B.GaussianSet.empty(V, A * K, nf, True)
    room = {k: torch.full((getattr(empty, k).numel() + 256,), 7.0, device="cuda") for k in FIELDS}
    out = B.GaussianSet(*(room[k][:getattr(empty, k).numel()].view(getattr(empty, k).shape) for k in FIELDS), True)
    R.decode(ad, md, cams, out=out)
    torch.cuda.synchronize()
    for v, cam in enumerate(cams):
        ref = reference(anc, mlp, cam, K, nf)
        for k in FIELDS:
            if ref[k].size:
                err = np.abs(getattr(out, k)[v].cpu().numpy() - ref[k])
                assert err.max() < 1e-2 and err.mean() < 1e-4, (k, v, err.max(), err.mean())
    for k in FIELDS:
        assert (room[k][getattr(empty, k).numel():] == 7.0).all(), k
    R.close()
