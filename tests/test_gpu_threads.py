"""Calls of different sizes on several native threads at once: a server's slots, and
servers whose scenes differ in K.  The limit of a kernel's dynamic shared memory
belongs to the kernel on the device, not to the launch, so no call may set it to less
than another one asks for.

Every request must be done without an error and equal the same request alone: loss
within the forward bar (1e-5 + 1e-4 relative), pose gradient within 2e-3 relative L2
(atomic accumulation order is free).
"""
import pytest

from gpu_cases import rel_l2, round_cams, round_dict
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def server(A, K, nf=16, slots=1, **cfg):
    anc = round_dict(scenes.anchors(A, A, K))
    mlp = round_dict(scenes.mlp_weights(K, K, nf, bias_sigma=0.1))
    return B.Server(*B.anchors_to_device(anc, mlp), n_feat=nf, k=K, slots=slots, batching=False, **cfg)


def flood(servers, jobs, fresh=40, rounds=4):
    """servers() -> [Server]; jobs: (server index, kind, width, height, views).  Rounds of one
    request of each job on servers that have just been made: their workers start on a round
    at the same time, and allocate between their launches in the first."""
    import torch
    srvs = servers()
    reqs = []
    for k, kind, W, H, n in jobs:
        cams = round_cams(scenes.cameras(3, n, W, H, 0.9 * W))
        P = n * W * H
        tgt = dict(color=torch.rand(3 * P, device="cuda"), depth=torch.rand(P, device="cuda"),
                   feat=torch.rand(srvs[k].n_feat * P, device="cuda"))
        reqs.append((k, kind, cams, tgt, torch.zeros(fresh * rounds + 1, 4 + 6 * n, device="cuda")))
    torch.cuda.synchronize()

    def submit(req, i):
        k, kind, cams, tgt, buf = req
        return srvs[k], srvs[k].submit(kind, cams, tgt, buf[i, :1], buf[i, 4:], levels=1)

    bad = []

    def finish(tickets):
        bad.extend(s.last_error() for s, t in tickets if s.wait(t)["status"] != B.UPS_OK)

    for r in reqs:
        finish([submit(r, fresh * rounds)])
    assert not bad
    for i in range(fresh * rounds):
        if i % rounds == 0:
            for s in srvs:
                s.close()
            srvs = servers()
        finish([submit(r, i) for r in reqs[::(-1) ** i]])
    for s in srvs:
        s.close()
    torch.cuda.synchronize()
    assert not bad, (len(bad), bad[0])
    for _, _, _, _, buf in reqs:
        out = buf.cpu().numpy().astype(float)
        assert abs(out[:-1, 0] - out[-1, 0]).max() <= 1e-5 + 1e-4 * abs(out[-1, 0])
        assert max(rel_l2(o, out[-1, 4:]) for o in out[:-1, 4:]) < 2e-3


def test_decodes_of_two_sizes():
    flood(lambda: [server(3000, 10, slots=2)], [(0, B.TRACK, 64, 48, 1), (0, B.MAP, 64, 48, 12)])


@pytest.mark.parametrize("bf16,ka,kb", [(0, 4, 10), (1, 3, 16)])
def test_decodes_of_two_widths(bf16, ka, kb):
    nf = 0 if kb == 16 else 16
    flood(lambda: [server(3000, k, nf, decode_bf16=bf16, decode_bwd_bf16=bf16) for k in (ka, kb)],
          [(i, B.TRACK, 64, 48, 1) for i in range(2)])


def test_frames_of_two_sizes():
    flood(lambda: [server(300, 4, 0, slots=2)], [(0, B.TRACK, 1280, 720, 1), (0, B.TRACK, 1237, 693, 1)])
