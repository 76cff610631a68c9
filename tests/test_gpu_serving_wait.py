"""Server.wait (ups_wait): returns when the request is done, reports a cancelled
one and refuses an unknown ticket, from several threads at once.
"""
import threading

import pytest

from gpu_cases import round_cams, round_dict
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_wait():
    import torch
    A, K, nf = 300, 4, 16
    anc, mlp = round_dict(scenes.anchors(1, A, K)), round_dict(scenes.mlp_weights(2, K, nf, bias_sigma=0.1))
    cam = round_cams(scenes.cameras(3, 1, 64, 48, 60.0))
    ad, md = B.anchors_to_device(anc, mlp)
    P = sum((64 >> l) * (48 >> l) for l in range(3))
    tgt = dict(color=torch.rand(3 * P, device="cuda"), depth=torch.rand(P, device="cuda"),
               feat=torch.rand(nf * P, device="cuda"), weight=torch.ones(P, device="cuda"))
    out = [(torch.zeros(1, device="cuda"), torch.zeros(6, device="cuda")) for _ in range(8)]
    torch.cuda.synchronize()
    srv = B.Server(ad, md, n_feat=nf, k=K, slots=1)
    tickets = [srv.submit(B.TRACK, cam, tgt, loss, pose, levels=3) for loss, pose in out]
    # from several threads, each its own tickets
    res = {}
    ts = [threading.Thread(target=lambda i=i: res.update({t: srv.wait(t) for t in tickets[i::2]})) for i in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join(60)
    assert sorted(res) == sorted(tickets) and all(r["status"] == B.UPS_OK for r in res.values())
    torch.cuda.synchronize()
    for loss, pose in out[1:]:
        assert loss.item() == pytest.approx(out[0][0].item(), rel=1e-5)
    with pytest.raises(B.UpsError):  # taken already
        srv.wait(tickets[0])
    t = srv.submit(B.TRACK, cam, tgt, *out[0], levels=3)
    if srv.cancel(t) == B.UPS_OK:
        assert srv.wait(t)["status"] != B.UPS_OK
    else:
        srv.wait(t)
    srv.close()
