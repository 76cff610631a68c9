"""ups_wait's timeouts: without end (infinity), none, a short one that ends, NaN."""
import ctypes as C
import math
import time

import pytest

from gpu_cases import round_cams, round_dict
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_timeouts():
    import torch
    A, K = 20_000, 10
    anc, mlp = round_dict(scenes.anchors(1, A, K)), round_dict(scenes.mlp_weights(2, K, 0, bias_sigma=0.1))
    cam = round_cams(scenes.cameras(3, 1, 320, 240, 300.0))
    P = 320 * 240
    tgt = dict(color=torch.rand(3 * P, device="cuda"), depth=torch.rand(P, device="cuda"))
    out = [(torch.zeros(1, device="cuda"), torch.zeros(6, device="cuda")) for _ in range(24)]
    torch.cuda.synchronize()
    srv = B.Server(*B.anchors_to_device(anc, mlp), n_feat=0, k=K, slots=1, batching=False)
    wait = lambda t, ms: srv._L.ups_wait(srv._h, t, C.c_double(ms), C.byref(B.Result()))
    tickets = [srv.submit(B.TRACK, cam, tgt, loss, pose, levels=1) for loss, pose in out]
    # the last of 24 requests that run one after another: not done yet
    t0 = time.perf_counter()
    early = [wait(tickets[-1], ms) for ms in (0.0, -1.0, -math.inf, 0.01)]
    assert time.perf_counter() - t0 < 1.0 and early == [B.UPS_PENDING] * 4
    assert wait(tickets[-1], math.nan) == 2  # UPS_ERR_ARG, the request stays
    for t, ms in zip(tickets[::-1], (math.inf, 1e300, 1e18) * 8):
        assert wait(t, ms) == B.UPS_OK
    srv.close()
