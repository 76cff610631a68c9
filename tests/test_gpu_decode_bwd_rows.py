"""The decode backward over the rows with a gradient (csrc/decode.cu).

Without MLP gradients only (anchor, view) rows whose dL/dG is not all zero are
evaluated; with them all rows are.  Both must agree on the anchor and pose
gradients whatever share of the rows is zero (FP32 sums of atomic adds in
another order: 1e-5 relative).
"""
import numpy as np
import pytest

from gpu_cases import rel_l2
from paper_2505_22335_gb300 import binding as B
from test_gpu_decode_bwd import _built, gpu_grads, make_case  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A,K,nf,V,live", [(1, 10, 16, 1, 1.0), (257, 4, 0, 3, 0.02), (600, 10, 16, 2, 0.1),
                                           (300, 7, 32, 1, 0.0), (513, 16, 16, 1, 1.0)])
def test_zero_rows_change_nothing(A, K, nf, V, live):
    case = make_case(A + K, A, K, nf, V)
    rng = np.random.default_rng(A)
    for v, g in enumerate(case["dG"]):
        for a in np.nonzero(rng.uniform(size=A) >= live)[0]:
            for k in g:
                g[k][a * K:(a + 1) * K] = 0.0
        if live == 0.1:  # one value alone keeps its row
            g["feat"][3 * K + K - 1, nf - 1] = 1.0
    some = gpu_grads(case, False, mask=B.GRAD_POSE | B.GRAD_ANCHOR)
    full = gpu_grads(case, False)
    for k in ("pos", "feat", "offsets", "scaling", "pose"):
        assert rel_l2(some[k], full[k]) < 1e-5, k
        if live == 0.0:
            assert not np.any(some[k]), k
