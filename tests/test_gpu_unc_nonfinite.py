"""The uncertainty MLP (csrc/unc_mlp.cu) with hidden units whose pre-activation is not a
finite number: a unit that is off adds nothing to any gradient, one that is on adds what
its formula gives (dL/dz2 times its value).

A bias of -inf or NaN gives the unit, for every pixel, what a bias of -1e30 gives: off.  Both
calls then do the same arithmetic, but for the order of the atomic sums over cells
(300 of them at most, 300 x 2^-24 of the summed magnitudes): bar 1e-4 relative L2.
"""
import math

import numpy as np
import pytest

from gpu_cases import rel_l2
from paper_2505_22335_gb300 import binding as B
from paper_2505_22335_gb300 import scenes

pytestmark = pytest.mark.gpu

NH, PATCH = 24, 14


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def run(change):
    import torch
    rng = np.random.default_rng(7)
    W, H = 131, 90
    mlp = dict(w1=rng.normal(size=(128, NH)) * 0.2, b1=rng.normal(size=128) * 0.1, w2=rng.normal(size=128) * 0.2,
               b2=np.array([0.2]))
    grid = rng.normal(size=(-(-H // PATCH), -(-W // PATCH), NH))
    res = rng.uniform(0, 1.5, (H, W))
    change(mlp, grid)
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    R = B.Renderer(n_feat=0, k=1)
    R.forward(B.to_set(scenes.plain_gaussians(1, 50, 0)), [scenes.Camera(60.0, 60.0, W / 2, H / 2, W, H)])
    dm = {k: torch.zeros(v.shape, dtype=torch.float32, device="cuda") for k, v in mlp.items()}
    loss, out = R.uncertainty_mlp(dev(grid), dev(res), {k: dev(v) for k, v in mlp.items()}, n_h=NH, patch=PATCH,
                                  lam=1.0, scale=0.3, d_mlp=dm)
    torch.cuda.synchronize()
    R.close()
    return float(loss.item()), out["sigma"].cpu().numpy(), {k: v.cpu().numpy().astype(np.float64) for k, v in dm.items()}


@pytest.mark.parametrize("off", [-math.inf, math.nan])
@pytest.mark.parametrize("units", [[5], [64, 65, 66, 67], [0, 9, 127]])
def test_off_units(units, off):
    def bias(x):
        def change(mlp, grid):
            mlp["b1"][units] = x
        return change
    (l0, s0, g0), (l1, s1, g1) = run(bias(off)), run(bias(-1e30))
    assert np.array_equal(s0, s1) and l0 == pytest.approx(l1, rel=1e-5)
    assert not g0["w2"][units].any() and not g0["b1"][units].any() and not g0["w1"][units].any()
    for k in g0:
        assert np.isfinite(g0[k]).all() and rel_l2(g0[k], g1[k]) < 1e-4, k


def test_infinite_corner_values():
    # a lane's four units (12 .. 15) infinite at every corner, their weights positive: on,
    # sigma infinite, dL/dz2 zero and zero times infinity their dL/dw2
    def change(mlp, grid):
        grid[..., 0] = np.abs(grid[..., 0]) + 0.1
        mlp["w1"][12:16, 0] = math.inf
        mlp["w2"][12:16] = 0.3
    _, s, g = run(change)
    y, x = PATCH, PATCH  # a pixel inside a cell: all four weights positive
    assert np.isinf(s.reshape(90, 131)[y, x])
    assert np.isnan(g["w2"][12:16]).all()
