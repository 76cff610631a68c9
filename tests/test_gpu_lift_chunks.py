"""Chunks of the lifting kernel (csrc/lift.cu, 16 channels): cells of the patch
grid from one pixel to several chunks of 64, whose last chunk takes 1 to 4 steps
of 16 pixels.  Tolerances as in test_gpu_lift.py.
"""
import pytest

from paper_2505_22335_gb300 import scenes
from test_gpu_lift import _built, run_case  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("patch,W,H", [(1, 17, 9), (3, 33, 20), (4, 32, 16), (7, 40, 31), (8, 48, 24), (9, 37, 29),
                                       (21, 70, 45)])
def test_cell_sizes(patch, W, H):
    run_case(scenes.cameras(patch, 2, W, H, 1.2 * W), 16, 24, patch, patch, weighted=patch % 2 == 1)
