"""The D-SSIM strips (csrc/ssim.cu) at their edges: images narrower and shorter
than the window, one column short of, at and past a 128-column strip, heights
around the 11-row rotation; bars of tests/test_gpu_ssim.py."""
import pytest

from paper_2505_22335_gb300 import scenes
from test_gpu_ssim import _built, run_case  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(1, 1), (3, 40), (10, 11), (127, 12), (128, 10), (129, 33), (139, 91), (300, 5)])
def test_strip_edges(W, H):
    cams = [scenes.Camera(60.0, 60.0, W / 2, H / 2, W, H), scenes.Camera(60.0, 60.0, 8.0, 7.0, 17, 14)]
    run_case(cams, W + H, weighted=W % 2 == 1)
