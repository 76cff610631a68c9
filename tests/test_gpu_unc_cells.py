"""The uncertainty MLP's cells (csrc/unc_mlp.cu) at their edges: patches of one
pixel, cells of more than the 224 pixels of a unit in one row (a patch wider
than a unit) and in several, one-patch views, views of different sizes in one
call, feature widths around the parts of the patch product; bars of
tests/test_gpu_unc_mlp.py."""
import pytest

from paper_2505_22335_gb300 import scenes
from test_gpu_unc_mlp import _built, run_case  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,nh,patch", [([(9, 7)], 8, 1), ([(500, 3)], 16, 300), ([(40, 30), (17, 90)], 24, 32),
                                            ([(5, 4)], 64, 14), ([(64, 48), (33, 20), (16, 16)], 260, 16),
                                            ([(230, 230)], 20, 15)])
def test_cell_edges(sizes, nh, patch):
    run_case([scenes.Camera(60.0, 60.0, w / 2, h / 2, w, h) for w, h in sizes], nh, patch, nh + patch)
