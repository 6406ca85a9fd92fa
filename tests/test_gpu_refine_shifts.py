"""The half-warp refinement (window half-size 5) over every search radius,
odd keypoint counts, windows at the level's edges and saturated differences,
against the oracle."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes
from parity_util import params_from
from test_gpu_refine import J, _pair  # noqa: F401  (fixture and comparison)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("search", range(1, 8))
@pytest.mark.parametrize("contrast", [False, True])
def test_refine_every_radius(J, oracle, search, contrast):  # noqa: F811
    pair = scenes.planes_pair(401, 299, 0, 21, 22, max_disp=40)
    left, right = pair.left, pair.right
    if contrast:  # differences of 0 and 255
        left, right = ((v > 128).astype(np.uint8) * 255 for v in (left, right))
    p = params_from(oracle, levels=3, max_feats=333, fast_thresh_lo=7, border=16)
    _pair(J, oracle, left, right, p, w=5, L=search)
