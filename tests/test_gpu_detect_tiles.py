"""The bit-sliced detection kernel where its tiles can go wrong: cell sizes
that divide neither 32 nor a word, one-cell tiles, several keypoints a cell
with ties, flat and noisy images (no corners, corners everywhere), batches of
fewer and of many more tiles than CTAs, and every chosen tile size, against
the oracle."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes
from parity_util import compare_keypoints, frontend_for, params_from

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def J():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_04090_gb300 import build
    build.build()
    from paper_2410_04090_gb300 import jslam
    return jslam


def _image(kind, h, w):
    if kind == "noise":  # corners at the fallback threshold almost everywhere
        return np.random.default_rng(4).integers(90, 150, (h, w)).astype(np.uint8)
    if kind == "steps":  # saturated thresholds on both sides
        img = np.zeros((h, w), np.uint8)
        img[(np.arange(h)[:, None] // 5 + np.arange(w)[None, :] // 7) % 2 == 0] = 255
        return img
    return scenes.random_image(h, w, 8)


@pytest.mark.parametrize("width,height,levels,cell,k,arc,kind,pairs,tile", [
    (641, 479, 4, 31, 1, 0, "scene", 1, None), (641, 479, 3, 13, 3, 0, "scene", 2, None),
    (333, 251, 3, 7, 8, 0, "noise", 1, None), (500, 333, 3, 128, 1, 0, "scene", 1, None),
    (500, 333, 2, 101, 2, 1, "noise", 1, None), (320, 240, 4, 32, 1, 0, "steps", 1, None),
    (320, 240, 3, 1, 1, 0, "scene", 1, None), (640, 480, 4, 32, 2, 1, "scene", 60, None),
    (752, 480, 5, 32, 1, 0, "noise", 1, (32, 8)), (752, 480, 5, 32, 1, 0, "scene", 1, (36, 40)),
    (752, 480, 5, 19, 2, 0, "scene", 1, (128, 128)), (752, 480, 5, 32, 1, 0, "steps", 1, (64, 128)),
])
def test_detect_parity(J, oracle, width, height, levels, cell, k, arc, kind, pairs, tile):
    import torch
    p = params_from(oracle, levels=levels, max_feats=6000, cell=cell, k_per_cell=k, fast_thresh_lo=7,
                    response_mode=arc)
    img = _image(kind, height, width)
    flat = np.full_like(img, 77)
    want = oracle.extract_image(img, p)
    fe = frontend_for(J, p, max_width=width, max_height=height, max_pairs=pairs)
    if tile:
        fe.set_tuning(*tile)
    a, z = torch.from_numpy(img).cuda(), torch.from_numpy(flat).cuda()
    torch.cuda.synchronize()
    fe.extract_batch([J.Job(a, z, levels=levels, scale=p.scale, fast_thresh=p.fast_thresh, cell=cell, max_feats=6000)]
                     * pairs)
    fe.sync()
    compare_keypoints(J.to_numpy(fe.keypoints(pairs - 1, 0)), want, "left")
    assert fe.keypoints(pairs - 1, 1)["count"] == 0
    fe.close()
