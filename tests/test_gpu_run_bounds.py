"""Detection for every pair of run bounds 1 <= P_min <= P_max <= 16, the run
test being chosen at run time outside the default ones, against the oracle."""
import numpy as np
import pytest

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


def _runs(h, w, seed):
    """Centres of random contrast inside rings with one or two random runs,
    noise between: every run length, both polarities, 0 and 255."""
    rng = np.random.default_rng(seed)
    dx = [0, 1, 2, 3, 3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1]
    dy = [3, 3, 2, 1, 0, -1, -2, -3, -3, -3, -2, -1, 0, 1, 2, 3]
    img = rng.integers(118, 138, (h, w)).astype(np.uint8)
    for y in range(20, h - 20, 8):
        for x in range(20, w - 20, 8):
            for polarity in rng.permutation([0, 255])[:rng.integers(1, 3)]:
                start, length = rng.integers(0, 16), rng.integers(1, 17)
                for q in range(start, start + length):
                    img[y + dy[q & 15], x + dx[q & 15]] = polarity
            img[y, x] = rng.choice([0, 100, 128, 255])
    return img


@pytest.mark.parametrize("p_min", range(1, 17))
@pytest.mark.parametrize("options", [dict(), dict(k_per_cell=3, cell=16, response_mode=1, fast_thresh_lo=7)])
def test_run_bounds(J, oracle, p_min, options):
    import torch
    img = _runs(122, 171, p_min)
    dev = torch.from_numpy(img).cuda()
    torch.cuda.synchronize()
    for p_max in range(p_min, 17):
        p = params_from(oracle, levels=1, max_feats=2000, p_min=p_min, p_max=p_max, **options)
        fe = frontend_for(J, p, max_width=171, max_height=122, max_pairs=1)
        fe.extract_batch([J.Job(dev, dev, levels=1, scale=p.scale, fast_thresh=p.fast_thresh, cell=p.cell,
                                max_feats=p.max_feats)])
        fe.sync()
        compare_keypoints(J.to_numpy(fe.keypoints(0, 0)), oracle.extract_image(img, p), f"{p_min} {p_max}")
        fe.close()
