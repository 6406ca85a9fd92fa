"""The pyramid kernel at the edges of its strips and of its ways to read the
source: every raw and blurred level equals the oracle's, byte for byte."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes

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


# widths at whole strips of 120 columns and one off, heights at and around a
# strip's rows; scales whose taps fit one window, two, or neither (beyond 512
# bytes of source a strip), each with levels down to the smallest accepted
@pytest.mark.parametrize("width,height,levels,scale,pairs", [
    (119, 40, 1, 1.2, 1), (120, 39, 1, 1.2, 1), (121, 45, 2, 1.1, 1), (241, 64, 2, 1.2, 1), (361, 58, 1, 1.2, 70),
    (363, 131, 3, 1.3, 40), (480, 117, 2, 1.99, 3), (725, 175, 2, 2.01, 3), (1241, 376, 8, 1.2, 1),
    (640, 301, 5, 1.5, 2), (1000, 330, 2, 4.0, 1), (1000, 330, 2, 4.1, 1), (901, 703, 3, 3.9, 1), (700, 640, 2, 15.9, 1),
])
@pytest.mark.parametrize("shift", [0, 3])
def test_levels_equal_the_oracle(J, oracle, width, height, levels, scale, pairs, shift):
    import torch
    left = scenes.random_image(height, width, 5)
    right = scenes.random_image(height, width, 6)
    # rows `shift` bytes after the buffer's start, at an odd pitch
    buf = torch.zeros((2, height, width + 9), dtype=torch.uint8, device="cuda")
    buf[0, :, shift:shift + width] = torch.from_numpy(left).cuda()
    buf[1, :, shift:shift + width] = torch.from_numpy(right).cuda()
    fe = J.Frontend(device=0, max_width=width, max_height=height, max_levels=levels, max_feats=64, max_pairs=pairs)
    torch.cuda.synchronize()
    job = J.Job(buf[0, :, shift:shift + width], buf[1, :, shift:shift + width], levels=levels, scale=scale, max_feats=64)
    fe.extract_batch([job] * pairs)
    fe.sync()
    for n in range(levels):
        for side, img in ((0, left), (1, right)):
            want = img if n == 0 else oracle.pyramid_level(img, scale, n)
            got = fe.level(pairs - 1, side, n)
            assert np.array_equal(got["raw"].cpu().numpy(), want), (n, side)
            assert np.array_equal(got["blurred"].cpu().numpy(), oracle.blur(want)), (n, side)
    fe.close()
