"""Stage times of batches from host memory are device durations of the stages:
the pyramid's does not hold the upload, and results are the same either way."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,levels,pairs", [(640, 480, 1, 100), (1241, 376, 8, 25)])
def test_pyramid_stage_without_the_upload(J, width, height, levels, pairs):
    """100 pairs of 640x480 are 61 MB, 15 us a megabyte at 64 GB/s and far more
    than the pyramid's own time at one level: the host batch's stage may take
    no more than half as long again as the same frames' on the device."""
    import torch
    f = scenes.planes_pair(width, height, 0, 3, 4)
    pinned = torch.empty((pairs, 2, height, width), dtype=torch.uint8).pin_memory()
    host = pinned.numpy()
    for i in range(pairs):
        host[i, 0], host[i, 1] = np.roll(f.left, i, axis=1), np.roll(f.right, i, axis=1)
    dev = pinned.cuda()
    torch.cuda.synchronize()
    fe = J.Frontend(max_width=width, max_height=height, max_levels=8, max_feats=500, max_pairs=pairs)
    job = lambda a, b: J.Job(a, b, levels=levels, max_feats=500)
    batches = {"host": fe.prepare_batch([job(host[i, 0], host[i, 1]) for i in range(pairs)]),
               "device": fe.prepare_batch([job(dev[i, 0], dev[i, 1]) for i in range(pairs)])}
    best, keypoints = {}, {}
    for name, batch in batches.items():
        fe.extract_batch(batch)  # without timing
        fe.sync()
        plain = J.to_numpy(fe.keypoints(pairs - 1, 1))
        fe.enable_stage_timing(True)
        t = []
        for _ in range(12):
            fe.extract_batch(batch)
            fe.sync()
            t.append(fe.stage_times()["pyramid"])
        fe.enable_stage_timing(False)
        best[name] = min(t)
        keypoints[name] = J.to_numpy(fe.keypoints(pairs - 1, 1))
        for k in plain:
            assert np.array_equal(plain[k], keypoints[name][k]), (name, k)
    for k in keypoints["host"]:
        assert np.array_equal(keypoints["host"][k], keypoints["device"][k]), k
    assert best["host"] <= 1.5 * best["device"], best
    fe.close()
