"""Batches of host frames uploaded in parts: the results of the same frames on
the device, for one to four parts, uneven ones, pairs of several sizes, frames
that do not lie in one run, and frames replaced between calls."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("sizes,order", [
    ([(752, 480)] * 5, 1), ([(752, 480)] * 12, 1), ([(752, 480)] * 23, 1), ([(752, 480)] * 23, -1),
    ([(1920, 1080)] * 3, 1), ([(641, 479)] * 9 + [(1241, 376)] * 10 + [(1919, 1079)] * 2, 1),
])
@pytest.mark.parametrize("mode", [0, 1])
def test_host_batch_equals_device_batch(J, sizes, order, mode):
    import torch
    n = len(sizes)
    total = sum(2 * w * h for w, h in sizes)
    pinned = torch.empty(total, dtype=torch.uint8).pin_memory()
    flat = pinned.numpy()
    views, at = [], 0
    for w, h in sizes:
        pair = []
        for _ in range(2):
            pair.append(flat[at:at + w * h].reshape(h, w))
            at += w * h
        views.append(pair)
    args = dict(levels=4, max_feats=500)
    make = lambda: J.Frontend(max_width=1920, max_height=1080, max_feats=500, fast_thresh_lo=7, max_pairs=n,
                              pyramid_mode=mode)
    fh, fd = make(), make()
    pairs = views[::order]
    batch = fh.prepare_batch([J.Job(a, b, **args) for a, b in pairs])
    for seed in (1, 2, 3):
        rng = np.random.default_rng(seed)
        for a, b in views:
            small = rng.integers(0, 256, (a.shape[0] // 8 + 1, a.shape[1] // 8 + 1)).astype(np.uint8)
            a[:] = np.kron(small, np.ones((8, 8), np.uint8))[:a.shape[0], :a.shape[1]]
            b[:] = np.roll(a, -7, axis=1)
        fh.extract_batch(batch)
        fh.match()
        fh.sync()
        dev = [[torch.from_numpy(im.copy()).cuda() for im in p] for p in pairs]
        torch.cuda.synchronize()
        fd.extract_batch([J.Job(a, b, **args) for a, b in dev])
        fd.match()
        fd.sync()
        for p in range(n):
            for side in (0, 1):
                got, want = J.to_numpy(fh.keypoints(p, side)), J.to_numpy(fd.keypoints(p, side))
                assert got["count"] == want["count"] > 0
                for k in want:
                    assert np.array_equal(got[k], want[k]), (p, side, k)
            got, want = J.to_numpy(fh.matches(p)), J.to_numpy(fd.matches(p))
            for k in want:
                assert np.array_equal(got[k], want[k]), (p, k)
    fh.close()
    fd.close()
