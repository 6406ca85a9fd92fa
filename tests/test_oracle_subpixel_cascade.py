"""The oracle's refinement on a cascaded pyramid: the windows come from the
levels the keypoints were found on, each resampled from the one above."""
import numpy as np
import pytest

from test_oracle_subpixel import smooth_texture


@pytest.mark.parametrize("mode", [0, 1])
def test_sads_come_from_the_levels_of_the_mode(oracle, mode):
    p = oracle.FrontendParams()
    p.levels, p.max_feats, p.fast_thresh, p.pyramid_mode = 4, 500, 15, mode
    left, right = smooth_texture(300, 420, 0.0, 11), smooth_texture(300, 420, 10.25, 11)
    kl, kr, m = oracle.extract_pair(left, right, p)
    w, L = 4, 3
    got = oracle.subpixel(left, right, kl, kr, m[0], p, w, L, 0.0)["sad"]
    W, H, _ = oracle.level_geometry(420, 300, p.levels, p.scale, p.cell)
    lev = []
    for img in (left, right):
        raw = [img]
        for n in range(1, p.levels):
            raw.append(oracle.pyramid_level_sized(raw[n - 1], p.scale, 1, int(W[n]), int(H[n])) if mode
                       else oracle.pyramid_level(img, p.scale, n))
        lev.append([r.astype(np.int64) for r in raw])
    seen = 0
    for i in range(kl["count"]):
        j, n = m[0][i], int(kl["level"][i])
        if j < 0 or n < 2:
            continue
        x, y = int(kl["x"][i]), int(kl["y"][i])
        xr = int(np.floor(float(kr["X"][j]) / oracle.level_scale(p.scale, n) + 0.5))
        if x < w or x + w >= W[n] or y < w or y + w >= H[n] or xr < L + w or xr + L + w >= W[n]:
            assert got[i] == 0xFFFFFFFF
            continue
        a = lev[0][n][y - w:y + w + 1, x - w:x + w + 1]
        sads = []
        for t in range(-L, L + 1):
            b = lev[1][n][y - w:y + w + 1, xr + t - w:xr + t + w + 1]
            sads.append(np.abs((a - a[w, w]) - (b - b[w, w])).sum())
        assert got[i] == min(sads), (i, n)
        seen += 1
    assert seen > 20
