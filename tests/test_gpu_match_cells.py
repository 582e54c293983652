"""The cell-sharing matcher (grid step 4, windows up to 31) against the FP64 oracle, whole numbers equal: tile edges
(references per row and column around 8), grids whose last row and column are off the step, both Eq. 9 planes in
one tile, every group size, ties, and more near candidates than a warp's list holds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _image(kind, C, H, W, rng):
    yy, xx = np.mgrid[0:H, 0:W]
    if kind == "noise":
        return rng.uniform(0, 255, (C, H, W))
    if kind == "planes":  # green dominates in patches, so that neighbouring references differ in Eq. 9's plane
        base = np.where(((yy // 9) + (xx // 7)) % 2, 1.6, 0.6)
        img = rng.uniform(20, 90, (3, H, W))
        img[1] *= base
        return img[:C]
    if kind == "flat":
        return np.full((C, H, W), 37.0)
    if kind == "stripes":
        return 90.0 + 60.0 * np.sin(2 * np.pi * (xx - yy) / 7.0)[None] + 0.01 * rng.standard_normal((C, H, W))
    return np.clip(np.repeat(((yy // 16) * 40.0 + (xx // 12) * 7.0)[None], C, 0) + 5.0 * rng.standard_normal((C, H, W)),
                   0, 255)


@pytest.mark.parametrize("kind,C,H,W,K,win", [
    ("noise", 1, 36, 36, 16, 21), ("noise", 1, 40, 40, 8, 21), ("steps", 3, 37, 71, 16, 31),
    ("planes", 3, 68, 45, 16, 31), ("planes", 3, 41, 42, 32, 21), ("noise", 1, 12, 75, 16, 31),
    ("noise", 3, 75, 12, 4, 15), ("noise", 1, 20, 20, 2, 3), ("steps", 1, 51, 50, 32, 31), ("flat", 1, 40, 44, 16, 21),
    ("flat", 3, 30, 33, 8, 9), ("stripes", 1, 64, 64, 16, 31), ("stripes", 3, 48, 49, 32, 29), ("noise", 1, 9, 9, 2, 31),
    ("noise", 1, 64, 96, 32, 31), ("steps", 1, 60, 61, 16, 33),  # 33: the reference-per-warp matcher
])
def test_groups_equal_the_oracle(kind, C, H, W, K, win, oracle):
    import torch

    from paper_2512_23569_gb300 import hts

    img = _image(kind, C, H, W, np.random.default_rng(H * W + K)).astype(np.float32)
    want, wgreen, _ = oracle.match(img, oracle.Params(K=K, win=win))
    idx, green = hts.match(torch.from_numpy(img).cuda(), p=hts.params(K=K, win=win))
    np.testing.assert_array_equal(green.cpu().numpy(), wgreen)
    np.testing.assert_array_equal(idx.cpu().numpy(), want)
