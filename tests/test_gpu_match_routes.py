"""FP32 matching against the FP64 oracle, whole numbers equal, through both matchers: the cell-sharing one on the sizes
it takes (grids of 500 to 40000 references, by window and channels; grids cut around its tiles of eight, last rows and
columns off the step), and the reference-per-warp one at every other grid step and at windows above 31.  Both Eq. 9
planes in one tile, ties, near ties that FP64 decides, and more near candidates than a warp's list holds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _image(kind, C, H, W):
    rng = np.random.default_rng(H * W + C)
    yy, xx = np.mgrid[0:H, 0:W]
    if kind == "noise":
        return rng.uniform(0, 255, (C, H, W))
    if kind == "planes":  # green dominates in patches, so that neighbouring references differ in Eq. 9's plane
        img = rng.uniform(20, 90, (3, H, W))
        img[1] *= np.where(((yy // 9) + (xx // 7)) % 2, 1.6, 0.6)
        return img[:C]
    if kind == "flat":
        return np.full((C, H, W), 37.0)
    if kind == "stripes":
        return 90.0 + 60.0 * np.sin(2 * np.pi * (xx - yy) / 7.0)[None] + 0.01 * rng.standard_normal((C, H, W))
    return np.clip(np.repeat(((yy // 16) * 40.0 + (xx // 12) * 7.0)[None], C, 0) + 5.0 * rng.standard_normal((C, H, W)),
                   0, 255)


def _check(oracle, kind, C, H, W, K, win, step):
    import torch

    from paper_2512_23569_gb300 import build, hts

    build.build()
    img = _image(kind, C, H, W).astype(np.float32)
    want, wgreen, _ = oracle.match(img, oracle.Params(K=K, win=win, step=step))
    idx, green = hts.match(torch.from_numpy(img).cuda(), p=hts.params(K=K, win=win, step=step))
    np.testing.assert_array_equal(green.cpu().numpy(), wgreen)
    np.testing.assert_array_equal(idx.cpu().numpy(), want)


@pytest.mark.parametrize("kind,C,H,W,K,win", [
    ("steps", 1, 93, 102, 16, 21), ("stripes", 1, 96, 96, 32, 31), ("flat", 1, 100, 92, 16, 21), ("noise", 1, 100, 101, 8, 25),
    ("noise", 1, 140, 136, 2, 21), ("steps", 1, 227, 230, 16, 19), ("noise", 1, 230, 229, 4, 17),
    ("steps", 1, 341, 343, 32, 13), ("noise", 1, 345, 340, 16, 15), ("noise", 1, 812, 812, 8, 7), ("noise", 1, 812, 813, 4, 5),
    ("planes", 3, 229, 231, 16, 31), ("planes", 3, 228, 230, 32, 21), ("steps", 3, 232, 227, 16, 17),
    ("stripes", 3, 228, 228, 16, 31), ("flat", 3, 228, 229, 8, 21), ("planes", 3, 343, 341, 16, 11),
    ("planes", 3, 812, 810, 8, 7), ("planes", 3, 97, 100, 32, 31), ("stripes", 3, 98, 99, 32, 29),
])
def test_cell_matcher(kind, C, H, W, K, win, oracle):
    _check(oracle, kind, C, H, W, K, win, 4)


@pytest.mark.parametrize("kind,C,H,W,K,win,step", [
    ("noise", 1, 41, 43, 16, 21, 1), ("planes", 3, 40, 37, 16, 21, 1), ("planes", 3, 45, 52, 32, 31, 2),
    ("steps", 1, 50, 61, 2, 9, 3), ("planes", 3, 63, 58, 8, 33, 3), ("stripes", 3, 64, 61, 16, 21, 5),
    ("flat", 1, 44, 40, 16, 21, 5), ("flat", 3, 41, 46, 32, 21, 8), ("planes", 3, 90, 97, 16, 63, 8),
    ("noise", 1, 83, 85, 32, 63, 4), ("stripes", 3, 70, 81, 32, 33, 4), ("steps", 3, 81, 70, 2, 33, 4),
    ("stripes", 1, 64, 64, 8, 41, 7), ("planes", 3, 42, 41, 4, 31, 6),
])
def test_reference_per_warp_matcher(kind, C, H, W, K, win, step, oracle):
    _check(oracle, kind, C, H, W, K, win, step)
