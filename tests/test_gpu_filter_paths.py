"""The tensor-core filter's two inverse paths at partly filled batches and tiles, every group size and channel count, on
inputs whose decisions no rounding can turn, so that a misplaced pixel, row or group shows in any one pixel.

All kept: a zero threshold keeps every coefficient of a noise image, detail rows included.  No detail: the image repeats a
2 x 2 pattern of whole numbers, every group's members are equal (36 positions at an even offset in the smallest window),
the detail rows are exact zeros, the first row's few coefficients lie far above the threshold (38 and more against 14 to
17) and the others, zero but for the rounding of the FP16 operands, below 6.  Either way the output is the image, up to
the FP16 rounding of operands and coefficients: the suite's reconstruction bound, 0.5 at most; its mean bound, 0.05,
holds for the noise image, where the rounding differs from pixel to pixel (a 2 x 2 pattern repeats the same four)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _image(kind, C, H, W):
    rng = np.random.default_rng(100 * H + W + C)
    if kind == "noise":
        return rng.uniform(0, 255, (C, H, W))
    tile = np.array([[220, 90], [140, 30]])[None] - rng.integers(0, 20, (C, 1, 1))
    return np.tile(tile, (1, -(-H // 2), -(-W // 2)))[:, :H, :W]


@pytest.mark.parametrize("kind,sigma", [("noise", 0.0), ("tiles", 4.0)])
@pytest.mark.parametrize("K", [8, 16, 32])
@pytest.mark.parametrize("H,W,C,win", [(24, 20, 1, 21), (24, 20, 3, 21), (27, 32, 3, 31), (61, 77, 1, 21), (67, 53, 3, 31)])
def test_the_filter_returns_the_image(H, W, C, win, K, kind, sigma):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    img = _image(kind, C, H, W).astype(np.float32)
    out = hts.denoise(torch.from_numpy(img).cuda(), sigma=sigma, p=hts.params(K=K, win=win, precision=2)).cpu().numpy()
    assert hts.last_stats()["tau"] == 0.0 if sigma == 0.0 else hts.last_stats()["tau"] > 12.0
    err = np.abs(out.astype(np.float64) - img)
    assert np.max(err) <= 0.5
    assert kind == "tiles" or np.mean(err) <= 0.05
