"""FP32 matching of an image with a NaN pixel: a distance over it is no number, so the references whose patch covers the
pixel have no candidates and repeat themselves, no other group takes a patch that covers it, and every index is a patch
of the image (the kernels behind read pixels at them).  Both matchers, gray and colour."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grid(n, step):
    return sorted(set(range(0, n - 7, step)) | {n - 8})


@pytest.mark.parametrize("C,H,W,K,win,step", [(1, 40, 44, 16, 21, 3), (3, 36, 41, 8, 21, 4), (1, 96, 101, 16, 21, 4),
                                              (1, 97, 98, 32, 31, 4), (3, 229, 231, 16, 31, 4)])
def test_groups_stay_inside_the_image_and_off_the_pixel(C, H, W, K, win, step):
    import torch

    from paper_2512_23569_gb300 import build, hts

    build.build()
    img = np.random.default_rng(H).uniform(0, 255, (C, H, W)).astype(np.float32)
    y, x = H // 2, W // 2
    img[:, y, x] = np.nan
    idx, _ = hts.match(torch.from_numpy(img).cuda(), p=hts.params(K=K, win=win, step=step))
    idx = idx.cpu().numpy().astype(np.int64)
    py, px = idx // W, idx % W
    assert idx.min() >= 0 and py.max() <= H - 8 and px.max() <= W - 8
    covers = (py <= y) & (y < py + 8) & (px <= x) & (x < px + 8)
    refs = np.array([r * W + c for r in _grid(H, step) for c in _grid(W, step)])
    np.testing.assert_array_equal(idx[:, 0], refs)
    hit = covers[:, 0]
    assert hit.any()
    np.testing.assert_array_equal(idx[hit], np.repeat(refs[hit, None], K, 1))
    assert not covers[~hit].any()
