"""The tensor-core filter's inverse (a tensor-memory lane per pixel, a column per Haar row) at every group size and
channel count, with partly filled batches and tiles, against the FP32 filter on the same exact groups."""

import math

import numpy as np
import pytest

from paper_2512_23569_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [4.0, 40.0])  # most groups keep detail coefficients, few do
@pytest.mark.parametrize("K", [8, 16, 32])
@pytest.mark.parametrize("H,W,C,win", [(12, 16, 1, 21), (24, 20, 3, 21), (61, 77, 1, 21), (67, 53, 3, 31)])
def test_tensor_core_filter_follows_the_fp32_filter(H, W, C, win, K, sigma):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    _, noisy = synth.make_config_image(H, W, C, sigma, 1000 * K + H)
    x = torch.from_numpy(np.ascontiguousarray(noisy, dtype=np.float32)).cuda()
    want = hts.denoise(x, sigma=sigma, p=hts.params(K=K, win=win, precision=0)).cpu().double()
    got = hts.denoise(x, sigma=sigma, p=hts.params(K=K, win=win, precision=2)).cpu().double()
    diff = (got - want).abs()
    # FP16 rounding: 0.05 in the mean, the bound of the same groups at full size.  A coefficient within it of the
    # threshold may be kept on one side only: tau |u v h| <= tau / 32 on the pixels of its group's patches; four
    # such groups are allowed for.
    n_ref = (-(-(H - 8) // 4) + 1) * (-(-(W - 8) // 4) + 1)
    tau = sigma * math.sqrt(2.0 * math.log(C * K * 64))
    assert float(diff.max()) <= 12.0
    assert float(diff.mean()) <= 0.05 + 4.0 * (tau / 32.0) / n_ref
