"""The exhaustive matcher behind the tensor-core matcher (references whose bins may have lost a candidate): on integer
images, where FP32 distances are exact, every group equals the definition's, ties included.  Stripes whose equally
good candidates crowd few bins, without noise (whole lattices tie: the list of candidates at the bound overflows into
the exact one) and with a little; windows cut by the border, every group size the bins overflow for, one to three
channels."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a,b,period,C,H,W,K,win,noise", [
    (1, 3, 16, 1, 96, 96, 16, 21, 0), (1, 3, 16, 3, 80, 128, 16, 31, 1), (3, 1, 16, 3, 80, 128, 16, 31, 0),
    (3, 1, 16, 1, 96, 96, 32, 21, 1), (3, 1, 16, 1, 96, 96, 8, 31, 0), (1, 3, 4, 1, 96, 96, 32, 21, 4),
    (1, 1, 8, 3, 80, 128, 16, 31, 4),
])
def test_listed_references_match_the_definition(a, b, period, C, H, W, K, win, noise, oracle):
    import torch

    from paper_2512_23569_gb300 import hts

    yy, xx = np.mgrid[0:H, 0:W]
    rng = np.random.default_rng(1)
    base = np.round(128 + 60 * np.sin(2 * np.pi * (a * xx + b * yy) / period))
    img = np.stack([base + rng.integers(0, noise + 1, base.shape) for _ in range(C)]).astype(np.float32)
    want, _, _ = oracle.match(img, oracle.Params(K=K, win=win))
    idx, _ = hts.match(torch.from_numpy(img).cuda(), p=hts.params(K=K, win=win, precision=1))
    assert hts.last_stats()["match_fallback"] >= 50
    np.testing.assert_array_equal(idx.cpu().numpy(), want)
