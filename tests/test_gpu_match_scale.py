"""Tensor-core matcher: the distances' scale (a power of two per tile) leaves the groups alone, for every bin shape.
Multiplying an image by a power of two multiplies every distance exactly, so the groups are those of the image."""

import numpy as np
import pytest

from paper_2512_23569_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [4, 8, 16, 32])
@pytest.mark.parametrize("H,W,C,win", [(45, 61, 1, 21), (67, 53, 3, 31)])
def test_groups_do_not_depend_on_a_power_of_two(H, W, C, win, K):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    _, noisy = synth.make_config_image(H, W, C, 20.0, 100 * K + H)
    x = torch.from_numpy(np.ascontiguousarray(noisy, dtype=np.float32)).cuda()
    p = hts.params(K=K, win=win, precision=1)
    idx, green = hts.match(x, p=p)
    exact, _ = hts.match(x, p=hts.params(K=K, win=win, precision=0))
    # BF16 keys, FP32 re-rank of the nearest 2 K: nearly all groups are the exact ones
    assert float((idx == exact).all(dim=1).float().mean()) >= 0.9
    for e in (-40, -12, 9, 40):
        scaled, g = hts.match(x * 2.0**e, p=p)
        assert torch.equal(scaled, idx) and (C == 1 or torch.equal(g, green))  # gray has no plane flags
