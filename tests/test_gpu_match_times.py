"""Matching times that must not turn over: a smaller search window holds fewer candidates, so the FP32 matcher may not
take longer for it (device times, the least of several)."""

import numpy as np
import pytest

from paper_2512_23569_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _match_us(hts, x, **kw):
    p = hts.params(**kw)
    hts.match(x, p=p)
    times = []
    for _ in range(7):
        hts.profile_begin()
        hts.match(x, p=p)
        r = hts.profile_end()
        times.append(1e3 * sum(r[k][0] for k in ("k_match", "k_match_fallback")))
    return min(times)


@pytest.mark.parametrize("H,W,C,K,win,wide", [
    (301, 417, 1, 16, 9, 21), (512, 640, 1, 16, 9, 21), (512, 640, 3, 4, 9, 21),
    (24, 30, 1, 16, 7, 21), (96, 128, 3, 16, 7, 31), (203, 317, 3, 2, 9, 21),  # the reference-per-warp matcher's sizes
])
def test_a_smaller_window_takes_no_longer(H, W, C, K, win, wide):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    _, noisy = synth.make_config_image(H, W, C, 20.0, 7 * H + W)
    x = torch.from_numpy(np.ascontiguousarray(noisy, dtype=np.float32)).cuda()
    assert _match_us(hts, x, K=K, win=win) <= _match_us(hts, x, K=K, win=wide)
