"""Matching times that must not turn over: a smaller search window holds fewer candidates, so the FP32 matcher may not
take longer for it (device times, the least of several)."""

import numpy as np
import pytest

from paper_2512_23569_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _match_us(hts, x, params):
    """The least matching time of each set of parameters, the sets timed in turn."""
    for p in params:
        hts.match(x, p=p)
    times = [[] for _ in params]
    for _ in range(21):
        for p, t in zip(params, times):
            hts.profile_begin()
            hts.match(x, p=p)
            r = hts.profile_end()
            t.append(1e3 * sum(r[k][0] for k in ("k_match", "k_match_fallback")))
    return [min(t) for t in times]


@pytest.mark.parametrize("H,W,C,K,win,wide", [
    (301, 417, 1, 16, 9, 21), (512, 640, 1, 16, 9, 21), (512, 640, 3, 4, 9, 21),
    (24, 30, 1, 16, 7, 21), (96, 128, 3, 16, 7, 31), (203, 317, 3, 2, 9, 21),  # the reference-per-warp matcher's sizes
])
def test_a_smaller_window_takes_no_longer(H, W, C, K, win, wide):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    _, noisy = synth.make_config_image(H, W, C, 20.0, 7 * H + W)
    x = torch.from_numpy(np.ascontiguousarray(noisy, dtype=np.float32)).cuda()
    small, large = _match_us(hts, x, [hts.params(K=K, win=win), hts.params(K=K, win=wide)])
    assert small <= large


@pytest.mark.parametrize("C,win,step,noise,share", [(1, 31, 4, 1, 0.32), (3, 45, 2, 0, 0.19)])
def test_the_exhaustive_pass_over_a_few_references_stays_short(C, win, step, noise, share):
    """Some dozens of the references, ties among their candidates, against the tensor-core matching of all of them."""
    from paper_2512_23569_gb300 import build, hts

    build.build()
    img = synth.make_config_image(400, 400, C, 20.0, 5)[noise]
    x = torch.from_numpy(np.ascontiguousarray(img, dtype=np.float32)).cuda()
    p = hts.params(K=16, win=win, step=step, precision=1)
    hts.match(x, p=p)
    assert 0 < hts.last_stats()["match_fallback"] < 100
    times = []
    for _ in range(21):
        hts.profile_begin()
        hts.match(x, p=p)
        r = hts.profile_end()
        times.append([r[k][0] for k in ("k_match_rescue", "k_match_tc")])
    assert min(t[0] for t in times) <= share * min(t[1] for t in times)
