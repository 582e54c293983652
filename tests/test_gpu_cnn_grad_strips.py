"""The training step's weight-gradient strips (8 x 64 pixels, up to one block per strip and SM) at their edges:
smallest image, exact and one-over strips, more strips than blocks; and the packed weights after an Adam step.

Tolerance of the gradients: as the training-step test, 2e-3 of a layer's norm (a stored FP16 value can move by one
unit where FP32 and FP64 accumulation round apart)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _theta(co, C, rng):
    parts = []
    for cout, cin in co.layer_shapes(C):
        parts.append(rng.standard_normal(cout * cin * 9) * np.sqrt(2.0 / (9 * cin)))
        parts.append(rng.standard_normal(cout) * 0.05)
    return np.concatenate(parts).astype(np.float32)


@pytest.mark.parametrize("C,H,W", [(1, 12, 12), (3, 16, 64), (3, 9, 65), (1, 16, 128), (3, 160, 513)])
def test_gradients_at_strip_edges_and_after_adam(C, H, W):
    import torch

    from oracle import cnn_oracle as co
    from paper_2512_23569_gb300 import hts

    rng = np.random.default_rng(31 * H + W + C)
    net = hts.Cnn(C, seed=2)
    net.set_params(_theta(co, C, rng))
    p = hts.params()
    cen = co.ref_centres(H, W)
    img = rng.uniform(0, 255, size=(C, H, W)).astype(np.float32)
    tgt = rng.uniform(1.0, 3.5, size=len(cen)).astype(np.float32)
    x, t = torch.from_numpy(img).cuda(), torch.from_numpy(tgt).cuda()
    for step in range(2):  # the second on the weights the Adam step wrote
        th16 = co.fp16(net.get_params().astype(np.float64))
        want_loss, want = co.grad_act16(th16, img, cen, tgt)
        net.zero_grad()
        net.accumulate_grad(x, t, p)
        assert net.take_loss() == pytest.approx(want_loss, rel=1e-3)
        got = net.get_grad().astype(np.float64)
        o = 0
        for cout, cin in co.layer_shapes(C):
            n = cout * cin * 9 + cout
            assert np.linalg.norm(got[o:o + n] - want[o:o + n]) <= 2e-3 * np.linalg.norm(want[o:o + n]) + 1e-9
            o += n
        net.adam_step(1e-3)
