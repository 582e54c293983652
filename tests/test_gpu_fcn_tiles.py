"""The enhancement network's GEMM tiles at their edges: sample counts around the 64-sample tile, the 16-sample slab
and the parts of the weight gradients, against the FP64 oracle.

Tolerances: every value is a chain of at most 208 (layers) or n (gradients, in parts) fused multiply-adds in FP32,
so its error is below (208 + 3 layers' propagation) u relative to the sum of absolute products -- 1e-4 of the norm
leaves a factor of ten."""

import numpy as np
import pytest

from oracle import fcn_oracle as fo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,K,n", [(1, 8, 1), (3, 16, 3), (1, 16, 63), (3, 16, 64), (3, 16, 65), (1, 32, 129),
                                   (3, 8, 1000), (3, 16, 4097)])
def test_refine_and_gradients_at_tile_edges(C, K, n):
    import torch

    from paper_2512_23569_gb300 import hts

    rng = np.random.default_rng(17 * n + C)
    f = hts.Fcn(C, K, seed=n)
    theta = f.get_params() + 0.01 * rng.standard_normal(f.nparams).astype(np.float32)
    f.set_params(theta)
    noisy = (60.0 * rng.standard_normal((n, C * 64))).astype(np.float32)
    clean = (noisy + 12.0 * rng.standard_normal((n, C * 64))).astype(np.float32)
    sigma = rng.uniform(30, 75, n).astype(np.float32)
    dn, dc, ds = (torch.from_numpy(a).cuda() for a in (noisy, clean, sigma))
    want = fo.refine(theta, noisy, sigma, C, K)
    got = f.refine(dn, ds).cpu().numpy()
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
    f.zero_grad()
    for _ in range(2):  # gradients and losses add up
        f.accumulate_grad(dn, dc, ds)
    out, cache = fo.forward(theta, fo.features(noisy, sigma, C, K), C)
    loss, dout = fo.loss_and_dout(out, noisy, clean, sigma, K)
    grad = 2.0 * fo.backward(theta, cache, dout, C)
    o = 0
    g = f.get_grad().astype(np.float64)
    for n_out, n_in in fo.layer_shapes(C):
        for size in (n_out * n_in, n_out):
            a, b = g[o:o + size], grad[o:o + size]
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b) + 1e-9
            o += size
    assert abs(f.take_loss() - 2.0 * loss) <= 1e-5 * loss
