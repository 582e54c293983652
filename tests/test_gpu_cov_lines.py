"""Covariance sums over chunks of grid lines, with entries taken from the entry one step before them (step 4 to 7):
every grid step, grids with and without a last line off the step, one to several lines and chunks per block."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [1, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("H,W,C", [(8, 16, 3), (12, 9, 1), (16, 15, 3), (23, 301, 1), (129, 40, 3), (150, 263, 3)])
def test_eigenvalues_match_oracle(oracle, H, W, C, step):
    from paper_2512_23569_gb300 import build, hts

    build.build()
    rng = np.random.default_rng(1000 * H + step)
    x = rng.integers(0, 256, size=(C, H, W)).astype(np.float32)  # whole numbers: the cover counts multiply exactly
    _, want, _ = oracle.estimate_basis(x, oracle.Params(K=8, step=step))
    b, got = hts.estimate_basis(torch.from_numpy(x).cuda(), p=hts.params(K=8, step=step)).read()
    # the bound of the suite's eigenvalue comparisons
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-10 * np.max(np.abs(want)))
