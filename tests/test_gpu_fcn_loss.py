"""The enhancement network's loss is summed in 64 bits.  With a zero network and one error e for every value, e^2 has
48 significant bits, every partial sum of equal terms k e^2 (k < 32 times a power of two) fits FP64's 53 and the mean is
e^2 to the last bit; a sum held in fewer bits rounds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,n", [(1, 64), (3, 64), (3, 4096)])
def test_the_mean_of_equal_squares_is_exact(C, n):
    import torch

    from paper_2512_23569_gb300 import hts

    f = hts.Fcn(C, 16, seed=1)
    f.set_params(np.zeros(f.nparams, dtype=np.float32))
    noisy = torch.zeros(n, C * 64, device="cuda")
    sigma = torch.full((n,), 4.0, device="cuda")  # 4 / sqrt(K) = 1: errors in grey levels
    for e in (1.6369617, -1.0165277, 1.9127556, 1.6066358e-15, -1.7294966e15):
        e = np.float32(e)
        f.accumulate_grad(noisy, torch.full((n, C * 64), float(e), device="cuda"), sigma)
        assert f.take_loss() == float(e) ** 2
