"""Device memory of the noise-map network's calls: log_sigma_map writes the caller's map, so the network allocates its
two FP16 activation buffers (32 channels each) and nothing per pixel besides."""

import gc

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_the_noise_map_call_allocates_its_activations_only():
    from paper_2512_23569_gb300 import build, hts

    build.build()
    H, W = 2048, 4096
    net = hts.Cnn(1, seed=1)
    x = torch.zeros(1, H, W, device="cuda")
    net.log_sigma_map(x[:, :64, :64].contiguous())  # the kernels loaded, torch's pool warm
    net = hts.Cnn(1, seed=1)
    out = torch.empty(H, W, device="cuda")  # the map's place in torch's pool
    del out
    gc.collect()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net.log_sigma_map(x)
    torch.cuda.synchronize()
    taken = before - torch.cuda.mem_get_info()[0]
    planes = 2 * 32 * 2 * H * W
    assert planes <= taken < planes + 4 * H * W // 2  # less than half a map more (allocation granularity)
