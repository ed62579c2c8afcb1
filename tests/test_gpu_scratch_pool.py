"""The scratch that moving_forward keeps between calls (needs a GPU): at most 8 GiB,
given back to the device by set_moving_scratch; the call after that gives the same
result (to the rounding of the output sums, 1e-12 of the largest value)."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


def test_kept_scratch_goes_back(dev):
    from paper_2312_16263_gb300 import moving_forward, set_moving_scratch
    P, nt, O = 4096, 512, 8
    g = torch.Generator(device=dev).manual_seed(1)
    k = np.arange(P) + 0.5
    z = 1.0 - 2.0 * k / P
    r, ph = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    n0 = torch.as_tensor(np.stack([r * np.cos(ph), r * np.sin(ph), z], 1), device=dev)
    y = (n0[None] + 0.1 * 0.02 * torch.arange(nt, dtype=torch.float64, device=dev)[:, None, None]).contiguous()
    n, v = n0.expand(nt, P, 3).contiguous(), torch.full((nt, P, 3), 0.1, dtype=torch.float64, device=dev)
    f = 1e-3 * torch.randn((nt, 5, P), dtype=torch.float64, device=dev, generator=g)
    out = torch.empty((O, nt), dtype=torch.float64, device=dev)

    def call():
        return moving_forward(y, n, v, np.full(P, 4 * np.pi / P), 1.0, 1.0, 0.02, f,
                              observers_circle(12.0, O), out=out)[0].clone()

    set_moving_scratch()
    first = call()           # also loads the kernels
    set_moving_scratch()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    call()
    kept = free - torch.cuda.mem_get_info()[0]
    assert 2 * 8 * nt * P * O <= kept <= 8 << 30      # two columns of nt per (panel, observer)
    set_moving_scratch()
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    torch.testing.assert_close(call(), first, rtol=1e-12, atol=1e-12 * first.abs().max().item())
    set_moving_scratch()
