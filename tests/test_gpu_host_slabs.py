"""Host fields of small surfaces, copied in slabs of 128 frames and more (needs a GPU).

A slab holds 4 MB or 64 frames, whichever is more: 128 frames of 1700 panels, 256 of
1000, 704 of 300, 2752 of 77; past 128 frames the scatter runs in segments of a whole
chunk of the tile shape, the short segment first.  Record lengths around the slabs'
and segments' edges, against the same fields in one copy, one prep and one scatter.
The series are the same bits; FP32 sums split at other segment ends agree to their
rounding, 1e-6 relative L2 per observer (rows left over from the larger record before
would be O(1))."""
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


@pytest.mark.parametrize("cfg", [-1, 2])
@pytest.mark.parametrize("panels,nts", [
    (1700, (256, 257, 372, 383, 384, 385, 700)), (1000, (257, 504, 505, 511, 512, 513, 769, 1008)),
    (300, (705, 756, 1407, 1408, 1409, 2113)), (77, (2753, 2772, 5505))])
def test_slabs_of_small_surfaces(dev, panels, nts, cfg):
    from paper_2312_16263_gb300 import FWH
    k = np.arange(panels) + 0.5
    z = 1.0 - 2.0 * k / panels
    r, ph = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    n = np.stack([r * np.cos(ph), r * np.sin(ph), z], 1)
    g = torch.Generator(device=dev).manual_seed(panels)

    def handle():
        s = FWH(0.1 * n, n, np.full(panels, 0.04 * np.pi / panels), 0.4, 0.1, 0.02, "mixed",
                observers=observers_circle(20.0, 7))
        s.set_tile_config(cfg)
        return s

    host, ref = handle(), handle()
    host.forward(0.1 * torch.randn((nts[-1] + 300, 5, panels), device=dev, generator=g))
    for nt in nts:
        f = 1e-3 * torch.randn((nt, 5, panels), device=dev, generator=g)
        want = ref.forward(f).cpu()
        _, nv = ref.window(nt)
        got = host.forward(f.cpu().pin_memory())
        host.check()
        for o, m in enumerate(nv):
            assert m > nt - 30
            err = torch.linalg.norm(got[o, :m] - want[o, :m]) / torch.linalg.norm(want[o, :m])
            assert err.item() <= 1e-6, (nt, o, err)
            assert torch.all(got[o, m:] == 0)
    host.close()
    ref.close()
