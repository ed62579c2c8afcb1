"""Record ends of the series prep (needs a GPU): the signals of records around
the lengths where blocks, chunks and the filters' exact starts change, against
the oracle, in both precisions.

The prep walks 64-row blocks of X (row r holds sample r - 1); H + 3 samples
(H = 16 mixed, 32 FP64) is the shortest record it filters, and the last sample,
the ghost after it and the block it lies in move with the length.  Random
fields make every sample count.  Bars: FP64 1e-11, mixed 1e-5 relative L2 per
observer (rounding of sums of 77 panels; a wrong end sample is O(1e-2))."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle, uv_sphere
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-11), ("mixed", 1e-5)])
@pytest.mark.parametrize("nts", [(3, 4, 5, 17, 18, 19, 20, 21), (33, 34, 35, 36, 37, 62, 63, 64, 65), (95, 96, 97, 125, 126, 127, 128, 129),
                                 (145, 157, 158, 159, 160, 161, 189, 190), (191, 192, 193, 253, 254, 256)])
def test_lengths_around_block_and_chunk_ends(dev, prec, bar, nts):
    from paper_2312_16263_gb300 import FWH
    surf = uv_sphere(0.02, 7, 11)           # small: nearly the whole record is valid
    obs = observers_circle(6.0, 3)
    s = FWH(surf.centroids, surf.normals, surf.areas, 0.4, 0.1, 0.03, prec, observers=obs)
    orc = Oracle(surf.centroids, surf.normals, surf.areas, 0.4, 0.1, 0.03)
    rng = np.random.default_rng(5)
    for nt in nts:
        f = torch.as_tensor(rng.normal(size=(nt, 5, surf.n_panels)) * 1e-3, dtype=s.dtype, device=dev)
        p = s.forward(f).cpu().numpy()
        s.check()
        _, nv = s.window(nt)
        ref, _, nv_ref = orc.forward(f.double().cpu().numpy(), obs)
        for o in range(3):
            n = int(min(nv[o], nv_ref[o]))
            assert n >= nt - 2, (nt, o, n)
            err = np.linalg.norm(p[o, :n] - ref[o, :n]) / np.linalg.norm(ref[o, :n])
            assert err <= bar, (nt, o, err)
    s.close()
