"""A mean pressure far above the fluctuation, on flat faces (needs a GPU).

A box whose faces' normals lie along the axes carries p' = 1 with a fluctuation of
1e-3; the integrands are then exact, and the far field of the fluctuation comes from
differences in source time that the mean must not spoil.  Compared with the oracle
less each signal's mean.  Bars: the offset's share of a panel's term is about 16
times the fluctuation's (c_L against c_L' at 20 units and 10 rad per unit of time), a
window sums 25 panels of one face in the type of the fields with a few roundings a
panel: 6e-8 x 16 x 25 x 8 = 2e-4 in FP32, 1.1e-16 x 3200 = 4e-13 in FP64.  A
difference of rounded spline coefficients left 6e-4, integrands scaled by a factor
that is no power of two 1e-12."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle
from oracle import Oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


def _box(m):
    g = (np.arange(m) + 0.5) / m - 0.5
    a, b = (v.ravel() for v in np.meshgrid(g, g, indexing="ij"))
    pos, nrm = [], []
    for axis in range(3):
        for sign in (-1.0, 1.0):
            q, n = np.zeros((m * m, 3)), np.zeros((m * m, 3))
            q[:, (axis + 1) % 3], q[:, (axis + 2) % 3], q[:, axis] = a, b, 0.5 * sign
            n[:, axis] = sign
            pos.append(q)
            nrm.append(n)
    return np.concatenate(pos), np.concatenate(nrm), np.full(6 * m * m, 1.0 / (m * m))


@pytest.mark.parametrize("prec,bar", [("mixed", 2e-4), ("fp64", 4e-13)])
@pytest.mark.parametrize("nt", [128, 191, 256, 600, 1000])
def test_fluctuation_under_a_mean(dev, prec, bar, nt):
    from paper_2312_16263_gb300 import FWH
    pos, nrm, area = _box(5)
    obs = observers_circle(20.0, 5)
    rng = np.random.default_rng(3)
    f = np.zeros((nt, 5, len(area)))
    f[:, 4] = 1.0 + 1e-3 * np.sin(0.1 * np.arange(nt)[:, None] + rng.uniform(0, 2 * np.pi, len(area)))
    f = f.astype(np.float32)
    s = FWH(pos, nrm, area, 0.3, 0.1, 0.01, prec, observers=obs)
    p = s.forward(torch.as_tensor(f, device=dev).to(s.dtype)).cpu().numpy()
    s.check()
    _, nv = s.window(nt)
    s.close()
    ref, _, nv_ref = Oracle(pos, nrm, area, 0.3, 0.1, 0.01).forward(f.astype(np.float64), obs)
    for o in range(5):
        n = int(min(nv[o], nv_ref[o]))
        assert n > nt // 3
        a, b = p[o, :n] - p[o, :n].mean(), ref[o, :n] - ref[o, :n].mean()
        err = np.linalg.norm(a - b) / np.linalg.norm(b)
        assert err <= bar, (o, err)
