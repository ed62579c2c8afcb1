"""Observers whose windows end far apart, in one warp (needs a GPU).

The kernels work, chunk by chunk, only on the observers with a valid bin in
reach.  A long row of panels seen end on (few or no valid bins) and broadside
(nearly all) makes every mixture of them; against the oracle, with zeros past
each window.  Bars, relative to the RMS of all signals: FP64 1e-11, mixed 1e-5
(rounding of sums of 203 panels; a chunk or a tail left out is O(1)).  The
gradient, frame by frame against the largest frame: FP64 1e-10, mixed 1e-4."""
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


def _row(rng, n):
    pos = np.stack([12.0 * np.sort(rng.random(n)), 0.1 * rng.random(n), 0.1 * rng.random(n)], 1)
    nrm = rng.normal(size=(n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    return pos, nrm, rng.uniform(0.5, 1.5, n)


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-11), ("mixed", 1e-5)])
@pytest.mark.parametrize("n_obs", [5, 41])
def test_windows_far_apart(dev, prec, bar, n_obs):
    from paper_2312_16263_gb300 import FWH
    rng = np.random.default_rng(8)
    n = 203
    pos, nrm, area = _row(rng, n)
    obs = observers_circle(60.0, n_obs)
    s = FWH(pos, nrm, area, 0.4, 0.1, 0.03, prec, observers=obs)
    orc = Oracle(pos, nrm, area, 0.4, 0.1, 0.03)
    for nt in (300, 509, 1100):
        f = torch.as_tensor(rng.normal(size=(nt, 5, n)) * 1e-3, dtype=s.dtype, device=dev)
        p = s.forward(f).cpu().numpy()
        s.check()
        _, nv = s.window(nt)
        ref, _, nv_ref = orc.forward(f.double().cpu().numpy(), obs)
        assert max(nv_ref) - min(nv_ref) > 200, nv_ref
        k = [int(min(a, b)) for a, b in zip(nv, nv_ref)]
        rms = np.sqrt(sum(np.sum(ref[o, :k[o]] ** 2) for o in range(n_obs)) / sum(k))
        for o in range(n_obs):
            assert abs(int(nv[o]) - int(nv_ref[o])) <= 1
            assert np.all(p[o, int(nv[o]):] == 0.0)
            err = np.sqrt(np.sum((p[o, :k[o]] - ref[o, :k[o]]) ** 2) / max(k[o], 1)) / rms
            assert err <= bar, (nt, o, k[o], err)
    s.close()


@pytest.mark.parametrize("prec,bar", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("shape,n_obs,nts", [
    ("sphere", 3, (3, 4, 62, 63, 64, 65, 66, 126, 127, 128, 129, 130, 131)),  # ends around the chunks' edges
    ("sphere", 40, (65, 129, 193)),
    ("row", 41, (300, 509))])                                             # reordered, most windows short
def test_gradient_at_record_ends_and_past_windows(dev, prec, bar, shape, n_obs, nts):
    from paper_2312_16263_gb300 import FWH
    rng = np.random.default_rng(9)
    if shape == "row":
        pos, nrm, area = (v[::-1].copy() for v in _row(rng, 203))
        mix = rng.permutation(203)
        pos, nrm, area = pos[mix], nrm[mix], area[mix]
        obs = observers_circle(60.0, n_obs)
    else:
        sf = uv_sphere(0.02, 7, 11)             # small: nearly the whole record is valid
        pos, nrm, area = sf.centroids, sf.normals, sf.areas
        obs = observers_circle(6.0, n_obs)
    s = FWH(pos, nrm, area, 0.4, 0.1, 0.03, prec, observers=obs)
    orc = Oracle(pos, nrm, area, 0.4, 0.1, 0.03)
    for nt in nts:
        f = torch.as_tensor(rng.normal(size=(nt, 5, len(area))) * 1e-3, dtype=s.dtype, device=dev)
        gp = torch.as_tensor(rng.normal(size=(n_obs, nt)), device=dev)
        g = s.backward(f, gp).double().cpu().numpy().reshape(nt, -1)
        s.check()
        ref = orc.backward(f.double().cpu().numpy(), obs, gp.cpu().numpy()).reshape(nt, -1)
        err = np.linalg.norm(g - ref, axis=1).max() / np.linalg.norm(ref, axis=1).max()
        assert err <= bar, (nt, err)
    s.close()
