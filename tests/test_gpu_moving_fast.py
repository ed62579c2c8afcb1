"""Fast motion with coarse steps in fwh_forward_moving (needs a GPU).

A sphere spinning at a tip Mach number of 0.9 with 18 to 31 frames a revolution,
seen from two and five radii: the arrival times curve strongly within a source
interval, so the root tau* of each bin needs every step of Newton's method.
Against the FP64 oracle, which bisects, at rest and moving observers.  Bars,
relative L2 per observer, from a long-double model of the same sum: at 31 frames
three FP64 steps leave rounding (4e-14; ten times that is allowed for), at 18 they
leave 1e-11 (the usual 1e-10 is the bar); an FP32 quotient from the tangent
without a clamp left 1e-12 and 1e-9."""
import numpy as np
import pytest
import torch

from oracle.oracle import forward_moving as oracle_moving

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


def _spinning(mach, dt, nt, P):
    rng = np.random.default_rng(17)
    k = np.arange(P) + 0.5
    z = 1.0 - 2.0 * k / P
    r, ph = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    n0 = np.stack([r * np.cos(ph), r * np.sin(ph), z], 1)
    tau = np.arange(nt) * dt
    c, s = np.cos(mach * tau)[:, None], np.sin(mach * tau)[:, None]
    y = np.stack([c * n0[:, 0] - s * n0[:, 1], s * n0[:, 0] + c * n0[:, 1],
                  np.broadcast_to(n0[:, 2], (nt, P))], -1)
    v = np.cross(np.array([0.0, 0.0, mach]), y)
    # five smooth modes a component, up to a fifth of the sampling rate
    f = np.zeros((nt, 5, P))
    for comp in range(5):
        for w in 2 * np.pi * rng.uniform(0.5 / (nt * dt), 0.1 / dt, 5):
            d = rng.normal(size=3)
            f[:, comp] += 0.005 * np.cos(w * (tau[:, None] - n0 @ d / np.linalg.norm(d))
                                         + rng.uniform(0, 2 * np.pi))
    return y, y.copy(), v, np.full(P, 4 * np.pi / P), f


@pytest.mark.parametrize("w", [(0.0, 0.0, 0.0), (0.05, -0.02, 0.0)])
@pytest.mark.parametrize("step,bar", [(0.2, 4e-13), (0.35, 1e-10)])
def test_tip_mach_09_matches_oracle(dev, step, bar, w):
    from paper_2312_16263_gb300 import moving_forward
    mach, nt, P = 0.9, 90, 300
    dt = step / mach
    y, n, v, dS, f = _spinning(mach, dt, nt, P)
    obs = np.array([[3.0, 0.3, 0.0], [-1.0, 4.9, 0.5]])
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    p, ts, nv = moving_forward(t(y), t(n), t(v), dS, 1.0, 1.0, dt, t(f), obs, w)
    p = p.cpu().numpy()
    ref, _, nv_ref = oracle_moving(y, n, v, dS, 1.0, 1.0, dt, f, obs, np.array(w))
    for o in range(2):
        assert abs(int(nv[o]) - int(nv_ref[o])) <= 1
        m = int(min(nv[o], nv_ref[o]))
        assert m > 40
        err = np.linalg.norm(p[o, :m] - ref[o, :m]) / np.linalg.norm(ref[o, :m])
        assert err <= bar, (o, err)
