"""Rounding of fwh_forward_moving against long double (needs a GPU).

A coarsely sampled sphere spinning at a tip Mach number of 0.3, observers twelve radii
away: what is left of the error is the rounding of the delays, half a unit of the last
place of 12 (9e-16) in steps of 0.078, 1.1e-14 of an interval in the root tau*, times
the slope of signals of up to 0.2 of the sampling rate (0.6 a step): 7e-15 relative,
and a tenth more is allowed for.  Splines of the whole delays left 1.1e-14."""
import numpy as np
import pytest
import torch

from fwh_inputs.geometry import observers_circle

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from __graft_entry__ import build
    build()
    return torch.device("cuda:0")


def _case(mach, dt, nt, P):
    rng = np.random.default_rng(23)
    k = np.arange(P) + 0.5
    z = 1.0 - 2.0 * k / P
    r, ph = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    n0 = np.stack([r * np.cos(ph), r * np.sin(ph), z], 1)
    tau = np.arange(nt) * dt
    c, s = np.cos(mach * tau)[:, None], np.sin(mach * tau)[:, None]
    y = np.stack([c * n0[:, 0] - s * n0[:, 1], s * n0[:, 0] + c * n0[:, 1],
                  np.broadcast_to(n0[:, 2], (nt, P))], -1)
    v = np.stack([-mach * y[..., 1], mach * y[..., 0], np.zeros((nt, P))], -1)
    f = np.zeros((nt, 5, P))
    for w in np.exp(rng.uniform(np.log(2.0 / (nt * dt)), np.log(0.2 / dt), 8)):
        d, q, p0 = rng.normal(size=3), rng.normal(size=4), rng.uniform(0, 2 * np.pi)
        arg = 2 * np.pi * w * (tau[:, None] - n0 @ d / np.linalg.norm(d)) + p0
        f[:, 1:4] += 0.005 * np.cos(arg)[:, None] * q[:3, None]
        f[:, 4] += 0.0005 * np.sin(arg) * q[3]
    f[:, 0] = f[:, 4]
    return y, v, f


def _diff(F, dt):
    return np.concatenate([-3 * F[:1] + 4 * F[1:2] - F[2:3], F[2:] - F[:-2],
                           3 * F[-1:] - 4 * F[-2:-1] + F[-3:-2]]) / (2 * LD(dt))


def _moments(F, h):
    m, inv = np.zeros_like(F), [LD(0)] * F.shape[0]
    for i in range(1, F.shape[0] - 1):
        inv[i] = 1 / (4 - inv[i - 1])
        m[i] = (6 * (F[i + 1] - 2 * F[i] + F[i - 1]) / (h * h) - m[i - 1]) * inv[i]
    for i in range(F.shape[0] - 2, 0, -1):
        m[i] -= m[i + 1] * inv[i]
    return m


def _long_double(y, v, f, x0, dt, ts, bins):
    """One observer's signal of unit panels of area 4 pi on a unit sphere, c0 = rho0 = 1."""
    y, v, f = (a.astype(LD) for a in (y, v, f))
    h, u, rho, pp = LD(dt), np.moveaxis(f[:, 1:4], 1, 2), 1 + f[:, 0], f[:, 4]
    un, vn = (u * y).sum(-1), (v * y).sum(-1)
    Q, L = vn + rho * (un - vn), pp[..., None] * y + (rho * (un - vn))[..., None] * u
    b = x0.astype(LD) - y
    r = np.sqrt((b * b).sum(-1))
    rh = b / r[..., None]
    Mr, Lr = (v * rh).sum(-1), (L * rh).sum(-1)
    D, K = 1 - Mr, r * (_diff(v, dt) * rh).sum(-1) + Mr - (v * v).sum(-1)
    g = (_diff(Q, dt) + (_diff(L, dt) * rh).sum(-1)) / (r * D ** 2) + (Lr - (L * v).sum(-1)) / (
        r ** 2 * D ** 2) + (Q + Lr) * K / (r ** 2 * D ** 3)
    t = np.arange(len(y))[:, None] * h + r
    mg, mt, ar = _moments(g, h), _moments(t, h), np.arange(y.shape[1])
    out = np.empty(bins, LD)
    for j in range(bins):
        tj = LD(ts) + j * h
        k = np.clip((t <= tj).sum(0) - 1, 0, len(y) - 2)
        t0, t1, m0, m1 = t[k, ar], t[k + 1, ar], mt[k, ar], mt[k + 1, ar]
        B = np.clip((tj - t0) / (t1 - t0), 0, 1)
        for _ in range(8):
            A = 1 - B
            e = A * t0 + B * t1 + ((A ** 3 - A) * m0 + (B ** 3 - B) * m1) * h * h / 6 - tj
            B = np.clip(B - e / (t1 - t0 + ((1 - 3 * A * A) * m0 + (3 * B * B - 1) * m1) * h * h / 6), 0, 1)
        A = 1 - B
        out[j] = (A * g[k, ar] + B * g[k + 1, ar]
                  + ((A ** 3 - A) * mg[k, ar] + (B ** 3 - B) * mg[k + 1, ar]) * h * h / 6).sum()
    return out


def test_rounding_of_coarse_steps(dev):
    from paper_2312_16263_gb300 import moving_forward
    dt, nt, P, O = 0.078, 64, 300, 6
    y, v, f = _case(0.3, dt, nt, P)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)
    obs = observers_circle(12.0, O)
    p, ts, nv = moving_forward(t(y), t(y), t(v), np.full(P, 4 * np.pi), 1.0, 1.0, dt, t(f), obs)
    p = p.cpu().numpy()
    err = ref2 = 0.0
    for o in range(O):
        m = int(nv[o]) - 1
        ref = _long_double(y, v, f, obs[o], dt, ts[o], m)
        err += float(((p[o, :m] - ref) ** 2).sum())
        ref2 += float((ref ** 2).sum())
    assert (err / ref2) ** 0.5 <= 7.7e-15, (err / ref2) ** 0.5
