"""The work that is timed: calls of the public entry points over the sizes, options and
directions a user of this framework runs.

  forward  FWH.forward on device fields (mixed and fp64), or on pinned host fields
  step     fwh_apply and the gradient of a misfit (forward and adjoint)
  batch    batch_forward over uneven surfaces
  moving   moving_forward, the general moving-surface form (FP64)
  psd      welch_psd of far-field signals

listed() are the fixed cases, draw() gives more of the same ranges, prepare() makes what a
program holds before the call, run() is one pass, work() its unavoidable bytes and
operations, exact() the same result from plain torch in 64 bits.

The signals of a mixed handle are kept in the type of its fields, FP32, as the program that
chose the mixed form does (its FP64 output type serves the sums over panel sets).
"""
from __future__ import annotations

import math

import numpy as np
import torch

DEG = math.pi / 180.0
N_MODES = 32


def listed():
    return [
        # the small validation case of a convected monopole: launches and latency count
        {"name": "monopole-mixed", "kind": "forward", "precision": "mixed", "shape": "sphere",
         "n1": 32, "n2": 64, "nt": 256, "obs": 8, "mach": 0.3, "dt": 0.05},
        {"name": "monopole-fp64", "kind": "forward", "precision": "fp64", "shape": "sphere",
         "n1": 32, "n2": 64, "nt": 256, "obs": 8, "mach": 0.3, "dt": 0.05},
        # the directivity of a dipole, the workload bench.py reports, in both precisions
        {"name": "dipole-mixed", "kind": "forward", "precision": "mixed", "shape": "sphere",
         "n1": 128, "n2": 256, "nt": 2048, "obs": 72, "mach": 0.5, "dt": 0.01},
        {"name": "dipole-fp64", "kind": "forward", "precision": "fp64", "shape": "sphere",
         "n1": 128, "n2": 256, "nt": 2048, "obs": 72, "mach": 0.5, "dt": 0.01},
        # the airfoil-like surface with a long broadband record, the largest single surface
        {"name": "contour-mixed", "kind": "forward", "precision": "mixed", "shape": "contour",
         "n1": 1200, "n2": 64, "nt": 4096, "obs": 36, "mach": 0.17, "dt": 1.264e-3},
        # an unstructured surface (panels in no spatial order), odd sizes everywhere
        {"name": "ragged-mixed", "kind": "forward", "precision": "mixed", "shape": "scattered",
         "n1": 20011, "n2": 1, "nt": 1501, "obs": 37, "mach": 0.4, "dt": 0.013},
        # fields that a solver left in pinned host memory, signals back on the host
        {"name": "host-mixed", "kind": "host", "precision": "mixed", "shape": "sphere",
         "n1": 64, "n2": 256, "nt": 1024, "obs": 36, "mach": 0.5, "dt": 0.01},
        # one step of an inverse problem: signals, misfit and its gradient over the fields
        {"name": "step-mixed", "kind": "step", "precision": "mixed", "shape": "sphere",
         "n1": 64, "n2": 256, "nt": 1024, "obs": 36, "mach": 0.5, "dt": 0.01},
        {"name": "step-fp64", "kind": "step", "precision": "fp64", "shape": "sphere",
         "n1": 51, "n2": 101, "nt": 701, "obs": 19, "mach": 0.3, "dt": 0.02},
        # eight uneven surfaces in one call, many observers around each
        {"name": "surfaces-mixed", "kind": "batch", "precision": "mixed", "n": 8, "panels": 65536,
         "nt": 2048, "obs": 512, "mach": 0.5, "dt": 0.01},
        # a spinning permeable surface (rotor-like), observers at rest
        {"name": "spinning-fp64", "kind": "moving", "n1": 64, "n2": 128, "nt": 2048, "obs": 16,
         "dt": 0.025},
        # spectra of the dipole case's signals
        {"name": "spectra", "kind": "psd", "signals": 72, "nt": 2048, "nperseg": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _step(dt, spread, nt):
    """A time step with which a surface's arrivals (spread out over that time) leave an
    observer window of at least 0.4 nt steps."""
    return round(max(dt, spread / (0.6 * nt)), 6)


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward", "host", "step", "batch", "moving", "psd"])
    if kind == "psd":
        L = 1 << rng.randint(5, 12)
        return {"kind": kind, "signals": _log(rng, 1, 1024), "nt": _log(rng, 512, 8192),
                "nperseg": L}
    if kind == "moving":
        nt = _log(rng, 64, 2048)
        return {"kind": kind, "n1": _log(rng, 8, 64), "n2": _log(rng, 16, 128), "nt": nt,
                "obs": _log(rng, 1, 16), "dt": _step(0.025, 3.0, nt)}
    if kind == "batch":
        nt, mach = _log(rng, 256, 2048), round(rng.uniform(0.2, 0.5), 3)
        return {"kind": kind, "precision": "mixed", "n": rng.randint(2, 8),
                "panels": _log(rng, 4096, 65536), "nt": nt, "obs": _log(rng, 16, 512),
                "mach": mach, "dt": _step(0.01, mach * 5.5 / (1.0 - mach), nt)}
    precision = "mixed" if kind == "host" else rng.choice(["mixed", "mixed", "fp64"])
    shape = rng.choice(["sphere", "contour", "scattered"])
    cap = 1e10 if precision == "mixed" else 1e9
    top = {"forward": (76800, 4096, 128), "host": (32768, 2048, 72), "step": (16384, 1024, 72)}[kind]
    P, nt, O = _log(rng, 512, top[0]), _log(rng, 48, top[1]), _log(rng, 1, top[2])
    while float(P) * nt * O > cap:
        P = max(512, int(P * 0.7))
    if shape == "contour":
        n2 = rng.choice([8, 16, 64]) + rng.randint(0, 1)
        n1, mach = max(16, P // n2), 0.17
        dt = _step(1.264e-3, mach * 7.4 / (1.0 - mach), nt)
    else:
        n1 = max(8, int(math.sqrt(P / 2))) if shape == "sphere" else P
        n2 = max(8, P // n1) if shape == "sphere" else 1
        mach = round(rng.uniform(0.2, 0.6), 3)
        dt = _step(rng.uniform(0.01, 0.05), mach * 3.0 / (1.0 - mach), nt)
    return {"kind": kind, "precision": precision, "shape": shape, "n1": n1, "n2": n2, "nt": nt,
            "obs": O, "mach": mach, "dt": dt}


# ---- surfaces, observers and fields -----------------------------------------------------


def _sphere(n1, n2, radius=1.5, center=(0.0, 0.0, 0.0)):
    """Polar x azimuth patches: centroids, outward normals, exact patch areas."""
    th, ph = np.linspace(0.0, np.pi, n1 + 1), np.linspace(0.0, 2 * np.pi, n2 + 1)
    T, F = np.meshgrid(0.5 * (th[1:] + th[:-1]), 0.5 * (ph[1:] + ph[:-1]), indexing="ij")
    n = np.stack([np.sin(T) * np.cos(F), np.sin(T) * np.sin(F), np.cos(T)], -1).reshape(-1, 3)
    a = radius ** 2 * (np.cos(th[:-1]) - np.cos(th[1:]))[:, None] * np.diff(ph)[None, :]
    return radius * n + np.asarray(center), n, a.reshape(-1)


def _contour(n1, n2, span=1.0 / 9.0):
    """A closed curve around a chord and its wake (n1 segments), extruded over n2 strips."""
    t = np.linspace(0.0, 2 * np.pi, n1, endpoint=False)
    pts = np.stack([2.5 + 3.7 * np.cos(t), 1.15 * np.sin(t) * (1.0 - 0.15 * np.cos(t))], -1)
    nxt = np.roll(pts, -1, 0)
    d = nxt - pts
    length = np.linalg.norm(d, axis=1)
    z = (np.arange(n2) + 0.5) * span / n2 - 0.5 * span
    y, n = np.zeros((n1 * n2, 3)), np.zeros((n1 * n2, 3))
    mid = 0.5 * (pts + nxt)
    for c in range(2):
        y[:, c] = np.repeat(mid[:, c], n2)
    n[:, 0], n[:, 1] = np.repeat(d[:, 1] / length, n2), np.repeat(-d[:, 0] / length, n2)
    y[:, 2] = np.tile(z, n1)
    return y, n, np.repeat(length, n2) * span / n2


def _scattered(P, radius=1.5):
    """P panels of equal area on a sphere, in random order (an unstructured mesh)."""
    k = np.arange(P) + 0.5
    z = 1.0 - 2.0 * k / P
    r, phi = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    n = np.stack([r * np.cos(phi), r * np.sin(phi), z], -1)[np.random.RandomState(7).permutation(P)]
    return radius * n, n, np.full(P, 4 * np.pi * radius ** 2 / P)


def _surface(case):
    if case["shape"] == "sphere":
        return _sphere(case["n1"], case["n2"])
    if case["shape"] == "contour":
        return _contour(case["n1"], case["n2"])
    return _scattered(case["n1"])


def _circle(O, radius, center=(0.0, 0.0, 0.0)):
    """O observers on a circle in the x-y plane (the paper's directivity arcs)."""
    a = 2 * np.pi * np.arange(O) / O + 0.1
    return np.stack([radius * np.cos(a), radius * np.sin(a), np.zeros(O)], -1) + np.asarray(center)


def _ball(O, radius, center):
    k = np.arange(O) + 0.5
    z = 1.0 - 2.0 * k / O
    r, phi = np.sqrt(1.0 - z * z), np.pi * (3.0 - np.sqrt(5.0)) * k
    return radius * np.stack([r * np.cos(phi), r * np.sin(phi), z], -1) + np.asarray(center)


def _aoa(case):
    return (5.5 if case.get("shape") == "contour" else 10.0) * DEG


def _observers(case):
    return _circle(case["obs"], 10.0 if case["shape"] == "contour" else 100.0)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields(y, mach, dt, nt, seed, dtype):
    """Convected random modes with a -5/3 energy spectrum up to 0.4 Nyquist, rms 0.01:
    pulsations rho', u', v', w', p' as [nt][5][P] on the device."""
    dev, rng = _device(), np.random.RandomState(seed)
    f_hi = 0.2 / dt
    f = np.exp(np.linspace(math.log(max(f_hi / 300.0, 2.0 / (nt * dt))), math.log(f_hi), N_MODES))
    a = f ** (-5.0 / 6.0)
    a *= math.sqrt(2.0) * 0.01 / math.sqrt(float(np.sum(a * a)))
    w = rng.normal(size=(N_MODES, 3))
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    q = rng.normal(size=(N_MODES, 3))
    q *= math.sqrt(3.0) / np.linalg.norm(q, axis=1, keepdims=True)
    ph = rng.uniform(0.0, 2 * np.pi, (2, N_MODES))
    om = 2 * np.pi * f

    def to(v):
        return torch.as_tensor(v, dtype=torch.float64, device=dev)
    theta = to(om)[:, None] * (to(w) @ to(y).T)
    wt = to(dt * np.arange(nt))[:, None] * to(om)[None, :]
    basis = torch.cat([torch.cos(wt), torch.sin(wt)], 1).to(dtype)
    out = torch.empty((nt, 5, y.shape[0]), dtype=dtype, device=dev)
    for k in range(2):
        arg = to(ph[k])[:, None] - theta
        C, S = to(a)[:, None] * torch.cos(arg), -to(a)[:, None] * torch.sin(arg)
        for c in range(3) if k == 0 else (3,):
            s = to(q[:, c])[:, None] if k == 0 else 1.0
            out[:, 1 + c] = basis @ torch.cat([C * s, S * s], 0).to(dtype)
    out[:, 0] = out[:, 4] * (mach * mach)
    return out


def _batch_surfaces(case):
    """Uneven sphere surfaces: each about half the panels of the one before."""
    share = [0.5 ** min(i, 4) for i in range(case["n"])]
    out = []
    for i, s in enumerate(share):
        P = max(64, int(case["panels"] * s / sum(share)))
        n1 = max(4, int(math.sqrt(P / 2)))
        c = (4.0 * i, 0.0, 0.0)
        y, n, a = _sphere(n1, max(8, P // n1), 1.0 + 0.25 * i, c)
        out.append((y, n, a, _ball(case["obs"], 100.0, c)))
    return out


def _motion(case):
    """A unit sphere spinning at 0.3 c0: positions, normals, velocities [nt][P][3]."""
    dev = _device()
    y, n, a = _sphere(case["n1"], case["n2"], 1.0)
    y, n = (torch.as_tensor(v, dtype=torch.float64, device=dev) for v in (y, n))
    tau = case["dt"] * torch.arange(case["nt"], dtype=torch.float64, device=dev)
    c, s = torch.cos(0.3 * tau)[:, None], torch.sin(0.3 * tau)[:, None]

    def turn(v):
        return torch.stack([c * v[:, 0] - s * v[:, 1], s * v[:, 0] + c * v[:, 1],
                            v[:, 2].expand(case["nt"], -1)], -1).contiguous()
    yt = turn(y)
    vt = torch.stack([-0.3 * yt[..., 1], 0.3 * yt[..., 0], torch.zeros_like(yt[..., 0])], -1)
    return yt, turn(n), vt.contiguous(), a


def _signals(case, seed):
    """Far-field-like signals: tones over noise, with a mean; ragged valid lengths."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    ns, nt = case["signals"], case["nt"]
    p = torch.randn((ns, nt), dtype=torch.float64, device=_device(), generator=g)
    t = torch.arange(nt, dtype=torch.float64, device=p.device)
    p = 1e-3 * (p + 5.0 * torch.sin(0.13 * t)[None, :] + 0.4)
    nv = nt - (np.arange(ns) * 37 + seed) % max(1, nt // 16)
    return p, nv.astype(np.int64)


# ---- the calls ------------------------------------------------------------------------------


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def prepare(case, seed):
    kind = case["kind"]
    if kind == "psd":
        p, nv = _signals(case, seed)
        return {"case": case, "p": p, "nv": nv}
    if kind == "moving":
        y, n, v, a = _motion(case)
        f = _fields(y[0].cpu().numpy(), 0.3, case["dt"], case["nt"], seed, torch.float64)
        return {"case": case, "y": y, "n": n, "v": v, "a": a, "f": f,
                "x0": _circle(case["obs"], 12.0)}
    from paper_2312_16263_gb300 import FWH
    dt, mach, prec = case["dt"], case["mach"], case["precision"]
    if kind == "batch":
        surf = _batch_surfaces(case)
        s = [FWH(y, n, a, mach, _aoa(case), dt, prec, observers=x) for y, n, a, x in surf]
        f = [_fields(y, mach, dt, case["nt"], seed + i, _dtype(case))
             for i, (y, _, _, _) in enumerate(surf)]
        outs = [torch.empty((case["obs"], case["nt"]), dtype=torch.float64, device=_device())
                for _ in surf]
        return {"case": case, "s": s, "f": f, "outs": outs}
    y, n, a = _surface(case)
    st = {"case": case, "f": _fields(y, mach, dt, case["nt"], seed, _dtype(case)),
          "s": FWH(y, n, a, mach, _aoa(case), dt, prec, observers=_observers(case))}
    if kind == "host":
        st["f"] = st["f"].cpu().pin_memory()
        st["out"] = torch.empty((case["obs"], case["nt"]), dtype=torch.float64).pin_memory()
    if kind == "step":
        st["target"] = _target(case, seed)
        st["f"].requires_grad_(True)
    return st


def _target(case, seed):
    g = torch.Generator(device=_device()).manual_seed(seed + 1)
    return 1e-5 * torch.randn((case["obs"], case["nt"]), dtype=torch.float64, device=_device(),
                              generator=g)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "psd":
        from paper_2312_16263_gb300 import welch_psd
        return welch_psd(st["p"], 100.0, case["nperseg"], st["nv"])
    if kind == "moving":
        from paper_2312_16263_gb300 import moving_forward
        p, t_start, _ = moving_forward(st["y"], st["n"], st["v"], st["a"], 1.0, 1.0, case["dt"],
                                       st["f"], st["x0"])
        return p, t_start
    if kind == "batch":
        from paper_2312_16263_gb300 import batch_forward
        return [p.to(_dtype(case)) for p in batch_forward(st["s"], st["f"], st["outs"])]
    if kind == "step":
        from paper_2312_16263_gb300 import fwh_apply
        p = fwh_apply(st["s"], st["f"])
        g, = torch.autograd.grad(((p - st["target"]) ** 2).sum(), st["f"])
        return p.detach().to(g.dtype), g
    if kind == "host":
        return st["s"].forward(st["f"], st["out"]).to(_dtype(case))
    return st["s"].forward(st["f"]).to(_dtype(case))


def work(case):
    """Inputs read once, outputs written once; per (panel, sample, observer) a dot product
    with the eight coefficients and the four weights of a cubic spline, 12 multiply-adds."""
    kind = case["kind"]
    if kind == "psd":
        L, nt = case["nperseg"], case["nt"]
        seg = max(0, (nt - L) // (L // 2) + 1)
        return {"bytes": case["signals"] * 8.0 * (nt + L // 2 + 1),
                "flops": case["signals"] * seg * 2.5 * L * math.log2(L)}
    nt, O = case["nt"], case["obs"]
    if kind == "moving":
        P = case["n1"] * case["n2"]
        # root, bracket of pT + pL, two spline solves, the bin's root and spline: about 100
        return {"bytes": 8.0 * nt * (14 * P + O), "flops": 100.0 * P * nt * O}
    if kind == "batch":
        P = sum(len(a) for _, _, a, _ in _batch_surfaces(case))
        return {"bytes": 20.0 * P * nt + 8.0 * case["n"] * O * nt, "flops": 24.0 * P * nt * O}
    P = case["n1"] * case["n2"]
    size = 8 if case["precision"] == "fp64" else 4
    field, out = 5.0 * size * P * nt, 8.0 * O * nt
    if kind == "step":
        return {"bytes": 2 * (field + out), "flops": 48.0 * P * nt * O}
    return {"bytes": field + out, "flops": 24.0 * P * nt * O}


# ---- the same results in 64 bits, plain torch ---------------------------------------------


class _Solve(torch.autograd.Function):
    """tridiag(1, 4, 1) x = r along dim 0 on rows 1 .. n - 2, x = 0 at both ends (symmetric)."""

    @staticmethod
    def forward(ctx, r):
        n = r.shape[0]
        x, inv = torch.zeros_like(r), 0.25
        piv = [0.0] * n
        for i in range(1, n - 1):
            piv[i] = inv
            torch.mul(r[i] - x[i - 1], inv, out=x[i])
            inv = 1.0 / (4.0 - inv)
        for i in range(n - 3, 0, -1):
            x[i].sub_(x[i + 1], alpha=piv[i])
        return x

    @staticmethod
    def backward(ctx, g):
        return _Solve.forward(ctx, g)


def _moments(F, dt):
    r = torch.zeros_like(F)
    r[1:-1] = (F[2:] - 2.0 * F[1:-1] + F[:-2]) * (6.0 / (dt * dt))
    return _Solve.apply(r)


def _diff(F, dt):
    """Second-order source-time derivative: central, one-sided at the ends."""
    return torch.cat([(-3.0 * F[:1] + 4.0 * F[1:2] - F[2:3]), F[2:] - F[:-2],
                      (3.0 * F[-1:] - 4.0 * F[-2:-1] + F[-3:-2])], 0) * (0.5 / dt)


def _series(f, n, U, dt):
    """The integrand Q_n, L_i, their derivatives, and the spline moments of all eight:
    lists of [nt][P] in the order Q', Q, L'(3), L(3)."""
    f = f.to(torch.float64)
    un = f[:, 1] * n[:, 0] + f[:, 2] * n[:, 1] + f[:, 3] * n[:, 2]
    Un = n @ U
    r1 = 1.0 + f[:, 0]
    Q = f[:, 0] * Un + r1 * un
    L = [f[:, 4] * n[:, c] + r1 * f[:, 1 + c] * (Un + un) for c in range(3)]
    F = [_diff(Q, dt), Q] + [_diff(v, dt) for v in L] + L
    return F, [_moments(v, dt) for v in F]


def _geometry(y, a, x, mach, U):
    """Convected distance and the eight coefficients of one observer, per panel."""
    d = x - y
    ud = d @ U
    beta2 = 1.0 - mach * mach
    R = (torch.sqrt((mach * ud) ** 2 + beta2 * (d * d).sum(1)) - mach * ud) / beta2
    Rh = (d - mach * R[:, None] * U) / R[:, None]
    MR = -mach * (Rh @ U)
    D, S = 1.0 - MR, a / (4 * math.pi)
    m = MR - mach * mach
    c = [S / (R * D ** 2), S * m / (mach * R ** 2 * D ** 3)]
    c += [S * mach * Rh[:, i] / (R * D ** 2) for i in range(3)]
    c += [S * (Rh[:, i] * (1.0 + m / D) + mach * U[i]) / (R ** 2 * D ** 2) for i in range(3)]
    return R, c


def _signal(F, M, R, c, mach, dt, nt):
    """One observer's signal [nt]: the splines of all panels' source signals at tau = t_j - M0 R."""
    delta = mach * (R.max() - R) / dt
    i0 = torch.floor(delta)
    b = delta - i0
    a = 1.0 - b
    w = [a, b, (a ** 3 - a) * (dt * dt / 6.0), (b ** 3 - b) * (dt * dt / 6.0)]
    span = (nt - 1) * dt + mach * float(R.min()) - mach * float(R.max())
    nv = max(0, min(nt, math.floor(span / dt) + 1))
    if nv == 0:
        return F[0].new_zeros(nt)
    g, m = F[0] * c[0], M[0] * c[0]
    for q in range(1, 8):
        g = torch.addcmul(g, F[q], c[q])
        m = torch.addcmul(m, M[q], c[q])
    left, right = w[0] * g + w[2] * m, w[1] * g + w[3] * m
    k = torch.arange(nv, device=R.device)[:, None] + i0.to(torch.int64)[None, :]
    s = left.gather(0, k.clamp(0, nt - 1)) + right.gather(0, (k + 1).clamp(0, nt - 1))
    return torch.cat([s.sum(1), s.new_zeros(nt - nv)])


def _exact_surface(f, y, n, a, x, mach, aoa, dt):
    """[O][nt] signals of one surface and a function giving the gradient over f."""
    nt, dev = f.shape[0], f.device
    y, n, a, x = (torch.as_tensor(v, dtype=torch.float64, device=dev) for v in (y, n, a, x))
    U = torch.tensor([math.cos(aoa), math.sin(aoa), 0.0], dtype=torch.float64, device=dev)
    with torch.no_grad():
        F, M = _series(f, n, U, dt)
        out = torch.stack([_signal(F, M, *_geometry(y, a, xo, mach, U), mach, dt, nt) for xo in x])

    def gradient(gp):
        leaf = [v.detach().requires_grad_(True) for v in F + M]
        for o, xo in enumerate(x):
            s = _signal(leaf[:8], leaf[8:], *_geometry(y, a, xo, mach, U), mach, dt, nt)
            s.backward(gp[o])
        f64 = f.detach().to(torch.float64).requires_grad_(True)
        Fs, Ms = _series(f64, n, U, dt)
        g, = torch.autograd.grad(Fs + Ms, f64, [v.grad for v in leaf])
        return g
    return out, gradient


def _exact_moving(case, seed):
    dt, nt, O = case["dt"], case["nt"], case["obs"]
    y, n, v, a = _motion(case)
    f = _fields(y[0].cpu().numpy(), 0.3, dt, nt, seed, torch.float64)
    dev = y.device
    a = torch.as_tensor(a, dtype=torch.float64, device=dev)
    x0 = torch.as_tensor(_circle(O, 12.0), dtype=torch.float64, device=dev)
    rho, u, p = 1.0 + f[:, 0], f[:, 1:4].transpose(1, 2), f[:, 4]
    Q = ((v + rho[..., None] * (u - v)) * n).sum(-1)
    L = p[..., None] * n + (rho * ((u - v) * n).sum(-1))[..., None] * u
    Qd, Ld, vd = _diff(Q, dt), _diff(L, dt), _diff(v, dt)
    tau = dt * torch.arange(nt, dtype=torch.float64, device=dev)[:, None]
    out, start = torch.zeros((O, nt), dtype=torch.float64, device=dev), []
    for o in range(O):  # observers at rest, c0 = rho0 = 1
        d = x0[o] - y
        r = torch.linalg.vector_norm(d, dim=-1)
        rh = d / r[..., None]
        Mr, D = (v * rh).sum(-1), 1.0 - (v * rh).sum(-1)
        K = r * (vd * rh).sum(-1) + Mr - (v * v).sum(-1)
        Lr = (L * rh).sum(-1)
        g = Qd / (r * D ** 2) + Q * K / (r ** 2 * D ** 3) + (Ld * rh).sum(-1) / (r * D ** 2) \
            + (Lr - (L * v).sum(-1)) / (r ** 2 * D ** 2) + Lr * K / (r ** 2 * D ** 3)
        g, t = g * (a / (4 * math.pi)), tau + r
        mg, mt = _moments(g, dt), _moments(t, dt)
        ts, te = float(t[0].max()), float(t[-1].min())
        start.append(ts)
        nv = max(0, min(nt, math.floor((te - ts) / dt) + 1))
        tj = ts + dt * torch.arange(nv, dtype=torch.float64, device=dev)[:, None]
        k = torch.searchsorted(t.T.contiguous(), tj.expand(-1, t.shape[1]).T.contiguous()).T
        k = (k - 1).clamp(0, nt - 2)
        t0, t1, m0, m1 = t.gather(0, k), t.gather(0, k + 1), mt.gather(0, k), mt.gather(0, k + 1)
        h = dt * dt / 6.0
        B = ((tj - t0) / (t1 - t0)).clamp(0.0, 1.0)
        for _ in range(6):
            A = 1.0 - B
            e = A * t0 + B * t1 + ((A ** 3 - A) * m0 + (B ** 3 - B) * m1) * h - tj
            de = t1 - t0 + ((1.0 - 3.0 * A * A) * m0 + (3.0 * B * B - 1.0) * m1) * h
            B = (B - e / de).clamp(0.0, 1.0)
        A = 1.0 - B
        s = A * g.gather(0, k) + B * g.gather(0, k + 1) + (
            (A ** 3 - A) * mg.gather(0, k) + (B ** 3 - B) * mg.gather(0, k + 1)) * h
        out[o, :nv] = s.sum(1)
    return out, np.asarray(start)


def exact(case, seed):
    kind = case["kind"]
    if kind == "moving":
        return _exact_moving(case, seed)
    if kind == "psd":
        p, nv = _signals(case, seed)
        L = case["nperseg"]
        w = 0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(L, dtype=torch.float64) / L).to(p.device)
        out = p.new_full((case["signals"], L // 2 + 1), math.nan)
        for i, N in enumerate(nv):
            if N >= L:
                seg = p[i, :N].unfold(0, L, L // 2)
                X = torch.fft.rfft((seg - seg.mean(1, keepdim=True)) * w)
                out[i] = (X.real ** 2 + X.imag ** 2).mean(0) / (100.0 * (w * w).sum())
        out[:, 1:L // 2] *= 2.0
        return out
    mach, dt = case["mach"], case["dt"]
    if kind == "batch":
        return [_exact_surface(_fields(y, mach, dt, case["nt"], seed + i, _dtype(case)), y, n, a, x,
                               mach, _aoa(case), dt)[0]
                for i, (y, n, a, x) in enumerate(_batch_surfaces(case))]
    y, n, a = _surface(case)
    f = _fields(y, mach, dt, case["nt"], seed, _dtype(case))
    p, gradient = _exact_surface(f, y, n, a, _observers(case), mach, _aoa(case), dt)
    if kind == "step":
        return p, gradient(2.0 * (p - _target(case, seed)))
    return p
