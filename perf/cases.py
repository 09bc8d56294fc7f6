"""What a user of the channel library has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes what a program holds before
the call (a channel, batch or problem statement with seeded inputs), ``run`` is
one pass through the public entry points and returns its results, ``exact`` is
the same pass in plain FP64 torch or numpy, straight from the equations of
arXiv:1603.01955.

Three kinds of case:
* channel: ``steps`` time steps of one channel, then the observables (the
  convergence check of a run to steady state) and the populations read back
  into the caller's pinned host array;
* batch: a Knudsen sweep of many periodic channels, its scalars and states;
* adjoint: the checkpointed forward pass and the gradient of the flow sum.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1603_01955_gb300 import clb

# ------------------------------------------------------------------- cases


def _channel(name, nx, ny, storage, steps, drive="pressure", kn=0.1, value=2.0, kn_mode=0, sigma=1.0):
    return dict(name=name, kind="channel", nx=nx, ny=ny, storage=storage, steps=steps, drive=drive, kn=kn,
                value=value, kn_mode=kn_mode, sigma=sigma)


def listed():
    return [
        # the L/H = 100 throughput channel (6.55 M nodes) in the default FP32 storage: the largest
        # production run, advanced between two looks at the flow
        _channel("pressure_25601x256_fp32s", 25601, 256, "fp32s", 200, value=2.47),
        # the same channel where memory or time is short and a few per cent of error will do
        _channel("pressure_25601x256_fp16s", 25601, 256, "fp16s", 200, value=2.47),
        # the same channel as FP64 reference run that the other storages are judged against
        _channel("pressure_25601x256_fp64", 25601, 256, "fp64", 16, value=2.47),
        # a periodic channel of 1.6 M nodes with ragged sides, BF16 storage
        _channel("force_12803x127_bf16s", 12803, 127, "bf16s", 150, drive="body_force", value=1e-5),
        # a middle resolution of the L/H = 100 channel, as in a grid refinement study
        _channel("pressure_6401x64_fp32s", 6401, 64, "fp32s", 500),
        # the L/H = 100 channel of the steady-state study (16 rows), one chunk of 1000 steps
        # between two convergence checks
        _channel("pressure_1601x16_fp32s", 1601, 16, "fp32s", 1000),
        # the same chunk for the mass-flow curve: FP64, centreline Knudsen number, sigma = 0.93
        _channel("curve_801x8_fp64", 801, 8, "fp64", 1000, kn=0.2, value=1.8, kn_mode=1, sigma=0.93),
        # the same chunk for the periodic channel compared with the slip-Poiseuille profile
        _channel("periodic_4x32_fp64", 4, 32, "fp64", 1000, drive="body_force", value=1e-6),
        # a transient watched closely: few steps between looks, launches and latency count
        _channel("transient_2101x33_fp16s", 2101, 33, "fp16s", 5, drive="body_force", kn=0.3, value=1e-6),
        # the Knudsen-minimum sweep: 48 periodic channels of 16 to 128 rows
        dict(name="knudsen_48_fp32s", kind="batch", n=48, nx=4, ny_lo=16, ny_hi=128, kn_lo=0.01, kn_hi=10.0,
             storage="fp32s", steps=5000),
        # one gradient of the calibration of r_b and a to a mass-flow curve
        dict(name="calibration_4x64_fp32s", kind="adjoint", nx=4, ny=64, kn=0.1, storage="fp32s", steps=20000,
             every=141),
        # a gradient on a grid too large for one block's shared memory
        dict(name="gradient_100x50_fp32s", kind="adjoint", nx=100, ny=50, kn=0.3, storage="fp32s", steps=500,
             every=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("channel", "batch", "adjoint"), (8, 2, 2))[0]
    if kind == "batch":
        ny_lo = round(_log(rng, 6, 30))
        return dict(kind=kind, n=rng.randint(8, 96), nx=rng.randint(1, 5), ny_lo=ny_lo,
                    ny_hi=round(_log(rng, ny_lo + 8, 160)), kn_lo=0.01 * rng.uniform(1, 3), kn_hi=rng.uniform(1, 10),
                    storage=rng.choice(("fp32s", "fp32s", "fp64")), steps=round(_log(rng, 300, 3000)))
    if kind == "adjoint":
        big = rng.random() < 0.3
        nodes = _log(rng, 3000, 20000) if big else _log(rng, 8, 600)
        ny = min(round(_log(rng, 4, 128)), round(nodes))
        return dict(kind=kind, nx=max(1, round(nodes / ny)), ny=ny, kn=_log(rng, 0.05, 1.0),
                    storage=rng.choice(("fp32s", "fp32s", "fp64")),
                    steps=round(_log(rng, 100, 600) if big else _log(rng, 300, 4000)), every=rng.choice((0, 0, 37, 100)))
    storage = rng.choice(("fp32s", "fp32s", "fp64", "fp16s", "bf16s"))
    # BF16's few bits leave nothing of the pressure's deviation from its linear course
    drive = "body_force" if storage == "bf16s" else rng.choice(("pressure", "pressure", "body_force"))
    ny = round(_log(rng, 5, 320))
    # pressure channels are long (in a short one these ratios would drive the gas at the speed of sound);
    # periodic ones have any length; up to the nodes of the largest listed one
    nx = round(ny * rng.uniform(60, 110)) if drive == "pressure" or rng.random() < 0.5 else round(_log(rng, 4, 4000))
    if nx * ny > 6_500_000:
        ny = ny * 6_500_000 // (nx * ny)
        nx = min(nx, 6_500_000 // ny)
    # a pass of a third of a millisecond to 15 ms: a step costs about 3 us, or its nodes
    us = max(12.0 if storage == "fp64" else 3.0, nx * ny * {"fp64": 2.2e-4, "fp32s": 1.1e-5}.get(storage, 7e-6))
    steps = max(1, round(_log(rng, 300, 15000) / us))
    if storage in ("fp16s", "bf16s"):
        steps = min(steps, 150)  # later a channel at rest is all rounding
    centre = drive == "pressure" and rng.random() < 0.2
    return dict(kind=kind, nx=nx, ny=ny, storage=storage, steps=steps, drive=drive, kn=_log(rng, 0.05, 1.0),
                value=rng.uniform(1.3, 2.5) if drive == "pressure" else _log(rng, 1e-6, 1e-5),
                kn_mode=1 if centre else 0, sigma=rng.uniform(0.8, 1.0))


# ------------------------------------------------------------------- inputs

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _initial(nx, ny, rho_in, rho_out, seed):
    """A flow in mid-development: the end densities joined linearly, with a few long waves of density
    and velocity and a little noise from the seed, as equilibrium populations [9][ny][nx] in FP64."""
    dev = _device()
    host = np.random.default_rng(seed)
    g = torch.Generator(dev).manual_seed(int(host.integers(1 << 62)))
    x = torch.linspace(0, 1, nx, dtype=torch.float64, device=dev)[None, :]
    y = ((torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) / ny)[:, None]

    def waves(amp):
        f = torch.zeros(ny, nx, dtype=torch.float64, device=dev)
        for _ in range(3):
            kx, ky = host.integers(0, 4, 2)
            px, py, a = host.uniform(0, 2 * math.pi, 3)
            f += amp * math.sin(a) * torch.sin(2 * math.pi * float(kx) * x + px) * torch.sin(2 * math.pi * float(ky) * y + py)
        return f

    rho = (rho_in + (rho_out - rho_in) * x) * (1 + waves(0.01))
    ux = waves(0.01) + 0.01 * y * (1 - y)
    uy = waves(0.002)
    f = torch.empty(9, ny, nx, dtype=torch.float64, device=dev)
    u2 = 1.5 * (ux * ux + uy * uy)
    for i in range(9):
        eu = EX[i] * ux + EY[i] * uy
        f[i] = W[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - u2)
        f[i] *= 1 + 0.001 * (2 * torch.rand(ny, nx, dtype=torch.float64, device=dev, generator=g) - 1)
    return f


def _ends(case):
    return (case["value"], 1.0) if case["drive"] == "pressure" else (1.0, 1.0)


def _rows(case):
    """Rows of each channel of a batch: ny_lo .. ny_hi, doubling and starting again."""
    ny, out = case["ny_lo"], []
    while len(out) < case["n"]:
        out.append(ny)
        ny = case["ny_lo"] if ny * 2 > case["ny_hi"] else ny * 2
    return out


def _knudsen(case):
    n = case["n"]
    return [case["kn_lo"] * (case["kn_hi"] / case["kn_lo"]) ** (k / max(1, n - 1)) for k in range(n)]


def _theta(seed):
    """The point (r_b, a, G) at which a calibration asks for a gradient."""
    host = np.random.default_rng(seed)
    return float(host.uniform(0.5, 0.9)), float(host.uniform(1.5, 2.5)), float(host.uniform(0.5e-6, 2e-6))


SCALARS = ("mass_flow", "q_norm", "u_slip", "total_mass", "ux_max")


def prepare(case, seed):
    if case["kind"] == "channel":
        nx, ny = case["nx"], case["ny"]
        ch = clb.Channel(nx, ny, case["kn"], drive=case["drive"], drive_value=case["value"],
                         storage=case["storage"], kn_mode=case["kn_mode"], sigma=case["sigma"])
        host = torch.empty((9, ny, nx), dtype=torch.float64, pin_memory=True)
        host.copy_(_initial(nx, ny, *_ends(case), seed))
        clb.clb_set_state(ch.sim, host.data_ptr())
        # the profile and the column sums of the flow; along a pressure channel its centreline too
        cols = dict(ux_prof=np.empty(ny), m_of_x=np.empty(nx))
        if case["drive"] == "pressure":
            cols.update(p_centre=np.empty(nx), dp_nonlin=np.empty(nx))
        return dict(case=case, ch=ch, host=host, cols=cols, scalars=clb.clb_scalars())
    if case["kind"] == "batch":
        ny, kn = _rows(case), _knudsen(case)
        b = clb.Batch([case["nx"]] * case["n"], ny, kn, g=1e-6, storage=case["storage"])
        for k in range(case["n"]):
            b.set_state(k, _initial(case["nx"], ny[k], 1.0, 1.0, [seed, k]).cpu().numpy())
        b.tune()
        return dict(case=case, b=b)
    return dict(case=case, theta=_theta(seed))


def run(state):
    case = state["case"]
    if case["kind"] == "channel":
        ch = state["ch"]
        c, s = state["cols"], state["scalars"]
        ch.step(case["steps"])
        clb.clb_observables(ch.sim, -1, s, c["ux_prof"], None, c.get("p_centre"), c.get("dp_nonlin"), c["m_of_x"])
        clb.clb_get_state(ch.sim, state["host"].data_ptr())
        return dict(c, f=state["host"], **{k: getattr(s, k) for k in SCALARS})
    if case["kind"] == "batch":
        b = state["b"]
        b.step(case["steps"])
        obs = b.observables()
        out = {k: np.array([o[k] for o in obs]) for k in ("mass_flow", "q_norm", "u_slip", "total_mass", "step")}
        out["f"] = np.concatenate([b.state(k).ravel() for k in range(case["n"])])
        return out
    r, a, g = state["theta"]
    fg = clb.FlowGradient(case["nx"], case["ny"], case["kn"], a, r, g, case["steps"], storage=case["storage"],
                          checkpoint_every=case["every"])
    out = dict(J=fg.J, q=fg.q_norm, grad=fg.grad())
    fg.close()
    return out


def work(case):
    """Bytes: the stored state once in and once out, and the results.  Flops: the collision of each node
    and step (about 156 operations, 200 with the body force); a gradient needs the states twice (the
    forward pass and the recomputation between checkpoints) and their reversal, at least twice one step."""
    elem = {"fp64": 8, "fp32s": 4, "fp16s": 2, "bf16s": 2}[case["storage"]]
    if case["kind"] == "channel":
        nodes = case["nx"] * case["ny"]
        per = 156 if case["drive"] == "pressure" else 200
        return dict(bytes=nodes * 9 * (2 * elem + 8), flops=nodes * case["steps"] * per)
    if case["kind"] == "batch":
        nodes = case["nx"] * sum(_rows(case))
        return dict(bytes=nodes * 9 * (2 * elem + 8), flops=nodes * case["steps"] * 200)
    nodes = case["nx"] * case["ny"]
    return dict(bytes=nodes * 9 * 2 * elem, flops=nodes * case["steps"] * 200 * 4)


# ------------------------------------------------------------------- exact values


def _rates(kn, ny, a=2.0, b2=0.55):
    """s_v of Eq. 18 and s_q of Eq. 21 at a local Knudsen number."""
    tau = math.sqrt(6 / math.pi) * ny * kn / (1 + a * kn)
    return 1 / (0.5 + tau), 1 / (0.5 + (3 + 4 * math.pi * tau * tau * b2) / (16 * tau))


def _r_of(sigma):
    return 1 / (1 + (1 - 0.1817 * sigma) * (2 - sigma) / sigma * math.sqrt(math.pi / 6))


def _collide(f, fx, sv, sq, s3=1.1, s8=1.2):
    """Eq. 4 with the cascade of Eq. 6-10 on nine populations (any number type with arithmetic)."""
    a57, a68, d57, d86 = f[5] + f[7], f[6] + f[8], f[5] - f[7], f[8] - f[6]
    kxx, kyy, kxy = f[1] + f[3] + a57 + a68, f[2] + f[4] + a57 + a68, a57 - a68
    kxxy, kxyy, kxxyy = d57 - d86, d57 + d86, a57 + a68
    rho = f[0] + f[1] + f[3] + f[2] + f[4] + kxxyy
    ux = (f[1] - f[3] + kxyy) / rho + 0.5 * fx
    uy = (f[2] - f[4] + kxxy) / rho
    ux2, uy2, uxy = ux * ux, uy * uy, ux * uy
    F = rho * fx
    g3 = s3 / 12 * (2 / 3 * rho + rho * (ux2 + uy2) - (kxx + kyy) - F * ux)
    g4 = sv / 4 * (rho * (ux2 - uy2) - (kxx - kyy) - F * ux)
    g5 = sv / 4 * (rho * uxy - kxy - 0.5 * F * uy)
    p, m = 0.5 * (3 * g3 + g4), 0.5 * (3 * g3 - g4)
    g6 = sq / 4 * (2 * rho * ux * uxy + kxxy - 2 * ux * kxy - uy * kxx - F * uxy) - uy * p - 2 * ux * g5
    g7 = sq / 4 * (2 * rho * uy * uxy + kxyy - 2 * uy * kxy - ux * kyy - 0.5 * F * uy2) - ux * m - 2 * uy * g5
    g8 = s8 / 4 * (rho / 9 + 3 * rho * uxy * uxy - (kxxyy - 2 * ux * kxyy - 2 * uy * kxxy + ux2 * kyy + uy2 * kxx
                                                    + 4 * uxy * kxy) - F * ux * uy2) \
        - 2 * g3 - uy2 * p - ux2 * m - 4 * uxy * g5 - 2 * uy * g6 - 2 * ux * g7
    # Eq. 9: the source's raw moments (x, xx+yy, xx-yy, xy, xxy, xyy, xxyy), through T^-1
    m1, m3, m5, m6, m7, m8 = F, 2 * F * ux, F * uy, 2 * F * uxy, F * uy2, 2 * F * ux * uy2
    c = m3 - 2 * m8
    return [f[0] - 4 * g3 + 4 * g8 - m3 + m8,
            f[1] - g3 + g4 + 2 * g7 - 2 * g8 + 0.25 * (c + m3 + 2 * (m1 - m7)),
            f[2] - g3 - g4 + 2 * g6 - 2 * g8 + 0.25 * (c - m3 - 2 * m6),
            f[3] - g3 + g4 - 2 * g7 - 2 * g8 + 0.25 * (c + m3 - 2 * (m1 - m7)),
            f[4] - g3 - g4 - 2 * g6 - 2 * g8 + 0.25 * (c - m3 + 2 * m6),
            f[5] + 2 * g3 + g5 - g6 - g7 + g8 + 0.25 * (m5 + m6 + m7 + m8),
            f[6] + 2 * g3 - g5 - g6 + g7 + g8 + 0.25 * (-m5 + m6 - m7 + m8),
            f[7] + 2 * g3 + g5 + g6 + g7 + g8 + 0.25 * (m5 - m6 - m7 + m8),
            f[8] + 2 * g3 - g5 + g6 - g7 + g8 + 0.25 * (-m5 - m6 + m7 + m8)]


def _equilibrium(rho, ux, uy):
    """Eq. 11 through the closed form of T^-1."""
    x2, y2 = ux * ux, uy * uy
    m3, m4, m5 = 2 / 3 * rho + rho * (x2 + y2), rho * (x2 - y2), rho * ux * uy
    m6, m7 = rho * uy * (1 / 3 + x2), rho * ux * (1 / 3 + y2)
    m8 = rho * (1 / 9 + (x2 + y2) / 3 + x2 * y2)
    c, jx, jy = m3 - 2 * m8, rho * ux, rho * uy
    return [rho - m3 + m8, 0.25 * (c + m4 + 2 * (jx - m7)), 0.25 * (c - m4 + 2 * (jy - m6)),
            0.25 * (c + m4 - 2 * (jx - m7)), 0.25 * (c - m4 - 2 * (jy - m6)), 0.25 * (m5 + m6 + m7 + m8),
            0.25 * (-m5 + m6 - m7 + m8), 0.25 * (m5 - m6 - m7 + m8), 0.25 * (-m5 - m6 + m7 + m8)]


class _Flow:
    """Channels side by side as flat nodes, their populations f [9][nodes]; a step is one gather (Eq. 5),
    the wall rows (Eq. 20), the pressure columns (Sec. 3.2) and the collision."""

    def __init__(self, shapes, r, pressure):
        self.shapes, self.r = shapes, r
        idx, wall, at = [[] for _ in range(9)], {"b": [], "t": []}, 0
        total = sum(nx * ny for nx, ny in shapes)
        for nx, ny in shapes:
            x, y = np.meshgrid(np.arange(nx), np.arange(ny))
            for i in range(9):
                sx = np.clip(x - EX[i], 0, nx - 1) if pressure else (x - EX[i]) % nx
                idx[i].append((i * total + at + np.clip(y - EY[i], 0, ny - 1) * nx + sx).ravel())
            c = np.arange(nx)
            left, right = (np.clip(c - 1, 0, None), np.clip(c + 1, None, nx - 1)) if pressure else ((c - 1) % nx, (c + 1) % nx)
            for key, row in (("b", 0), ("t", ny - 1)):
                wall[key].append(at + row * nx + np.stack([c, left, right]))
            at += nx * ny
        dev = _device()
        self.idx = torch.from_numpy(np.stack([np.concatenate(v) for v in idx])).to(dev)
        self.b, self.t = (torch.from_numpy(np.concatenate(wall[k], axis=1)).to(dev) for k in ("b", "t"))

    def pull(self, f):
        o = f.view(-1)[self.idx]
        r, q = self.r, 1 - self.r
        for (c, left, right), a, up in ((self.b, (2, 5, 6), (4, 7, 8)), (self.t, (4, 7, 8), (2, 5, 6))):
            o[a[0], c] = f[up[0], c]
            # the specular part comes from the column the population left
            sides = (left, right) if a[0] == 2 else (right, left)
            o[a[1], c] = r * f[up[1], c] + q * f[up[2], sides[0]]
            o[a[2], c] = r * f[up[2], c] + q * f[up[1], sides[1]]
        return o


def _obs_of(case, f):
    """Observables of the post-collision state f [9][ny][nx] (Sec. 3.1, 3.2)."""
    nx, ny = case["nx"], case["ny"]
    press = case["drive"] == "pressure"
    gx = 0.0 if press else case["value"]
    rho = f.sum(0)
    mx = f[1] - f[3] + f[5] - f[7] + f[8] - f[6] - 0.5 * gx * rho
    col = nx - 1 if press else 0
    ux = mx[:, col] / rho[:, col]
    pin, pout = (v / 3 for v in _ends(case))
    pc = 0.5 * (rho[(ny - 1) // 2] + rho[ny // 2]) / 3
    length = max(1, nx - 1)
    x = torch.arange(nx, dtype=torch.float64, device=f.device)
    m = float(mx.sum()) / nx
    if press:
        mu = math.sqrt(6 / math.pi) * case["kn"] * ny / 3
        q = m / (ny ** 3 * (pin * pin - pout * pout) / (8 * mu * length))
    else:
        q = float((mx / rho).sum()) / nx / (3 * gx * ny * ny * math.sqrt(1 / 6))
    slip = 0.5 * (1.5 * ux[0] - 0.5 * ux[1] + 1.5 * ux[-1] - 0.5 * ux[-2]) if ny > 1 else ux[0]
    out = dict(mass_flow=m, q_norm=q, u_slip=float(slip), total_mass=float(rho.sum()), ux_max=float(ux.max()),
               ux_prof=ux.cpu().numpy(), m_of_x=mx.sum(0).cpu().numpy())
    if press:
        out.update(p_centre=pc.cpu().numpy(),
                   dp_nonlin=((pc - (pin - (pin - pout) * x / length)) / pout).cpu().numpy())
    return out


def _exact_channel(case, seed):
    nx, ny, press = case["nx"], case["ny"], case["drive"] == "pressure"
    if case["steps"] * (1.2e-3 + nx * ny * 1.5e-9) > 15:
        return None
    f = _initial(nx, ny, *_ends(case), seed).reshape(9, -1)
    flow = _Flow([(nx, ny)], _r_of(case["sigma"]), press)
    sv, sq = _rates(case["kn"], ny)
    for _ in range(case["steps"]):
        o = flow.pull(f)
        if press:
            v = o.view(9, ny, nx)
            for edge, one, two, rho_b in ((0, 1, 2, case["value"]), (nx - 1, nx - 2, nx - 3, 1.0)):
                mac = []
                for c in (one, two):
                    n = v[:, :, c]
                    rho = n.sum(0)
                    mac.append((rho, (n[1] - n[3] + n[5] - n[7] + n[8] - n[6]) / rho,
                                (n[2] - n[4] + n[5] - n[7] + n[6] - n[8]) / rho))
                (r1, ux1, uy1), (_, ux2, uy2) = mac
                e1 = _equilibrium(r1, ux1, uy1)
                eb = _equilibrium(torch.full_like(r1, rho_b), 2 * ux1 - ux2, 2 * uy1 - uy2)
                v[:, :, edge] = torch.stack(eb) + (v[:, :, one] - torch.stack(e1))
            if case["kn_mode"]:  # the centreline density of the step before, for the whole column
                rows = f.view(9, ny, nx)[:, [(ny - 1) // 2, ny // 2]].sum(0)
                rho = (0.5 * (rows[0] + rows[1])).expand(ny, nx).reshape(-1)
            else:
                rho = o.sum(0)
            kn = case["kn"] / rho
            tau = math.sqrt(6 / math.pi) * ny * kn / (1 + 2 * kn)
            sv, sq = 1 / (0.5 + tau), 1 / (0.5 + (3 + 4 * math.pi * 0.55 * tau * tau) / (16 * tau))
        f = torch.stack(_collide(o, 0.0 if press else case["value"], sv, sq))
    f = f.view(9, ny, nx)
    return dict(_obs_of(case, f), f=f.cpu())


def _exact_batch(case, seed):
    if case["steps"] > 9000:
        return None
    ny, kn, nx, g = _rows(case), _knudsen(case), case["nx"], 1e-6
    f = torch.cat([_initial(nx, ny[k], 1.0, 1.0, [seed, k]).reshape(9, -1) for k in range(case["n"])], 1)
    flow = _Flow([(nx, n) for n in ny], _r_of(1.0), False)
    per = [np.repeat(v, [nx * n for n in ny]) for v in zip(*(_rates(k, n) for k, n in zip(kn, ny)))]
    sv, sq = (torch.from_numpy(v).to(f.device) for v in per)
    for _ in range(case["steps"]):
        f = torch.stack(_collide(flow.pull(f), g, sv, sq))
    out, at = {k: [] for k in ("mass_flow", "q_norm", "u_slip", "total_mass", "f")}, 0
    for n in ny:
        c = f[:, at:at + nx * n].reshape(9, n, nx)
        at += nx * n
        o = _obs_of(dict(drive="body_force", value=g, nx=nx, ny=n, kn=1.0), c)
        for k in out:
            out[k].append(c.cpu().numpy().ravel() if k == "f" else o[k])
    return {k: np.concatenate(v) if k == "f" else np.array(v) for k, v in out.items()} | dict(step=None)


def _exact_adjoint(case, seed):
    """Complex step (Im/h) in r_b, a and G of one column: a channel at rest and driven uniformly stays
    uniform along x.  Three perturbed runs side by side."""
    if case["steps"] * 2.5e-4 > 15:
        return None
    ny, h = case["ny"], 1e-30
    r, a, g = (v + 1j * h * np.eye(3)[k][:, None] for k, v in enumerate(_theta(seed)))
    sv, sq = _rates(case["kn"], ny, a)
    f = [np.full((3, ny), w, dtype=complex) for w in W]
    for _ in range(case["steps"]):
        o = list(f)
        for i in (2, 5, 6, 4, 7, 8):
            o[i] = np.empty_like(f[i])
        for i in (2, 5, 6):
            o[i][:, 1:] = f[i][:, :-1]
        for i in (4, 7, 8):
            o[i][:, :-1] = f[i][:, 1:]
        for (i, j, k), (p, q, s), y in (((2, 5, 6), (4, 7, 8), slice(0, 1)), ((4, 7, 8), (2, 5, 6), slice(ny - 1, ny))):
            o[i][:, y] = f[p][:, y]
            o[j][:, y] = r * f[q][:, y] + (1 - r) * f[s][:, y]
            o[k][:, y] = r * f[s][:, y] + (1 - r) * f[q][:, y]
        f = _collide(o, g, sv, sq)
    J = ((f[1] - f[3] + f[5] - f[7] + f[8] - f[6]) / sum(f) - 0.5 * g).sum(1)
    value = float(J[0].real)
    return dict(J=value, q=value / (3 * float(g[0, 0].real) * ny * ny * math.sqrt(1 / 6)),
                grad=[float(v) for v in J.imag / h])


def exact(case, seed):
    return {"channel": _exact_channel, "batch": _exact_batch, "adjoint": _exact_adjoint}[case["kind"]](case, seed)
