"""Performance cases of the FGA library: what a user's program has it do, through the public binding.

Sizes come from this repository's own workloads, tests and benchmark (``workloads.py``, ``bench.py``):

* whole forward solves in the smooth gridded medium: a parity-test sized one (launches and host work), the smallest
  and an ordinary request of the serving mix, and the medium size of the benchmark with its snapshot;
* the homogeneous experiment in FP64 with point receivers;
* the layered crust, with flat and with undulating interfaces, where beams split;
* the point-force experiment: decomposition with beam selection, propagation, sum on the receiver patch;
* single steps a program calls by themselves: the wave-packet transform, and the Gaussian sum of a propagated
  beam set at scattered points and on a volume lattice;
* one source of the crosswell gradient: forward solve, L2 misfit and backward through ``adjoint``.

``exact`` restates the method in 64 bits with plain torch (transform, beam initialisation, RK4, Hermite records,
windowed sums); it shares nothing with the library.
"""
import math

import numpy as np
import torch

from paper_1810_06760_gb300 import adjoint, fga
from paper_1810_06760_gb300 import workloads as W

DEV = "cuda"
SQRT3 = math.sqrt(3.0)
C64, C128, F64 = torch.complex64, torch.complex128, torch.float64


def listed():
    return [
        # a solve of the parity tests' size: 13,500 beams, 40 steps; launches, allocations and host work show
        dict(name="solve_tiny", kind="solve", k=64.0, nq=5, np=3, ny=24, nsteps=40, dt=0.0025, n_times=30, rx0=7,
             rx1=7, snap=5, grid=33),
        # the smallest request of the serving mix (N = 1e5): 442 k beams, 200 steps, 256 receivers x 200 samples
        dict(name="solve_serving_small", kind="solve", k=32.0, nq=6, np=8, ny=48, nsteps=200, dt=0.0025, n_times=200,
             rx0=16, rx1=16, snap=0, grid=128),
        # an ordinary request of the serving mix: 2.7 M beams
        dict(name="solve_serving", kind="solve", k=64.0, nq=11, np=8, ny=64, nsteps=200, dt=0.0025, n_times=200,
             rx0=16, rx1=16, snap=0, grid=128),
        # the benchmark's medium size: 8.4 M beams, 400 receivers x 250 samples and a 64^3 snapshot
        dict(name="solve_snapshot", kind="solve", k=64.0, nq=16, np=8, ny=96, nsteps=100, dt=0.0025, n_times=250,
             rx0=20, rx1=20, snap=64, grid=128),
        # the homogeneous experiment at its stated size, FP64, 1,000 scattered receivers, the field at T
        dict(name="homogeneous_fp64", kind="homogeneous", k=32.0, nq=12, np=6, ny=96, nsteps=100, dt=0.005, n_times=1,
             n_rx=1000),
        # flat 3-layer crust: 442 k beams that split at the interfaces, 256 surface stations every 0.1 s
        dict(name="layered_flat", kind="layered", shape="planes", nq=6, np=8, ny=40, nsteps=300, dt=0.02, every=5,
             rx=16),
        # the same crust with undulating interfaces
        dict(name="layered_undulating", kind="layered", shape="undulating", nq=6, np=8, ny=40, nsteps=300, dt=0.02,
             every=5, rx=16),
        # point-force experiment: selection out of 4 x 22 M mesh points, 79 steps, a 41 x 1 x 17 patch
        dict(name="point_force", kind="point_force", k=0.15, nq=20, np=14, nsteps=79, rx0=41, rx2=17),
        # the wave-packet transform alone at the benchmark's shape
        dict(name="transform", kind="transform", k=64.0, nq=24, np=8, ny0=128, ny1=128, ny2=128),
        # Gaussian sum of a propagated set (1.05 M beams) at scattered points, an odd count
        dict(name="sum_points", kind="sum_points", k=64.0, nq=8, np=8, ny=64, nsteps=60, dt=0.0025, n=5003),
        # the same on a volume lattice with ragged tiles
        dict(name="sum_lattice", kind="sum_lattice", k=64.0, nq=8, np=8, ny=64, nsteps=60, dt=0.0025, n0=61, n1=64,
             n2=57),
        # one source of the crosswell inversion: seismograms, L2 misfit, gradient of the node fields
        dict(name="gradient", kind="gradient", k=64.0, nq=8, np=8, ny=64, nsteps=200, dt=0.0025, n_times=100, rx=16,
             grid=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "homogeneous", "layered", "point_force", "transform", "sum_points",
                       "sum_lattice", "gradient"])
    k = rng.choice([32.0, 64.0, 128.0])
    ny = 8 * int(math.ceil(math.sqrt(k)))
    if kind == "solve":
        nsteps = _log(rng, 40, 200)
        return dict(kind=kind, k=k, nq=_log(rng, 4, 11), np=rng.choice([4, 5, 6, 7, 8]), ny=ny + rng.randrange(8),
                    nsteps=nsteps, dt=0.0025, n_times=_log(rng, 20, 250), rx0=rng.randrange(5, 24),
                    rx1=rng.randrange(5, 24), snap=rng.choice([0, 0, 13, 30]), grid=rng.choice([33, 64, 128]))
    if kind == "homogeneous":
        return dict(kind=kind, k=rng.choice([16.0, 32.0]), nq=_log(rng, 4, 12), np=rng.randrange(3, 7),
                    ny=48 + rng.randrange(48), nsteps=_log(rng, 30, 100), dt=0.005, n_times=rng.choice([1, 2, 5]),
                    n_rx=_log(rng, 50, 1000))
    if kind == "layered":
        return dict(kind=kind, shape=rng.choice(["planes", "undulating", "spheres"]), nq=_log(rng, 3, 6),
                    np=rng.choice([4, 6, 8]), ny=rng.randrange(28, 48), nsteps=5 * _log(rng, 16, 60), dt=0.02,
                    every=rng.choice([1, 5, 10]), rx=rng.randrange(5, 17))
    if kind == "point_force":
        return dict(kind=kind, k=rng.choice([0.12, 0.15, 0.2]), nq=rng.randrange(9, 17),
                    np=rng.choice([8, 10, 12]), nsteps=_log(rng, 20, 79), rx0=rng.randrange(9, 42), rx2=rng.randrange(5, 18))
    if kind == "transform":
        n = [_log(rng, 24, 128) for _ in range(3)]
        return dict(kind=kind, k=k, nq=_log(rng, 5, 24), np=rng.randrange(3, 9), ny0=n[0], ny1=n[1], ny2=n[2])
    if kind == "sum_points":
        return dict(kind=kind, k=k, nq=_log(rng, 4, 8), np=rng.randrange(5, 9), ny=ny, nsteps=_log(rng, 10, 60),
                    dt=0.0025, n=_log(rng, 1, 6000))
    if kind == "sum_lattice":
        return dict(kind=kind, k=k, nq=_log(rng, 4, 8), np=rng.randrange(5, 9), ny=ny, nsteps=_log(rng, 10, 60),
                    dt=0.0025, n0=_log(rng, 5, 64), n1=_log(rng, 5, 64), n2=_log(rng, 3, 64))
    return dict(kind=kind, k=rng.choice([32.0, 64.0]), nq=_log(rng, 4, 8), np=rng.choice([4, 6, 8]), ny=ny,
                nsteps=_log(rng, 60, 200), dt=0.0025, n_times=_log(rng, 20, 100), rx=rng.randrange(6, 17),
                grid=rng.choice([33, 64]))


# ---------------------------------------------------------------------------------------------
# inputs, from the case and the seed alone
# ---------------------------------------------------------------------------------------------
def _t(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device=DEV)


def _mesh(nq, qc, rq, np_, pc, rp):
    """Cell-centred tensor mesh qc +- rq, pc +- rp (per axis)."""
    rq, rp = np.broadcast_to(rq, (3,)), np.broadcast_to(rp, (3,))
    dq, dp = 2.0 * rq / nq, 2.0 * rp / np_
    return dict(nq=nq, np=np_, q0=np.asarray(qc) - rq + 0.5 * dq, dq=dq, p0=np.asarray(pc) - rp + 0.5 * dp, dp=dp)


def _grid_axes(y0, dy, ny):
    return [_t(y0[a] + dy[a] * np.arange(ny[a])) for a in range(3)]


def _packet(k, x0, pol, d, ny, half):
    """pol exp(-k|y-x0|^2/2 + i k d.y) on a cell-centred grid over x0 +- half."""
    ny = np.broadcast_to(ny, (3,))
    dy = 2.0 * half / ny
    y0 = np.asarray(x0) - half + 0.5 * dy
    ax = _grid_axes(y0, dy, ny)
    e = [torch.exp(-0.5 * k * (a - x0[i]) ** 2 + 1j * k * d[i] * a) for i, a in enumerate(ax)]
    f = e[0][:, None, None] * e[1][None, :, None] * e[2][None, None, :]
    return (f[..., None] * _t(pol)).contiguous(), y0, dy


def _sine_fields(n, amp):
    """c_p = 2 + amp sin sin sin with gradient and Hessian on an n^3 FP32 node grid, and c_s = c_p/sqrt 3."""
    w = 2.0 * math.pi
    x = torch.linspace(0.0, 1.0, n, dtype=F64, device=DEV)
    s, c = torch.sin(w * x), torch.cos(w * x)
    S = [s[:, None, None], s[None, :, None], s[None, None, :]]
    Co = [c[:, None, None], c[None, :, None], c[None, None, :]]
    sss = S[0] * S[1] * S[2]
    out = torch.stack([2.0 + amp * sss, amp * w * Co[0] * S[1] * S[2], amp * w * S[0] * Co[1] * S[2],
                       amp * w * S[0] * S[1] * Co[2], -amp * w * w * sss, amp * w * w * Co[0] * Co[1] * S[2],
                       amp * w * w * Co[0] * S[1] * Co[2], -amp * w * w * sss, amp * w * w * S[0] * Co[1] * Co[2],
                       -amp * w * w * sss], -1)
    return out.float().contiguous(), (out.float().double() / SQRT3).float().contiguous()


def _explosion(y0, dy, ny, x0, ell, sigma):
    """grad[exp(-r^2/(2 sigma^2)) cos(2 pi r/ell)] on the y grid."""
    ax = _grid_axes(y0, dy, (ny,) * 3)
    Y = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1) - _t(x0)
    r = Y.pow(2).sum(-1).sqrt()
    rs = torch.where(r == 0, torch.ones_like(r), r)
    w = 2.0 * math.pi / ell
    d = torch.exp(-r * r / (2 * sigma ** 2)) * (-r / sigma ** 2 * torch.cos(w * r) - w * torch.sin(w * r))
    return ((d / rs)[..., None] * Y).to(C128).contiguous()


POINT = dict(x0=(64.0, 64.0, 64.0), force=(1.0, 1.0, 1.0), rho=1.0, cp=8.0, cs=4.619, f=1.4702, T0=0.1768, sigma=0.8660,
             t0=3.0, t1=6.93)


def _inputs(case, seed):
    rng = np.random.default_rng([int(seed), 71])
    kind = case["kind"]
    I = dict(case)
    k = I.get("k", 0.0)
    sk = math.sqrt(k) if k else 0.0
    if kind in ("solve", "sum_points", "sum_lattice", "gradient", "transform"):
        # a packet of random place, polarisation and direction; where there are receivers on x3 = 0 (x1 = 0.9 for
        # the crosswell) it travels towards them
        x0 = rng.uniform(0.3, 0.7, 3)
        if kind == "gradient":
            x0[0] = 0.1 + 0.02 * rng.uniform()
            to = np.array([0.9, rng.uniform(0.3, 0.7), rng.uniform(0.3, 0.7)])
        elif kind == "solve":
            x0[2] = rng.uniform(0.2, 0.45)
            to = np.array([rng.uniform(0.3, 0.7), rng.uniform(0.3, 0.7), 0.0])
        else:
            to = x0 + rng.normal(size=3)
        d = (to - x0) / np.linalg.norm(to - x0)
        b = rng.normal(size=3)
        b = b / np.linalg.norm(b) + d * rng.choice([-0.7, 0.7])   # both P and S excited
        b /= np.linalg.norm(b)
        ny = (I["ny0"], I["ny1"], I["ny2"]) if kind == "transform" else (I["ny"],) * 3
        I["f"], I["y0"], I["dy"] = _packet(k, x0, b, d, ny, 6.0 / sk)
        I["g"] = None
        I["mesh"] = _mesh(I["nq"], x0, 6.0 / sk, I["np"], d, 4.8 / sk)
        I["classes"] = (0, 1, 2, 3)
        I["rw"] = 6.0 / sk
        if kind != "transform":
            n = I.get("grid", 64)
            I["fields"] = _sine_fields(n, 0.2 * rng.uniform(0.8, 1.2))
            I["h"] = 1.0 / (n - 1)
        T = I.get("nsteps", 0) * I.get("dt", 0.0)
        if kind in ("solve", "gradient"):
            I["times"] = T * np.arange(1, I["n_times"] + 1) / I["n_times"]
        if kind == "solve":
            I["rx_axes"] = tuple((np.arange(n) + 0.5) / n for n in (I["rx0"], I["rx1"])) + (np.zeros(1),)
            s = (np.arange(I["snap"]) + 0.5) / max(I["snap"], 1)
            I["snap_axes"] = (s, s, s) if I["snap"] else None
        elif kind == "gradient":
            r = (np.arange(I["rx"]) + 0.5) / I["rx"]
            R1, R2 = np.meshgrid(r, r, indexing="ij")
            I["rx_pts"] = np.stack([np.full(R1.size, 0.9), R1.ravel(), R2.ravel()], -1)
            I["observed_seed"] = int(rng.integers(1 << 30))
        elif kind == "sum_points":
            I["points"] = rng.uniform(0.0, 1.0, (I["n"], 3))
        elif kind == "sum_lattice":
            I["axes"] = tuple((np.arange(n) + 0.5) / n for n in (I["n0"], I["n1"], I["n2"]))
    elif kind == "homogeneous":
        x0 = np.array([0.5, 0.5, 0.5]) + rng.uniform(-0.02, 0.02, 3)
        e1 = np.array([1.0, 0.0, 0.0])
        I["f"], I["y0"], I["dy"] = _packet(k, x0, e1, e1, (I["ny"],) * 3, 6.0 / sk)
        I["g"] = -1j * k * 2.0 * I["f"]
        I["mesh"] = _mesh(I["nq"], x0, 4.8 / sk, I["np"], e1, 4.8 / sk)
        I["classes"] = (0,)
        I["rw"] = 6.0 / sk
        I["rx_pts"] = rng.uniform(0.0, 1.0, (I["n_rx"], 3))
        I["times"] = I["nsteps"] * I["dt"] * np.arange(1, I["n_times"] + 1) / I["n_times"]
        I["const"] = (2.0, 1.0)
    elif kind == "layered":
        ell = 5.8 / 2.0
        sigma = 0.45 * ell
        k = I["k"] = 2.0 * math.pi / ell
        x0 = np.array([0.0, 0.0, 10.0]) + rng.uniform(-1.0, 1.0, 3)
        half = 3.2 * sigma
        I["dy"] = np.full(3, 2.0 * half / I["ny"])
        I["y0"] = x0 - half + 0.5 * I["dy"]
        I["f"], I["g"] = _explosion(I["y0"], I["dy"], I["ny"], x0, ell, sigma), None
        I["mesh"] = _mesh(I["nq"], x0, 2.2 * sigma, I["np"], (0.0, 0.0, 0.0), 1.5)
        I["classes"] = (0, 1, 2, 3)
        I["rw"] = 6.0 / math.sqrt(k)
        I["times"] = I["dt"] * np.arange(I["every"], I["nsteps"] + 1, I["every"])
        r = 6.0 * (np.arange(I["rx"]) - 0.5 * (I["rx"] - 1))   # stations 6 km apart
        I["rx_axes"] = (r, r, np.zeros(1))
        q = np.linspace(-15.0, 15.0, I["rx"])
        R1, R2 = np.meshgrid(q, q, indexing="ij")
        I["rx_pts"] = np.stack([R1.ravel(), R2.ravel(), (60.0 - np.sqrt(3600.0 - R1 ** 2 - R2 ** 2)).ravel()], -1)
    elif kind == "point_force":
        w = 1.0 / sk
        T = POINT["t1"] - POINT["t0"]
        m = 7.0 * w
        shift = rng.uniform(-0.5, 0.5, 3)
        r1 = np.linspace(24.0, 44.0, I["rx0"]) + shift[0]
        s3 = np.linspace(-4.0, 4.0, I["rx2"]) + shift[2]
        I["rx_axes"] = (64.0 + r1, np.array([64.0 + shift[1]]), 64.0 + s3)
        lo = np.array([64.0 + 24.0 - POINT["cp"] * T - m, 60.0 - m, 60.0 - m])
        hi = np.array([64.0 + 44.0 - POINT["cs"] * T + m, 68.0 + m, 68.0 + m])
        xi = (2.0 * math.pi * POINT["f"] + 2.0 * math.sqrt(math.log(1e3)) / POINT["sigma"]) / POINT["cs"]
        px, pl = (xi + 3.0 * math.sqrt(2.0 * k)) / k, (0.4 * xi + 3.0 * math.sqrt(2.0 * k)) / k
        # an even np keeps p = 0 off the mesh
        I["mesh"] = _mesh(I["nq"], 0.5 * (lo + hi), 0.5 * (hi - lo), I["np"], (0.0, 0.0, 0.0), np.array([px, pl, pl]))
        ylo, yhi = lo - 3.0 * w, hi + 3.0 * w
        I["nyv"] = np.ceil((yhi - ylo) / 0.8).astype(int)
        I["dy"] = (yhi - ylo) / I["nyv"]
        I["y0"] = ylo + 0.5 * I["dy"]
        I["classes"] = (0, 1, 2, 3)
        I["rw"] = 5.0 * w
        I["dt"] = T / 79
        I["const"] = (POINT["cp"], POINT["cs"])
        # radiated field of the force as data: a smooth shell of the pulse's width, P along and S across the radius
        ax = _grid_axes(I["y0"], I["dy"], I["nyv"])
        Y = torch.stack(torch.meshgrid(*ax, indexing="ij"), -1) - _t(POINT["x0"])
        r = Y.pow(2).sum(-1).sqrt().clamp_min(1e-3)
        n = Y / r[..., None]
        F = _t(POINT["force"]) * _t(rng.uniform(0.8, 1.2, 3))
        nF = (n * F).sum(-1, keepdim=True)

        def pulse(c):
            t = POINT["t0"] + POINT["T0"] - r / c
            w2 = 2.0 * math.pi * POINT["f"]
            env = torch.exp(-t * t / POINT["sigma"] ** 2) / r
            s = torch.cos(w2 * t) * env
            sd = (-w2 * torch.sin(w2 * t) - 2.0 * t / POINT["sigma"] ** 2 * torch.cos(w2 * t)) * env
            return s[..., None] / c ** 2, sd[..., None] / c ** 2

        (sp, vp), (ss, vs) = pulse(POINT["cp"]), pulse(POINT["cs"])
        I["f"] = (nF * n * sp + (F - nF * n) * ss).to(C128).contiguous()
        I["g"] = (nF * n * vp + (F - nF * n) * vs).to(C128).contiguous()
    return I


def _desc(I, precision, **kw):
    m = I["mesh"]
    return fga.init_desc(I["k"], I["f"], I["g"], I["y0"], I["dy"],
                         W.MeshSpec(m["nq"], m["q0"], m["dq"], m["np"], m["p0"], m["dp"]), I["classes"], precision, **kw)


def _grid_model(I):
    m = fga.Model("grid", grid_p=I["fields"][0], grid_s=I["fields"][1], origin=(0, 0, 0), spacing=(I["h"],) * 3)
    torch.cuda.synchronize()
    return m


def prepare(case, seed):
    I = _inputs(case, seed)
    kind = case["kind"]
    S = dict(kind=kind, I=I)
    if kind == "solve":
        S["model"], S["desc"] = _grid_model(I), _desc(I, fga.PREC_FP32)
    elif kind == "homogeneous":
        S["model"], S["desc"] = fga.Model("const", cp0=2.0, cs0=1.0), _desc(I, fga.PREC_FP64)
        S["rx"] = _t(I["rx_pts"])
    elif kind == "layered":
        kw = dict(layer_cp=(5.8, 6.5, 8.04), layer_cs=(3.46, 3.85, 4.47), layer_rho=(2.72, 2.92, 3.32),
                  layer_shape=case["shape"])
        if case["shape"] == "planes":
            kw["z_interfaces"] = (15.0, 35.0)
        elif case["shape"] == "undulating":
            kw.update(z_interfaces=(15.0, 35.0), layer_amp=(3.0, -2.0), layer_wavelength=(20.0, 30.0))
        else:
            kw.update(z_interfaces=(45.0, 25.0), layer_center=(0.0, 0.0, 60.0))
        S["model"] = fga.Model("layered", **kw)
        S["desc"] = fga.set_layered_options(_desc(I, fga.PREC_FP32, psi_rel_min=1e-6), growth=8.0)
        S["rx"] = _t(I["rx_pts"]) if case["shape"] == "spheres" else None
    elif kind == "point_force":
        S["model"] = fga.Model("const", cp0=POINT["cp"], cs0=POINT["cs"])
        S["desc"] = _desc(I, fga.PREC_FP32, psi_rel_min=1e-5)
    elif kind == "transform":
        S["desc"] = _desc(I, fga.PREC_FP32)
    elif kind in ("sum_points", "sum_lattice"):
        S["model"] = _grid_model(I)
        S["beams"] = fga.decompose(S["model"], _desc(I, fga.PREC_FP32))
        fga.propagate(S["model"], S["beams"], I["dt"], I["nsteps"])
        if kind == "sum_points":
            S["x"] = _t(I["points"])
    elif kind == "gradient":
        S["spec"] = adjoint.SourceSpec(_desc(I, fga.PREC_FP32), I["dt"], I["nsteps"], I["times"], _t(I["rx_pts"]), I["rw"],
                                       (0.0, 0.0, 0.0), (I["h"],) * 3, 20)
        S["fields"] = [f.clone().requires_grad_(True) for f in I["fields"]]
        # observed data: seismograms of the same size as the synthetic's
        rx, nt = case["rx"] ** 2, case["n_times"]
        gen = torch.Generator(DEV).manual_seed(I["observed_seed"])
        with torch.no_grad():
            u = adjoint.seismograms(I["fields"][0], I["fields"][1], S["spec"])
            noise = torch.randn((nt, rx, 3), dtype=C64, device=DEV, generator=gen)
            S["observed"] = 0.8 * u + 0.3 * u.abs().pow(2).mean().sqrt() * noise
    torch.cuda.synchronize()
    return S


def run(S):
    I, kind = S["I"], S["kind"]
    if kind == "solve":
        u, snap = fga.solve(S["model"], S["desc"], I["dt"], I["nsteps"], I["times"], rw=I["rw"], rx_axes=I["rx_axes"],
                            snap_axes=I["snap_axes"])
        return [u] if snap is None else [u, snap]
    if kind == "homogeneous":
        return fga.solve(S["model"], S["desc"], I["dt"], I["nsteps"], I["times"], S["rx"], rw=I["rw"])[0]
    if kind == "layered":
        axes = None if S["rx"] is not None else I["rx_axes"]
        return fga.solve(S["model"], S["desc"], I["dt"], I["nsteps"], I["times"], S["rx"], rw=I["rw"], rx_axes=axes)[0]
    if kind == "point_force":
        beams = fga.decompose(S["model"], S["desc"])
        fga.propagate(S["model"], beams, I["dt"], I["nsteps"])
        u = fga.reconstruct_lattice(beams, I["rx_axes"], rw=I["rw"])
        beams.close()
        return u
    if kind == "transform":
        return fga.transform(S["desc"])
    if kind == "sum_points":
        return fga.reconstruct(S["beams"], S["x"], rw=I["rw"])
    if kind == "sum_lattice":
        return fga.reconstruct_lattice(S["beams"], I["axes"], rw=I["rw"])
    for f in S["fields"]:
        f.grad = None
    u = adjoint.seismograms(S["fields"][0], S["fields"][1], S["spec"])
    adjoint.misfit(u, S["observed"]).backward()
    return [u.detach(), S["fields"][0].grad, S["fields"][1].grad]


# ---------------------------------------------------------------------------------------------
# work that a pass cannot do without
# ---------------------------------------------------------------------------------------------
STEP_FLOPS = 4300       # one RK4 step of one beam: four right-hand sides and the combination
CONST_STEP_FLOPS = 400  # the same where the speed is constant: straight ray, linear dzQ, amplitude from det Z


def work(case):
    kind = case["kind"]
    if kind == "transform":
        n, A = (case["ny0"], case["ny1"], case["ny2"]), case["nq"] * case["np"]
        flops = 8 * 3 * (n[0] * n[1] * n[2] * A + n[0] * n[1] * A * A + n[0] * A ** 3)
        return dict(bytes=48 * n[0] * n[1] * n[2] + 24 * A ** 3, flops=flops)
    if kind == "point_force":
        sk = math.sqrt(case["k"])
        half = np.array([20.0 + (POINT["cp"] - POINT["cs"]) * 3.93, 8.0, 8.0]) + 20.0 / sk
        ny = int(np.prod(np.ceil(half / 0.8)))
    else:
        ny = case["ny"] ** 3
    M = case["nq"] ** 3 * case["np"] ** 3 * (1 if kind == "homogeneous" else 4)
    steps = case["nsteps"]
    if kind in ("sum_points", "sum_lattice"):
        # the records' fields of every beam once, and the separable product of each beam with each point row
        pts = case["n"] if kind == "sum_points" else case["n0"] * case["n1"] * case["n2"]
        per = 26 if kind == "sum_points" else 24
        return dict(bytes=40 * M + 24 * pts, flops=0.5 * per * M * pts)
    per = STEP_FLOPS if kind in ("solve", "gradient") else CONST_STEP_FLOPS
    if kind == "solve":
        # beams near the receivers: a separable product per sample (columns x rows x 3 components)
        rx = case["rx0"] * case["rx1"]
        out = 24 * (rx * case["n_times"] + case["snap"] ** 3)
        sums = 0.3 * M * 24 * (rx * case["n_times"] + case["snap"] ** 3)
        grid = 80 * case["grid"] ** 3
    elif kind == "homogeneous":
        out, grid = 48 * case["n_rx"] * case["n_times"], 0
        sums = 0.3 * M * 43 * case["n_rx"] * case["n_times"]
    elif kind == "layered":
        nt = steps // case["every"]
        out, grid = 24 * case["rx"] ** 2 * nt, 0
        sums = 0.02 * M * 24 * case["rx"] ** 2 * nt
    elif kind == "point_force":
        M *= 0.3   # survivors of the selection, about
        out, grid = 24 * case["rx0"] * case["rx2"], 0
        sums = 0.1 * M * 24 * case["rx0"] * case["rx2"]
    else:
        # forward, forward again between checkpoints, and the reverse sweep (about twice a forward step)
        out = 24 * case["rx"] ** 2 * case["n_times"] + 80 * case["grid"] ** 3
        sums = 3 * 0.2 * M * 43 * case["rx"] ** 2 * case["n_times"]
        grid, per = 80 * case["grid"] ** 3, 4 * STEP_FLOPS
    return dict(bytes=48 * ny + grid + out, flops=M * steps * per + sums)


# ---------------------------------------------------------------------------------------------
# 64-bit values, plain torch
# ---------------------------------------------------------------------------------------------
def _exact_transform(I, f):
    """F(q,p) = sum_y f(y) exp(-i k p.(y-q) - k |y-q|^2/2) dy^3 on the pair mesh, [A, A, A, 3]."""
    m, k = I["mesh"], I["k"]
    for a in (2, 1, 0):
        q = _t(m["q0"][a] + m["dq"][a] * np.arange(m["nq"])).repeat_interleave(m["np"])
        p = _t(m["p0"][a] + m["dp"][a] * np.arange(m["np"])).repeat(m["nq"])
        y = _t(I["y0"][a] + I["dy"][a] * np.arange(f.shape[a]))
        d = y[None, :] - q[:, None]
        K = torch.exp(-1j * k * p[:, None] * d - 0.5 * k * d * d)
        f = torch.movedim(torch.tensordot(K, f, dims=([1], [a])), 0, a)
    return f * float(np.prod(I["dy"]))


def _exact_frame(P, e1):
    z = torch.zeros_like(P[:, 0])
    v = torch.where(e1[:, None], torch.stack([z, -P[:, 2], P[:, 1]], -1), torch.stack([-P[:, 1], P[:, 0], z], -1))
    vn = v.norm(dim=-1, keepdim=True)
    sh = v / vn
    return torch.linalg.cross(sh, P / P.norm(dim=-1, keepdim=True)), sh, vn[:, 0]


def _exact_speed(I, wave, Q):
    """c, grad c, Hess c at Q: constant, or trilinear in every field of the node grid (clamped outside)."""
    n = Q.shape[0]
    if "const" in I:
        return (torch.full((n,), I["const"][wave], dtype=F64, device=DEV), torch.zeros((n, 3), dtype=F64, device=DEV),
                None)
    G = I["fields"][wave]
    N = G.shape[0]
    t = (Q / I["h"]).clamp(0.0, N - 1.0)
    i = t.floor().long().clamp(max=N - 2)
    fr = t - i
    flat = G.reshape(-1, 10)
    out = torch.zeros((n, 10), dtype=F64, device=DEV)
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                w = ((fr[:, 0] if a else 1 - fr[:, 0]) * (fr[:, 1] if b else 1 - fr[:, 1]) *
                     (fr[:, 2] if c else 1 - fr[:, 2]))
                out += w[:, None] * flat[((i[:, 0] + a) * N + i[:, 1] + b) * N + i[:, 2] + c].double()
    H = out[:, [4, 5, 6, 5, 7, 8, 6, 8, 9]].reshape(n, 3, 3)
    return out[:, 0], out[:, 1:4], H


def _exact_rhs(I, wave, sg, e1, y):
    Q, P, DQ, DP, A = y
    c, g, H = _exact_speed(I, wave, Q)
    pn = P.norm(dim=-1)
    Ph = P / pn[:, None]
    dQ = sg * c[:, None] * Ph
    dP = -sg * pn[:, None] * g
    v = (DP * Ph[:, None, :]).sum(-1)
    u = (DQ * g[:, None, :]).sum(-1)
    cip = (c / pn)[:, None]
    dDQ = sg * (cip[..., None] * DP + (u - cip * v)[..., None] * Ph[:, None, :])
    dDP = torch.zeros_like(DP) if H is None else -sg * (pn[:, None, None] * (DQ @ H.to(C128)) + v[..., None] * g[:, None, :])
    Z, Zd = DQ + 1j * DP, dDQ + 1j * dDP
    Cf = torch.stack([torch.linalg.cross(Z[:, 1], Z[:, 2]), torch.linalg.cross(Z[:, 2], Z[:, 0]),
                      torch.linalg.cross(Z[:, 0], Z[:, 1])], 1)
    gam = sg * (g * Ph).sum(-1) + 0.5 * (Cf * Zd).sum((1, 2)) / (Z[:, 0] * Cf[:, 0]).sum(-1)
    dA = gam[:, None] * A
    if wave:
        sv, sh, vn = _exact_frame(P, e1)
        z = torch.zeros_like(dP[:, 0])
        w = torch.where(e1[:, None], torch.stack([z, -dP[:, 2], dP[:, 1]], -1), torch.stack([-dP[:, 1], dP[:, 0], z], -1))
        om = (w * sv).sum(-1) / vn
        dA = dA + torch.stack([-om * A[:, 1], om * A[:, 0]], -1)
    return dQ, dP, dDQ, dDP, dA


def _exact_beams(I, cls, F, G, eps):
    """Initial state of the beams of one class (mesh order), |psi|^2 of each."""
    m, k, wave = I["mesh"], I["k"], cls >= 2
    nq, np_ = m["nq"], m["np"]

    def pairs(T):   # [a0, a1, a2, 3] -> [mesh point, 3]
        return T.reshape(nq, np_, nq, np_, nq, np_, 3).permute(0, 2, 4, 1, 3, 5, 6).reshape(-1, 3)

    def nodes(lo, h, n):
        ax = [_t(lo[a] + h[a] * np.arange(n)) for a in range(3)]
        return torch.stack(torch.meshgrid(*ax, indexing="ij"), -1).reshape(-1, 3)

    Q = nodes(m["q0"], m["dq"], nq).repeat_interleave(np_ ** 3, 0)
    P = nodes(m["p0"], m["dp"], np_).repeat(nq ** 3, 1)
    pn = P.norm(dim=-1)
    e1 = (P[:, 0] ** 2 + P[:, 1] ** 2) < 0.01 * pn * pn
    n = (P / pn[:, None],) if not wave else _exact_frame(P, e1)[:2]
    Fp = pairs(F)
    sg = -1.0 if cls & 1 else 1.0
    A = []
    for d in n:
        a = (Fp * d).sum(-1)
        if G is not None:
            a = a + sg * 1j * (pairs(G) * d).sum(-1) / (k * _exact_speed(I, int(wave), Q)[0] * pn)
        A.append(math.sqrt(2.0) * a)
    A = torch.stack(A if wave else [A[0], torch.zeros_like(A[0])], -1)
    return Q, P, e1, A


def _axpy(y, h, k):
    return tuple(a + h * b for a, b in zip(y, k))


def _records(wave, e1, w, Q, P, A):
    if not wave:
        return Q, P, w * A[:, :1] * (P / P.norm(dim=-1, keepdim=True))
    sv, sh, _ = _exact_frame(P, e1)
    return Q, P, w * (A[:, :1] * sv + A[:, 1:] * sh)


def _sum_at_points(k, rw, x, rec):
    u = torch.zeros((x.shape[0], 3), dtype=C128, device=DEV)
    step = max(1, 40_000_000 // x.shape[0])
    for b in range(0, rec[0].shape[0], step):
        Q, P, A = (r[b:b + step] for r in rec)
        d = x[:, None, :] - Q[None]
        r2 = d.pow(2).sum(-1)
        ph = k * (d * P[None]).sum(-1)
        e = torch.where(r2 <= rw * rw, torch.exp(-0.5 * k * r2), torch.zeros_like(r2))
        u += torch.complex(e * torch.cos(ph), e * torch.sin(ph)) @ A
    return u


def _sum_on_lattice(k, axes, rec):
    ax = [_t(a) for a in axes]
    n = [a.numel() for a in ax]
    u = torch.zeros((n[0] * 3, n[1] * n[2]), dtype=C128, device=DEV)
    step = max(256, 30_000_000 // (3 * n[0] + n[1] * n[2]))
    for b in range(0, rec[0].shape[0], step):
        Q, P, A = (r[b:b + step] for r in rec)
        E = []
        for i in range(3):
            d = ax[i][None, :] - Q[:, i:i + 1]
            r, ph = torch.exp(-0.5 * k * d * d), k * P[:, i:i + 1] * d
            E.append(torch.complex(r * torch.cos(ph), r * torch.sin(ph)))
        X = (E[0][:, :, None] * A[:, None, :]).reshape(-1, 3 * n[0])
        Y = (E[1][:, :, None] * E[2][:, None, :]).reshape(-1, n[1] * n[2])
        u += X.T @ Y
    return u.reshape(n[0], 3, n[1], n[2]).permute(0, 2, 3, 1)


def exact(case, seed):
    kind = case["kind"]
    # the layered crust's interface events and the gradient's reverse sweep have no short 64-bit restatement
    if kind in ("layered", "gradient"):
        return None
    M = case["nq"] ** 3 * case["np"] ** 3 * (1 if kind == "homogeneous" else 4)
    if kind != "transform":
        lat = kind in ("solve", "point_force")
        pts = (case["rx0"] * case.get("rx1", case.get("rx2", 1)) if lat else case.get("n_rx", 0)) * case.get("n_times", 1)
        if lat:
            pts += case.get("snap", 0) ** 3
        if kind in ("sum_points", "sum_lattice"):
            pts = case["n"] if kind == "sum_points" else case["n0"] * case["n1"] * case["n2"]
        if M * case["nsteps"] > 2.0e8 or M * pts > 3.0e11:   # over about 20 seconds
            return None
    I = _inputs(case, seed)
    F = _exact_transform(I, I["f"])
    if kind == "transform":
        return F
    G = None if I["g"] is None else _exact_transform(I, I["g"])
    k, m = I["k"], I["mesh"]
    w = float(np.prod(m["dq"]) * np.prod(m["dp"])) / (2.0 * math.pi / k) ** 4.5
    dt, nsteps = I["dt"], I["nsteps"]
    times = I.get("times", np.zeros(0))
    beams = {c: _exact_beams(I, c, F, G, 0.0) for c in I["classes"]}
    keep = {c: None for c in beams}
    if kind == "point_force":
        mag = {c: b[3].abs().pow(2).sum(-1) for c, b in beams.items()}
        top = max(float(v.max()) for v in mag.values())
        keep = {c: v > 1e-10 * top for c, v in mag.items()}
    at = np.minimum(np.floor(times / dt).astype(int), nsteps - 1)
    seis = snap = None
    field = lambda rec: (_sum_on_lattice(k, I["rx_axes"], rec) if kind == "solve" else  # noqa: E731
                         _sum_at_points(k, I["rw"], _t(I["rx_pts"]), rec))
    for c, (Q, P, e1, A) in beams.items():
        if keep[c] is not None:
            Q, P, e1, A = (v[keep[c]] for v in (Q, P, e1, A))
        eye = torch.eye(3, dtype=C128, device=DEV).expand(Q.shape[0], 3, 3)
        y = (Q, P, eye.clone(), (-1j * eye).clone(), A)
        wave, sg = int(c >= 2), (-1.0 if c & 1 else 1.0)
        got = []
        j = 0
        k1 = _exact_rhs(I, wave, sg, e1, y)
        for n in range(nsteps):
            k2 = _exact_rhs(I, wave, sg, e1, _axpy(y, 0.5 * dt, k1))
            k3 = _exact_rhs(I, wave, sg, e1, _axpy(y, 0.5 * dt, k2))
            k4 = _exact_rhs(I, wave, sg, e1, _axpy(y, dt, k3))
            y1 = tuple(a + dt / 6.0 * (b + 2.0 * d + 2.0 * e + f) for a, b, d, e, f in zip(y, k1, k2, k3, k4))
            kn = _exact_rhs(I, wave, sg, e1, y1) if n + 1 < nsteps or len(times) else None
            while j < len(times) and at[j] == n:
                t = times[j] / dt - n
                h = (2 * t ** 3 - 3 * t * t + 1, (t ** 3 - 2 * t * t + t) * dt, 3 * t * t - 2 * t ** 3, (t ** 3 - t * t) * dt)
                q, p = (h[0] * y[s] + h[1] * k1[s] + h[2] * y1[s] + h[3] * kn[s] for s in (0, 1))
                got.append(field(_records(wave, e1, w, q, p, (1 - t) * y[4] + t * y1[4])))
                j += 1
            y, k1 = y1, kn
        if got:
            got = torch.stack(got)
            seis = got if seis is None else seis + got
        rec = _records(wave, e1, w, y[0], y[1], y[4])
        end = None
        if kind == "sum_points":
            end = _sum_at_points(k, I["rw"], _t(I["points"]), rec)
        elif kind in ("sum_lattice", "point_force"):
            end = _sum_on_lattice(k, I["axes" if kind == "sum_lattice" else "rx_axes"], rec)
        elif I.get("snap_axes") is not None:
            end = _sum_on_lattice(k, I["snap_axes"], rec)
        if end is not None:
            snap = end if snap is None else snap + end
    if kind == "solve":
        return [seis] if snap is None else [seis, snap]
    return seis if kind == "homogeneous" else snap
