"""Work that programs using this framework have it do, as measurable cases.

Each case is a dict of plain values; prepare() builds what a program holds
before the call (a lattice handle with its bodies, a batch, trajectories, shell
start positions), run() makes one pass through the public entry points and
returns what the program reads back, and exact() gives the same values from a
plain torch FP64 evaluation of the model (D3Q19 lattice Boltzmann with MRT or
BGK relaxation, friction-coupled rigid raspberries, pore and channel walls).

FP32 lattices hand their results back as doubles; they are returned here in
FP32, the precision they are held in.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1604_01829_gb300 import lb
from paper_1604_01829_gb300 import workloads as W

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
WCA_BEADS = (5.0, 6.25, 0.5, 1e-3)       # pore-wall beads: spacing, radii, epsilon (grid of 1 nm)


# ------------------------------------------------------------------- the cases
def _lattice(name, n, **kw):
    c = dict(kind="lattice", nx=n[0], ny=n[1], nz=n[2], precision=32, collision="mrt", nu=W.NU_PAPER, kT=0.0,
             pore_R=0.0, pore_axis=2, wall_beads=False, channel=False, bodies=1, semi_a=3.0, semi_b=3.0, fixed=0,
             substeps=1, force=1e-4, body_force=0.0, compensate=0, gamma=20.0, flow=True, steps=100, io=False, probe=8192)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the validation run: one sphere pulled through a small periodic box in FP64
        _lattice("sphere_32_fp64", (32, 32, 32), precision=64, collision="bgk", nu=1 / 6, compensate=1, steps=200,
                 probe=0),
        # a host control loop: new forces in, one step, forces and torques out, again and again
        _lattice("control_64_fp32", (64, 64, 64), kT=1e-4, bodies=4, semi_a=6.0, semi_b=2.5, steps=20, io=True),
        # confinement as the paper runs it: pore, thermal noise, wall beads, two MD steps per LB step
        _lattice("pore_thermal_fp32", (48, 48, 96), kT=1e-4, pore_R=20.0, wall_beads=True, semi_a=4.0, semi_b=4.0,
                 substeps=2, force=0.0, steps=200),
        # pore drag protocol: pulled sphere, driven fluid, momentum and velocity sampled every 100 steps
        _lattice("pore_drag_fp64", (48, 48, 96), precision=64, collision="bgk", nu=1 / 6, pore_R=20.0, semi_a=4.0,
                 semi_b=4.0, fixed=2, force=1e-3, body_force=1e-6, steps=100),
        # thermal FP64 box of the paper's largest diffusion boxes, ragged sizes
        _lattice("thermal_fp64", (94, 81, 103), precision=64, kT=1e-4, semi_a=8.0, semi_b=3.0, steps=50),
        # resistance: raspberries held in a deterministic FP32 flow, odd edges
        _lattice("held_ragged_fp32", (150, 97, 203), bodies=3, semi_a=7.0, semi_b=3.0, fixed=1, steps=50),
        # the headline workload: 256^3, thermal, 64 prolate ellipsoids
        _lattice("ellipsoids_256_fp32", (256, 256, 256), kT=1e-4, bodies=64, semi_a=8.0, semi_b=3.0, force=0.0,
                 flow=False, steps=40, probe=65536),
        # many uneven boxes and pores at once (parameter scans)
        dict(name="batch_uneven_fp32", kind="batch", count=256, lo=24, hi=64, pores=True, kT=0.0, precision=32, steps=24),
        # diffusion statistics: replicas of a small thermal box, trajectories recorded
        dict(name="batch_brownian_fp32", kind="batch", count=64, lo=24, hi=24, pores=False, kT=1e-4, precision=32, steps=100),
        # drag gradient: forward and reverse sweep through a pulled ellipsoid's run
        dict(name="adjoint_96_fp32", kind="adjoint", n=96, precision=32, a=15.0, b=5.0, steps=200, window=50, schedule=0, snapshots=0),
        # raspberry construction: the shells of 64 ellipsoidal raspberries relaxed together
        dict(name="construction_64", kind="shells", raspberries=64, a_lo=4.0, a_hi=8.0, precision=32, steps=1000, density=1.0),
        # transport analysis of recorded trajectories
        dict(name="msd_64", kind="msd", bodies=64, records=4000, lags=400),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "pore", "pore", "channel", "fp32", "fp32", "thermal", "io", "batch", "adjoint", "shells", "msd"])
    if kind in ("fp64", "fp32", "thermal", "io"):
        p = 64 if kind == "fp64" or (kind == "thermal" and rng.random() < 0.3) else 32
        hi = 128 if p == 64 else (220 if kind != "io" else 96)
        n = tuple(_log(rng, 20, hi) for _ in range(3))
        mrt = kind in ("thermal", "io") or rng.random() < 0.5
        thermal = kind == "thermal" or (kind == "io" and rng.random() < 0.5)
        nodes = n[0] * n[1] * n[2]
        a = rng.uniform(2.0, 6.0)
        return _lattice(None, n, precision=p, collision="mrt" if mrt else "bgk", nu=W.NU_PAPER if mrt else 1 / 6,
                        kT=1e-4 if thermal else 0.0, bodies=min(8, 1 + nodes // 60000) if rng.random() < 0.7 else 1,
                        semi_a=a, semi_b=rng.uniform(0.45, 1.0) * a, compensate=int(rng.random() < 0.5), fixed=1 if kind == "fp32" else 0, steps=rng.randint(12, 40),
                        io=kind == "io", substeps=rng.choice([1, 1, 2, 3]), probe=4096)
    if kind == "pore":
        R = rng.randint(8, 28)
        ax = rng.randint(0, 2)
        across, along = 2 * R + rng.randint(2, 9), rng.randint(24, 110)
        n = [across, across + rng.randint(0, 3), across + rng.randint(0, 2)]
        n[ax] = along
        p = rng.choice([32, 64])
        thermal = rng.random() < 0.5
        a = rng.uniform(1.8, 0.3 * R)
        return _lattice(None, tuple(n), precision=p, collision="mrt" if thermal else "bgk", nu=W.NU_PAPER if thermal else 1 / 6,
                        kT=1e-4 if thermal else 0.0, pore_R=float(R), pore_axis=ax, wall_beads=rng.random() < 0.5, semi_a=a,
                        semi_b=a, substeps=rng.choice([1, 2]), force=1e-4, body_force=1e-6, steps=rng.randint(20, 100), probe=4096)
    if kind == "channel":
        n = tuple(_log(rng, 20, 90) for _ in range(3))
        return _lattice(None, n, precision=rng.choice([32, 64]), collision="bgk", nu=1 / 6, channel=True,
                        semi_a=rng.uniform(2.0, 6.0), semi_b=2.0, fixed=1, steps=rng.randint(20, 100), probe=4096)
    if kind == "batch":
        thermal = rng.random() < 0.5
        lo = rng.randint(16, 32)
        return dict(kind="batch", count=_log(rng, 4, 200), lo=lo, hi=lo + rng.randint(0, 28), pores=rng.random() < 0.5, kT=1e-4 if thermal else 0.0,
                    precision=rng.choice([32, 32, 64]), steps=rng.randint(12, 24))
    if kind == "adjoint":
        n = _log(rng, 32, 96)
        b = rng.uniform(2.0, n / 16)
        return dict(kind="adjoint", n=n, precision=rng.choice([32, 32, 64]) if n < 60 else 32, a=b * rng.uniform(1.0, 2.5), b=b,
                    steps=rng.randint(60, 200), window=rng.randint(10, 50), schedule=rng.randint(0, 1), snapshots=rng.choice([0, 8, 16]))
    if kind == "shells":
        a = rng.uniform(3.0, 9.0)
        return dict(kind="shells", raspberries=_log(rng, 1, 96), a_lo=a, a_hi=a * rng.uniform(1.0, 1.5), precision=32,
                    steps=_log(rng, 100, 1000), density=1.0)
    records = _log(rng, 500, 4000)
    return dict(kind="msd", bodies=_log(rng, 1, 64), records=records, lags=max(2, int(records * rng.uniform(0.02, 0.12))))


# ------------------------------------------------------------- inputs (shared)
@functools.lru_cache(maxsize=512)
def _beads(a, b):
    return W.sphere_raspberry(a) if a == b else W.ellipsoid_raspberry(a, b, b, seed=7)


def _params(c, seed, compensate=0, body_force=0.0, substeps=1, axis=2):
    g = [0.0, 0.0, 0.0]
    g[axis] = body_force
    p = dict(collision=1 if c["collision"] == "mrt" else 0, rho0=1.0, kT=c["kT"], gamma_bead=W.paper_gamma_to_lattice(c["gamma"]),
             seed=seed * 7919 + 11, precision=c["precision"], compensate_force=compensate, md_substeps=substeps, body_force=tuple(g))
    if c["collision"] == "mrt":
        p.update(W.mrt_rates(c["nu"]))
    else:
        p.update(tau=3.0 * c["nu"] + 0.5)
    return p


def _scene(c, seed):
    """Parameters, bodies, walls, forces and read-out nodes of a lattice case."""
    rng = np.random.default_rng([seed, c["nx"], c["ny"], c["nz"]])
    n = np.array([c["nx"], c["ny"], c["nz"]], float)
    a, b, ax = round(c["semi_a"], 2), round(c["semi_b"], 2), c["pore_axis"]
    pore = c["pore_R"] > 0.0
    s = dict(n=(c["nx"], c["ny"], c["nz"]), pore=(c["pore_R"], ax) if pore else None, wall_beads=WCA_BEADS if c["wall_beads"] else None,
             u_lo=None, u_hi=None, init=None,
             params=_params(c, seed, c["compensate"], c["body_force"], c["substeps"], ax if pore else 2), bodies=[])
    if c["channel"]:
        s["u_lo"], s["u_hi"] = (-0.01, 0.0, 0.004), (0.012, 0.0, -0.003)
    shape = [(a, b)] if pore or c["bodies"] == 1 else [(a, b), (round(0.9 * a, 2), round(0.8 * b, 2)), (round(0.8 * a, 2), b)]
    placed = []
    for k in range(c["bodies"]):
        sa, sb = shape[k % len(shape)]
        for _ in range(200):
            if pore or c["channel"]:
                X = n / 2 + rng.uniform(-1.5, 1.5, 3)
            else:
                X = rng.random(3) * n
            d = [np.abs(X - Y) for Y in placed]
            if all(np.linalg.norm(np.minimum(v, n - v)) > 2 * a + 1 for v in d):
                break
        placed.append(X)
        mass = 4.0 / 3.0 * math.pi * sa * sb * sb
        F = rng.standard_normal(3)
        T = rng.standard_normal(3)
        s["bodies"].append(dict(beads=_beads(sa, sb), X=X, q=W.random_unit_quaternion(rng), mass=mass,
                                inertia=W.solid_ellipsoid_inertia(mass, sa, sb, sb), fixed=c["fixed"],
                                F_ext=c["force"] * F / np.linalg.norm(F), T_ext=c["force"] * T / np.linalg.norm(T)))
    N = c["nx"] * c["ny"] * c["nz"]
    if c["flow"]:
        s["init"] = rng.uniform(0, 2 * math.pi, 12)
    if c["io"]:
        s["io"] = c["force"] * rng.standard_normal((c["steps"], 2, 3 * c["bodies"]))
    if c["probe"]:
        nodes = rng.choice(N, min(4 * c["probe"] if pore else c["probe"], N), replace=False, shuffle=False)
        if pore:
            nodes = nodes[~_is_wall(s, nodes)]
            nodes = np.resize(nodes, c["probe"])
        s["nodes"] = nodes
    return s


def _is_wall(s, nodes):
    nx, ny, nz = s["n"]
    xyz = [nodes % nx, nodes // nx % ny, nodes // (nx * ny)]
    R, ax = s["pore"]
    d2 = sum((xyz[k] + 0.5 - s["n"][k] / 2) ** 2 for k in range(3) if k != ax)
    return d2 >= R * R


_C = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0], [1, -1, 0],
               [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1], [0, 1, -1], [0, -1, 1]])
_OPP = np.array([0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)])
_WQ = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _flow(s):
    """Populations [19, N] of a developed flow: a drift and shear waves of a few percent of the lattice speed."""
    nx, ny, nz = s["n"]
    ph = s["init"]
    x, y, z = (2 * math.pi * (torch.arange(m, dtype=F64, device=DEV) + 0.5) / m for m in s["n"])
    u = torch.empty((3, nz, ny, nx), dtype=F64, device=DEV)
    u[0] = 0.004 + 0.01 * torch.sin(y + ph[0])[None, :, None] + 0.006 * torch.sin(2 * z + ph[1])[:, None, None]
    u[1] = -0.003 + 0.01 * torch.sin(z + ph[2])[:, None, None] + 0.006 * torch.sin(x + ph[3])[None, None, :]
    u[2] = 0.002 + 0.01 * torch.sin(x + ph[4])[None, None, :] + 0.006 * torch.sin(2 * y + ph[5])[None, :, None]
    u = u.reshape(3, -1)
    c = torch.tensor(_C, dtype=F64, device=DEV)
    cu = c @ u
    w = torch.tensor(_WQ, dtype=F64, device=DEV)[:, None]
    return w * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))


def _batch_scenes(c, seed):
    rng = np.random.default_rng([seed, c["count"], c["lo"]])
    sizes = np.random.default_rng(c["count"]).integers(c["lo"], c["hi"] + 1, c["count"])
    out = []
    for k, L in enumerate(int(v) for v in sizes):
        pore, n = None, (L, L, L)
        if c["pores"] and k % 2:
            R = max(8, (L - 4) // 2)
            n, pore = (2 * R + 4, 2 * R + 4, min(48, 2 * L)), (float(R), 2)
        a = round(float(rng.choice([2.0, 2.5, 3.0, 4.0])), 2)
        a = min(a, pore[0] - 4.0) if pore else min(a, L / 6)
        b = round(a / 1.5, 2) if k % 3 == 0 and not c["kT"] else a
        mass = 4.0 / 3.0 * math.pi * a * b * b
        cc = dict(collision="mrt", nu=W.NU_PAPER if not c["kT"] else 1 / 6, kT=c["kT"], gamma=20.0 if not c["kT"] else 90.0, precision=c["precision"])
        p = _params(cc, seed, 0 if pore or c["kT"] else 1)
        p["instance"] = k
        F = (0.0, 0.0, 0.0 if c["kT"] else 1e-3)
        body = dict(beads=_beads(a, b), X=np.array(n) / 2 + rng.uniform(-1, 1, 3), q=W.random_unit_quaternion(rng), mass=mass,
                    inertia=W.solid_ellipsoid_inertia(mass, a, b, b), F_ext=F, T_ext=(0.0, 0.0, 0.0), fixed=0)
        out.append(dict(n=n, pore=pore, wall_beads=None, u_lo=None, u_hi=None, init=None, params=p, bodies=[body]))
    return out


def _adjoint_scene(c, seed):
    rng = np.random.default_rng([seed, c["n"]])
    a, b = round(c["a"], 2), round(c["b"], 2)
    mass = 4.0 / 3.0 * math.pi * a * b * b
    p = _params(dict(collision="mrt", nu=W.NU_PAPER, kT=0.0, gamma=20.0, precision=c["precision"]), seed, 1)
    body = dict(beads=_beads(a, b), X=c["n"] / 2 + rng.uniform(-1, 1, 3), q=np.array([1.0, 0, 0, 0]), mass=mass,
                inertia=W.solid_ellipsoid_inertia(mass, a, b, b), F_ext=(1e-3, 0.0, 0.0), T_ext=(0.0, 0.0, 0.0), fixed=2)
    return dict(n=(c["n"],) * 3, pore=None, wall_beads=None, u_lo=None, u_hi=None, init=rng.uniform(0, 2 * math.pi, 12), params=p, bodies=[body])


@functools.lru_cache(maxsize=4096)
def _shell_start(a, b, n):
    return W.spread_shell_start(a, b, b, n, seed=3)


def _shells(c, seed):
    rng = np.random.default_rng([seed, c["raspberries"]])
    axes, xyz = [], []
    for r in range(c["raspberries"]):
        t = r % 16 / 15
        a = round(c["a_lo"] + t * (c["a_hi"] - c["a_lo"]), 1)
        b = round(max(2.0, a / (2 + r % 3)), 1)
        for (sa, sb, _), n in W.raspberry_shells(a, b, b, c["density"]):
            P = _shell_start(round(sa, 2), round(sb, 2), n)
            axes.append((round(sa, 2), round(sb, 2), round(sb, 2)))
            xyz.append(P * (1.0 + 0.02 * rng.uniform(-1, 1, (n, 1))))
    return np.array(axes), xyz


def _trajectories(c, seed):
    """Brownian centres and orientations of free bodies."""
    rng = np.random.default_rng([seed, c["bodies"], c["records"]])
    nb, nr = c["bodies"], c["records"]
    X = 30.0 + np.cumsum(0.05 * rng.standard_normal((nb, nr, 3)), axis=1)
    w = 0.03 * rng.standard_normal((nb, nr, 3))
    q = np.zeros((nb, nr, 4))
    cur = np.stack([W.random_unit_quaternion(rng) for _ in range(nb)])
    for k in range(nr):
        h = 0.5 * w[:, k]
        v0, v1 = cur[:, :1], cur[:, 1:]
        s0 = np.sqrt(1.0 - (h * h).sum(1, keepdims=True))
        cur = np.concatenate([v0 * s0 - (v1 * h).sum(1, keepdims=True), v0 * h + s0 * v1 + np.cross(v1, h)], axis=1)
        q[:, k] = cur
    q /= np.linalg.norm(q, axis=2, keepdims=True)
    return np.ascontiguousarray(X), q


# -------------------------------------------------------------- prepare and run
def _handle(s):
    h = lb.LB(*s["n"], **s["params"])
    if s["pore"]:
        h.lb_set_pore(*s["pore"])
    if s["u_lo"]:
        h.lb_set_channel_walls(s["u_lo"], s["u_hi"])
    if s["wall_beads"]:
        h.lb_set_pore_beads(*s["wall_beads"])
    for b in s["bodies"]:
        h.lb_add_raspberry(b["beads"], b["X"], b["q"], b["mass"], b["inertia"], b["F_ext"], b["T_ext"], b["fixed"])
    if s["init"] is not None:
        h.lb_set_populations(_flow(s).cpu().numpy())
    return h


def prepare(case, seed):
    k = case["kind"]
    if k == "lattice":
        s = _scene(case, seed)
        st = dict(case=case, h=_handle(s), nodes=s.get("nodes"))
        if case["io"]:
            st["io"] = s["io"]
        return st
    if k == "batch":
        scenes = _batch_scenes(case, seed)
        B = lb.LBBatch([dict(s["params"], nx=s["n"][0], ny=s["n"][1], nz=s["n"][2]) for s in scenes])
        for i, s in enumerate(scenes):
            if s["pore"]:
                B.lb_batch_set_pore(i, *s["pore"])
            for b in s["bodies"]:
                B.lb_batch_add_raspberry(i, b["beads"], b["X"], b["q"], b["mass"], b["inertia"], b["F_ext"], b["T_ext"], b["fixed"])
        B.lb_batch_record_bodies(max(1, case["steps"] // 4), 64)
        return dict(case=case, h=B)
    if k == "adjoint":
        return dict(case=case, h=_handle(_adjoint_scene(case, seed)))
    if k == "shells":
        axes, xyz = _shells(case, seed)
        return dict(case=case, axes=axes, xyz=xyz)
    X, q = _trajectories(case, seed)
    return dict(case=case, X=X, q=q)


def run(state):
    c, k = state["case"], state["case"]["kind"]
    if k == "lattice":
        h = state["h"]
        out = {}
        nb = c["bodies"]
        F, T = np.zeros(3 * nb), np.zeros(3 * nb)
        if c["io"]:
            series = np.zeros((c["steps"], 2, 3 * nb))
            for t in range(c["steps"]):
                h.lb_step_io(state["io"][t, 0], state["io"][t, 1], series[t, 0], series[t, 1])
            out["series"] = series
        else:
            h.lb_step(c["steps"])
            h.lb_forces_all(F, T)
            out["F"], out["T"] = F, T
        if nb <= 8:
            bodies = [h.lb_get_body(b) for b in range(nb)]
            for key in ("X", "V", "q", "w"):
                out[key] = np.stack([b[key] for b in bodies])
            out["beads"] = np.concatenate([h.lb_forces(b, per_bead=True)[2] for b in range(nb)])
        if c["body_force"]:
            mass, mom = h.lb_conservation()
            out["mass"], out["momentum"] = np.array([mass]), mom
        out["f"] = h.lb_get_populations() if state["nodes"] is None else h.lb_sample_populations(state["nodes"])
        return _held(out, c["precision"])
    if k == "batch":
        B = state["h"]
        B.lb_batch_step(c["steps"])
        got = [B.lb_batch_get_body(i) for i in range(B.n)]
        out = {key: np.stack([g[key] for g in got]) for key in ("X", "V", "q", "w")}
        out["F"] = np.stack([B.lb_batch_forces(i)[0] for i in range(B.n)])
        out["path"] = np.stack([B.lb_batch_get_trajectory(i)[1][-4:] for i in range(min(B.n, 64))])
        out["f"] = [B.lb_batch_get_populations(i) for i in (0, 2 * (B.n // 4))]
        return _held(out, c["precision"])
    if k == "adjoint":
        J, dg, ds, _ = state["h"].lb_adjoint_drag_ex(c["steps"], c["window"], 0, 0, c["schedule"], c["snapshots"])
        return _held(dict(J=np.array([J]), dJ_dgamma=np.array([dg]), dJ_dbeads=ds), c["precision"])
    if k == "shells":
        got = lb.lb_relax_shells(state["axes"], state["xyz"], c["steps"], precision=c["precision"])
        return _held(dict(beads=np.concatenate(got)), c["precision"])
    return dict(msd=lb.lb_msd_trajectory(state["X"], state["q"], c["lags"]))


def _held(out, precision):
    """Results in the precision the lattice holds them in."""
    if precision == 64:
        return out
    return {k: [x.astype(np.float32) for x in v] if isinstance(v, list) else v.astype(np.float32) for k, v in out.items()}


# ----------------------------------------------------------------------- work
def _fluid(n, pore):
    if not pore:
        return n[0] * n[1] * n[2]
    return int(math.pi * pore[0] ** 2) * n[pore[1]]


def work(case):
    k = case["kind"]
    if k == "lattice":
        pore = (case["pore_R"], case["pore_axis"]) if case["pore_R"] else None
        N = _fluid((case["nx"], case["ny"], case["nz"]), pore) * case["steps"]
        return dict(bytes=N * 38 * case["precision"] // 8, flops=N * 363)
    if k == "batch":
        L = 0.5 * (case["lo"] + case["hi"])
        N = case["count"] * L ** 3 * (0.85 if case["pores"] else 1.0) * case["steps"]
        return dict(bytes=N * 38 * case["precision"] // 8, flops=N * 363)
    if k == "adjoint":
        # a forward step, and a reversed one that reads the populations, the adjoint and the forces
        N = case["n"] ** 3 * case["steps"]
        return dict(bytes=N * (38 + 69) * case["precision"] // 8, flops=N * (363 + 800))
    if k == "shells":
        n = sum(m for r in range(case["raspberries"])
                for _, m in W.raspberry_shells(*(lambda a: (a, max(2.0, a / (2 + r % 3)), max(2.0, a / (2 + r % 3))))(
                    case["a_lo"] + r % 16 / 15 * (case["a_hi"] - case["a_lo"]))))
        # per bead and step: a few steps of a root search, the neighbours within the repulsion's range, the update
        return dict(bytes=n * 48, flops=n * case["steps"] * 400)
    n = case["bodies"] * case["records"]
    return dict(bytes=n * 56 + case["bodies"] * case["lags"] * 80, flops=n * case["lags"] * 60)


# ----------------------------------------------------------- plain FP64 model
def _basis():
    c = _C.astype(float)
    x, y, z = c.T
    c2 = (c * c).sum(1)
    E = np.stack([np.ones(19), x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x,
                  (3 * c2 - 5) * x, (3 * c2 - 5) * y, (3 * c2 - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                  3 * c2 * c2 - 6 * c2 + 1, (2 * c2 - 3) * (3 * x * x - c2), (2 * c2 - 3) * (y * y - z * z)])
    return E, (_WQ * E * E).sum(1)


def _philox(c, key):
    """Philox4x32-10 of four int64 counters (tensors or numbers below 2^32)."""
    M = (0xD2511F53, 0xCD9E8D57)

    def mul(a, m):
        return (((a >> 16) * m + (((a & 0xFFFF) * m) >> 16)) >> 16), (a * m) & 0xFFFFFFFF

    k0, k1 = key
    for _ in range(10):
        h0, l0 = mul(c[0], M[0])
        h1, l1 = mul(c[2], M[1])
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _rot(q):
    w, x, y, z = q
    return torch.stack([torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)]),
                        torch.stack([2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)]),
                        torch.stack([2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)])])


class _Model:
    """The coupled step in plain torch, FP64, pre-collision populations f[19, N]."""

    def __init__(self, s, dev=DEV):
        p = s["params"]
        self.s, self.p, self.dev = s, p, dev
        t = functools.partial(torch.tensor, dtype=F64, device=dev)
        nx, ny, nz = self.n = s["n"]
        self.N = nx * ny * nz
        E, b = _basis()
        self.E, self.b, self.w, self.c = t(E), t(b), t(_WQ), t(_C)
        self.back = self.w[:, None] * self.E.T / self.b
        if p["collision"] == 1:
            g = [0.0] * 4 + [p["gamma_bulk"]] + [p["gamma_shear"]] * 5 + [p["gamma_odd"]] * 6 + [p["gamma_even"]] * 3
        else:
            g = [0.0] * 4 + [1.0 - 1.0 / p["tau"]] * 15
        self.g = t(g)
        self.sig = (torch.sqrt(3.0 * p["kT"] * self.b * (1 - self.g ** 2)) * math.sqrt(12.0))[4:]
        idx = torch.arange(self.N, device=dev)
        self.xyz = torch.stack([idx % nx, idx // nx % ny, idx // (nx * ny)])
        self.wall = None
        if s["pore"]:
            self.wall = torch.from_numpy(_is_wall(s, np.arange(self.N))).to(dev)
        self.nfluid = self.N if self.wall is None else int((~self.wall).sum())
        self.f = _flow(s).to(dev) if s["init"] is not None else (self.w[:, None] * p["rho0"]).repeat(1, self.N)
        self.key = (p["seed"] & 0xFFFFFFFF, p["seed"] >> 32)
        self.inst, self.t = p.get("instance", 0), 0
        self.gamma = t(p["gamma_bead"])
        self.F = torch.zeros((3, self.N), dtype=F64, device=dev)
        self.bodies = []
        first = 0
        for B in s["bodies"]:
            self.bodies.append(dict(s=t(B["beads"]), X=t(B["X"]), V=t([0.0] * 3), q=t(B["q"]) / t(B["q"]).norm(), w=t([0.0] * 3), M=B["mass"],
                                    I=t(B["inertia"]), fixed=B["fixed"], Fe=t(B["F_ext"]), Te=t(B["T_ext"]), Fl=t([0.0] * 3), Tl=t([0.0] * 3),
                                    first=first, F=t([0.0] * 3), T=t([0.0] * 3), fb=torch.zeros((len(B["beads"]), 3), dtype=F64, device=dev)))
            first += len(B["beads"])
        self.set_force()

    def set_force(self):
        g = torch.tensor(self.p["body_force"], dtype=F64, device=self.dev)
        if self.p["compensate_force"]:
            for B in self.bodies:
                if B["fixed"] != 1:
                    g = g - B["Fe"] / self.nfluid
        self.gf = g

    # rigid bodies
    def drift(self, B, dt):
        if B["fixed"] != 1:
            B["V"] = B["V"] + 0.5 * dt * B["Fl"] / B["M"]
            B["X"] = B["X"] + dt * B["V"]
            if B["fixed"] == 0:
                w = B["w"]
                w = w + 0.5 * dt * (B["Tl"] - torch.linalg.cross(w, B["I"] * w)) / B["I"]
                B["w"] = w
                wn = w.norm()
                if wn > 0:
                    d0, d = torch.cos(0.5 * wn * dt), torch.sin(0.5 * wn * dt) / wn * w
                    q0, q = B["q"][0], B["q"][1:]
                    B["q"] = torch.cat([(q0 * d0 - (q * d).sum())[None], q0 * d + d0 * q + torch.linalg.cross(q, d)])
                B["q"] = B["q"] / B["q"].norm()
            else:
                B["w"] = torch.zeros_like(B["w"])
        B["R"] = _rot(B["q"])

    def kick(self, B, dt):
        B["F"], B["T"] = B["aF"] + B["Fe"], B["aT"] + B["Te"]
        Tb = B["R"].T @ B["T"]
        B["Fl"], B["Tl"] = B["F"], Tb
        if B["fixed"] == 1:
            return
        B["V"] = B["V"] + 0.5 * dt * B["F"] / B["M"]
        if B["fixed"] == 2:
            return
        w0 = w = B["w"]
        for _ in range(6):
            w = w0 + 0.5 * dt * (Tb - torch.linalg.cross(w, B["I"] * w)) / B["I"]
        B["w"] = w

    def wall_beads(self, B, rel):
        spacing, rp, rr, eps = self.s["wall_beads"]
        R, ax = self.s["pore"]
        a1, a2 = [k for k in range(3) if k != ax]
        Rc, L = R + rp, self.n[ax]
        nt, nr = max(3, round(2 * math.pi * Rc / spacing)), max(1, round(L / spacing))
        j, k = torch.meshgrid(torch.arange(nt, dtype=F64, device=self.dev), torch.arange(nr, dtype=F64, device=self.dev), indexing="ij")
        P = torch.empty((nt * nr, 3), dtype=F64, device=self.dev)
        P[:, a1] = (self.n[a1] / 2 + Rc * torch.cos(2 * math.pi * j / nt)).reshape(-1)
        P[:, a2] = (self.n[a2] / 2 + Rc * torch.sin(2 * math.pi * j / nt)).reshape(-1)
        P[:, ax] = ((k + 0.5) * L / nr).reshape(-1)
        d = (B["X"] + rel)[:, None] - P[None]
        d[..., ax] -= L * torch.floor(d[..., ax] / L + 0.5)
        d2 = (d * d).sum(-1)
        s6 = ((rp + rr) ** 2 / d2) ** 3
        m = torch.where(d2 < 2 ** (1 / 3) * (rp + rr) ** 2, 24 * eps * (2 * s6 * s6 - s6) / d2, 0.0)
        return (m[..., None] * d).sum(1)

    def couple(self, F, sub, dt):
        p = self.p
        for B in self.bodies:
            rel = B["s"] @ B["R"].T
            wl = B["R"] @ B["w"]
            v = B["V"] + torch.linalg.cross(wl.expand_as(rel), rel)
            tq = B["X"] + rel - 0.5
            fl = torch.floor(tq.detach())
            fr = tq - fl
            o = torch.tensor([[c & 1, c >> 1 & 1, c >> 2] for c in range(8)], device=self.dev)
            raw = fl.long()[:, None] + o[None]
            wt = torch.where(o[None] == 1, fr[:, None], 1 - fr[:, None]).prod(-1)
            n3 = torch.tensor(self.n, device=self.dev)
            pos = raw % n3
            idx = (pos[..., 0] + self.n[0] * (pos[..., 1] + self.n[1] * pos[..., 2])).reshape(-1)
            fluid = torch.ones(idx.shape, dtype=torch.bool, device=self.dev) if self.wall is None else ~self.wall[idx]
            fn = self.f[:, idx]
            u = ((self.c.T @ fn) + 0.5 * (self.gf[:, None] + self.F[:, idx])) / fn.sum(0)
            if self.s["u_lo"]:
                y = raw[..., 1].reshape(-1)
                for out, uw in ((y < 0, self.s["u_lo"]), (y >= self.n[1], self.s["u_hi"])):
                    u = torch.where(out, torch.tensor(uw, dtype=F64, device=self.dev)[:, None], u)
                    fluid = fluid & ~out
            else:
                u = torch.where(fluid, u, 0.0)
            ub = (wt[..., None] * u.T.reshape(-1, 8, 3)).sum(1)
            Fb = -self.gamma * (v - ub)
            if p["kT"] > 0:
                nb = len(rel)
                k = torch.arange(nb, device=self.dev) + B["first"]
                z = torch.zeros_like(k)
                r = _philox((k, z + self.t, z + self.inst, z + 4 + sub), self.key)
                xi = torch.stack(r[:3], 1).to(F64)
                Fb = Fb + torch.sqrt(2.0 * p["kT"] * self.gamma / dt) * math.sqrt(12.0) * ((xi + 0.5) / 2.0 ** 32 - 0.5)
            B["fb"] = Fb
            share = torch.where(fluid[:, None], (-dt * wt[..., None] * Fb[:, None]).reshape(-1, 3), 0.0)
            F = F.index_add(1, idx, share.T)
            B["aF"], B["aT"] = Fb.sum(0), torch.linalg.cross(rel, Fb).sum(0)
            if self.s["wall_beads"]:
                Fw = self.wall_beads(B, rel)
                B["aF"], B["aT"] = B["aF"] + Fw.sum(0), B["aT"] + torch.linalg.cross(rel, Fw).sum(0)
        return F

    def collide(self, f, F):
        m = self.E @ f
        rho = m[0]
        Ft = F + self.gf[:, None]
        u = (m[1:4] + 0.5 * Ft) / rho
        x, y, z = u
        X, Y, Z = Ft
        eq = torch.stack([rho * (x * x + y * y + z * z), rho * (2 * x * x - y * y - z * z), rho * (y * y - z * z), rho * x * y, rho * y * z, rho * z * x])
        S = torch.stack([2 * (x * X + y * Y + z * Z), 2 * (2 * x * X - y * Y - z * Z), 2 * (y * Y - z * Z), x * Y + y * X, y * Z + z * Y, z * X + x * Z])
        g = self.g[4:, None]
        r = g * m[4:]
        r = torch.cat([r[:6] + (1 - g[:6]) * eq + 0.5 * (1 + g[:6]) * S, r[6:]])
        if self.p["kT"] > 0:
            k = torch.arange(self.N, device=self.dev)
            z64 = torch.zeros((), dtype=torch.int64, device=self.dev)
            for call in (0, 1):
                q = _philox((k, z64 + self.t, z64 + self.inst, z64 + call), self.key)
                for h in range(8):
                    mode = 8 * call + h
                    if mode < 15:
                        v = (q[h // 2] >> 16) if h % 2 == 0 else (q[h // 2] & 0xFFFF)
                        r[mode] += torch.sqrt(rho) * self.sig[mode] * ((v.to(F64) + 0.5) / 65536.0 - 0.5)
        return self.back @ torch.cat([m[:1], m[1:4] + Ft, r])

    def stream(self, post):
        nx, ny, nz = self.n
        out = []
        wall = self.wall
        for i in range(19):
            cx, cy, cz = (int(v) for v in _C[i])
            v = torch.roll(post[i].reshape(nz, ny, nx), (cz, cy, cx), (0, 1, 2)).reshape(-1)
            if i and wall is not None:
                up = torch.roll(wall.reshape(nz, ny, nx), (cz, cy, cx), (0, 1, 2)).reshape(-1)
                v = torch.where(up, post[int(_OPP[i])], v)
            if cy and self.s["u_lo"]:
                at = self.xyz[1] == (0 if cy > 0 else ny - 1)
                uw = self.s["u_lo"] if cy > 0 else self.s["u_hi"]
                term = 6.0 * _WQ[i] * self.p["rho0"] * float(np.dot(_C[i], uw))
                v = torch.where(at, post[int(_OPP[i])] + term, v)
            out.append(v)
        return torch.stack(out)

    def step(self):
        n = self.p["md_substeps"]
        dt = 1.0 / n
        F = torch.zeros_like(self.F)
        for sub in range(n):
            for B in self.bodies:
                if sub:
                    self.kick(B, dt)
                self.drift(B, dt)
            F = self.couple(F, sub, dt)
        self.f = self.stream(self.collide(self.f, F))
        self.F = F
        for B in self.bodies:
            self.kick(B, dt)
        self.t += 1


def _bodies_of(m, keys):
    return {k: torch.stack([B[k] for B in m.bodies]) for k in keys}


def _exact_lattice(c, seed):
    s = _scene(c, seed)
    m = _Model(s)
    out, nb = {}, c["bodies"]
    series = np.zeros((c["steps"], 2, 3 * nb))
    for t in range(c["steps"]):
        if c["io"]:
            for b, B in enumerate(m.bodies):
                B["Fe"], B["Te"] = (torch.tensor(s["io"][t, k, 3 * b:3 * b + 3], dtype=F64, device=DEV) for k in (0, 1))
            m.set_force()
        m.step()
        if c["io"]:
            for b, B in enumerate(m.bodies):
                series[t, 0, 3 * b:3 * b + 3], series[t, 1, 3 * b:3 * b + 3] = B["F"].cpu().numpy(), B["T"].cpu().numpy()
    if c["io"]:
        out["series"] = series
    else:
        got = _bodies_of(m, ("F", "T"))
        out["F"], out["T"] = got["F"].reshape(-1), got["T"].reshape(-1)
    if nb <= 8:
        out.update(_bodies_of(m, ("X", "V", "q", "w")))
        out["beads"] = torch.cat([B["fb"] for B in m.bodies])
    if c["body_force"]:
        f = m.f if m.wall is None else m.f[:, ~m.wall]
        out["mass"], out["momentum"] = f.sum().reshape(1), (m.c.T @ f).sum(1)
    out["f"] = m.f if not c["probe"] else m.f[:, torch.from_numpy(s["nodes"]).to(DEV)].T
    return out


def _exact_batch(c, seed):
    scenes = _batch_scenes(c, seed)
    every, keep = max(1, c["steps"] // 4), (0, 2 * (c["count"] // 4))
    out = dict(X=[], V=[], q=[], w=[], F=[], path=[], f=[])
    for i, s in enumerate(scenes):
        m = _Model(s)
        path = []
        for t in range(c["steps"]):
            m.step()
            if (t + 1) % every == 0:
                path.append(m.bodies[0]["X"])
        for k in ("X", "V", "q", "w", "F"):
            out[k].append(m.bodies[0][k])
        if i < 64:
            out["path"].append(torch.stack(path[-4:]))
    for i in keep:
        m = _Model(scenes[i])
        for _ in range(c["steps"]):
            m.step()
        out["f"].append(m.f)
    return {k: v if k == "f" else torch.stack(v) for k, v in out.items()}


def _exact_adjoint(c, seed):
    """Reverse-mode differentiation of the plain model, the graph of one step at a time."""
    m = _Model(_adjoint_scene(c, seed))
    B = m.bodies[0]
    names = ("X", "V", "Fl")

    def advance(x):
        m.f, m.F = x[0], x[1]
        for k, v in zip(names, x[2:5]):
            B[k] = v
        m.gamma, B["s"] = x[5], x[6]
        m.step()
        return [m.f, m.F] + [B[k] for k in names]

    gamma, s = m.gamma, B["s"]
    x = [m.f, m.F] + [B[k] for k in names]
    tape, V = [], []
    with torch.no_grad():
        for _ in range(c["steps"]):
            tape.append(x)
            x = advance(x + [gamma, s])
            V.append(float(x[3][0]))
    lam = [torch.zeros_like(v) for v in x]
    dg, ds = torch.zeros_like(gamma), torch.zeros_like(s)
    for t in reversed(range(c["steps"])):
        if t >= c["steps"] - c["window"]:
            lam[3][0] += 1.0 / c["window"]
        leaves = [v.detach().requires_grad_(True) for v in tape.pop() + [gamma, s]]
        got = torch.autograd.grad(advance(leaves), leaves, lam, allow_unused=True)
        lam = [torch.zeros_like(l) if g is None else g for g, l in zip(got[:5], leaves)]
        lam = [v.clone() for v in lam]
        dg, ds = dg + got[5], ds + got[6]
    return dict(J=np.array([np.mean(V[-c["window"]:])]), dJ_dgamma=dg.reshape(1), dJ_dbeads=ds)


def _surface(P, A):
    """Nearest points of the ellipsoids A[S, 1, 3] to P[S, M, 3], by bisection."""
    m = A.min(-1, keepdim=True).values
    xm = torch.where(A == m, P.abs(), 0.0).max(-1, keepdim=True).values
    lo = -m * m + m * xm
    hi = torch.maximum(A.max(-1, keepdim=True).values * P.norm(dim=-1, keepdim=True), lo)
    PA, A2 = P * A, A * A
    for _ in range(56):
        mid = 0.5 * (lo + hi)
        pos = ((PA / (mid + A2)) ** 2).sum(-1, keepdim=True) > 1.0
        lo, hi = torch.where(pos, mid, lo), torch.where(pos, hi, mid)
    t = 0.5 * (lo + hi)
    return P * A2 / (t + A2)


def _exact_shells(c, seed):
    axes, xyz = _shells(c, seed)
    k, sigma, eps, dt, eta = 1000.0, 1.4, 0.1, 1e-3, 1000.0
    M = max(len(x) for x in xyz)
    P = torch.zeros((len(xyz), M, 3), dtype=F64, device=DEV)
    live = torch.zeros((len(xyz), M), dtype=torch.bool, device=DEV)
    for i, x in enumerate(xyz):
        P[i, :len(x)] = torch.tensor(x, device=DEV)
        P[i, len(x):] = 1.0 + torch.arange(M - len(x), device=DEV)[:, None]
        live[i, :len(x)] = True
    A = torch.tensor(axes, dtype=F64, device=DEV)[:, None]
    pairs = live[:, :, None] & live[:, None, :] & ~torch.eye(M, dtype=torch.bool, device=DEV)
    V = torch.zeros_like(P)
    for _ in range(c["steps"]):
        F = -2.0 * k * (P - _surface(P, A))
        d = [P[:, :, None, q] - P[:, None, :, q] for q in range(3)]
        d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        near = pairs & (d2 < 2 ** (1 / 3) * sigma ** 2)
        s6 = (sigma ** 2 / torch.where(near, d2, 1.0)) ** 3
        f = torch.where(near, 24 * eps * (2 * s6 * s6 - s6) / d2, 0.0)
        F = F + torch.stack([(f * d[q]).sum(2) for q in range(3)], -1)
        V = torch.where(live[..., None], (1 - eta * dt) * V + dt * F, 0.0)
        P = P + dt * V
    return dict(beads=torch.cat([_surface(P, A)[i, :len(x)] for i, x in enumerate(xyz)]))


def _exact_msd(c, seed):
    X, q = (torch.tensor(v, dtype=F64, device=DEV) for v in _trajectories(c, seed))
    w, x, y, z = q.unbind(-1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w), 2 * (x * y + z * w), 1 - 2 * (x * x + z * z),
                     2 * (y * z - x * w), 2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1).reshape(*q.shape[:2], 3, 3)
    a0, a1 = R[:, :-1], R[:, 1:]                       # columns are the body axes in the lab frame
    zero = torch.zeros((X.shape[0], 1, 3), dtype=F64, device=DEV)
    Xb = torch.cumsum(torch.cat([zero, (a0 * (X[:, 1:] - X[:, :-1])[..., None]).sum(2)], 1), 1)

    def dot(i, j):
        return (a1[..., i] * a0[..., j]).sum(-1)

    ang = torch.stack([torch.atan2(dot(2, 1), dot(2, 2)), torch.atan2(dot(0, 2), dot(0, 0)), torch.atan2(dot(1, 0), dot(1, 1))], -1)
    Th = torch.cumsum(torch.cat([zero, ang], 1), 1)
    p = R[..., 0]
    out = torch.empty((X.shape[0], c["lags"], 10), dtype=F64, device=DEV)
    for l in range(1, c["lags"] + 1):
        out[:, l - 1, 0:3] = ((X[:, l:] - X[:, :-l]) ** 2).mean(1)
        out[:, l - 1, 3:6] = ((Xb[:, l:] - Xb[:, :-l]) ** 2).mean(1)
        cr = torch.linalg.cross(p[:, :-l], p[:, l:])
        out[:, l - 1, 6] = (torch.atan2(cr.norm(dim=-1), (p[:, :-l] * p[:, l:]).sum(-1)) ** 2).mean(1)
        out[:, l - 1, 7:] = ((Th[:, l:] - Th[:, :-l]) ** 2).mean(1)
    return dict(msd=out)


def exact(case, seed):
    k = case["kind"]
    if k == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        return {"lattice": _exact_lattice, "batch": _exact_batch, "shells": _exact_shells, "msd": _exact_msd}[k](case, seed)
