"""The marches a user of this library runs, as measured cases.

A case is one scatterer (or three marched together), a time step, a mode with
its precisions, a number of incident waves and a number of steps, taken through
the package's own entry points (`Solver.step`, `Solver.march`,
`Solver.step_v_async`, `march_many`, `Solver.history_eval`, `Solver.mlp_train`).
The context (mesh, operators, trees) is what a program keeps; the incident
waves and, where the caller supplies them, the right-hand sides come from the
seed.  A pass starts the march afresh, so it can be repeated on one context.
"""
import functools
import math

import numpy as np
import torch

import workloads
from paper_2303_05006_gb300 import Solver, march_many
from workloads.configs import Pulse, pulse_star, random_plane_waves, sin2_pulse
from workloads.meshes import (cube_jittered, cylinder_cone, ellipsoid_uv, geodesic_sphere, icosphere,
                              mean_edge_length, octa_ellipsoid)

# arithmetic codes of include/tdbem.h
FP32, TF32X3, F16X3, FP64, FP24 = 0, 4, 5, 6, 7

# A plain case: the defaults of Solver except where a case says otherwise.
BASE = {"mesh": "ico", "size": 3, "mode": "direct", "p2p_prec": FP64, "m2l_prec": F16X3, "p": 4, "n_rhs": 1,
        "dt_per_h": 0.5, "solve_tol": 1e-13, "call": "march", "steps": 64}


def listed():
    return [
        # The smallest call: one step at a time on a 120-RWG body, each current handed back before the next
        # step is asked for (a solver coupled to another code).  Launches and latency only.
        dict(BASE, name="steps_sphere120", size=1, call="step", steps=24),
        # The default march of a small body (1920 RWG), everything at its default.
        dict(BASE, name="march_sphere1920", size=3, steps=96),
        # The exact direct march of an odd-sized, non-spherical body: 5292 RWG, no block size divides it;
        # theta = zeta = 3 as for every body here that is not a sphere.
        dict(BASE, name="march_ellipsoid5292", mesh="octa_ellipsoid", size=21, steps=40),
        # The headline use: the 7680-RWG sphere with FP32 coefficients, streamed end to end with the
        # incident field produced on the host (pinned arrays, a few steps in flight).
        dict(BASE, name="stream_sphere7680_fp32", size=4, p2p_prec=FP32, call="stream", steps=80),
        # The paper's test problem, case 1 (sphere of radius 0.5, 1280 triangles, dt = 0.005): a time step
        # far below the edge length, so that lag windows and the history are long.
        dict(BASE, name="march_paper_case1", mesh="geodesic", size=8, dt_per_h=0.0, steps=48),
        # Several incident waves on one body through the exact direct method.
        dict(BASE, name="waves8_sphere1920", size=3, n_rhs=8, steps=24),
        # The fast method on the 7680-RWG sphere at the paper's solve tolerance.
        dict(BASE, name="fast_sphere7680", mode="fast", size=4, solve_tol=1e-8, steps=96),
        # The fast method at a higher order, where the M2L products dominate.
        dict(BASE, name="fast_p6_sphere1920", mode="fast", size=3, p=6, m2l_prec=TF32X3, solve_tol=1e-8, steps=48),
        # Two bodies, 12864 RWG, three far levels (the precision sweep's pair, the cube a little coarser).
        dict(BASE, name="fast_sphere_cube", mode="fast", mesh="sphere_cube", size=12, m2l_prec=TF32X3,
             solve_tol=1e-8, steps=64),
        # Many incident waves on one body through the fast method (4608 RWG, slivers at the cone tips).
        dict(BASE, name="fast_waves16_cylinder", mode="fast", mesh="cylinder", size=48, n_rhs=16, solve_tol=1e-8,
             steps=16),
        # Three scatterers marched together: a sphere, a cylinder and an ellipsoid, whose solves differ widely.
        dict(BASE, name="many_fast", mode="fast", mesh="trio", size=21, solve_tol=1e-8, call="many", steps=24),
        # Training the learned warm start on recorded steps (width 256, on the tensor cores).
        dict(BASE, name="train_256", size=3, call="train", width=256, steps=24, batch=4096),
    ]


def draw(rng):
    """One more case of the same ranges: small bodies to some 6000 RWG (direct) or 9000 (fast), every
    precision, odd sizes, few or many steps and waves."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["direct", "direct", "direct_waves", "stream", "step", "fine", "fast", "fast", "fast_p",
                       "fast_waves", "many", "history", "train"])
    c = dict(BASE, wave=rng.randrange(1 << 20))
    body = rng.choice(["octa_sphere", "octa_ellipsoid"])
    if kind in ("direct", "stream"):
        c.update(mesh=body, size=log_int(5, 22), p2p_prec=rng.choice([FP64, FP32, FP24]), steps=log_int(24, 90),
                 call="stream" if kind == "stream" else "march")
    elif kind == "direct_waves":
        c.update(mesh=body, size=log_int(4, 13), n_rhs=rng.choice([2, 3, 5, 8, 13]), steps=log_int(8, 24))
    elif kind == "step":
        c.update(mesh=body, size=log_int(3, 12), call="step", steps=log_int(12, 48))
    elif kind == "fine":
        c.update(mesh="geodesic", size=rng.randrange(6, 10), dt_per_h=0.0, steps=log_int(16, 48))
    elif kind == "fast":
        c.update(mode="fast", mesh=body, size=log_int(10, 28), m2l_prec=rng.choice([F16X3, TF32X3, FP32]),
                 solve_tol=rng.choice([1e-8, 1e-13]), steps=log_int(24, 90))
    elif kind == "fast_p":
        c.update(mode="fast", mesh=body, size=log_int(9, 16), p=rng.choice([3, 5, 6]),
                 m2l_prec=rng.choice([F16X3, TF32X3]), solve_tol=1e-8, steps=log_int(16, 48))
    elif kind == "fast_waves":
        c.update(mode="fast", mesh=rng.choice([body, "cylinder"]), size=log_int(9, 20),
                 n_rhs=rng.choice([2, 5, 8, 16]), solve_tol=1e-8, steps=log_int(8, 16))
        if c["mesh"] == "cylinder":
            c.update(size=2 * rng.randrange(12, 25))
    elif kind == "many":
        c.update(mode="fast", mesh="trio", size=rng.randrange(13, 22), solve_tol=1e-8, call="many",
                 steps=log_int(12, 24))
    elif kind == "history":
        c.update(mode=rng.choice(["direct", "fast"]), mesh=body, size=log_int(5, 16), call="history",
                 steps=log_int(12, 48))
    else:
        c.update(call="train", size=2, mesh="ico", width=rng.choice([64, 256]), steps=log_int(16, 40),
                 batch=128 * rng.choice([8, 16, 31]))
    return c


@functools.lru_cache(maxsize=8)
def _mesh(kind, size):
    """(verts, tris, theta, edge length of the time step), generated once per process."""
    if kind == "ico":
        v, t = icosphere(1.0, size)
    elif kind == "geodesic":
        v, t = geodesic_sphere(0.5, size)
    elif kind == "octa_sphere":
        v, t = octa_ellipsoid((1.0, 1.0, 1.0), size)
    elif kind == "octa_ellipsoid":
        v, t = octa_ellipsoid(freq=size)
    elif kind == "cylinder":
        v, t = cylinder_cone(n_around=size)
    elif kind == "uv":
        v, t = ellipsoid_uv(n_lat=size)
    else:  # sphere_cube: a sphere beside a jittered cube
        vs, ts = icosphere(1.0, 4)
        vc, tc = cube_jittered(2.0, size, 0.02, 3, centre=(3.5, 0.0, 0.0))
        v, t = np.concatenate([vs, vc]), np.concatenate([ts, tc + len(vs)]).astype(np.int32)
        return v, t, 3.0, mean_edge_length(vs, ts)
    return v, t, 1.0 if kind in ("ico", "geodesic", "octa_sphere") else 3.0, mean_edge_length(v, t)


def _bodies(case):
    if case["mesh"] == "trio":
        return [("ico", 3), ("cylinder", 40), ("uv", case["size"])]
    return [(case["mesh"], case["size"])]


def _dt(case, h):
    return case["dt_per_h"] * h if case["dt_per_h"] else 0.005  # 0.005: the paper's test problem


def _pulses(case, v, rng):
    """Plane waves of seeded direction, polarisation and, a little, strength of the carrier."""
    out = []
    for k, pol in random_plane_waves(case["n_rhs"], int(rng.integers(1 << 30))):
        if case["dt_per_h"] == 0.0:
            out.append(sin2_pulse(v, k=k, pol=pol))
        else:
            # three widths before its peak (1% of it), so that a short march carries currents in every step
            p = pulse_star(v, k, pol, f_scale=float(rng.uniform(0.7, 1.0)))
            out.append(Pulse(p.k, p.pol, p.f0, p.sigma, 3.0 * p.sigma, p.z_min))
    return out


def _solver(case, body, rng, Nt):
    v, t, theta, h = _mesh(*body)
    s = Solver(v, t, _dt(case, h), Nt, theta=theta, zeta=theta, mode=1 if case["mode"] == "fast" else 0,
               p_s=case["p"], p_t=case["p"], p2p_prec=case["p2p_prec"], m2l_prec=case["m2l_prec"],
               n_rhs=case["n_rhs"], solve_tol=case["solve_tol"])
    for r, p in enumerate(_pulses(case, v, rng)):
        s.set_incident_plane(p, r)
    return s


def prepare(case, seed):
    rng = np.random.default_rng([int(seed), int(case.get("wave", 0))])
    n = case["steps"]
    ss = [_solver(case, b, rng, n + 4) for b in _bodies(case)]
    st = {"case": case, "solvers": ss}
    if case["call"] == "stream":
        # a host program's right-hand sides: the wave's own tested field of each step
        s = ss[0]
        V = torch.empty(n, s.ne, dtype=torch.float64).pin_memory()
        for a in range(n):
            V[a] = torch.from_numpy(s.history_eval(a + 1, np.zeros((0, s.ne))))
        st["V"] = V
    elif case["call"] == "many":
        st["out"] = [torch.empty(n, s.ne, dtype=torch.float64, device="cuda") for s in ss]
    elif case["call"] == "history":
        # band-limited currents: a sinusoid per function, with its own period and phase
        s = ss[0]
        per, ph = rng.uniform(15, 60, s.ne), rng.uniform(0, 2 * np.pi, s.ne)
        st["J"] = np.sin(2 * np.pi * np.arange(n)[:, None] / per + ph) * rng.uniform(0.5, 1.5, s.ne)
    elif case["call"] == "train":
        s = ss[0]
        s.mlp_set_width(case["width"])
        F, H = s.MLP_FEATURES, case["width"]
        st["theta"] = np.concatenate([rng.standard_normal(F * H) / math.sqrt(F), rng.standard_normal(H * H) / math.sqrt(H),
                                      0.1 * rng.standard_normal(H) / math.sqrt(H)]).astype(np.float32)
        s.mlp_record(n * s.ne)
        s.march(n)
    return st


def run(st):
    case, ss = st["case"], st["solvers"]
    s, n = ss[0], case["steps"]
    if case["call"] == "train":
        s.mlp_set_weights(st["theta"])
        loss = s.mlp_train(2, case["batch"], 1e-4, seed=5)
        return {"loss": loss, "weights": s.mlp_get_weights()}
    if case["call"] == "history":
        return s.history_eval(n + 1, st["J"])
    for x in ss:
        x.reset()
    if case["call"] == "step":
        return np.stack([s.step()[0] for _ in range(n)])
    if case["call"] == "stream":
        V = st["V"].numpy()
        J = torch.empty(n, s.ne, dtype=torch.float64, pin_memory=True).numpy()
        for a in range(n):
            s.step_v_async(V[a], J[a])
            if a >= 2:  # the currents are taken two steps later
                s.step_wait()
        s.step_wait()
        s.step_wait()
        return J
    if case["call"] == "many":
        march_many(ss, [n] * len(ss), [o.data_ptr() for o in st["out"]])
        return st["out"]
    return s.march(n)


@functools.lru_cache(maxsize=64)
def _lags(kind, size, dt):
    """Mean stored lags per pair of functions, from a sample of rows: a pair couples at the lags m with
    m - r/(c dt) in (0, 3) for some distance r between the two supports."""
    v, t, _, _ = _mesh(kind, size)
    e = np.unique(np.sort(np.concatenate([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), axis=1), axis=0)
    mid, rad = v[e].mean(1), np.linalg.norm(v[e[:, 0]] - v[e[:, 1]], axis=1)
    rows = np.random.default_rng(1).choice(len(e), min(64, len(e)), replace=False)
    d = np.linalg.norm(mid[rows][:, None] - mid[None], axis=2)
    ext = rad[rows][:, None] + rad[None]
    return len(e), float(np.mean((np.minimum(2 * d, 2 * ext)) / dt + 3.0)), float(np.mean(d < 3.0 * ext))


def work(case):
    """Bytes: the stored operators and the incident field read once, the currents written once.  Flops:
    two per coefficient, step and wave; for the fast method an estimate of its near field and M2L."""
    n, R = case["steps"], case["n_rhs"]
    if case["call"] == "train":
        ne = 480 if case["size"] == 2 else 1920
        H, S = case["width"], n * ne
        return {"bytes": S * 27 * 4.0 + 8.0 * (25 * H + H * H), "flops": 2 * 6.0 * S * (25 * H + H * H + H)}
    nb = fl = 0.0
    for kind, size in _bodies(case):
        ne, lags, near = _lags(kind, size, _dt(case, _mesh(kind, size)[3]))
        nb += 16.0 * n * ne * R
        steps = 1 if case["call"] == "history" else n
        if case["mode"] == "direct":
            nval = lags * ne * ne
            nb += nval * {FP64: 8, FP32: 4, FP24: 3}[case["p2p_prec"]]
            fl += 2.0 * nval * R * steps
        else:
            P, cells = case["p"] ** 4, ne / 32.0
            nb += 4.0 * lags * near * ne * ne
            # 7 components, about 27 far cells and 3 lags for each, once per interval of about 6 steps
            fl += R * n * (2.0 * lags * near * ne * ne + 2.0 * P * P * 7 * 27 * 3 * cells / 6)
    return {"bytes": nb, "flops": fl}


def exact(case, seed):
    # The operators are exact retarded integrals over all pairs of functions: in 64 bits without the library
    # they take hours on the host, so no case has an independent value here.
    return None
