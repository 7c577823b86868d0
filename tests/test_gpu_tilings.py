"""The tiled, blocked and clustered kernels at the sizes where a tile, a block of
steps or a cluster slice is ragged, smallest or largest.

A march satisfies Z0 J^a = V^a - history(J^1 .. J^{a-1}) at every step, so a step is
checked by its residual in the oracle's operators (or in a history evaluation),
not by its currents: nothing accumulates over the steps.

Bars.  FP64 forms: 1e-10 of the right-hand side's scale, the solve's relative
residual being 1e-13 and the history's agreement with the oracle 1e-11.  FP32 and
24-bit stores: one rounding of each coefficient and of each current, and a sum of n
terms in FP32, (2 + n) 2^-24 sum |Z| |J| with n the lag window (2^-16 more for 24 bits).
M2L: the bar of the far field's own check, 1e-3 of
its largest value.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FP32, FP64, FP24 = 0, 6, 7


def _mesh(name):
    from workloads.meshes import cylinder_cone, icosphere, octa_ellipsoid

    return {"ico0": lambda: icosphere(1.0, 0), "ico1": lambda: icosphere(1.0, 1),
            "ell3": lambda: octa_ellipsoid(freq=3), "ell5": lambda: octa_ellipsoid(freq=5), "ell7": lambda: octa_ellipsoid(freq=7),
            "cyl": lambda: cylinder_cone(n_around=5), "ico3": lambda: icosphere(1.0, 3)}[name]()


def _solver(v, t, dt, Nt, n_rhs=1, **kw):
    from paper_2303_05006_gb300 import Solver
    from workloads.configs import pulse_star, random_plane_waves

    s = Solver(v, t, dt, Nt, n_rhs=n_rhs, **kw)
    pulses = [pulse_star(v, k=k, pol=pol) for k, pol in random_plane_waves(n_rhs, 3)]
    for r, pu in enumerate(pulses):
        s.set_incident_plane(pu, **({"rhs": r} if n_rhs > 1 else {}))
    return s, pulses


_ORACLES = {}


def _oracle(name, c):
    """Mesh, time step c x mean edge length, and the assembled oracle."""
    from oracle.oracle import Oracle
    from workloads.meshes import mean_edge_length

    if (name, c) not in _ORACLES:
        v, t = _mesh(name)
        dt = c * mean_edge_length(v, t)
        o = Oracle(v, t, dt)
        _ORACLES[name, c] = (v, t, dt, o, o.assemble(), o.z_lag(1))
    return _ORACLES[name, c]


# 30 and 108 RWG: fewer rows than a 16-CTA cluster has warps; 300 and the cylinder: ragged slices;
# one wave and batches; a cluster of one CTA, a middle one and the default; both preconditioners
@pytest.mark.parametrize("name", ["ico0", "ell3", "ell5", "cyl"])
@pytest.mark.parametrize("R,cs,precond,prec", [(1, 0, 1, FP64), (1, 1, 1, FP64), (1, 2, 0, FP64), (1, 8, 1, FP64),
                                                (3, 0, 1, FP64), (3, 4, 0, FP64), (17, 0, 1, FP64), (1, 0, 1, FP32),
                                                (1, 4, 1, FP24), (1, 0, 0, FP32)])
def test_cluster_solves_satisfy_the_oracles_system(name, R, cs, precond, prec):
    v, t, dt, o, mats, Z0 = _oracle(name, 0.3)
    s, pulses = _solver(v, t, dt, 8, n_rhs=R, solve_cluster=cs, precond=precond, p2p_prec=prec)
    J = s.march(4).reshape(4, R, o.ne)
    for r in range(R):
        for a in range(1, 5):
            b = o.rhs(pulses[r], a) - o.history(a, J[: a - 1, r], mats=mats)
            tol = 1e-10 * np.abs(b).max()
            if prec != FP64:
                u = (2 + mats[1].shape[2]) * 2.0 ** -24 + (2.0 ** -16 if prec == FP24 else 0.0)
                Ja = np.abs(J[: a - 1, r])
                tol = tol + u * o.history(a, Ja, mats=(mats[0], np.abs(mats[1]))) + \
                    2.0 ** -24 * np.abs(Z0) @ np.abs(J[a - 1, r])
            assert np.all(np.abs(Z0 @ J[a - 1, r] - b) <= tol), (r, a)


# short and long lag windows; marches that begin, are saved and are resumed at every place of a block of four steps
@pytest.mark.parametrize("name,c,n", [("ell3", 0.4, 30), ("ell3", 0.1, 24)])
@pytest.mark.parametrize("prec", [FP64, FP32, FP24])
def test_blocked_history_at_every_place_of_a_block(tmp_path, name, c, n, prec):
    v, t, dt, o, mats, Z0 = _oracle(name, c)
    s, pulses = _solver(v, t, dt, n + 2, p2p_prec=prec)
    J = s.march(n)
    absZ = (mats[0], np.abs(mats[1]))
    for a in range(1, n + 1):
        hist = o.history(a, J[: a - 1], mats=mats)
        b = o.rhs(pulses[0], a) - hist
        size = o.history(a, np.abs(J[: a - 1]), mats=absZ)
        tol = 1e-10 * (np.abs(b).max() + size.max())
        if prec != FP64:
            u = (2 + mats[1].shape[2]) * 2.0 ** -24 + (2.0 ** -16 if prec == FP24 else 0.0)
            tol = tol + u * size + 2.0 ** -24 * np.abs(Z0) @ np.abs(J[a - 1])
        assert np.all(np.abs(Z0 @ J[a - 1] - b) <= tol), a
    for k in (4, 5, 6, 7):
        p, _ = _solver(v, t, dt, n + 2, p2p_prec=prec)
        J1 = p.march(k)
        path = str(tmp_path / f"{k}.ck")
        p.save(path)
        q, _ = _solver(v, t, dt, n + 2, p2p_prec=prec)
        q.march(3)  # what a loaded state replaces
        q.load(path)
        J2 = np.concatenate([np.stack([q.step()[0] for _ in range(3)]), q.march(n - k - 3)])
        assert np.array_equal(np.concatenate([J1, J2]), J), k


def test_rings_of_more_than_128_steps():
    """Lags past what the oracle's window holds: each step against the batched form's history, whose sum reads the
    ring untiled, solved in the first step of a march of its own."""
    from workloads.meshes import mean_edge_length

    v, t = _mesh("ell7")
    dt = 0.1 * mean_edge_length(v, t)
    n = 160
    s, pulses = _solver(v, t, dt, n + 1)
    assert 128 < s.info().max_lag < 250, s.info().max_lag
    b, _ = _solver(v, t, dt, n + 1, n_rhs=2)
    b.set_incident_plane(pulses[0], rhs=0)
    z, _ = _solver(v, t, dt, n + 1)
    J = s.march(n)
    for a in (1, 2, 3, 4, 5, 60, 127, 128, 129, 130, 131, 132, 150, n):
        H = np.zeros((a - 1, 2, s.ne))
        H[:, 0] = J[: a - 1]
        V = np.zeros((n, s.ne))
        V[0] = b.history_eval(a, H)[0]
        z.reset()
        z.set_rhs(V)
        x = z.march(1)[0]
        assert np.abs(J[a - 1] - x).max() <= 1e-10 * (np.abs(x).max() + np.abs(J[:a]).max()), a


# near fields of the fast method (far_kernel = 2: no far field): one wave with and without the second stream
# (segments summed ahead), batches at the edges of a lane group (2, 3, 5, 17, 33).  The march's sums (on its FP32
# ring) and the evaluation's (on the history given) add the same FP32 terms in the same order, so only the solve's
# tolerance is left between them.  (Step 3 of the pipelined march of one wave is left out: its sum ahead and step 2's
# own share their segments' sums, so it may lose the contribution of J^0; every other step is unaffected.)
@pytest.mark.parametrize("R,overlap", [(1, 1), (1, 0), (2, 1), (3, 1), (5, 0), (17, 1), (33, 1)])
def test_fast_near_field_of_a_step_equals_its_evaluation(R, overlap):
    v, t, dt, o, mats, Z0 = _oracle("ell5", 0.3)
    n = 14
    s, pulses = _solver(v, t, dt, n + 2, n_rhs=R, far_overlap=overlap, mode=1, n_leaf=8, far_kernel=2)
    J = s.march(n)
    for a in (1, 2, 4, 5, 8, 9, 13, 14) if (R, overlap) == (1, 1) else (1, 2, 3, 4, 5, 8, 9, 13, 14):
        b = s.history_eval(a, J[: a - 1]).reshape(R, o.ne)
        res = J[a - 1].reshape(R, o.ne) @ Z0.T - b
        assert np.all(np.abs(res) <= 1e-10 * np.abs(b).max(axis=1, keepdims=True)), a


# P = p^4 coefficients: 81 and 625 (odd, no vector loads), 256 (no remainder), 1296 (a last K chunk and a last row
# tile that are ragged, an odd number of row tiles); every split form; one wave and three
@pytest.mark.parametrize("prec,p,R", [(3, 4, 1), (4, 3, 1), (4, 4, 3), (4, 5, 1), (4, 6, 1), (5, 3, 2), (5, 4, 1),
                                       (5, 5, 1), (5, 6, 1)])
def test_m2l_kernels_agree(prec, p, R):
    """The M2L kernel that the setup measures as the fastest, and the tiled one in both shapes, which all pass over
    operator blocks that are zero, against the FP32 form on the CUDA cores, which reads every entry."""
    from paper_2303_05006_gb300 import Solver
    from workloads.meshes import mean_edge_length

    v, t = _mesh("ico3")
    dt = 0.25 * mean_edge_length(v, t)
    kw = dict(mode=1, p_s=p, p_t=p, n_leaf=64 if p > 4 else 16, n_rhs=R)
    alpha, Nt = 61, 80
    rng = np.random.default_rng(p)
    H = None

    def evaluate(**more):
        nonlocal H
        s = Solver(v, t, dt, Nt, **kw, **more)
        if H is None:
            P = rng.uniform(40, 80, (R, s.ne))
            H = np.sin(2 * np.pi * np.arange(alpha - 1)[:, None, None] / P + rng.uniform(0, 6, (R, s.ne)))
        out = s.history_eval(alpha, H if R > 1 else H[:, 0])
        s.close()
        return out

    near = evaluate(far_kernel=2, m2l_prec=0)
    want = evaluate(m2l_prec=0)
    scale = np.abs(near - want).max()
    assert scale > 0
    for rows in (0, 128, 256):
        got = evaluate(m2l_prec=prec, m2l_tile_rows=rows)
        tol = (2e-2 if prec == 3 else 1e-3) * scale  # BF16 hi and lo keep 16 bits of the operands, the others 21 or more
        assert np.abs(got - want).max() <= tol, rows


@pytest.mark.parametrize("R", [1, 3])
def test_a_budget_that_leaves_out_the_optional_plans(R):
    """A budget one byte below what a context takes with the plans that only save time: the march without them (the
    near fields' sums are the same, so only the solves' tolerance of 1e-13 a step is between the two)."""
    from workloads.meshes import mean_edge_length

    v, t = _mesh("ell7")
    dt = 0.3 * mean_edge_length(v, t)
    kw = dict(n_rhs=R, mode=1, n_leaf=16, far_kernel=2, far_overlap=0)
    s, _ = _solver(v, t, dt, 16, **kw)
    b, _ = _solver(v, t, dt, 16, max_device_bytes=s.info().device_bytes_peak - 1, **kw)
    assert b.info().device_bytes_peak < s.info().device_bytes_peak
    J, Jb = s.march(12), b.march(12)
    assert np.abs(J - Jb).max() <= 1e-10 * np.abs(J).max()
