"""Sums launched ahead on a second stream, at the steps where a march has to do without them or meets them with
something else in between: its first steps, the steps after a load, after a load that is refused, and after a
history evaluation.

Each step is checked by its residual: Z0 J^{a-1} against V^{a-1} minus the history, evaluated by the same context
(two contexts of the fast method differ in the last bits of their coefficients).  March and evaluation add the same
terms in the same order, so the solve's tolerance of 1e-13 is all that is left between them; the bar is 1e-10 of the
right-hand side's scale.  A context's own marches of the same steps are equal to the last bit.
"""
import numpy as np
import pytest

from test_gpu_tilings import _oracle, _solver

pytestmark = pytest.mark.gpu


def _residuals_hold(J, Z0, evaluate, steps, bar=1e-10):
    for a in steps:
        b = evaluate(a, J[: a - 1])
        assert np.abs(Z0 @ J[a - 1] - b).max() <= bar * np.abs(b).max(), a


# far_kernel = 2: no far field, whose atomics would be above the bar
def _fast(v, t, dt, n):
    return _solver(v, t, dt, n + 2, mode=1, n_leaf=8, far_kernel=2)[0]


@pytest.mark.parametrize("name,c", [("ell5", 0.3), ("cyl", 0.3)])
def test_every_step_of_the_fast_march(tmp_path, name, c):
    v, t, dt, o, mats, Z0 = _oracle(name, c)
    n, k = 14, 6
    s = _fast(v, t, dt, n)
    J = s.march(n)
    _residuals_hold(J, Z0, s.history_eval, range(1, n + 1))
    # a state loaded over another march's
    s.reset()
    J1 = s.march(k)
    path = str(tmp_path / "fast.ck")
    s.save(path)
    q = _fast(v, t, dt, n)
    q.march(4)
    q.load(path)
    J2 = np.concatenate([J1, q.march(n - k)])
    _residuals_hold(J2, Z0, q.history_eval, range(k + 1, n + 1))
    # a load that is refused leaves the march as it was
    s.reset()
    J1 = s.march(k)
    from paper_2303_05006_gb300 import TdbemError

    with pytest.raises(TdbemError):
        s.load(str(tmp_path / "missing.ck"))
    assert np.array_equal(np.concatenate([J1, s.march(n - k)]), J)


def test_an_evaluation_between_two_steps_of_the_fast_march():
    v, t, dt, o, mats, Z0 = _oracle("ell5", 0.3)
    n = 14
    s = _fast(v, t, dt, n)
    J = s.march(n)
    s.reset()
    for a in range(1, n + 1):
        b = s.history_eval(a, J[: a - 1])
        x = s.step()[0]
        assert np.array_equal(x, J[a - 1]), a
        assert np.abs(Z0 @ x - b).max() <= 1e-10 * np.abs(b).max(), a


# The direct march forms its far pairs' sums four steps a pass where its store is 64 MiB or more (8, 4 or 3 bytes a
# coefficient): 1452 RWG.  Every step from its evaluation, solved in the first step of a march of its own, and every
# other way to the same steps bit for bit.
@pytest.mark.parametrize("prec,size", [(6, 8), (0, 4), (7, 3)])
def test_every_step_of_the_blocked_direct_march(tmp_path, prec, size):
    from paper_2303_05006_gb300 import TdbemError
    from workloads.meshes import mean_edge_length, octa_ellipsoid

    v, t = octa_ellipsoid(freq=11)
    dt = 0.25 * mean_edge_length(v, t)
    n = 27
    s, pulses = _solver(v, t, dt, n + 2, p2p_prec=prec)
    assert s.info().near_coef_bytes // 8 * size >= 64 << 20
    J = s.march(n)
    z, _ = _solver(v, t, dt, n + 2, p2p_prec=prec)
    batch = None
    if prec == 6:  # the batched form's sum reads the ring untiled
        batch, _ = _solver(v, t, dt, n + 2, n_rhs=2)
        batch.set_incident_plane(pulses[0], rhs=0)
    for a in range(1, n + 1):
        b = [s.history_eval(a, J[: a - 1])]
        if batch is not None:
            H = np.zeros((a - 1, 2, s.ne))
            H[:, 0] = J[: a - 1]
            b.append(batch.history_eval(a, H)[0])
        for x in b:
            V = np.zeros((n + 1, s.ne))
            V[0] = x
            z.reset()
            z.set_rhs(V)
            x = z.march(1)[0]
            assert np.abs(J[a - 1] - x).max() <= 1e-10 * (np.abs(x).max() + np.abs(J[:a]).max()), a
    z.close()
    missing = str(tmp_path / "missing.ck")
    q, _ = _solver(v, t, dt, n + 2, p2p_prec=prec)
    for k in range(1, 14):
        s.reset()  # whatever is in flight after step k - 1's sums ahead
        J1 = s.march(k)
        path = str(tmp_path / f"{k}.ck")
        s.save(path)
        with pytest.raises(TdbemError):
            s.load(missing)
        s.history_eval(k + 1, J[:k])
        assert np.array_equal(np.concatenate([J1, s.march(n - k)]), J), k
        q.reset()
        q.march(3)
        q.load(path)
        assert np.array_equal(q.march(n - k), J[k:]), k
        s.reset()
        s.march_dev(k)
    s.close()
    for Nt in (7, 8, 9, 10):  # marches that end where a block's sums ahead would begin
        e, _ = _solver(v, t, dt, Nt, p2p_prec=prec)
        for _ in range(3):
            e.reset()
            assert np.array_equal(e.march(Nt - 1), J[: Nt - 1]), Nt
        e.close()


# what is not finite in the history reaches the rows that have an entry there, in its own right-hand side, and no other
@pytest.mark.parametrize("R", [2, 3, 17])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e200])
def test_values_that_are_not_finite_stay_in_their_rows(R, value):
    v, t, dt, o, mats, Z0 = _oracle("ell5", 0.3)
    one, _ = _solver(v, t, dt, 6, mode=1, n_leaf=8, far_kernel=2, far_overlap=0)
    s, _ = _solver(v, t, dt, 6, n_rhs=R, mode=1, n_leaf=8, far_kernel=2)
    H = np.random.default_rng(1).standard_normal((1, R, s.ne))
    H[0, 1, 0] = value
    got = s.history_eval(2, H)
    want = np.stack([one.history_eval(2, H[:, r]) for r in range(R)])
    reached = np.nonzero(~np.isfinite(want[1]))[0]
    assert 0 < len(reached) < s.ne // 4 and np.isfinite(want[[r for r in range(R) if r != 1]]).all()
    assert np.array_equal(np.isfinite(got), np.isfinite(want))


def test_a_value_that_is_not_finite_stays_on_its_side_of_the_body():
    """The direct march's stores pad the windows of 32 neighbouring rows to the longest, with zero coefficients, so
    what is not finite may reach rows beside those that have an entry there, but no row across the body."""
    from workloads.meshes import mean_edge_length, octa_ellipsoid

    v, t = octa_ellipsoid(freq=11)
    s, _ = _solver(v, t, 0.25 * mean_edge_length(v, t), 6)
    assert s.info().near_coef_bytes >= 64 << 20  # four steps a pass, near pairs apart
    ev = s.edges()[0]
    mid = v[ev].mean(axis=1)
    far = np.linalg.norm(mid - mid[0], axis=1)
    far = np.nonzero(far > 0.7 * far.max())[0]
    H = np.random.default_rng(1).standard_normal((1, s.ne))
    for value in (np.nan, np.inf):
        H[0, 0] = value
        for a in (3, 4, 5):
            got = s.history_eval(a, H)
            assert not np.isfinite(got).all() or a == 3
            assert np.isfinite(got[far]).all(), a
