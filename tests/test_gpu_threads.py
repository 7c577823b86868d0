"""Contexts of different kinds created and evaluated by several threads at once give what one thread gives."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_contexts_of_several_threads():
    from paper_2303_05006_gb300 import Solver
    from workloads.meshes import icosphere, mean_edge_length, octa_ellipsoid

    bodies = {"ico": icosphere(1.0, 3), "ell": octa_ellipsoid(freq=11)}
    # lag windows, orders, M2L kernels, numbers of right-hand sides and solves of their own
    kinds = [("ico", 0.25, dict(mode=1, m2l_prec=4, m2l_tile_rows=2, n_leaf=16)),
             ("ell", 0.1, dict(mode=1, n_leaf=8)),
             ("ico", 0.5, dict(mode=1, m2l_prec=5, m2l_tile_rows=1, n_leaf=16, n_rhs=3)),
             ("ell", 0.25, dict()),
             ("ico", 0.5, dict(p2p_prec=0)),
             ("ell", 0.5, dict(n_rhs=2))]
    n = 20

    def run(k):
        body, c, kw = kinds[k]
        v, t = bodies[body]
        s = Solver(v, t, c * mean_edge_length(v, t), n + 1, **kw)
        rng = np.random.default_rng(k)
        for r in range(kw.get("n_rhs", 1)):
            s.set_rhs(np.sin(np.arange(n)[:, None] / rng.uniform(2, 6, s.ne) + rng.uniform(0, 6, s.ne)), r)
        J = s.march(n)
        s.close()
        return J

    want = [run(k) for k in range(len(kinds))]
    got = [None] * len(kinds)

    def work(k):
        for _ in range(3):
            got[k] = run(k)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(kinds))]
    for x in ts:
        x.start()
    for x in ts:
        x.join()
    for k, (w, g) in enumerate(zip(want, got)):
        assert g is not None, k
        # the far field's FP32 atomics leave 1e-6 between two runs of one march
        bar = 1e-5 if kinds[k][2].get("mode") else 1e-12
        assert np.abs(w - g).max() <= bar * np.abs(w).max(), k
