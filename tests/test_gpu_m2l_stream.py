"""The streamed M2L kernel by itself: every split form at the orders where a K chunk, a row tile or the vector form of
the loads and adds is ragged, against the FP32 form on the CUDA cores.

Bar: twice what the tiled kernel of the same form is off by.  The two take the same products of the same hi and lo
parts (22 bits of an operand in TF32 and scaled FP16, 16 in BF16) and differ in the order of FP32 sums alone, 2^-24 of
the terms; a lost cross product would be 2^-11 of them (2^-8 in BF16).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BF16X3, TF32X3, F16X3 = 3, 4, 5


# P = p^4: 81 and 625 (odd: single adds), 256 (no remainder), 1296 (ragged last chunk, an odd number of 128-row tiles);
# p_t = 2 and 6 take the pairwise adds
@pytest.mark.parametrize("prec", [BF16X3, TF32X3, F16X3])
@pytest.mark.parametrize("p,pt,R", [(3, 3, 1), (3, 3, 2), (4, 4, 1), (4, 4, 3), (4, 2, 1), (5, 5, 1), (6, 6, 1)])
def test_the_streamed_kernel_agrees_with_the_fp32_form(prec, p, pt, R):
    from paper_2303_05006_gb300 import Solver
    from workloads.meshes import icosphere, mean_edge_length

    v, t = icosphere(1.0, 3)
    dt = 0.25 * mean_edge_length(v, t)
    kw = dict(mode=1, p_s=p, p_t=pt, n_leaf=64 if p > 4 else 16, n_rhs=R)
    alpha, Nt = 61, 80
    rng = np.random.default_rng(p)
    H = None

    def evaluate(**more):
        nonlocal H
        s = Solver(v, t, dt, Nt, **kw, **more)
        if H is None:
            per = rng.uniform(40, 80, (R, s.ne))
            H = np.sin(2 * np.pi * np.arange(alpha - 1)[:, None, None] / per + rng.uniform(0, 6, (R, s.ne)))
        out, info = s.history_eval(alpha, H if R > 1 else H[:, 0]), s.info()
        s.close()
        return out, info

    near, _ = evaluate(far_kernel=2, m2l_prec=0)
    want, _ = evaluate(m2l_prec=0)
    got, info = evaluate(m2l_prec=prec, m2l_tile_rows=2)
    levels = sum(1 << l for l in range(2, info.lmax + 1))
    assert info.m2l_streamed == levels and info.m2l_resident == 0
    tiled, info = evaluate(m2l_prec=prec, m2l_tile_rows=256)
    assert info.m2l_streamed == 0
    off, bar = np.abs(got - want).max(), 2 * np.abs(tiled - want).max()
    assert off <= bar and bar <= 2e-2 * np.abs(near - want).max()
    # nor is it the kernel of the other selections
    for rows in (1, 128):
        assert evaluate(m2l_prec=prec, m2l_tile_rows=rows)[1].m2l_streamed == 0
