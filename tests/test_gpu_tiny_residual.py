"""Refinement of a slice whose residual lies below the normal range of FP32 (a
right-hand side of about 1e-33: a product of many small rank-1 factors): the
correction's scale has to stay finite.  Tolerance as in test_gpu_parity.py
(complex64 1e-4; the systems of rank 1 have condition number 1)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu


def test_sweep_with_tiny_right_hand_sides():
    n, L, b, r, lam = 2048, 10, 2, 1, 1e-1
    i, j = synth.draw_pairs(n, 61440, 31)
    t = oracle.eval_entries(n, L, b, r, synth.random_factors(n, L, r, 901), i, j)
    X0 = synth.random_factors(n, L, r, 301)
    Xo, st_o = oracle.als_sweep(n, L, b, r, lam, X0, i, j, t, ridge_rel=2.0 ** -20)
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=bfc.PREC_C64) as c:
        c.set_factors(X0)
        st = c.sweep()
        Xg = c.get_factors()
    assert np.all(np.isfinite(Xg))
    assert abs(st["objective"] - st_o["objective"]) <= 1e-4 * st_o["objective"]
    assert rel_dev(oracle.eval_entries(n, L, b, r, Xg, i, j), oracle.eval_entries(n, L, b, r, Xo, i, j)) <= 1e-4
