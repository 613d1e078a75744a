"""The slice sums of the gradient, ADAM and ADF kernels at every rank, with
slices of more entries than a thread adds before a reduction (1024 entries;
64 terms times up to 32 threads per component), ragged and empty slices,
against the oracle.  Tolerances: FP64 1e-10; complex64 1e-4 of the largest
component (gradient) and of the entry values (ADAM, ADF), as in
test_gpu_parity.py and test_gpu_first_order.py."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev
from oracle import first_order as fo

pytestmark = pytest.mark.gpu

TOL = {bfc.PREC_FP64: 1e-10, bfc.PREC_C64: 1e-4}


def problem(r, ragged):
    n, L, b = (48, 2, 12) if ragged else (64, 1, 32)
    i, j = synth.draw_pairs(n, 701 if ragged else n * n, 60 + r)
    if ragged:
        keep = (i // b != 1) | (j // b < 3)
        i, j = i[keep], j[keep]
    X = synth.random_factors(n, L, r, 70 + r)
    t = oracle.eval_entries(n, L, b, r, X, i, j) + 0.1 * synth.SplitMix64(80 + r).cnormal(i.size)
    return n, L, b, 1e-3, i, j, t, synth.random_factors(n, L, r, 90 + r)


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("r", range(1, 13))
def test_gradient_every_rank(r, ragged, prec):
    n, L, b, lam, i, j, t, X0 = problem(r, ragged)
    go, f_o = oracle.grad(n, L, b, r, lam, X0, i, j, t, include_reg=True)
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec) as c:
        c.set_factors(X0)
        g, f = c.grad(True)
    assert abs(f - f_o) <= TOL[prec] * abs(f_o)
    assert np.abs(g - go).max() <= TOL[prec] * np.abs(go).max()


def check_entries(p, got, want, prec):
    n, L, b, r, i, j = p
    xg, xo = (oracle.eval_entries(n, L, b, r, X, i, j) for X in (got, want))
    assert rel_dev(xg, xo) <= TOL[prec]


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("r", [1, 2, 3, 5, 7, 8, 10, 12])
def test_adf_iteration_every_rank(r, prec):
    n, L, b, lam, i, j, t, X0 = problem(r, True)
    want, _ = fo.adf_iteration(n, L, b, r, lam, X0, i, j, t)
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec) as c:
        c.set_factors(X0)
        c.adf(1)
        check_entries((n, L, b, r, i, j), c.get_factors(), want, prec)


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("r", [2, 3, 5, 7, 8, 10, 12])
def test_adam_iterations_every_rank(r, prec):
    """Not rank 1: some component of this problem's gradient cancels there, and
    ADAM's step, m / sqrt(v), is then the ratio of two rounding errors."""
    n, L, b, lam, i, j, t, X0 = problem(r, True)
    M, V = np.zeros((X0.size, 2)), np.zeros((X0.size, 2))
    want = X0
    for it in (1, 2):
        want = fo.adam_iteration(n, L, b, r, lam, want, i, j, t, M, V, it)
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec) as c:
        c.set_factors(X0)
        c.adam(2)
        check_entries((n, L, b, r, i, j), c.get_factors(), want, prec)
