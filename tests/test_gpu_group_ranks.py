"""The grouped Gram at every rank (tile shapes, padded ranks 7 and 11, tiles
split over blocks, both group-sum kernels) against the oracle's sweep.

Tolerances as in test_gpu_parity.py: FP64 1e-10 relative on entry values and
the objective; complex64 max(1e-4, kappa_max 2^-24), kappa_max the largest
condition number of the sweep's block systems (a system solved from sums with
complex64 rounding is off by at most about that)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import block_conditions, rel_dev

pytestmark = pytest.mark.gpu

RIDGE = {bfc.PREC_FP64: 0.0, bfc.PREC_C64: 2.0 ** -20}


def problem(r, few):
    """(n, L, b, lam, entries, start): `few` leaves slices empty and groups of
    one or two entries; else 32 entries per row or column group at the outer
    middle levels (a warp per group) and 16 at the inner one."""
    n, L, b = (96, 3, 12) if few else (128, 3, 16)
    i, j = synth.draw_pairs(n, 8192 if not few else 1500, 40 + r)
    if few:
        keep = (i // b != 2) | (j // b < 4)     # some slices lose their entries
        i, j = i[keep], j[keep]
    X = synth.random_factors(n, L, r, 900 + r)
    t = oracle.eval_entries(n, L, b, r, X, i, j)
    return n, L, b, 1e-1 if few else 1e-6, i, j, t, synth.random_factors(n, L, r, 300 + r)


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("r", range(2, 13))
def test_grouped_sweep_parity(r, few, prec):
    n, L, b, lam, i, j, t, X0 = problem(r, few)
    Xo, st_o = oracle.als_sweep(n, L, b, r, lam, X0, i, j, t, ridge_rel=RIDGE[prec])
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec, group_ratio=2.0) as c:
        assert all(c.level_groups(m)[1] for m in range(1, L + 1))
        c.set_factors(X0)
        st = c.sweep()
        Xg = c.get_factors()
    tol = 1e-10
    if prec == bfc.PREC_C64:
        kappa = max(float(v.max()) for v in block_conditions(X0, Xo, i, j, t, n, L, b, r, lam, 2.0 ** -20) if v.size)
        tol = max(1e-4, kappa * 2.0 ** -24)
    assert abs(st["objective"] - st_o["objective"]) <= tol * abs(st_o["objective"])
    xg = oracle.eval_entries(n, L, b, r, Xg, i, j)
    assert rel_dev(xg, oracle.eval_entries(n, L, b, r, Xo, i, j)) <= tol


@pytest.mark.parametrize("r", [3, 5, 6, 7, 10, 12])
def test_default_grouping_by_rank(r):
    """Default rule: every level whose groups are below 0.9 of the entries in
    FP64 and above rank 8; next to the tensor-core kernel the levels for which
    the cost model (ns per slice, entry and group by rank) sees a gain."""
    n, L, b, lam, i, j, t, _ = problem(r, False)
    S = 2 << L
    for prec in (bfc.PREC_FP64, bfc.PREC_C64):
        with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec) as c:
            for m in range(1, L + 1):
                groups, on = c.level_groups(m)
                if prec == bfc.PREC_FP64 or r > 8:
                    want = groups < 0.9 * len(i)
                else:
                    base = (1.0, -12.0, -25.0, -49.0, -8.5, 19.0, 19.0)[r - 2]
                    per = (0.025, 0.1, 0.1, 0.375, 0.4, 1.0, 1.25)[r - 2]
                    want = (base * S + 0.105 * len(i) - per * groups) * max(1.0, 152.0 / S) > 5000.0
                    want = want or (r in (4, 8) and groups < 0.1 * len(i))
                assert on == want
