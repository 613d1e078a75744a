"""Both sides of three lines of the sweep's dispatch, against the oracle: rows
per fiber from which k_outer_gram takes tiles (complex64), slices per level from
which k_mid_solve takes one warp, groups per level from which FP64 rank 2 sums
by threads.  Tolerances as in test_gpu_group_ranks.py: FP64 1e-10 relative on
entry values and the objective; complex64 max(1e-4, kappa_max 2^-24)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import block_conditions, rel_dev

pytestmark = pytest.mark.gpu

RIDGE = {bfc.PREC_FP64: 0.0, bfc.PREC_C64: 2.0 ** -20}


def check(n, L, b, r, count, prec, lam=1e-1, **kw):
    i, j = synth.draw_pairs(n, count, 30 + r)
    X = synth.random_factors(n, L, r, 900 + r)
    t = oracle.eval_entries(n, L, b, r, X, i, j)
    X0 = synth.random_factors(n, L, r, 300 + r)
    Xo, st_o = oracle.als_sweep(n, L, b, r, lam, X0, i, j, t, ridge_rel=RIDGE[prec])
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=prec, **kw) as c:
        groups = [c.level_groups(m) for m in range(1, L + 1)]
        c.set_factors(X0)
        st = c.sweep()
        Xg = c.get_factors()
    tol = 1e-10
    if prec == bfc.PREC_C64:
        kappa = max(float(v.max()) for v in block_conditions(X0, Xo, i, j, t, n, L, b, r, lam, 2.0 ** -20) if v.size)
        tol = max(1e-4, kappa * 2.0 ** -24)
    assert abs(st["objective"] - st_o["objective"]) <= tol * abs(st_o["objective"])
    assert rel_dev(oracle.eval_entries(n, L, b, r, Xg, i, j), oracle.eval_entries(n, L, b, r, Xo, i, j)) <= tol
    return groups


@pytest.mark.parametrize("side", [-1, 0])
@pytest.mark.parametrize("r", range(1, 13))
def test_outer_gram_forms(r, side):
    rows = (45, 45, 90, 90, 140, 140, 85, 55, 70, 40, 28, 28)[r - 1]
    n = 6 * (rows // 2)                         # up to 1024 fibers: a third of the rows
    check(n, 0, n, r, rows * n // 3 + side, bfc.PREC_C64)


@pytest.mark.parametrize("L", [9, 10])      # 1024 and 2048 slices; 8 per SM lie between
@pytest.mark.parametrize("r,prec", [(1, bfc.PREC_C64), (2, bfc.PREC_C64), (3, bfc.PREC_C64), (4, bfc.PREC_C64),
                                    (5, bfc.PREC_C64), (1, bfc.PREC_FP64), (2, bfc.PREC_FP64)])
def test_solve_warps(r, prec, L):
    b = max(2, r)
    check(b << L, L, b, r, 30 * (2 << L), prec)


def test_group_sums_fp64_rank2():
    groups = check(4096, 10, 4, 2, 45_000, bfc.PREC_FP64, group_ratio=2.0)
    few, many = [g for g, _ in groups if g <= 64 * 148], [g for g, _ in groups if g > 64 * 160]
    assert all(on for _, on in groups) and few and many     # warps and threads
