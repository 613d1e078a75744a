"""What the default rule for grouped levels (group_ratio 0) has to keep to,
whatever its constants: above rank 8 in complex64 the levels whose slices span
fewer than r rows or columns stay per entry (and the sweep is the oracle's),
next to the tensor cores they may group; fewer groups never turn a level's
grouping off; levels of one entry per group never group.  Tolerance of the
sweep as in test_gpu_group_ranks.py: max(1e-4, kappa_max 2^-24)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import block_conditions, rel_dev

pytestmark = pytest.mark.gpu


def decisions(n, L, b, r, i, j, prec):
    t = np.ones(len(i), np.complex128)
    with bfc.Completion(n, L, b, r, 1e-6, i, j, t, prec=prec) as c:
        return [c.level_groups(m) for m in range(1, L + 1)]


def test_short_slices_stay_per_entry_above_rank_8():
    n, L, b, r, lam = 128, 5, 4, 12, 1e-1
    i, j = synth.draw_pairs(n, 9000, 3)
    X = synth.random_factors(n, L, r, 1)
    t = oracle.eval_entries(n, L, b, r, X, i, j)
    X0 = synth.random_factors(n, L, r, 2)
    Xo, st_o = oracle.als_sweep(n, L, b, r, lam, X0, i, j, t, ridge_rel=2.0 ** -20)
    with bfc.Completion(n, L, b, r, lam, i, j, t, prec=bfc.PREC_C64) as c:
        on = [c.level_groups(m)[1] for m in range(1, L + 1)]
        c.set_factors(X0)
        st = c.sweep()
        Xg = c.get_factors()
    assert [bool(x) for x in on] == [b << min(m - 1, L - m) >= r for m in range(1, L + 1)]   # levels 1, 2, 4, 5: no
    kappa = max(float(v.max()) for v in block_conditions(X0, Xo, i, j, t, n, L, b, r, lam, 2.0 ** -20) if v.size)
    tol = max(1e-4, kappa * 2.0 ** -24)
    assert st["singular_slices"] == st_o["singular"] == 0
    assert abs(st["objective"] - st_o["objective"]) <= tol * abs(st_o["objective"])
    assert rel_dev(oracle.eval_entries(n, L, b, r, Xg, i, j), oracle.eval_entries(n, L, b, r, Xo, i, j)) <= tol


@pytest.mark.parametrize("r", range(2, 13))
def test_fewer_groups_never_turn_grouping_off(r):
    """The same number of entries on all rows and columns, on half and on a
    quarter of them: each level's groups fall."""
    n, L, b = 1024, 6, 16
    for prec in (bfc.PREC_FP64, bfc.PREC_C64):
        for count in (4000, 15_000, 50_000):
            seen = []
            for part in (1, 2, 4):
                i, j = synth.draw_pairs(n // part, count, 5)
                # every part-th row and column of each leaf: the slices keep their shares
                seen.append(decisions(n, L, b, r, i * part, j * part, prec))
            for m in range(L):
                ordered = sorted((s[m][0], bool(s[m][1])) for s in seen)
                for (ga, a), (gb, z) in zip(ordered, ordered[1:]):
                    assert a or not z, (prec, count, m + 1, ordered)


@pytest.mark.parametrize("r", range(2, 13))
def test_extremes(r):
    """One entry per group: never grouped.  All entries of a matrix (16 to 64 per
    group): every level grouped where the alternative is the per-entry CUDA-core
    kernel."""
    n, L, b = 128, 3, 16
    i = np.arange(n, dtype=np.int32)
    full = np.divmod(np.arange(n * n), n)
    for prec in (bfc.PREC_FP64, bfc.PREC_C64):
        assert not any(on for _, on in decisions(n, L, b, r, i, i, prec))
        if prec == bfc.PREC_FP64 or r > 8:
            got = decisions(n, L, b, r, full[0].astype(np.int32), full[1].astype(np.int32), prec)
            assert all(on for _, on in got)
