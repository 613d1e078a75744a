"""The mat-vec's two FP64 forms on both sides of their rule (passes at ranks 5 ..
8 where the vectors fill the lanes, level by level otherwise), every split of
the levels, against the oracle (U = X V by its definition; FP64 1e-10)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu


def check(n, L, b, r, nvec):
    X = synth.random_factors(n, L, r, 11 + r)
    V = synth.SplitMix64(5).cnormal(n * nvec).reshape(n, nvec)
    i, j = synth.draw_pairs(n, min(20, n * n // 2), 3)
    with bfc.Completion(n, L, b, r, 1e-6, i, j, np.ones(len(i), complex), prec=bfc.PREC_FP64) as c:
        c.set_factors(X)
        c.profile(True)
        U = c.matvec(V)
        kernels = set(bfc.bfc_profile_read(c.ctx))
    assert ("mv_pass" in kernels) == (5 <= r <= 8 and nvec % 16 in (0, 14, 15))
    assert rel_dev(U, oracle.matvec(n, L, b, r, X, V)) <= 1e-10


@pytest.mark.parametrize("nvec", [13, 14, 16, 17])
@pytest.mark.parametrize("L", range(1, 11))
def test_level_splits(L, nvec):
    check(2 << L, L, 2, 6, nvec)


@pytest.mark.parametrize("r", [1, 4, 5, 8, 9, 12])
@pytest.mark.parametrize("nvec", [1, 16, 33, 64])
def test_ranks(r, nvec):
    check(96, 5, 3, r, nvec)
