"""Gauge fixing at the edges of its kernels: leaf blocks of 32 rows (the shared
memory kernel's largest) and 33, ranks 8 and 9 (a half and a whole warp per bond
group), rank-sized blocks, an odd number of bond groups.  Compared with
oracle.gauge; tolerance as in test_gpu_mlp.py (1e-10 of the largest entry), and
the orthogonality of the leaf blocks to 1e-14 r (twice the rounding of r
orthogonalized columns)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from oracle import gauge

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,b,r", [(64, 1, 32, 3), (66, 1, 33, 3), (128, 2, 32, 8), (132, 2, 33, 9), (144, 4, 9, 9),
                                     (96, 3, 12, 12), (128, 4, 8, 8), (40, 3, 5, 1), (24, 0, 24, 8), (31, 0, 31, 7),
                                     (33, 0, 33, 5)])
def test_canonical_gauge_shapes(n, L, b, r):
    rng = np.random.default_rng(n + 100 * r)
    P = oracle.num_params(n, L, b, r)
    X = rng.normal(size=P) + 1j * rng.normal(size=P)
    i, j = synth.draw_pairs(n, 200, 78)
    with bfc.Completion(n, L, b, r, 1e-6, i, j, np.ones(200, np.complex128), prec=bfc.PREC_FP64) as c:
        c.set_factors(X)
        c.canonicalize()
        C = c.get_factors()
    Co = gauge.canonicalize(n, L, b, r, X)
    assert np.max(np.abs(C - Co)) <= 1e-10 * np.max(np.abs(Co))
    Q = C[:n * r].reshape(n // b, b, r)
    err = np.einsum("pbi,pbj->pij", Q.conj(), Q) - np.eye(r)
    assert np.max(np.abs(err)) <= 1e-14 * r
