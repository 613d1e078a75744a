"""The mat-vec's passes over several levels: every split of the levels (L = 1 ..
10), every rank, vector counts around the 16-lane and block edges, against the
oracle (U = X V by its definition).  Tolerances as in test_gpu_first_order.py."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu

TOL = {bfc.PREC_FP64: 1e-10, bfc.PREC_C64: 1e-4}


def check(n, L, b, r, nvec, prec):
    X = synth.random_factors(n, L, r, 11 + r)
    V = synth.SplitMix64(5).cnormal(n * nvec).reshape(n, nvec)
    i, j = synth.draw_pairs(n, min(20, n * n // 2), 3)
    with bfc.Completion(n, L, b, r, 1e-6, i, j, np.ones(len(i), complex), prec=prec) as c:
        c.set_factors(X)
        U = c.matvec(V)
    assert rel_dev(U, oracle.matvec(n, L, b, r, X, V)) <= TOL[prec]


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("L", range(1, 11))
def test_level_splits(L, prec):
    check(2 << L, L, 2, 3 if L % 2 else 4, 5, prec)


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("r", range(1, 13))
def test_every_rank(r, prec):
    check(96, 5, 3, r, 3, prec)


@pytest.mark.parametrize("prec", [bfc.PREC_FP64, bfc.PREC_C64])
@pytest.mark.parametrize("nvec", [1, 15, 16, 17, 33, 63, 64, 65, 130])
def test_vector_counts(nvec, prec):
    check(96, 5, 3, 8, nvec, prec)


@pytest.mark.parametrize("shift", [0, 8])
def test_device_vectors_any_alignment(shift):
    """Device vectors at 16-byte addresses are used in place, others are copied;
    the result may overwrite the input."""
    torch = pytest.importorskip("torch")
    n, L, b, r, nvec = 96, 5, 3, 4, 7
    X = synth.random_factors(n, L, r, 2)
    V = synth.SplitMix64(6).cnormal(n * nvec).reshape(n, nvec)
    i, j = synth.draw_pairs(n, 20, 3)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    p = bfc.Params(n=n, L=L, b=b, r=r, lam=1e-6, prec=bfc.PREC_FP64, values_on_device=1)
    ctx = bfc.bfc_create(p, dev(i), dev(j), dev(np.ones(len(i), complex)))
    buf = torch.zeros(n * nvec * 16 + 64, dtype=torch.uint8, device="cuda")
    flat = buf[shift:shift + n * nvec * 16].view(torch.float64)
    flat.copy_(dev(V.ravel().view(np.float64)))
    bfc.bfc_set_factors(ctx, dev(X))
    torch.cuda.synchronize()
    bfc.bfc_matvec(ctx, nvec, flat, flat)
    U = flat.cpu().numpy().view(np.complex128).reshape(n, nvec)
    bfc.bfc_destroy(ctx)
    assert rel_dev(U, oracle.matvec(n, L, b, r, X, V)) <= 1e-10
