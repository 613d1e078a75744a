"""bfc_eval on host and device arrays around the sizes where its path changes
(4096: one copy of both index arrays; 65536: indices checked on the host), with
bad indices (the call is refused and the output left as it was), with an output
at an 8-byte address and one that overlaps the indices.  Tolerance as in
test_gpu_parity.py (FP64 1e-10)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu

N, L, B, R = 96, 3, 12, 3


def pairs(m):
    g = np.random.default_rng(m)
    return g.integers(0, N, m).astype(np.int32), g.integers(0, N, m).astype(np.int32)


@pytest.fixture(scope="module")
def factors():
    return synth.random_factors(N, L, R, 4)


@pytest.mark.parametrize("m", [1, 4095, 4096, 4097, 65536, 65537])
def test_host_arrays(factors, m):
    i, j = pairs(m)
    with bfc.Completion(N, L, B, R, 1e-6, [0], [0], [1.0 + 0j]) as c:
        c.set_factors(factors)
        got = c.eval(i, j)
        bad = i.copy()
        bad[-1] = N
        out = np.full(m, 7.0 + 0j)
        with pytest.raises(bfc.BfcError, match="outside"):
            bfc.bfc_eval(c.ctx, bad, j, out)
        assert np.all(out == 7.0)
    assert rel_dev(got, oracle.eval_entries(N, L, B, R, factors, i, j)) <= 1e-10


@pytest.mark.parametrize("where", ["aligned", "odd", "overlap"])
@pytest.mark.parametrize("m", [1, 5000])
def test_device_arrays(factors, where, m):
    torch = pytest.importorskip("torch")
    i, j = pairs(m)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    p = bfc.Params(n=N, L=L, b=B, r=R, lam=1e-6, prec=bfc.PREC_FP64, values_on_device=1)
    ctx = bfc.bfc_create(p, dev(np.zeros(1, np.int32)), dev(np.zeros(1, np.int32)), dev(np.ones(1, complex)))
    bfc.bfc_set_factors(ctx, dev(factors))
    buf = torch.full((2 * m + 3,), 7.0, dtype=torch.float64, device="cuda")
    out = buf[1:2 * m + 1] if where == "odd" else buf[:2 * m]
    di, dj = dev(i), dev(j)
    torch.cuda.synchronize()
    if where == "overlap":
        ints = buf.view(torch.int32)
        ints[:m].copy_(di)
        di = ints[:m]
    else:
        bad = di.clone()
        bad[0] = -1
        torch.cuda.synchronize()
        with pytest.raises(bfc.BfcError, match="outside"):
            bfc.bfc_eval(ctx, bad, dj, out)
        assert bool((buf == 7.0).all())
    torch.cuda.synchronize()
    bfc.bfc_eval(ctx, di, dj, out)
    got = out.cpu().numpy().copy().view(np.complex128)
    bfc.bfc_destroy(ctx)
    assert rel_dev(got, oracle.eval_entries(N, L, B, R, factors, i, j)) <= 1e-10
