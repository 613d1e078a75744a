"""bfc_eval on host arrays that work pending on the context's stream still
writes: the call sees what that work leaves there, in the indices it checks as
in those it evaluates, and an address that the host cannot read is left to the
runtime.  Tolerance as in test_gpu_parity.py (FP64 1e-10)."""
import numpy as np
import pytest

import oracle
import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu

N, L, B, R = 96, 3, 12, 3


@pytest.mark.parametrize("late_bad", [False, True])
@pytest.mark.parametrize("m", [1, 8192, 8193, 70000])
def test_indices_written_by_pending_work(m, late_bad):
    torch = pytest.importorskip("torch")
    g = np.random.default_rng(m)
    i, j = g.integers(0, N, m).astype(np.int32), g.integers(0, N, m).astype(np.int32)
    bad = i.copy()
    bad[-1] = N
    factors = synth.random_factors(N, L, R, 4)
    first, late = (i, bad) if late_bad else (bad, i)
    pin = torch.from_numpy(first.copy()).pin_memory()
    src = torch.from_numpy(late).cuda()
    stream = torch.cuda.Stream()
    with bfc.Completion(N, L, B, R, 1e-6, [0], [0], [1.0 + 0j]) as c:
        c.set_factors(factors)
        c.eval(i, j)
        bfc.bfc_set_stream(c.ctx, stream.cuda_stream)
        out = np.full(m, 7.0 + 0j)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(20_000_000)            # about 10 ms before the indices arrive
            pin.copy_(src, non_blocking=True)
        if late_bad:
            with pytest.raises(bfc.BfcError, match="outside"):
                bfc.bfc_eval(c.ctx, pin, j, out)
            assert np.all(out == 7.0)
        else:
            bfc.bfc_eval(c.ctx, pin, j, out)
            assert rel_dev(out, oracle.eval_entries(N, L, B, R, factors, i, j)) <= 1e-10
