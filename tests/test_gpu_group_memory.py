"""Memory of the group records: bounded (a level's slices run in batches), and
no reason to refuse a problem that fits without them.  The batched sums are the
same sums, so the sweep is compared with the per-entry kernel's: FP64 1e-10 on
the factors' entry values, as in test_gpu_parity.py."""
import numpy as np
import pytest

import paper_2510_17734_gb300 as bfc
import synth
from helpers import rel_dev

pytestmark = pytest.mark.gpu

n, L, B, R, LAM = 16384, 10, 16, 12, 1.0
MIB = 1 << 20
RECORD = 2736              # bytes of a group record at rank 12 in FP64


def data():
    i, j = synth.draw_pairs(n, 500_000, 9)
    return i, j, np.exp(1j * np.pi / 16 * np.hypot((i - j), 1.5 * n))


def free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def make(i, j, t, ratio):
    return bfc.Completion(n, L, B, R, LAM, i, j, t, prec=bfc.PREC_FP64, group_ratio=ratio)


def test_record_buffer_is_bounded():
    torch = pytest.importorskip("torch")
    i, j, t = data()
    X0 = synth.random_factors(n, L, R, 5)
    used, entries = {}, {}
    for ratio in (-1.0, 2.0):
        make(i, j, t, ratio).close()                     # modules and pools are there
        before = free(torch)
        with make(i, j, t, ratio) as c:
            used[ratio] = before - free(torch)
            groups = [c.level_groups(m) for m in range(1, L + 1)]
            c.set_factors(X0)
            c.sweep()
            entries[ratio] = c.eval(i[:20000], j[:20000])
    assert all(on for _, on in groups)
    # several batches: the largest level's records are more than the bound
    assert max(g for g, _ in groups) * RECORD > 512 * MIB
    # the bound, the groups' offsets (under 4 bytes per entry and level) and the allocator's granularity
    assert used[2.0] - used[-1.0] <= 256 * MIB + 4 * L * len(i) + 16 * MIB
    assert rel_dev(entries[2.0], entries[-1.0]) <= 1e-10


def test_fits_where_the_records_do_not():
    torch = pytest.importorskip("torch")
    i, j, t = data()
    X0 = synth.random_factors(n, L, R, 5)
    with make(i, j, t, 0.0) as c:                        # kernels loaded, both forms
        assert any(c.level_groups(m)[1] for m in range(1, L + 1))
        c.set_factors(X0)
        c.sweep()
    torch.cuda.empty_cache()
    before = free(torch)
    with make(i, j, t, -1.0) as c:
        need = before - free(torch)
        c.set_factors(X0)
        c.sweep()
        want = c.get_factors()
        alone = before - free(torch)
    # all but what the per-entry context needs and 100 to 196 MiB (records: 256)
    filler = None
    for spare in (100, 132, 164, 196):
        try:
            filler = torch.empty(free(torch) - max(need, alone) - spare * MIB, dtype=torch.uint8, device="cuda")
            break
        except torch.cuda.OutOfMemoryError:
            pass
    assert filler is not None
    try:
        with make(i, j, t, 0.0) as c:
            assert not any(c.level_groups(m)[1] for m in range(1, L + 1))
            c.set_factors(X0)
            c.sweep()
            assert np.array_equal(c.get_factors(), want)
    finally:
        del filler
        torch.cuda.empty_cache()
