"""An export of the diagonal alone does not walk the connected pairs: its values are those of the whole
export, and it takes less than a quarter of the time of the elements (it reads and writes 1 / 2,625 of
their bytes; what is left is each sample's set-up)."""
import pytest

from paper_2506_23809_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_diagonal_alone():
    import torch
    from paper_2506_23809_gb300 import binding as B
    ints = I.make_integrals(20, 8, 7)
    keys = B.keys_to_tensor(I.rank_weighted_samples(20, 5, 5, 3000, 5)).repeat(7, 1)[:20_000].contiguous()
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 40, 10)

    def best(**a):
        times = []
        for _ in range(10):
            b, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            b.record()
            out = B.qc_eloc_export(h, keys, **a)
            e.record()
            torch.cuda.synchronize()
            times.append(b.elapsed_time(e))
        return min(times[2:]), out

    try:
        te, (_, _, none) = best(keys=False, diag=False)
        td, (_, _, diag) = best(keys=False, elems=False)
        whole = B.qc_eloc_export(h, keys)[2]
    finally:
        B.qc_eloc_destroy(h)
    assert none is None and torch.equal(diag, whole)
    assert td <= 0.25 * te, (td, te)
