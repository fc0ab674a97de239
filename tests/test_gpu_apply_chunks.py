"""A sample's E_loc from qc_eloc_apply is the same, bit for bit, in whatever chunk it comes: its sum's
order depends on the number of connected pairs alone, not on how many samples share the call.  Sizes
on both sides of each rule that hands the sum to warps, CTAs or clusters."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb,n_elec,chunks", [
    (14, 6, (1, 3, 1400, 5000)), (24, 12, (7, 1300, 2500)), (28, 20, (1, 40, 1369, 3000)), (34, 10, (5, 1500)),
    (40, 10, (2, 305, 761, 1600)), (46, 10, (1, 121, 304, 305, 1217)), (52, 14, (1, 121, 456, 457, 1217)),
    (76, 20, (1, 60, 243, 300, 457)), (90, 30, (1, 40, 76, 244)), (104, 40, (1, 40, 130)), (120, 60, (1, 39, 58))])
def test_same_bits_in_any_chunk(n_orb, n_elec, chunks):
    import torch
    from paper_2506_23809_gb300 import binding as B
    K, most = n_orb // 2, max(chunks)
    h = B.qc_eloc_create(np.zeros((K, K)), np.zeros((K, K, K, K)), 0.0, n_orb, n_elec)
    try:
        P = B.qc_eloc_pairs_per_sample(h)
        g = torch.Generator(device="cuda")
        g.manual_seed(n_orb)

        def draw(*s):
            return torch.randn(*s, dtype=torch.float64, device="cuda", generator=g)

        elems, diag = draw(most * P), draw(most)
        conn, psi = torch.view_as_complex(draw(most * P, 2)), torch.view_as_complex(draw(most, 2))
        counts = torch.ones(most, dtype=torch.int64, device="cuda")

        def apply(lo, hi):
            return B.qc_eloc_apply(h, psi[lo:hi], counts[lo:hi], elems[lo * P:hi * P], diag[lo:hi],
                                   conn[lo * P:hi * P]).clone()

        whole = torch.view_as_real(apply(0, most))
        for n in chunks:
            for lo in {0, (most - n) // 2, most - n}:
                assert torch.equal(torch.view_as_real(apply(lo, lo + n)), whole[lo:lo + n]), (n, lo)
        # any order of summing P products in FP64 (twice, for torch's own sum), a division, an addition
        t, u = elems[:P] * conn[:P], 2.0 ** -53
        want = complex(t.sum() / psi[0] + diag[0])
        bound = 2 * (P + 8) * u * float(t.abs().sum() / psi[0].abs()) + 8 * u * abs(want)
        assert abs(complex(*whole[0].tolist()) - want) <= bound
    finally:
        B.qc_eloc_destroy(h)
