"""The Eq. 1 moments at the edges of the reduction's two forms (one cluster up to 8,192 rows, two
grid-wide passes above) and of its rows per thread, against numpy sums of the E_loc returned.

A sum of n rounded products, in any order, is off by at most (n + 1) 2^-53 sum |c E|."""
import numpy as np
import pytest

from paper_2506_23809_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_23809_gb300 import binding, build
    build.build()
    binding.load_library()
    return binding


@pytest.mark.parametrize("n_u", [1, 2, 255, 257, 2048, 2049, 8191, 8192, 8193, 20_000])
def test_moments(B, n_u):
    import torch
    ints = I.make_integrals(12, 24, 31)
    keys = I.rank_weighted_samples(12, 4, 4, n_u, seed=32)
    counts = I.zipf_counts(n_u, 50 * n_u, 33)
    psi = I.lognormal_psi(n_u, 34)
    if n_u > 2:
        psi[n_u - 1] = 0.0  # E_loc NaN: left out of every sum
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 24, 8)
    try:
        kt = B.keys_to_tensor(keys)
        ct, pt = torch.from_numpy(counts).cuda(), torch.from_numpy(psi).cuda()
        e, _ = B.qc_eloc_eval(h, kt, ct, pt)
        a = B.qc_eloc_summary_read(h)
        B.qc_eloc_eval(h, kt, ct, pt)
        b = B.qc_eloc_summary_read(h)
        neg = ct.clone()
        neg[n_u // 2] = -1
        B.qc_eloc_eval(h, kt, neg, pt)
        bad = B.qc_eloc_summary_read(h)
    finally:
        B.qc_eloc_destroy(h)
    assert a == b  # bit for bit
    e = e.cpu().numpy()
    ok = np.isfinite(e.real) & np.isfinite(e.imag)
    c, e = counts[ok].astype(np.longdouble), e[ok].astype(np.clongdouble)
    W, S = c.sum(), (c * e).sum()
    tol = (n_u + 2) * 2.0 ** -53 * float((c * abs(e)).sum())
    assert a["n_used"] == ok.sum() and a["w"] == float(W)
    assert abs(a["sum_ce_re"] - float(S.real)) <= tol and abs(a["sum_ce_im"] - float(S.imag)) <= tol
    m = S / W
    dm = 2.0 * tol / float(W)  # the mean's own rounding
    var = float((c * abs(e - m) ** 2).sum() / W)
    spread = float((c * abs(e - m)).sum() / W)
    assert abs(a["var"] - var) <= (n_u + 8) * 2.0 ** -53 * var + 2.0 * dm * spread + dm * dm
    assert bad["status"] == -12  # QC_ERR_COUNTS
