"""qc_eloc_apply over its splits -- a warp, 128 threads, 512 threads or a cluster of CTAs per
sample -- against the same sums in NumPy, at sizes on both sides of each rule and with sums that
do not divide by the threads or the cluster."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_orb,n_elec,n_u", [(4, 2, 3), (14, 6, 1), (14, 6, 5000), (24, 12, 7), (28, 20, 1300),
                                              (40, 10, 1216), (40, 10, 5001), (52, 14, 40), (52, 14, 301),
                                              (52, 14, 1300), (76, 20, 13), (90, 30, 1), (90, 30, 5)])
def test_apply_splits(n_orb, n_elec, n_u):
    import torch
    from paper_2506_23809_gb300 import binding as B
    K = n_orb // 2
    h = B.qc_eloc_create(np.zeros((K, K)), np.zeros((K, K, K, K)), 0.0, n_orb, n_elec)
    try:
        P = B.qc_eloc_pairs_per_sample(h)
        rng = np.random.default_rng(17 * n_u + P)
        elems, diag = rng.normal(size=n_u * P), rng.normal(size=n_u)
        conn = rng.normal(size=n_u * P) + 1j * rng.normal(size=n_u * P)
        psi = np.exp(rng.normal(size=n_u)) * np.exp(1j * rng.uniform(0, 6.28, size=n_u))
        up = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
        counts = up(np.ones(n_u, dtype=np.int64))
        args = (h, up(psi), counts, up(elems), up(diag), up(conn))
        got = B.qc_eloc_apply(*args).cpu().numpy()
        again = B.qc_eloc_apply(*args).cpu().numpy()
        assert np.array_equal(got.view(np.uint64), again.view(np.uint64))
        t = (elems * conn).reshape(n_u, P)
        want = diag + t.sum(1) / psi
        # any order of summing P products in FP64: P u sum |product| to first order (twice, for
        # NumPy's own sum), then a division and an addition
        u = 2.0 ** -53
        bound = 2 * (P + 8) * u * np.abs(t).sum(1) / np.abs(psi) + 8 * u * np.abs(want)
        assert np.all(np.abs(got - want) <= bound)
        assert B.qc_eloc_summary_read(h)["n_used"] == n_u
    finally:
        B.qc_eloc_destroy(h)
