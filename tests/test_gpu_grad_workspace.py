"""The gradient's partials buffer grown by one call holds every later call of no more rows and columns:
with the next device allocation made to fail, such calls still succeed (as a captured one must)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,later", [((2433, 300), [(2432, 300), (2383, 300), (2433, 257), (16, 300)]),
                                         ((3000, 257), [(3000, 256), (3000, 33), (2999, 255)])])
def test_smaller_calls_do_not_allocate(first, later):
    import torch
    from paper_2506_23809_gb300 import binding as B
    from paper_2506_23809_gb300 import inputs as I
    n, _ = first
    ints = I.make_integrals(12, 24, 3)
    keys = I.rank_weighted_samples(12, 4, 4, n, seed=4)
    counts = torch.ones(n, dtype=torch.int64, device="cuda")
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 24, 8)
    try:
        e, _ = B.qc_eloc_eval(h, B.keys_to_tensor(keys), counts, torch.from_numpy(I.lognormal_psi(n, 5)).cuda())
        calls = [(a, torch.randn(a[0], a[1], dtype=torch.complex128, device="cuda")) for a in [first] + later]
        B.qc_eloc_grad(h, e[:n], counts[:n], calls[0][1])
        for (rows, _), d in calls[1:]:
            B.qc_test_fail_alloc(0)
            B.qc_eloc_grad(h, e[:rows], counts[:rows], d)
        torch.cuda.synchronize()
    finally:
        B.qc_test_fail_alloc(-1)
        B.qc_eloc_destroy(h)
