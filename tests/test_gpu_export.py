"""qc_eloc_export over its work items -- ranges of a sample's output that end anywhere in a class
-- in the documented order: every key, and elements of every class against the oracle's
Slater-Condon rules, for one and two key words, odd list lengths and both precisions."""
import itertools

import numpy as np
import pytest

from paper_2506_23809_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _order(K, key):
    """The connected keys (Python integers) of one sample in the documented order."""
    x = int(key[0]) | int(key[1]) << 64
    occ = [[k for k in range(K) if x >> (2 * k + s) & 1] for s in (0, 1)]
    vir = [[k for k in range(K) if not x >> (2 * k + s) & 1] for s in (0, 1)]
    single = [[1 << (2 * i + s) | 1 << (2 * a + s) for i in occ[s] for a in vir[s]] for s in (0, 1)]
    out = single[0] + single[1]
    for s in (0, 1):
        colex = lambda v: [(p, q) for n, q in enumerate(v) for p in v[:n]]  # noqa: E731
        bits = lambda pq: 1 << (2 * pq[0] + s) | 1 << (2 * pq[1] + s)  # noqa: E731
        out += [bits(u) | bits(w) for u, w in itertools.product(colex(occ[s]), colex(vir[s]))]
    out += [u | w for u, w in itertools.product(single[0], single[1])]
    return [x ^ d for d in out], len(single[0])


@pytest.mark.parametrize("n_orb,n_elec,n_u,prec", [(4, 2, 3, 0), (6, 4, 5, 0), (14, 6, 700, 0), (24, 22, 2, 0),
                                                   (34, 8, 9, 1), (52, 14, 3, 1), (64, 32, 2, 0), (66, 2, 4, 0),
                                                   (66, 20, 1, 1), (90, 12, 1, 0), (128, 64, 1, 0), (128, 6, 2, 1)])
def test_export_order_and_elements(orc, n_orb, n_elec, n_u, prec):
    from paper_2506_23809_gb300 import binding as B
    K, o = n_orb // 2, n_elec // 2
    ints = I.make_integrals(K, 8, 700 + n_orb)
    keys = (I.uniform_samples(K, o, o, n_u, 701) if n_orb <= 14 else
            I.rank_weighted_samples(K, o, o, n_u, 702, batch=4096))
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, n_orb, n_elec, prec)
    try:
        P = B.qc_eloc_pairs_per_sample(h)
        k, e, d = B.qc_eloc_export(h, B.keys_to_tensor(keys))
        only = B.qc_eloc_export(h, B.keys_to_tensor(keys), keys=False, diag=False)[1]
        k, e, d = k.cpu().numpy().view(np.uint64), e.cpu().numpy(), d.cpu().numpy()
        assert np.array_equal(e, only.cpu().numpy())
        rng = np.random.default_rng(703)
        # an element is at most 1 + 3 n_elec / 2 integrals, each stored with relative error u (FP32
        # only) and added in the storage precision
        u = 2.0 ** -24 if prec else 2.0 ** -53
        tol = (3 * n_elec + 4) ** 2 * u * max(np.abs(ints.h).max(), np.abs(ints.eri).max())
        for s in sorted({0, n_u // 2, n_u - 1}):
            want, ns = _order(K, keys[s])
            got = k[s * P:(s + 1) * P]
            assert len(want) == P
            assert np.array_equal(got[:, 0], np.array([w & (2**64 - 1) for w in want], dtype=np.uint64))
            assert np.array_equal(got[:, 1], np.array([w >> 64 for w in want], dtype=np.uint64))
            ends = [0, ns - 1, ns, 2 * ns - 1, min(2 * ns, P - 1), P - ns * ns - 1, P - ns * ns, P - 1]
            for j in ends + list(rng.integers(0, P, 60)):
                v, _ = orc.slater_condon(ints.h, ints.eri, 0.0, n_orb, keys[s], got[j])
                assert abs(e[s * P + j] - v) <= tol, (s, j, P)
            v, _ = orc.slater_condon(ints.h, ints.eri, 0.0, n_orb, keys[s], keys[s])
            assert abs(d[s] - v) <= 1e-12 * max(1.0, abs(v))
    finally:
        B.qc_eloc_destroy(h)
