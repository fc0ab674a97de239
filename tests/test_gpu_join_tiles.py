"""The join index at the edges of its sort's tiles and digit widths: rows against tables of sizes
on both sides of each rule, through the join and without it.  The connected sets and their phases
are equal; the energies are two orders of the same sum of at most h hits, each within
(h + 2) 2^-53 sum |H psi(x') / psi(x)| of it (bounded here by h times the largest term seen)."""
import itertools

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


@pytest.fixture(scope="module")
def sector():
    """Every determinant of 26 spin orbitals and 8 electrons as ascending one-word keys."""
    s = np.array([sum(1 << (2 * i) for i in c) for c in itertools.combinations(range(13), 4)], dtype=np.uint64)
    return np.sort((s[:, None] | (s[None, :] << np.uint64(1))).ravel())


# tiles of 1,024 items up to 262,144 rows, of 2,048 above; at 131,072 rows the slot keys go from
# 20 to 21 bits (two digits of 10, then of 11); a partial last tile
@pytest.mark.parametrize("n_table", [2_000, 65_536, 131_071, 131_073, 262_144, 262_145, 400_001])
def test_join_index_sizes(B, sector, n_table):
    import torch
    rng = np.random.default_rng(n_table)
    lo = np.sort(rng.choice(sector, n_table, replace=False))
    tkeys = np.stack([lo, np.zeros_like(lo)], 1)
    tpsi = I.lognormal_psi(n_table, 3)
    pick = np.sort(rng.choice(n_table, 257, replace=False))
    ints = I.make_integrals(13, 26, 5)
    counts = torch.ones(len(pick), dtype=torch.int64, device="cuda")
    got = []
    for join in (1, 2):
        h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 26, 8)
        try:
            B.qc_eloc_set_option(h, B.QC_OPT_JOIN, join)
            e, d = B.qc_eloc_eval(h, B.keys_to_tensor(tkeys[pick]), counts, torch.from_numpy(tpsi[pick]).cuda(),
                                  B.keys_to_tensor(tkeys), torch.from_numpy(tpsi).cuda(), diagnostics=True)
            assert B.qc_eloc_summary_read(h)["status"] == 0
            assert (B.qc_eloc_last_config(h)["kernel"] in (4, 5)) == (join == 2)
            got.append((e.cpu().numpy(), {k: v.cpu().numpy() for k, v in d.items()}))
        finally:
            B.qc_eloc_destroy(h)
    (a, da), (b, db) = got
    for k in da:
        assert np.array_equal(da[k], db[k]), k
    hits = da["hit_count"].astype(np.float64)
    term = (np.abs(ints.h).max() + 26 * np.abs(ints.eri).max()) * np.abs(tpsi).max() / np.abs(tpsi[pick])
    assert (np.abs(a - b) <= 2 * (hits + 2) * 2.0 ** -53 * (np.abs(a) + hits * term)).all()
