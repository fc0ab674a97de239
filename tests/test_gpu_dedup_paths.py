"""qc_dedup's two ways -- distinct keys counted in a hash table and sorted, or the whole stream
sorted -- at the sizes between them: streams around the counting threshold, more distinct keys
than the hash table holds, one key, keys of one and two words up to the all-ones pattern, and
tiles and merge passes that end ragged.  Integer work: equal to NumPy's unique, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pool(n, bits, rng):
    lo = rng.integers(0, 2**64, n, dtype=np.uint64)
    hi = rng.integers(0, 2**64, n, dtype=np.uint64)
    if bits < 64:
        lo &= np.uint64((1 << bits) - 1)
    if bits <= 64:
        hi[:] = 0
    elif bits < 128:
        hi &= np.uint64((1 << (bits - 64)) - 1)
    return np.stack([lo, hi], 1)


@pytest.mark.parametrize("n,bits,distinct", [(2047, 52, 2047), (2048, 52, 30), (2049, 128, 2049), (4097, 100, 4000),
                                             (131073, 64, 1), (524287, 52, 9000), (524288, 52, 9000),
                                             (200000, 128, 200000), (262145, 64, 262145), (524289, 64, 1), (600001, 128, 600001), (600001, 64, 350000), (700001, 76, 17),
                                             (1000003, 52, 400000), (2500000, 30, 2500000), (3000001, 120, 100000)])
def test_dedup_paths(n, bits, distinct):
    import torch
    from paper_2506_23809_gb300 import binding as B
    rng = np.random.default_rng(n + bits)
    pool = _pool(distinct, bits, rng)
    pool[0] = np.uint64(2**64 - 1) if bits == 128 else 0
    if bits == 64:
        pool[0, 0] = np.uint64(2**64 - 1)
    # a few keys make up most of the stream, the others come at least once
    idx = np.concatenate([np.arange(distinct), (rng.zipf(1.3, n) - 1)[:n - distinct] % distinct])
    raw = pool[rng.permutation(idx)]
    dt = np.dtype([("hi", np.uint64), ("lo", np.uint64)])
    v = np.empty(n, dt)
    v["hi"], v["lo"] = raw[:, 1], raw[:, 0]
    order = np.lexsort((v["lo"], v["hi"]))
    v = v[order]
    head = np.ones(n, bool)
    head[1:] = v[1:] != v[:-1]
    at = np.flatnonzero(head)
    k, c, u = B.qc_dedup(torch.from_numpy(raw.view(np.int64)).cuda(), bits)
    u = int(u.item())
    assert u == len(at)
    k = k[:u].cpu().numpy().view(np.uint64)
    assert np.array_equal(k[:, 0], v["lo"][at]) and np.array_equal(k[:, 1], v["hi"][at])
    assert np.array_equal(c[:u].cpu().numpy(), np.diff(np.append(at, n)))


def test_dedup_over_the_raw_keys():
    """Outputs laid over the raw stream (which is then gone) and a bad bit in a counted stream."""
    import torch
    from paper_2506_23809_gb300 import binding as B
    rng = np.random.default_rng(5)
    raw = _pool(5000, 52, rng)[rng.integers(0, 5000, 600000)]
    t = torch.from_numpy(raw.view(np.int64)).cuda()
    k, c, u = (x.clone() for x in B.qc_dedup(t, 52))
    n = int(u.item())
    k2, c2, u2 = B.qc_dedup(t, 52, keys_out=t)
    assert int(u2.item()) == n and torch.equal(k2[:n], k[:n]) and torch.equal(c2[:n], c[:n])
    raw[777, 1] = np.uint64(1)
    assert int(B.qc_dedup(torch.from_numpy(raw.view(np.int64)).cuda(), 52)[2].item()) == -1
