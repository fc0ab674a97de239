"""Large products that cancel leave the small ones whole: the imaginary products' fixed-point sum
loses no bit of a product within its window to a larger one.

Rows of purely imaginary derivatives, two of which (equal weights, opposite derivatives, next to each
other in one thread's rows) cancel exactly.  Each remaining product is off by 2^-61 of itself at
most; then every chunk's sum, and the chunks', are FP64 sums of no more than n + 40 roundings."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", [0, 3, 101])
@pytest.mark.parametrize("bits", [20, 30, 40, 300])
def test_cancelling_pair(at, bits):
    import torch
    from paper_2506_23809_gb300 import binding as B
    from paper_2506_23809_gb300 import inputs as I
    n_u, P = 200, 300
    ints = I.make_integrals(12, 24, 7)
    counts = torch.from_numpy(I.zipf_counts(n_u, 50 * n_u, 13)).cuda()
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 24, 8)
    d = 1j * np.random.default_rng(bits).normal(size=(n_u, P))
    try:
        e, _ = B.qc_eloc_eval(h, B.keys_to_tensor(I.rank_weighted_samples(12, 4, 4, n_u, seed=11)), counts,
                              torch.from_numpy(I.lognormal_psi(n_u, 12)).cuda())
        e[at + 1], counts[at + 1] = e[at], counts[at]
        d[at] *= 2.0 ** bits
        d[at + 1] = -d[at]
        w, g = B.qc_eloc_grad(h, e, counts, torch.from_numpy(d).cuda())
    finally:
        B.qc_eloc_destroy(h)
    w, g = w.cpu().numpy(), g.cpu().numpy()
    assert w[at] == w[at + 1] and w[at].imag != 0
    rest = np.delete(np.arange(n_u), [at, at + 1])
    for p in range(P):
        x, y = -w.imag[rest], d.imag[rest, p]
        c = 134217729.0
        xh, yh = c * x - (c * x - x), c * y - (c * y - y)
        q = x * y
        low = ((xh * yh - q) + xh * (y - yh) + (x - xh) * yh) + (x - xh) * (y - yh)
        want = 2 * math.fsum(np.concatenate([q, low]))
        assert abs(g[p] - want) <= 2 * (n_u + 42) * 2.0 ** -53 * np.abs(q).sum(), (p, g[p], want)
