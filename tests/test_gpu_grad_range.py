"""The gradient's contraction at the edges of its row chunks, column tiles and number range,
against exactly summed products of the weights that the call itself returns.

The bound is that of an FP64 sum of n products taken one by one, (2 n + 4) 2^-53 sum |w d|,
plus the smallest subnormal once per product."""
import math

import numpy as np
import pytest

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


def _handle(B, n_u, rng, spread):
    """A handle whose last evaluation is of n_u samples: one determinant's energies stand in for them."""
    import torch
    from paper_2506_23809_gb300 import inputs as I
    ints = I.make_integrals(12, 24, 7)
    keys = I.rank_weighted_samples(12, 4, 4, n_u, seed=11)
    counts = np.maximum(1, np.exp2(rng.uniform(0, spread, n_u))).astype(np.int64)
    h = B.qc_eloc_create(ints.h, ints.eri, 0.0, 24, 8)
    ct = torch.from_numpy(counts).cuda()
    e, _ = B.qc_eloc_eval(h, B.keys_to_tensor(keys), ct, torch.from_numpy(I.lognormal_psi(n_u, 12)).cuda())
    return h, e, ct


def _split(a):
    c = 134217729.0 * a
    hi = c - (c - a)
    return hi, a - hi


def _exact(w, d):
    """Correctly rounded 2 sum Re(w d) and sum |w d| of one column (products split exactly)."""
    terms, mag = [], 0.0
    for x, y in ((w.real, d.real), (-w.imag, d.imag)):
        p = x * y
        (xh, xl), (yh, yl) = _split(x), _split(y)
        terms += [p, ((xh * yh - p) + xh * yl + xl * yh) + xl * yl]
        mag += np.abs(p).sum()
    return 2.0 * math.fsum(np.concatenate(terms)), 2.0 * mag


# rows: one, a partial load group, the edges of a 64-row chunk, and of a 256-row stage in use
# (above 131,072 rows of few columns a chunk has more than 256); columns: the edges of the 32- to
# 256-column tiles
@pytest.mark.parametrize("n_u,P", [(1, 1), (3, 33), (63, 32), (65, 31), (257, 300), (4000, 6145), (131_073, 65),
                                   (33_000, 640), (33_000, 768)])
def test_grad_edges(B, n_u, P):
    import torch
    rng = np.random.default_rng(n_u + P)
    h, e, ct = _handle(B, min(n_u, 4000), rng, 10)
    try:
        m = len(e)
        reps = -(-n_u // m)
        e, ct = e.repeat(reps)[:n_u].contiguous(), ct.repeat(reps)[:n_u].contiguous()
        D = torch.randn(n_u, P, dtype=torch.complex128, device="cuda")
        w, g = B.qc_eloc_grad(h, e, ct, D)
        _, g2 = B.qc_eloc_grad(h, e, ct, D, weights=False)
        assert torch.equal(g, g2)
        w, g = w.cpu().numpy(), g.cpu().numpy()
        for p in sorted({0, P // 2, P - 1, min(P - 1, 31), min(P - 1, 32)}):
            want, mag = _exact(w, D[:, p].cpu().numpy())
            assert abs(g[p] - want) <= (2 * n_u + 4) * 2.0 ** -53 * mag
    finally:
        B.qc_eloc_destroy(h)


@pytest.mark.parametrize("kind", ["wide", "rising", "falling", "cancel", "zeros", "subnormal", "huge"])
def test_grad_number_range(B, kind):
    import torch
    n_u, P = 700, 40
    rng = np.random.default_rng(5)
    h, e, ct = _handle(B, n_u, rng, 30)
    d = rng.normal(size=(n_u, P)) + 1j * rng.normal(size=(n_u, P))
    k = np.arange(n_u)[:, None] / n_u
    if kind == "wide":
        d *= np.exp2(rng.uniform(-200, 200, size=(n_u, P)))
    elif kind == "rising":
        d *= np.exp2(np.floor(-300 + 600 * k))
    elif kind == "falling":
        d *= np.exp2(np.floor(300 - 600 * k))
    elif kind == "zeros":
        d *= rng.random((n_u, P)) < 0.1
    elif kind == "subnormal":
        d *= 2.0 ** -1060
    elif kind == "huge":
        d *= 2.0 ** 900
    try:
        if kind == "cancel":  # a large pair that cancels, over small terms
            e[1], ct[1] = e[0], ct[0]
            d[1] = -d[0] * 2.0 ** 60
            d[0] *= 2.0 ** 60
        w, g = B.qc_eloc_grad(h, e, ct, torch.from_numpy(d).cuda())
        w, g = w.cpu().numpy(), g.cpu().numpy()
    finally:
        B.qc_eloc_destroy(h)
    scale = {"subnormal": 2.0 ** 400, "huge": 2.0 ** -400}.get(kind, 1.0)  # the oracle's splits stay in range
    for p in range(0, P, 7):
        want, mag = _exact(w, d[:, p] * scale)
        tiny = 2 * n_u * 2.0 ** -1074 * scale
        assert abs(g[p] * scale - want) <= (2 * n_u + 4) * 2.0 ** -53 * mag + 2 * tiny, (kind, p)


def test_grad_not_finite(B):
    """An infinity or NaN in a column reaches that column's sum as in FP64, and no other."""
    import torch
    n_u, P = 300, 64
    h, e, ct = _handle(B, n_u, np.random.default_rng(6), 4)
    D = torch.randn(n_u, P, dtype=torch.complex128, device="cuda")
    D[17, 3] = complex(0.0, float("inf"))
    D[18, 5] = complex(0.0, float("nan"))
    D[19, 40] = complex(float("-inf"), 0.0)
    try:
        w, g = B.qc_eloc_grad(h, e, ct, D)
    finally:
        B.qc_eloc_destroy(h)
    w, g = w.cpu().numpy(), g.cpu().numpy()
    assert g[3] == (-np.inf if w[17].imag > 0 else np.inf) and np.isnan(g[5])
    assert g[40] == (-np.inf if w[19].real > 0 else np.inf)
    assert np.isfinite(np.delete(g, [3, 5, 40])).all()
