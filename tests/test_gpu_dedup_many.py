"""qc_dedup on streams with too many distinct keys to count, or near it: found by a sample before the
counting, or counted all the same (few orbitals: every key has a slot of its own).  Results equal to
NumPy's unique, exactly; and the call takes no longer than sorting the whole stream at once, which
outputs laid over the raw keys ask for (a tenth allowed for the sample and the launches)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _stream(n, bits, distinct, seed):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    pool = torch.randint(0, 1 << bits, (distinct,), device="cuda", generator=g)
    idx = torch.cat([torch.arange(distinct, device="cuda"),
                     torch.randint(0, distinct, (n - distinct,), device="cuda", generator=g)])
    low = pool[idx[torch.randperm(n, device="cuda", generator=g)]]
    return torch.stack([low, torch.zeros_like(low)], 1).contiguous()


@pytest.mark.parametrize("n,bits,distinct", [(524288, 20, 524288), (524289, 19, 300000), (1500000, 20, 1500000),
                                             (1500000, 21, 1500000), (2200000, 21, 2200000), (2200000, 22, 2200000),
                                             (3000000, 28, 600000), (3000000, 40, 900000), (3000000, 28, 1000000),
                                             (3000000, 52, 1500000), (3000000, 28, 3000000), (600000, 40, 600000)])
def test_values(n, bits, distinct):
    import torch
    from paper_2506_23809_gb300 import binding as B
    raw = _stream(n, bits, distinct, n + bits)
    k, c, u = B.qc_dedup(raw, bits)
    want, counts = torch.unique(raw[:, 0], return_counts=True)
    u = int(u.item())
    assert u == len(want) and torch.equal(k[:u, 0], want) and torch.equal(c[:u], counts) and not k[:u, 1].any()
    raw[n // 3, 0] |= 1 << bits
    assert int(B.qc_dedup(raw, bits)[2].item()) == -1


def test_few_of_many_are_counted():
    """A key that is a third of the stream, over a tail that the table holds: the sample must not mistake it."""
    import torch
    from paper_2506_23809_gb300 import binding as B
    raw = _stream(4000000, 44, 400000, 5)
    raw[::3] = raw[0]
    k, c, u = B.qc_dedup(raw, 44)
    want, counts = torch.unique(raw[:, 0], return_counts=True)
    u = int(u.item())
    assert u == len(want) and torch.equal(k[:u, 0], want) and torch.equal(c[:u], counts)


@pytest.mark.parametrize("n,bits,distinct", [(3000000, 20, 1500000), (3000000, 28, 1500000), (3000000, 28, 3000000),
                                             (3000000, 32, 3000000), (6000000, 36, 4000000)])
def test_time(n, bits, distinct):
    import torch
    from paper_2506_23809_gb300 import binding as B
    raw = _stream(n, bits, distinct, n)
    keep = raw.clone()
    keys, counts = torch.zeros_like(raw), torch.zeros(n, dtype=torch.int64, device="cuda")
    nu = torch.zeros(1, dtype=torch.int64, device="cuda")
    work = torch.empty(B.qc_dedup_workspace_bytes(n) + 256, dtype=torch.uint8, device="cuda")

    def best(out):
        times = []
        for _ in range(12):
            raw.copy_(keep)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            B.qc_dedup(raw, bits, out, counts, nu, work)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[2:])

    plain, whole = best(keys), best(raw)
    assert plain <= 1.1 * whole, (plain, whole)
