"""The work that a user of the library has it do, as cases to be timed: local energies of sampled
bitstrings (alone, one rank's rows against the whole table, many molecules in one step), the energy
gradient, the sample table from a raw stream, and the accurate energy's export and apply.

Inputs are drawn on the GPU with the shapes and laws of the repository's own workloads: integrals
with 8-fold symmetry from random factors, bitstrings weighted by excitation rank (0.3**k against the
Aufbau determinant) or uniform in a small sector, Zipf(1.2) counts, log-normal complex amplitudes.
"""
import math

import numpy as np
import torch

from paper_2506_23809_gb300 import binding as B

SUMMARY_WORDS = 12  # a qc_eloc_summary is 6 doubles, 5 unsigned counters and two 32-bit words


def listed():
    return [
        # one small active space per optimisation step of a toy or a unit problem: launches and latency
        {"name": "eval_n14_e6_u1k", "op": "eval", "n_orb": 14, "n_elec": 6, "n_u": 1000, "fp32": False},
        # a diatomic in a minimal basis (20 spin orbitals), half of its sector sampled
        {"name": "eval_n20_e14_u7200", "op": "eval", "n_orb": 20, "n_elec": 14, "n_u": 7200, "fp32": False},
        # a transition-metal cluster's active space: more electrons than holes, dense connections
        {"name": "eval_n40_e30_u100k", "op": "eval", "n_orb": 40, "n_elec": 30, "n_u": 100_000, "fp32": False},
        # the benchmark's default workload
        {"name": "eval_n52_e14_u100k", "op": "eval", "n_orb": 52, "n_elec": 14, "n_u": 100_000, "fp32": False},
        # the precision form: FP32 integrals with compensated sums
        {"name": "eval_n76_e20_u200k_fp32", "op": "eval", "n_orb": 76, "n_elec": 20, "n_u": 200_000, "fp32": True},
        # the largest molecule of the paper's sweep, two-word keys and a 104 MB integral tensor
        {"name": "eval_n120_e60_u100k", "op": "eval", "n_orb": 120, "n_elec": 60, "n_u": 100_000, "fp32": False},
        # one rank of a data-parallel job: its own rows against the table of all ranks' samples
        {"name": "rows_n52_e14_u50001_of_200k", "op": "rows", "n_orb": 52, "n_elec": 14, "n_u": 50_001,
         "n_table": 200_000, "fp32": False},
        # several molecules (a bond scan, a data set) in one persistent launch
        {"name": "batch_16_molecules", "op": "batch", "n_mol": 16, "mol_seed": 6400, "fp32": True},
        # the gradient of one optimisation step: log-derivative rows of a small network
        {"name": "grad_u100k_p4096", "op": "grad", "n_u": 100_000, "n_par": 4096},
        # the sample table from ten million raw draws of the sampler
        {"name": "dedup_n52_10m", "op": "dedup", "n_orb": 52, "n_elec": 14, "n_raw": 10_000_000, "n_u": 100_000},
        # accurate energy: every connected bitstring of a chunk of samples, for the network to evaluate
        {"name": "export_n52_e14_u10k", "op": "export", "n_orb": 52, "n_elec": 14, "n_u": 10_000, "fp32": False},
        # accurate energy: the sums against the network's amplitudes; a large molecule's chunk is few samples
        {"name": "apply_n120_e60_u200", "op": "apply", "n_orb": 120, "n_elec": 60, "n_u": 200},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sector(n_orb, n_elec):
    return math.comb(n_orb // 2, n_elec // 2) ** 2


def _pairs(n_orb, n_elec):
    o, v = n_elec // 2, (n_orb - n_elec) // 2
    same = math.comb(o, 2) * math.comb(v, 2)
    return 2 * o * v + 2 * same + (o * v) ** 2


def _shape(rng, lo, hi):
    """Spin orbitals lo..hi and an even electron number from a quarter to three quarters of them."""
    n_orb = 2 * rng.randint(lo // 2, hi // 2)
    n_elec = 2 * rng.randint(max(1, n_orb // 8), max(1, (3 * n_orb) // 8))
    return n_orb, n_elec


def draw(rng):
    op = rng.choice(["eval"] * 5 + ["rows", "batch", "grad", "dedup", "export", "apply"])
    if op in ("eval", "rows"):
        n_orb, n_elec = _shape(rng, 14, 120)
        most = max(1, min(100_000, _sector(n_orb, n_elec) // 2))
        n_u = _log(rng, min(1000, most), most)
        c = {"op": op, "n_orb": n_orb, "n_elec": n_elec, "n_u": n_u, "fp32": rng.random() < 0.4}
        if op == "rows":
            c["n_table"] = n_u
            c["n_u"] = max(1, n_u // rng.randint(2, 8))
        return c
    if op == "batch":
        return {"op": op, "n_mol": rng.randint(2, 16), "mol_seed": rng.randrange(1 << 20), "fp32": rng.random() < 0.6}
    if op == "grad":
        n_u = _log(rng, 1000, 100_000)
        return {"op": op, "n_u": n_u, "n_par": _log(rng, 64, min(65_536, 400_000_000 // n_u))}
    if op == "dedup":
        n_orb, n_elec = _shape(rng, 20, 120)
        n_raw = _log(rng, 20_000, 10_000_000)
        most = max(1, min(n_raw, 400_000, _sector(n_orb, n_elec) // 2))
        return {"op": op, "n_orb": n_orb, "n_elec": n_elec, "n_raw": n_raw, "n_u": _log(rng, min(1000, most), most)}
    n_orb, n_elec = _shape(rng, 20, 120)
    p = _pairs(n_orb, n_elec)
    most = max(1, min(200_000_000 // p, 20_000, max(1, _sector(n_orb, n_elec) // 2)))
    c = {"op": op, "n_orb": n_orb, "n_elec": n_elec, "n_u": _log(rng, max(1, most // 64), most)}
    if op == "export":
        c["fp32"] = rng.random() < 0.3
    return c


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _integrals(K, g):
    """h (K x K) and (pq|rs) (K^4) on the GPU."""
    idx = torch.arange(K, device="cuda")
    off = torch.randn(K, K, dtype=torch.float64, device="cuda", generator=g)
    off = torch.triu(off * 0.1 * torch.exp(-(idx[:, None] - idx[None, :]).abs() / 2.0), 1)
    h = off + off.T
    h[idx, idx] = -(1.0 + 4.0 * torch.rand(K, dtype=torch.float64, device="cuda", generator=g))
    iu, ju = torch.triu_indices(K, K, device="cuda")
    L = 0.3 * torch.randn(2 * K, len(iu), dtype=torch.float64, device="cuda", generator=g)
    V = L.T @ L
    V = 0.5 * (V + V.T)
    pair = torch.zeros(K, K, dtype=torch.int64, device="cuda")
    pair[iu, ju] = torch.arange(len(iu), device="cuda")
    pair[ju, iu] = pair[iu, ju]
    flat = pair.reshape(-1)
    return h.contiguous(), V[flat][:, flat].reshape(K, K, K, K).contiguous()


def _strings(occ):
    """Occupation rows (bool, n x K with K <= 60) as integers."""
    w = torch.ones(occ.shape[1], dtype=torch.int64, device=occ.device) << torch.arange(occ.shape[1], device=occ.device)
    return (occ.to(torch.int64) * w).sum(1)


def _subset(n, k, g):
    """Row-wise random subsets of k[m] out of n."""
    r = torch.rand(len(k), n, dtype=torch.float64, device="cuda", generator=g)  # no ties
    if n == 0:
        return r.bool()
    thr = r.sort(1).values.gather(1, (k - 1).clamp(min=0)[:, None])
    return (r <= thr) & (k > 0)[:, None]


def _spread(w):
    """Bit k of a 32-bit integer to bit 2k."""
    w = (w | (w << 16)) & 0x0000FFFF0000FFFF
    w = (w | (w << 8)) & 0x00FF00FF00FF00FF
    w = (w | (w << 4)) & 0x0F0F0F0F0F0F0F0F
    w = (w | (w << 2)) & 0x3333333333333333
    return (w | (w << 1)) & 0x5555555555555555


def _keys(a, b):
    """Interleaved two-word keys of alpha and beta strings."""
    lo = _spread(a & 0xFFFFFFFF) | (_spread(b & 0xFFFFFFFF) << 1)
    hi = _spread(a >> 32) | (_spread(b >> 32) << 1)
    return torch.stack([lo, hi], 1)


def _unique_sorted(a, b):
    """Distinct (alpha, beta) pairs in ascending key order, with each one's first index."""
    k = _keys(a, b)
    sign = -(1 << 63)
    o = torch.sort(k[:, 0] ^ sign, stable=True).indices
    o = o[torch.sort(k[o, 1], stable=True).indices]
    k = k[o]
    new = torch.ones(len(o), dtype=torch.bool, device="cuda")
    new[1:] = (k[1:] != k[:-1]).any(1)
    return o[new]


def _samples(K, o, n_u, g):
    """n_u distinct (alpha, beta) strings, ascending by key. A small sector's are uniform; else rank k
    against the Aufbau determinant has weight 0.3**k, its alpha-beta split weighted by determinants
    (draws after the first batch leave out ranks 0 and 1, of which nearly all are there by then)."""
    v = K - o
    if _sector(2 * K, 2 * o) <= 1 << 18:
        import itertools
        s = torch.tensor([sum(1 << i for i in c) for c in itertools.combinations(range(K), o)], device="cuda")
        p = torch.randperm(len(s) ** 2, device="cuda", generator=g)[:n_u]
        a, b = s[p // len(s)], s[p % len(s)]
        u = _unique_sorted(a, b)
        return a[u], b[u]
    kmax = min(o, v)
    ks = [(ka, kb) for ka in range(kmax + 1) for kb in range(kmax + 1)]
    nd = [float(math.comb(o, ka) * math.comb(v, ka)) * float(math.comb(o, kb) * math.comb(v, kb)) for ka, kb in ks]
    per = {}
    for (ka, kb), n in zip(ks, nd):
        per[ka + kb] = per.get(ka + kb, 0.0) + n
    split = torch.tensor(ks, device="cuda")
    a = b = torch.empty(0, dtype=torch.int64, device="cuda")
    first = True
    while True:
        w = [(0.3 ** (ka + kb)) * n / per[ka + kb] if first or ka + kb >= 2 else 0.0 for (ka, kb), n in zip(ks, nd)]
        first = False
        cum = torch.tensor(w, dtype=torch.float64, device="cuda").cumsum(0)
        m = 4 * n_u + 1024
        r = torch.rand(m, dtype=torch.float64, device="cuda", generator=g) * cum[-1]
        k = split[torch.searchsorted(cum, r, right=True).clamp(max=len(ks) - 1)]
        new = []
        for s in (0, 1):
            occ = torch.cat([~_subset(o, k[:, s], g), _subset(v, k[:, s], g)], 1)
            new.append(_strings(occ))
        a, b = torch.cat([a, new[0]]), torch.cat([b, new[1]])
        u = _unique_sorted(a, b)
        if len(u) >= n_u:
            u = u.sort().values[:n_u]
            a, b = a[u], b[u]
            u = _unique_sorted(a, b)
            return a[u], b[u]
        u = u.sort().values
        a, b = a[u], b[u]


def _counts(n_u, total, g):
    """Zipf(1.2) over a random order, each at least 1."""
    w = torch.arange(1, n_u + 1, dtype=torch.float64, device="cuda") ** -1.2
    w = w[torch.randperm(n_u, device="cuda", generator=g)]
    return 1 + torch.floor(w / w.sum() * (total - n_u)).to(torch.int64)


def _psi(shape, g):
    la = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)
    ph = torch.rand(shape, dtype=torch.float64, device="cuda", generator=g) * (2 * math.pi)
    return torch.polar(torch.exp(la), ph)


class _Mol:
    """One molecule's inputs: integrals, strings, keys, counts and amplitudes."""

    def __init__(self, n_orb, n_elec, n_u, seed, salt=0, n_table=0):
        g = _gen(seed, salt)
        self.n_orb, self.n_elec, K, o = n_orb, n_elec, n_orb // 2, n_elec // 2
        self.h, self.eri = _integrals(K, g)
        self.ta, self.tb = _samples(K, o, n_table or n_u, g)
        self.tpsi = _psi(n_table or n_u, g)
        pick = None
        if n_table:
            pick = torch.randperm(n_table, device="cuda", generator=g)[:n_u].sort().values
        self.a, self.b = (self.ta, self.tb) if pick is None else (self.ta[pick], self.tb[pick])
        self.psi = self.tpsi if pick is None else self.tpsi[pick].contiguous()
        self.keys = _keys(self.a, self.b)
        self.tkeys = self.keys if pick is None else _keys(self.ta, self.tb)
        self.counts = _counts(n_u, 100 * n_u, g)

    def handle(self, fp32, mode=B.QC_SAMPLE):
        return B.qc_eloc_create(self.h.cpu().numpy(), self.eri.cpu().numpy(), 0.0, self.n_orb, self.n_elec,
                                B.QC_FP32_COMP if fp32 else B.QC_FP64, mode)


class _State(dict):
    """What a user's program keeps; its handles go with it."""

    def __del__(self):
        if self.get("batch") is not None:
            B.qc_batch_destroy(self["batch"])
        for h in self.get("handles", []):
            B.qc_eloc_destroy(h)


def _molecules(case, seed):
    """The shapes of a batch (spin orbitals 24..120, samples 1e3..1e5, at most a quarter of the sector)."""
    r = np.random.default_rng(case["mol_seed"])
    mols = []
    for m in range(case["n_mol"]):
        n = 2 * int(r.integers(12, 61))
        ne = n // 2 - 2 * int(r.integers(0, n // 4 + 1))
        ne = max(2, ne - ne % 2)
        n_u = min(int(round(10 ** r.uniform(3.0, 5.0))), max(1, _sector(n, ne) // 4))
        mols.append(dict(n_orb=n, n_elec=ne, n_u=n_u, seed=seed, salt=100 + m))
    return mols


GRAD_SHAPE = (28, 20)  # the gradient's own energies: a small system with enough determinants


def prepare(case, seed):
    op = case["op"]
    s = _State(op=op)
    if op in ("eval", "rows"):
        m = _Mol(case["n_orb"], case["n_elec"], case["n_u"], seed, n_table=case.get("n_table", 0))
        h = m.handle(case["fp32"])
        s.update(handles=[h], keys=m.keys, counts=m.counts, psi=m.psi)
        if op == "rows":
            s.update(tkeys=m.tkeys, tpsi=m.tpsi)
        B.qc_eloc_reserve(h, case["n_u"], case.get("n_table", case["n_u"]))
    elif op == "batch":
        s["handles"], s["eloc"], mols = [], [], []
        for q in _molecules(case, seed):
            m = _Mol(**q)
            mols.append((m.keys, m.counts, m.psi))
            s["handles"].append(m.handle(case["fp32"]))
        s["batch"] = B.qc_batch_create(s["handles"])
        for i, (k, c, p) in enumerate(mols):
            s["eloc"].append(torch.zeros(len(k), dtype=torch.complex128, device="cuda"))
            B.qc_batch_set_inputs(s["batch"], i, k, c, p, s["eloc"][i])
    elif op == "grad":
        m = _Mol(*GRAD_SHAPE, case["n_u"], seed)
        h = m.handle(False)
        eloc, _ = B.qc_eloc_eval(h, m.keys, m.counts, m.psi)
        d = torch.randn(case["n_u"], case["n_par"], 2, dtype=torch.float64, device="cuda", generator=_gen(seed, 7))
        s.update(handles=[h], eloc=eloc, counts=m.counts, dconj=torch.view_as_complex(d))
    elif op == "dedup":
        s.update(_raw(case, seed))
        n = case["n_raw"]
        s.update(n_orb=case["n_orb"], keys=torch.zeros(n, 2, dtype=torch.int64, device="cuda"),
                 counts=torch.zeros(n, dtype=torch.int64, device="cuda"),
                 n_unique=torch.zeros(1, dtype=torch.int64, device="cuda"),
                 work=torch.empty(B.qc_dedup_workspace_bytes(n) + 256, dtype=torch.uint8, device="cuda"))
    elif op == "export":
        m = _Mol(case["n_orb"], case["n_elec"], case["n_u"], seed)
        s.update(handles=[m.handle(case["fp32"], B.QC_FULL)], keys=m.keys)
    elif op == "apply":
        m = _Mol(case["n_orb"], case["n_elec"], case["n_u"], seed)
        s.update(handles=[m.handle(False, B.QC_FULL)], counts=m.counts, psi=m.psi, **_conn(case, seed))
    return s


def _raw(case, seed):
    """A sampler's raw stream: every determinant at least once, Zipf multiplicities, any order."""
    g = _gen(seed, 0)
    a, b = _samples(case["n_orb"] // 2, case["n_elec"] // 2, case["n_u"], g)
    n, n_u = case["n_raw"], case["n_u"]
    c = _counts(n_u, n, g)
    idx = torch.repeat_interleave(torch.arange(n_u, device="cuda"), c)
    more = torch.randint(0, n_u, (n - len(idx),), device="cuda", generator=g)
    idx = torch.cat([idx, more])
    idx = idx[torch.randperm(n, device="cuda", generator=g)]
    return {"raw": _keys(a, b)[idx].contiguous()}


def _conn(case, seed):
    """Elements, diagonal and amplitudes on the connected set, as the export and a network give them."""
    g = _gen(seed, 9)
    n, p = case["n_u"], _pairs(case["n_orb"], case["n_elec"])
    elems = 0.1 * torch.randn(n * p, dtype=torch.float64, device="cuda", generator=g)
    diag = -20.0 + torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    return {"elems": elems, "diag": diag, "conn": torch.view_as_complex(
        torch.randn(n * p, 2, dtype=torch.float64, device="cuda", generator=g))}


# ----------------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------------
def _summary(buf):
    """The page-locked summaries: moments and counters (the library fills them on the stream)."""
    f = buf.view(torch.float64).view(-1, SUMMARY_WORDS)
    i = buf.view(torch.int64).view(-1, SUMMARY_WORDS)
    w = buf.view(torch.int32).view(-1, 2 * SUMMARY_WORDS)
    return {"moments": f[:, :6], "counters": i[:, 6:11], "status": w[:, 22:24]}


def run(s):
    op = s["op"]
    if op == "eval":
        h = s["handles"][0]
        eloc, _ = B.qc_eloc_eval(h, s["keys"], s["counts"], s["psi"])
        return {"eloc": eloc, **_summary(h.summary_buf)}
    if op == "rows":
        h = s["handles"][0]
        eloc, _ = B.qc_eloc_eval(h, s["keys"], s["counts"], s["psi"], s["tkeys"], s["tpsi"])
        return {"eloc": eloc, **_summary(h.summary_buf)}
    if op == "batch":
        B.qc_batch_eval(s["batch"])
        return {"eloc": s["eloc"], **_summary(s["batch"].summary_buf)}
    if op == "grad":
        w, g = B.qc_eloc_grad(s["handles"][0], s["eloc"], s["counts"], s["dconj"])
        return {"w": w, "g": g}
    if op == "dedup":
        B.qc_dedup(s["raw"], s["n_orb"], s["keys"], s["counts"], s["n_unique"], s["work"])
        return {"keys": s["keys"], "counts": s["counts"], "n_unique": s["n_unique"]}
    if op == "export":
        k, e, d = B.qc_eloc_export(s["handles"][0], s["keys"])
        return {"keys": k, "elems": e, "diag": d}
    h = s["handles"][0]
    eloc = B.qc_eloc_apply(h, s["psi"], s["counts"], s["elems"], s["diag"], s["conn"])
    return {"eloc": eloc, **_summary(h.summary_buf)}


# ----------------------------------------------------------------------------------------------
# the least a pass has to do
# ----------------------------------------------------------------------------------------------
def _eval_bytes(n_orb, n_u, n_table, fp32):
    """Samples, amplitudes and counts read, energies written, a caller's table and the integrals read."""
    K = n_orb // 2
    return n_u * (16 + 16 + 8 + 16) + n_table * 32 + (K ** 4 + K ** 2) * (4 if fp32 else 8)


def work(case):
    op = case["op"]
    if op in ("eval", "rows"):
        # operations: the diagonal's pair terms (the connected terms depend on the samples)
        return {"bytes": _eval_bytes(case["n_orb"], case["n_u"], case.get("n_table", 0), case["fp32"]),
                "flops": case["n_u"] * case["n_elec"] ** 2}
    if op == "batch":
        ms = _molecules(case, 0)
        return {"bytes": sum(_eval_bytes(m["n_orb"], m["n_u"], 0, case["fp32"]) for m in ms),
                "flops": sum(m["n_u"] * m["n_elec"] ** 2 for m in ms)}
    if op == "grad":
        n, p = case["n_u"], case["n_par"]
        return {"bytes": 16 * n * p + n * (16 + 8 + 16) + 8 * p, "flops": 4 * n * p}
    if op == "dedup":
        return {"bytes": 16 * case["n_raw"] + 24 * case["n_u"], "flops": 0}
    n, p = case["n_u"], _pairs(case["n_orb"], case["n_elec"])
    if op == "export":
        return {"bytes": 24 * n * p + 24 * n + (case["n_orb"] // 2) ** 4 * (4 if case["fp32"] else 8), "flops": n * p}
    return {"bytes": 24 * n * p + 48 * n, "flops": 4 * n * p}


# ----------------------------------------------------------------------------------------------
# the same in plain 64-bit torch
# ----------------------------------------------------------------------------------------------
def _pop(x):
    """Set bits of non-negative integers below 2**62."""
    x = x - ((x >> 1) & 0x5555555555555555)
    x = (x & 0x3333333333333333) + ((x >> 2) & 0x3333333333333333)
    x = (x + (x >> 4)) & 0x0F0F0F0F0F0F0F0F
    x = x + (x >> 8)
    x = x + (x >> 16)
    return (x + (x >> 32)) & 127


def _bit(m):
    """Position of the only set bit."""
    return (torch.frexp(m.double())[1] - 1).to(torch.int64)


def _occupied_between(A, B_, p, q, spin):
    """Occupied spin orbitals strictly between spatial orbitals p and q of one spin, in the interleaved order."""
    lo, hi = torch.minimum(p, q), torch.maximum(p, q)
    one = torch.ones_like(lo)
    same = (one << hi) - (one << (lo + 1))
    other = (one << hi) - (one << lo) if spin == 0 else (one << (hi + 1)) - (one << (lo + 1))
    s, t = (A, B_) if spin == 0 else (B_, A)
    return _pop(s & same) + _pop(t & other)


def _sign(n):
    return 1.0 - 2.0 * (n & 1).double()


class _H:
    """Slater-Condon elements of 64-bit integrals on the GPU."""

    def __init__(self, h, eri):
        self.K = K = h.shape[0]
        self.h, self.eri = h, eri.reshape(-1)
        self.J = torch.einsum("kkll->kl", eri).contiguous()
        self.X = self.J - torch.einsum("kllk->kl", eri)
        self.Jt = torch.einsum("aikk->aik", eri).reshape(K * K, K).contiguous()
        self.Xt = torch.einsum("akki->aik", eri).reshape(K * K, K).contiguous()

    def occ(self, S):
        return ((S[:, None] >> torch.arange(self.K, device="cuda")) & 1).double()

    def diag(self, A, B_):
        a, b = self.occ(A), self.occ(B_)
        d = (a + b) @ self.h.diagonal()
        return d + 0.5 * (((a @ self.X) * a).sum(1) + ((b @ self.X) * b).sum(1)) + ((a @ self.J) * b).sum(1)

    def single(self, A, B_, i, a, spin):
        e = torch.empty(len(i), dtype=torch.float64, device="cuda")
        for c in range(0, len(i), 1 << 20):
            c = slice(c, c + (1 << 20))
            oa, ob, at = self.occ(A[c]), self.occ(B_[c]), a[c] * self.K + i[c]
            e[c] = self.h.reshape(-1)[at] + ((oa + ob) * self.Jt[at]).sum(1) - ((oa if spin == 0 else ob) * self.Xt[at]).sum(1)
        return e * _sign(_occupied_between(A, B_, i, a, spin))

    def _int(self, a, i, b, j):
        return self.eri[((a * self.K + i) * self.K + b) * self.K + j]

    def double(self, A, B_, i, a, j, b, s1, s2):
        """(i -> a of spin s1), then (j -> b of spin s2)."""
        n = _occupied_between(A, B_, i, a, s1)
        one = torch.ones_like(i)
        flip = (one << i) ^ (one << a)
        A2, B2 = (A ^ flip, B_) if s1 == 0 else (A, B_ ^ flip)
        n = n + _occupied_between(A2, B2, j, b, s2)
        e = self._int(a, i, b, j)
        if s1 == s2:
            e = e - self._int(a, j, b, i)
        return e * _sign(n)


def _low(m):
    return m & -m


def _eloc(H, n_elec, a, b, psi, ta, tb, tpsi):
    """E_loc of samples (a, b) against the table (ta, tb): all pairs by the overlap of their occupations."""
    def bits(x, y):
        return torch.cat([H.occ(x), H.occ(y)], 1).to(torch.bfloat16)

    X, Y = bits(a, b), bits(ta, tb).T.contiguous()
    acc = torch.zeros(len(a), 2, dtype=torch.float64, device="cuda")
    tp = torch.view_as_real(tpsi)
    step = max(1, 400_000_000 // Y.shape[1])
    for c in range(0, len(a), step):
        i, j = torch.nonzero((X[c:c + step] @ Y) >= n_elec - 2, as_tuple=True)
        i = i + c
        for q in range(0, len(i), 1 << 23):
            r, t = i[q:q + (1 << 23)], j[q:q + (1 << 23)]
            A, B_ = a[r], b[r]
            dA, dB = A ^ ta[t], B_ ^ tb[t]
            nA, nB = _pop(dA) // 2, _pop(dB) // 2
            e = torch.zeros(len(r), dtype=torch.float64, device="cuda")
            for ka, kb in ((1, 0), (0, 1), (2, 0), (0, 2), (1, 1)):
                s = torch.nonzero((nA == ka) & (nB == kb)).squeeze(1)
                if not len(s):
                    continue
                As, Bs = A[s], B_[s]
                if ka + kb == 1:
                    d, S = (dA[s], As) if ka else (dB[s], Bs)
                    e[s] = H.single(As, Bs, _bit(d & S), _bit(d & ~S), 0 if ka else 1)
                elif ka == 1:
                    x, y = dA[s], dB[s]
                    e[s] = H.double(As, Bs, _bit(x & As), _bit(x & ~As), _bit(y & Bs), _bit(y & ~Bs), 0, 1)
                else:
                    d, S = (dA[s], As) if ka else (dB[s], Bs)
                    ho, pa = d & S, d & ~S
                    l, k = _low(ho), _low(pa)
                    sp = 0 if ka else 1
                    e[s] = H.double(As, Bs, _bit(l), _bit(k), _bit(ho ^ l), _bit(pa ^ k), sp, sp)
            acc.index_add_(0, r, e[:, None] * tp[t])
    return H.diag(a, b) + torch.view_as_complex(acc) / psi


def _moments(e, counts):
    c = counts.double()
    w, s = c.sum(), (c * e).sum()
    m = s / w
    var = (c * (e - m).abs() ** 2).sum() / w
    return torch.stack([m.real, m.imag, var, w, s.real, s.imag])[None]


def _exact_eval(m):
    return _eloc(_H(m.h, m.eri), m.n_elec, m.a, m.b, m.psi, m.ta, m.tb, m.tpsi)


def _energies(e, counts):
    return {"eloc": e, "moments": _moments(e, counts), "counters": None, "status": None}


def _exact_export(m):
    """Elements in the documented order: singles (alpha, beta), alpha-alpha, beta-beta, alpha-beta doubles."""
    H, K, o = _H(m.h, m.eri), m.n_orb // 2, m.n_elec // 2
    v, n = K - o, len(m.a)
    ar = lambda k: torch.arange(k, device="cuda")  # noqa: E731

    def lists(S):
        order = torch.sort(1 - ((S[:, None] >> ar(K)) & 1), dim=1, stable=True).indices
        return order[:, :o], order[:, o:]

    def pairs(k):  # colex: (p < q) at q (q - 1) / 2 + p
        q, p = torch.tril_indices(k, k, -1, device="cuda")
        return p, q

    po, pv = pairs(o), pairs(v)
    ns, so, sv = o * v, ar(o * v) // v, ar(o * v) % v
    P = _pairs(m.n_orb, m.n_elec)
    out = torch.empty(n, P, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 23) // P)
    for c in range(0, n, step):
        A, B_ = m.a[c:c + step], m.b[c:c + step]
        r = len(A)
        (oa, va), (ob, vb) = lists(A), lists(B_)
        at = 0

        def put(e, k):
            nonlocal at
            out[c:c + step, at:at + k] = e.reshape(r, k)
            at += k

        def wide(x, k):
            return x[:, None].expand(r, k).reshape(-1)

        for spin, (oc, vi) in enumerate(((oa, va), (ob, vb))):
            put(H.single(wide(A, ns), wide(B_, ns), oc[:, so].reshape(-1), vi[:, sv].reshape(-1), spin), ns)
        for spin, (oc, vi) in enumerate(((oa, va), (ob, vb))):
            nu, nw = len(po[0]), len(pv[0])
            k = nu * nw
            if not k:
                continue
            u, w = ar(k) // nw, ar(k) % nw
            put(H.double(wide(A, k), wide(B_, k), oc[:, po[0][u]].reshape(-1), vi[:, pv[0][w]].reshape(-1),
                         oc[:, po[1][u]].reshape(-1), vi[:, pv[1][w]].reshape(-1), spin, spin), k)
        k = ns * ns
        u, w = ar(k) // ns, ar(k) % ns
        put(H.double(wide(A, k), wide(B_, k), oa[:, so[u]].reshape(-1), va[:, sv[u]].reshape(-1),
                     ob[:, so[w]].reshape(-1), vb[:, sv[w]].reshape(-1), 0, 1), k)
    return {"keys": None, "elems": out.reshape(-1), "diag": H.diag(m.a, m.b)}


def exact(case, seed):
    op = case["op"]
    if op == "dedup":
        return None  # whole numbers
    if op in ("eval", "rows"):
        m = _Mol(case["n_orb"], case["n_elec"], case["n_u"], seed, n_table=case.get("n_table", 0))
        return _energies(_exact_eval(m), m.counts)
    if op == "batch":
        es, mo = [], []
        for q in _molecules(case, seed):
            m = _Mol(**q)
            es.append(_exact_eval(m))
            mo.append(_moments(es[-1], m.counts))
        return {"eloc": es, "moments": torch.cat(mo), "counters": None, "status": None}
    if op == "grad":
        m = _Mol(*GRAD_SHAPE, case["n_u"], seed)
        e, c = _exact_eval(m), m.counts.double()
        w = c * (e - (c * e).sum() / c.sum()) / c.sum()
        d = torch.randn(case["n_u"], case["n_par"], 2, dtype=torch.float64, device="cuda", generator=_gen(seed, 7))
        g = 2.0 * (w.real @ d[..., 0] - w.imag @ d[..., 1])
        return {"w": w, "g": g}
    m = _Mol(case["n_orb"], case["n_elec"], case["n_u"], seed)
    if op == "export":
        return _exact_export(m)
    x = _conn(case, seed)
    n = case["n_u"]
    s = (x["elems"].reshape(n, -1) * x["conn"].reshape(n, -1)).sum(1)
    return _energies(x["diag"] + s / m.psi, m.counts)
