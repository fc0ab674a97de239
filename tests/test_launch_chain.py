"""Kernels launched while their predecessors still run (launch_early) may read what those write only
through coherent loads: non-coherent ones (__ldg, `const ... __restrict__` parameters) are defined for
data that nothing writes while the reading kernel is resident.  Held on the source text: the names
below are the handle's constants, the caller's inputs and what the host copied before the chain."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_23809_gb300", "csrc")
COMPLETE = {"keys", "samples", "T", "Tg", "T64", "mols", "slot_base", "row_base"}
UNITS = ("qc_device.cuh", "qc_main_kernel.cuh", "qc_kernels.cu", "qc_join.cu")  # the chain's kernels


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def _early_kernels():
    """name -> parameter list of every kernel that launch_early is given."""
    text = "\n".join(_read(n) for n in sorted(os.listdir(CSRC)) if n.endswith((".cu", ".cuh")))
    names = {n for n in re.findall(r"launch_early\(\s*(\w+)", text) if n != "k"} | {"eloc_main_kernel"}
    out = {}
    for n in names:
        m = re.search(r"__global__[^;{]*?\b" + n + r"\(([^{;]*?)\)\s*\{", text)
        if m:
            out[n] = m.group(1)
    return names, out


def test_parameters():
    names, params = _early_kernels()
    assert names - {"void"} == set(params) and len(params) >= 15
    for n, p in params.items():
        assert set(re.findall(r"__restrict__\s+(\w+)", p)) <= COMPLETE, n


def test_loads():
    for unit in UNITS:
        for base in re.findall(r"__ldg\(\s*([\w.\->]+)", _read(unit)):
            name = re.split(r"\.|->", base)[-1]
            assert name in COMPLETE | {"psi"} or base.startswith("sp."), (unit, base)
