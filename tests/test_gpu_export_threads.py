"""Threads that export with handles of different shared-memory needs at the same time (one thread per
handle, as the library allows): every call succeeds and writes what it writes alone."""
import ctypes
import threading

import pytest

from paper_2506_23809_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_export_threads():
    import torch
    from paper_2506_23809_gb300 import binding as B
    lib = B.load_library()
    jobs = []
    for n_orb in (128, 122, 124, 120):  # 62 to 58 empty orbitals a spin: 50 to 58 KB an item
        K = n_orb // 2
        ints = I.make_integrals(K, 8, n_orb)
        jobs.append([B.qc_eloc_create(ints.h, ints.eri, 0.0, n_orb, 4), None, [], None])
    key = torch.tensor([[15, 0]], dtype=torch.int64, device="cuda")

    def run(job):
        stream = torch.cuda.Stream()
        out = torch.empty_like(job[1])
        vp = ctypes.c_void_p
        args = (job[0].ptr, vp(key.data_ptr()), 1, None, vp(out.data_ptr()), None, vp(stream.cuda_stream))
        for _ in range(3000):
            if lib.qc_eloc_export(*args) != 0:
                job[2].append(lib.qc_eloc_last_error(job[0].ptr))
        stream.synchronize()
        job[3] = out

    try:
        for job in jobs:
            job[1] = B.qc_eloc_export(job[0], key, keys=False, diag=False)[1]
        torch.cuda.synchronize()
        threads = [threading.Thread(target=run, args=(job,)) for job in jobs]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for job in jobs:
            assert job[2] == [] and torch.equal(job[3], job[1])
    finally:
        for job in jobs:
            B.qc_eloc_destroy(job[0])
