"""Hierarchies of different sizes propagated by one kernel from several threads: every launch needs another amount of
dynamic shared memory, and none may lower what another thread's launch is allowed."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu

CALLS = 1500


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


def _context_calls(w, calls, out):
    s = torch.cuda.Stream()
    with heom.Context(w["params"], "fp32", stream=s) as c:
        # one CTA: the throughput engine caches all links of the hierarchy (16 to 130 KB with the exchange area)
        c.set_launch(mode=0, team_ctas=1, block_threads=512, node_threads=2)
        c.set_rho0(w["rho0"])
        for i in range(calls):
            c.propagate_device(0.1, 1, 1)
            if i % 50 == 0:
                c.synchronize()
        c.synchronize()
        out.append(c.rho())


def _static_calls(w, calls, out):
    vp = ctypes.c_void_p
    L = heom.lib()
    L.heom_propagate_static.argtypes = [ctypes.POINTER(heom._Params), vp, ctypes.c_double, ctypes.c_int64,
                                        ctypes.c_int64, vp, vp, vp, vp]
    L.heom_propagate_static.restype = ctypes.c_int
    keep = heom._Keep(w["params"], heom.FP32_MIXED)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        rho0 = torch.from_numpy(np.ascontiguousarray(w["rho0"], dtype=np.complex128)).cuda()
        rho = torch.zeros_like(rho0)
    for _ in range(calls // 4):
        heom._check(L.heom_propagate_static(ctypes.byref(keep.c), rho0.data_ptr(), 0.1, 1, 1, None, None,
                                            rho.data_ptr(), s.cuda_stream))
    out.append(rho.cpu().numpy())


def test_threads_launch_one_kernel_with_different_shared_memory():
    jobs = [(_context_calls, workloads.fmo_trap(K=6, nsteps=1)), (_context_calls, workloads.fmo_trap(K=4, nsteps=1)),
            (_context_calls, workloads.fmo_trap(K=5, nsteps=1)), (_static_calls, workloads.fmo_trap(K=4, nsteps=1))]
    alone = []
    for run, w in jobs:
        run(w, CALLS, alone)
    got, errors = [[] for _ in jobs], []

    def go(i):
        try:
            jobs[i][0](jobs[i][1], CALLS, got[i])
        except heom.HeomError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=go, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for a, g in zip(alone, got):
        assert np.array_equal(a, g[0])
