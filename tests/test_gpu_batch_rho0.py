"""heom_batch_set_rho0 around failures: it allocates nothing (its table of targets is made with the batch), a batch
whose creation runs out of memory is not made, and a call that fails leaves the next one right."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


def _instances():
    return [workloads.random_instance(N, K, seed=500 + N) for N, K in ((3, 3), (7, 2), (10, 1))]


def _check(b, ws, precision):
    tol = 1e-10 if precision == "fp64" else 1e-5
    rows = b.propagate(1.0, 20, 5)
    for v, r in zip(ws, rows):
        assert np.abs(r["pops"] - oracle.propagate(v["params"], v["rho0"], 1.0, 20, 5)["pops"]).max() < tol


class _Allocator:
    """Device memory from PyTorch's caching allocator; refuses the request number `refuse` (from 0)."""

    def __init__(self):
        self.calls, self.live, self.refuse = 0, 0, None

        def alloc(nbytes, _):
            self.calls += 1
            if self.refuse is not None and self.calls - 1 == self.refuse:
                return None
            self.live += 1
            return int(torch.cuda.caching_allocator_alloc(int(nbytes)))

        def free(p, nbytes, _):
            self.live -= 1
            torch.cuda.caching_allocator_delete(int(p))

        self.hooks = (heom.ALLOC_FN(alloc), heom.FREE_FN(free))

    def __enter__(self):
        heom._check(heom.lib().heom_set_allocator(self.hooks[0], self.hooks[1], None))
        return self

    def __exit__(self, *a):
        heom.use_torch_allocator(False)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_set_rho0_allocates_nothing_and_creation_fails_whole(precision):
    ws = _instances()
    ps, rho = [w["params"] for w in ws], [w["rho0"] for w in ws]
    with _Allocator() as a:
        with heom.Batch(ps, precision) as b:
            made = a.calls
            b.set_rho0(rho)
            b.set_rho0(rho)
            assert a.calls == made
            _check(b, ws, precision)
        assert a.live == 0
        for k in range(made):  # every allocation of the creation refused once
            a.calls, a.refuse = 0, k
            with pytest.raises(heom.HeomError) as e:
                heom.Batch(ps, precision)
            assert e.value.code == heom.ENOMEM and a.live == 0
        a.refuse = None
        with heom.Batch(ps, precision) as b:
            b.set_rho0(rho)
            _check(b, ws, precision)
    assert a.live == 0


def _cudart():
    for line in open("/proc/self/maps"):
        if "libcudart.so" in line:
            return ctypes.CDLL(line.split()[-1])
    raise RuntimeError("libcudart is not loaded")


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_set_rho0_refused_during_capture_works_afterwards(precision):
    """The first call made while the batch's stream is being captured (relaxed mode, so that allocations pass) is an
    error; after the capture the same call sets every rho(0)."""
    ws = _instances()
    rt = _cudart()
    s = torch.cuda.Stream()
    with heom.Batch([w["params"] for w in ws], precision, stream=s) as b:
        torch.cuda.synchronize()
        assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 2) == 0
        try:
            with pytest.raises(heom.HeomError) as e:
                b.set_rho0([w["rho0"] for w in ws])
            assert e.value.code == heom.ECUDA
        finally:
            g = ctypes.c_void_p()
            rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(g))
            if g.value:
                rt.cudaGraphDestroy(g)
            rt.cudaGetLastError()
        b.set_rho0([w["rho0"] for w in ws])
        for i, w in enumerate(ws):
            assert np.abs(b.rho(i) - w["rho0"]).max() < (1e-15 if precision == "fp64" else 1e-13)
        _check(b, ws, precision)
