"""A small hierarchy with its default launch shape, propagated while the caller captures its stream: every replay of the
graph continues the propagation as a direct call would (a one-step call is the one whose replay could read the words of
the run before in a dataflow launch)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


def _cudart():
    for line in open("/proc/self/maps"):
        if "libcudart.so" in line:
            return ctypes.CDLL(line.split()[-1])
    raise RuntimeError("libcudart is not loaded")


# one CTA by default; the dataflow engine by default (1120 and 3150 packed reals)
@pytest.mark.parametrize("N,K", [(2, 4), (4, 4), (5, 4)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nsteps", [1, 7])
def test_captured_default_replays(N, K, precision, nsteps):
    w = workloads.random_instance(N, K, seed=40 + N)
    rt, s = _cudart(), torch.cuda.Stream()
    vp = ctypes.c_void_p
    with heom.Context(w["params"], precision, stream=s) as c, heom.Context(w["params"], precision, stream=s) as direct:
        assert c.get_launch()["mode"] == 3
        for x in (c, direct):  # the first call makes its buffers
            x.propagate_device(1.0, nsteps, nsteps)
            x.synchronize()
            x.set_rho0(w["rho0"])
        assert rt.cudaStreamBeginCapture(vp(s.cuda_stream), 2) == 0
        graph, run = vp(), vp()
        try:
            c.propagate_device(1.0, nsteps, nsteps)
        finally:
            assert rt.cudaStreamEndCapture(vp(s.cuda_stream), ctypes.byref(graph)) == 0
        assert c.get_launch()["mode"] == 3
        assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, ctypes.c_ulonglong(0)) == 0
        for _ in range(3):
            assert rt.cudaGraphLaunch(run, vp(s.cuda_stream)) == 0
            direct.propagate_device(1.0, nsteps, nsteps)
        c.synchronize()
        direct.synchronize()
        tol = 1e-12 if precision == "fp64" else 1e-6
        assert np.abs(c.rho() - direct.rho()).max() < tol
        assert rt.cudaGraphExecDestroy(run) == 0 and rt.cudaGraphDestroy(graph) == 0
