"""Hierarchies small enough for the one-CTA kernel of launch mode 3 (a thread per
packed real: at most 992, 480 in FP64), at and around that limit, against the
FP64 oracle node by node.  Tolerances as in test_gpu_parity.py (1e-10 in FP64;
in mixed precision 1e-5, on the auxiliaries of the largest one).
"""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu

# (N, K): one real, a warp less one, full and one over; both limits from below and above; even and odd N
SIZES = [(1, 0), (1, 30), (1, 31), (1, 32), (2, 4), (2, 13), (2, 14), (2, 15), (2, 20), (2, 21), (3, 4), (3, 6), (4, 2),
         (4, 3), (5, 2), (6, 1), (7, 1), (7, 2), (8, 1)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["real", "complex_term", "scaled_low_temp"])
@pytest.mark.parametrize("N,K", SIZES)
def test_small_default(N, K, kind, precision):
    w = workloads.random_instance(N, K, seed=300 + 16 * N + K, complex_h=kind == "complex_term",
                                  terminator=1 if kind == "complex_term" else 0)
    w["params"]["scaled"] = w["params"]["low_temp"] = 1 if kind == "scaled_low_temp" else 0
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 21, 5, want_state=True)
    multi, _, _ = heom.build_index(N, K)
    pos = {tuple(m): i for i, m in enumerate(o["multi"].tolist())}
    ref = o["state"][np.array([pos[tuple(m)] for m in multi.tolist()])][:, :N, :N]
    tol = 1e-10 if precision == "fp64" else 1e-5
    with heom.Context(w["params"], precision) as c:
        c.set_rho0(w["rho0"])
        r = [c.propagate(1.0, n, 5) for n in (10, 11)]
        state, _ = c.state()
    pops = np.concatenate([r[0]["pops"], r[1]["pops"][1:]])
    eta = np.concatenate([r[0]["eta"], r[1]["eta"][1:]])
    assert np.abs(pops - o["pops"]).max() < tol
    assert np.abs(eta - o["eta"]).max() < tol
    assert np.abs(state - ref).max() < tol * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_stop_rule_and_partial_launch_shapes(precision):
    """The stop rule in the one-CTA kernel; team, block or node threads given alone still select a cluster launch; a
    batch of one small hierarchy still takes CUDA graphs; all rho(0) of a batch are set at once."""
    w = workloads.random_instance(3, 3, seed=78)
    w["params"]["trap"] = np.full(3, 40.0)
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 60, 1)
    step = int(np.argmax(o["trace"] < 0.5))
    assert 2 < step < 59 and abs(o["trace"][step] - 0.5) > 1e-4 and abs(o["trace"][step - 1] - 0.5) > 1e-4
    tol = 1e-10 if precision == "fp64" else 1e-5
    with heom.Context(w["params"], precision) as c:
        c.set_stop(0.5)
        for shape in (None, dict(team_ctas=16), dict(block_threads=64), dict(node_threads=8)):
            if shape:
                c.set_launch(**shape)
            c.set_rho0(w["rho0"])
            r = c.propagate(1.0, 60, 1)
            assert c.trapping_time()[1] == step
            assert np.abs(r["pops"][:step + 1] - o["pops"][:step + 1]).max() < tol
            assert np.all(np.isnan(r["pops"][step + 1:]))
    ws = [w, workloads.random_instance(10, 2, seed=5), workloads.random_instance(5, 4, seed=6)]
    for some in (ws[:1], ws):
        with heom.Batch([v["params"] for v in some], precision) as b:
            for _ in range(2):  # the second time over a propagated state
                b.set_rho0([v["rho0"] for v in some])
                for i, v in enumerate(some):
                    assert np.abs(b.rho(i) - v["rho0"]).max() < tol
                rows = b.propagate(1.0, 20, 5)
                for v, r in zip(some, rows):
                    assert np.abs(r["pops"] - oracle.propagate(v["params"], v["rho0"], 1.0, 20, 5)["pops"]).max() < tol
            if len(some) == 1:
                b.graph(1.0, 5, 5).close()
