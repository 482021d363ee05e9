"""The throughput engine (launch modes 0 and 1, node_threads 1, 2 and 4) at the
edges of its 32-node blocks, against the FP64 oracle node by node.

Tolerances as in test_gpu_parity.py: 1e-10 in FP64; in mixed precision 1e-5 on
populations and eta, and on the auxiliaries 1e-5 of the largest one.
"""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu

# one node; a block less one, full, and one over; odd and even N (the pairs at
# distance N/2); more blocks than sets, and more CTAs than blocks
SIZES = [(1, 0), (1, 30), (1, 31), (1, 32), (2, 7), (3, 4), (4, 0), (4, 3), (5, 3), (6, 2), (6, 4), (7, 2), (7, 4), (8, 1), (8, 3)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["real", "complex_term", "scaled_low_temp"])
@pytest.mark.parametrize("N,K", SIZES)
def test_block_edges(N, K, kind, precision):
    w = workloads.random_instance(N, K, seed=900 + 16 * N + K, complex_h=kind == "complex_term",
                                  terminator=1 if kind == "complex_term" else 0)
    w["params"]["scaled"] = w["params"]["low_temp"] = 1 if kind == "scaled_low_temp" else 0
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 21, 5, want_state=True)
    multi, _, _ = heom.build_index(N, K)
    pos = {tuple(m): i for i, m in enumerate(o["multi"].tolist())}
    ref = o["state"][np.array([pos[tuple(m)] for m in multi.tolist()])][:, :N, :N]
    tol = 1e-10 if precision == "fp64" else 1e-5
    for shape in (dict(mode=0, team_ctas=1, block_threads=64), dict(mode=0, team_ctas=16, block_threads=256),
                  dict(mode=1, block_threads=256)):
        with heom.Context(w["params"], precision) as c:
            c.set_launch(node_threads=4 if kind == "scaled_low_temp" else 2, **shape)
            c.set_rho0(w["rho0"])
            r = [c.propagate(1.0, n, 5) for n in (10, 11)]  # the state is put back into packed order in between
            state, extra = c.state()
        pops = np.concatenate([r[0]["pops"], r[1]["pops"][1:]])
        eta = np.concatenate([r[0]["eta"], r[1]["eta"][1:]])
        assert np.abs(pops - o["pops"]).max() < tol, shape
        assert np.abs(eta - o["eta"]).max() < tol, shape
        assert np.abs(state - ref).max() < tol * max(1.0, np.abs(ref).max()), shape


def test_block_stop_rule():
    """The stop rule takes the same step in cyclic order as the oracle's trace says."""
    w = workloads.random_instance(5, 3, seed=77)
    w["params"]["trap"] = np.full(5, 40.0)
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 60, 1)
    step = int(np.argmax(o["trace"] < 0.5))
    assert 2 < step < 59 and abs(o["trace"][step] - 0.5) > 1e-4 and abs(o["trace"][step - 1] - 0.5) > 1e-4
    for precision in ("fp64", "fp32"):
        for mode in (0, 1):
            with heom.Context(w["params"], precision) as c:
                c.set_launch(mode=mode, team_ctas=2, block_threads=128, node_threads=2)
                c.set_stop(0.5)
                c.set_rho0(w["rho0"])
                r = c.propagate(1.0, 60, 1)
                assert c.trapping_time()[1] == step
                assert np.abs(r["pops"][:step + 1] - o["pops"][:step + 1]).max() < (1e-10 if precision == "fp64" else 1e-5)
                assert np.all(np.isnan(r["pops"][step + 1:]))
