"""The 9..24-site kernel where (in FP64) the blocks of its last round are shared out among
CTAs by columns (team sizes that leave fewer blocks than sets after a full
round), and where they are not, against the FP64 oracle node by node.

Tolerances as in test_gpu_parity.py: 1e-10 in FP64; in mixed precision 1e-5 on
populations and eta, and on the auxiliaries 1e-5 of the largest one.
"""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu

# (N, K, blocks of 32 nodes): odd and even N, one and two sets per CTA, parts that do not divide N
SIZES = [(9, 4, 23), (10, 3, 9), (11, 3, 12), (13, 3, 18), (16, 3, 31), (17, 2, 6), (24, 2, 11)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["real", "complex_term", "scaled_low_temp"])
@pytest.mark.parametrize("N,K,blocks", SIZES)
def test_large_last_round(N, K, blocks, kind, precision):
    assert (heom.num_nodes(N, K) + 31) // 32 == blocks
    w = workloads.random_instance(N, K, seed=500 + 16 * N + K, complex_h=kind == "complex_term",
                                  terminator=1 if kind == "complex_term" else 0)
    w["params"]["scaled"] = w["params"]["low_temp"] = 1 if kind == "scaled_low_temp" else 0
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 9, 4, want_state=True)
    multi, _, _ = heom.build_index(N, K)
    pos = {tuple(m): i for i, m in enumerate(o["multi"].tolist())}
    ref = o["state"][np.array([pos[tuple(m)] for m in multi.tolist()])][:, :N, :N]
    tol = 1e-10 if precision == "fp64" else 1e-5
    for team in (1, 2, 4, 8, 16):
        with heom.Context(w["params"], precision) as c:
            c.set_launch(mode=0, team_ctas=team)
            c.set_rho0(w["rho0"])
            r = [c.propagate(1.0, n, 4) for n in (4, 5)]
            state, _ = c.state()
        pops = np.concatenate([r[0]["pops"], r[1]["pops"][1:]])
        eta = np.concatenate([r[0]["eta"], r[1]["eta"][1:]])
        assert np.abs(pops - o["pops"]).max() < tol, team
        assert np.abs(eta - o["eta"]).max() < tol, team
        assert np.abs(state - ref).max() < tol * max(1.0, np.abs(ref).max()), team
