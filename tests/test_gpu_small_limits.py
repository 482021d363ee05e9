"""The one-CTA kernel of small hierarchies at the end of its range: filtered hierarchies whose packed reals fill its
largest CTA (961 to 992 of 992, in FP64 449 to 480 of 480), and one node more, which the dataflow engine takes.  Against
the FP64 oracle on the same nodes; tolerances as in test_gpu_parity.py (1e-10, mixed precision 1e-5)."""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


# (N, K, nodes kept)
FULL = {"fp32": [(2, 22, 248), (3, 8, 110), (4, 4, 62), (5, 3, 39), (6, 2, 27), (7, 2, 20)],
        "fp64": [(2, 15, 120), (3, 5, 53), (4, 3, 30), (5, 2, 19), (6, 2, 13)]}


@pytest.mark.parametrize("precision,N,K,nodes", [(p, N, K, n + more) for p in FULL for N, K, n in FULL[p] for more in (0, 1)])
@pytest.mark.parametrize("complex_scaled", [False, True])
def test_full_cta(precision, N, K, nodes, complex_scaled):
    w = workloads.random_instance(N, K, seed=400 + 16 * N + K, complex_h=complex_scaled)
    w["params"]["scaled"] = w["params"]["low_temp"] = int(complex_scaled)
    M = heom.num_nodes(N, K)
    keep = (np.arange(M) < nodes).astype(np.uint8)  # by level: closed downwards
    multi, _, _ = heom.build_index(N, K)
    pos = {tuple(m): i for i, m in enumerate(oracle.multi_indices(N, K).tolist())}
    perm = np.array([pos[tuple(m)] for m in multi.tolist()])
    okeep = np.zeros(M, np.uint8)
    okeep[perm] = keep
    o = oracle.propagate(dict(w["params"], keep=okeep), w["rho0"], 1.0, 21, 5, want_state=True)
    ref = o["state"][perm][:nodes, :N, :N]
    tol = 1e-10 if precision == "fp64" else 1e-5
    with heom.Context(w["params"], precision, keep=keep) as c:
        assert c.nodes == nodes and c.get_launch()["mode"] == 3
        c.set_rho0(w["rho0"])
        r = [c.propagate(1.0, n, 5) for n in (10, 11)]
        state, _ = c.state()
    pops = np.concatenate([r[0]["pops"], r[1]["pops"][1:]])
    eta = np.concatenate([r[0]["eta"], r[1]["eta"][1:]])
    assert np.abs(pops - o["pops"]).max() < tol
    assert np.abs(eta - o["eta"]).max() < tol
    assert np.abs(state - ref).max() < tol * max(1.0, np.abs(ref).max())
