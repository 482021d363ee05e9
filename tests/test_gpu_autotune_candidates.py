"""The autotuners time each kernel shape once: of launch shapes that run the same kernel the same way, the one kept is
the representative (node_threads 2, 4 for scaled hierarchies; no more nodes per thread in mode 3 than are built; one shape
of the one-CTA kernel)."""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("N,K,precision,scaled", [(7, 8, "fp32", 0), (7, 8, "fp64", 0), (7, 8, "fp32", 1),
                                                  (8, 6, "fp32", 0), (2, 3, "fp32", 0), (2, 3, "fp64", 1)])
def test_context_keeps_a_representative(N, K, precision, scaled):
    w = workloads.random_instance(N, K, seed=60 + N)
    w["params"]["scaled"] = scaled
    with heom.Context(w["params"], precision) as c:
        for _ in range(3):
            c.autotune(trial_steps=20)
            shape = c.get_launch()
            if shape["mode"] == 3:
                assert shape["team_ctas"] <= (2 if N == 8 else 3), shape
            if shape["mode"] <= 1:
                assert shape["node_threads"] not in ((1, 2) if scaled else (1, 4)), shape
        c.set_rho0(w["rho0"])
        r = c.propagate(1.0, 10, 5)
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 10, 5)
    assert np.abs(r["pops"] - o["pops"]).max() < (1e-10 if precision == "fp64" else 1e-5)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("scaled", [0, 1])
def test_batch_keeps_a_representative(precision, scaled):
    ws = [workloads.random_instance(N, K, seed=70 + N) for N, K in ((3, 5), (7, 4), (10, 2))]
    for w in ws[:2]:
        w["params"]["scaled"] = scaled
    for some in (ws, ws[2:]):
        with heom.Batch([w["params"] for w in some], precision) as b:
            b.autotune(trial_steps=5)
            shape = b.get_launch(10)
            if shape["mode"] == 0:
                assert shape["node_threads"] in ((4 if scaled and len(some) > 1 else 2,) + ((8,) if len(some) > 1 else ()))
            b.set_rho0([w["rho0"] for w in some])
            for w, r in zip(some, b.propagate(1.0, 10, 5)):
                o = oracle.propagate(w["params"], w["rho0"], 1.0, 10, 5)
                assert np.abs(r["pops"] - o["pops"]).max() < (1e-10 if precision == "fp64" else 1e-5)
