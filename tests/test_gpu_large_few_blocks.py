"""The 9..24-site kernel on hierarchies of fewer node blocks than a team has sets: in FP64 every block, the root's among
them, is shared out among CTAs by columns, in mixed precision none is.  Against the FP64 oracle node by node, with the
stop rule and the running sums that the owners of the root's columns keep.

Tolerances as in test_gpu_parity.py: 1e-10 in FP64; in mixed precision 1e-5 on populations, eta and the trapping time's
integral per fs, and on the auxiliaries 1e-5 of the largest one.
"""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu

# (N, K): one block, two, three and six; odd and even N, one and two sets per CTA, parts that do not divide N
SIZES = [(9, 1), (10, 1), (17, 1), (24, 1), (9, 2), (12, 2), (17, 2)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["real", "complex_term", "scaled_low_temp"])
@pytest.mark.parametrize("N,K", SIZES)
def test_few_blocks(N, K, kind, precision):
    w = workloads.random_instance(N, K, seed=700 + 16 * N + K, complex_h=kind == "complex_term",
                                  terminator=1 if kind == "complex_term" else 0)
    w["params"]["scaled"] = w["params"]["low_temp"] = 1 if kind == "scaled_low_temp" else 0
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 9, 4, want_state=True)
    multi, _, _ = heom.build_index(N, K)
    pos = {tuple(m): i for i, m in enumerate(o["multi"].tolist())}
    ref = o["state"][np.array([pos[tuple(m)] for m in multi.tolist()])][:, :N, :N]
    tol = 1e-10 if precision == "fp64" else 1e-5
    shapes = [dict(mode=0, team_ctas=t) for t in (1, 2, 4, 8, 16)] + [dict(mode=1)]
    for shape in shapes:
        with heom.Context(w["params"], precision) as c:
            c.set_launch(**shape)
            c.set_rho0(w["rho0"])
            r = [c.propagate(1.0, n, 4) for n in (4, 5)]
            state, _ = c.state()
        pops = np.concatenate([r[0]["pops"], r[1]["pops"][1:]])
        eta = np.concatenate([r[0]["eta"], r[1]["eta"][1:]])
        assert np.abs(pops - o["pops"]).max() < tol, shape
        assert np.abs(eta - o["eta"]).max() < tol, shape
        assert np.abs(state - ref).max() < tol * max(1.0, np.abs(ref).max()), shape


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N,K", [(10, 1), (24, 1), (12, 2)])
def test_few_blocks_stop_rule_rows_and_batch(N, K, precision):
    w = workloads.random_instance(N, K, seed=79 + N)
    w["params"]["trap"] = np.full(N, 40.0)
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 60, 1)
    step = int(np.argmax(o["trace"] < 0.5))
    assert 2 < step < 59 and abs(o["trace"][step] - 0.5) > 1e-4 and abs(o["trace"][step - 1] - 0.5) > 1e-4
    tol = 1e-10 if precision == "fp64" else 1e-5
    t = np.arange(step + 1.0)
    mean = step * o["eta"][step] - np.trapezoid(o["eta"][:step + 1], t)  # <t>, up to the trapezoid rule's error
    for shape in (dict(mode=0, team_ctas=8), dict(mode=0, team_ctas=2), dict(mode=1)):
        with heom.Context(w["params"], precision) as c:
            c.set_launch(**shape)
            c.set_stop(0.5)
            c.set_rho0(w["rho0"])
            r = c.propagate(1.0, 60, 1)
            t_mean, done = c.trapping_time()
        assert done == step, shape
        assert np.abs(r["pops"][:step + 1] - o["pops"][:step + 1]).max() < tol, shape
        assert np.abs(r["eta"][:step + 1] - o["eta"][:step + 1]).max() < tol, shape
        assert np.all(np.isnan(r["pops"][step + 1:]))
        assert abs(t_mean - mean) < 0.02 * abs(mean) + 0.1, shape
    # instances of one and of more blocks in one launch, twice over
    ws = [w, workloads.random_instance(N, K + 1, seed=5), workloads.random_instance(N, 0, seed=6), w]
    with heom.Batch([v["params"] for v in ws], precision) as b:
        b.set_launch(mode=0, team_ctas=8)
        for _ in range(2):
            b.set_rho0([v["rho0"] for v in ws])
            for v, r in zip(ws, b.propagate(1.0, 12, 3)):
                assert np.abs(r["pops"] - oracle.propagate(v["params"], v["rho0"], 1.0, 12, 3)["pops"]).max() < tol
