"""heom_set_launch on a small hierarchy that still has its default shape."""
import numpy as np
import pytest

import oracle
from paper_1012_4382_gb300 import build as heom_build
from paper_1012_4382_gb300 import heom, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    heom_build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [dict(team_ctas=17), dict(block_threads=48), dict(node_threads=33), dict(mode=4),
                                 dict(mode=0, team_ctas=17)])
def test_refused_shape_leaves_the_default(bad, precision):
    w = workloads.random_instance(3, 3, seed=1)
    with heom.Context(w["params"], precision) as c:
        shape = c.get_launch()
        assert shape["mode"] == 3
        with pytest.raises(heom.HeomError) as e:
            c.set_launch(**bad)
        assert e.value.code == heom.EINVAL
        assert c.get_launch() == shape
        c.set_launch(node_threads=8)  # and the context still counts as one whose shape was never set
        assert c.get_launch()["mode"] != 3


# 5 sites, depth 5: 252 nodes, eight blocks of 32
@pytest.mark.parametrize("precision,call,mode,team", [
    ("fp64", dict(mode=0), 0, 8), ("fp64", dict(block_threads=128), 0, 8), ("fp64", dict(node_threads=8), 0, 8),
    ("fp64", dict(team_ctas=2), 0, 2), ("fp32", dict(mode=0), 0, 8), ("fp32", dict(mode=2), 2, 2),
    ("fp32", dict(node_threads=8), 2, 2), ("fp32", dict(node_threads=4), 0, 8)])
def test_values_left_out_are_those_of_a_cluster_launch(precision, call, mode, team):
    w = workloads.random_instance(5, 5, seed=12)
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 20, 5)
    tol = 1e-10 if precision == "fp64" else 1e-5
    with heom.Context(w["params"], precision) as c:
        c.set_launch(**call)
        shape = c.get_launch()
        assert (shape["mode"], shape["team_ctas"]) == (mode, team)
        c.set_rho0(w["rho0"])
        assert np.abs(c.propagate(1.0, 20, 5)["pops"] - o["pops"]).max() < tol


def test_mixed_hierarchy_that_one_cta_takes_at_once_stays_in_one():
    w = workloads.random_instance(4, 4, seed=13)  # 70 nodes, three blocks of 32 on the five sets of a CTA
    o = oracle.propagate(w["params"], w["rho0"], 1.0, 20, 5)
    with heom.Context(w["params"], "fp32") as c:
        c.set_launch(node_threads=4)
        assert c.get_launch()["team_ctas"] == 1
        c.set_rho0(w["rho0"])
        assert np.abs(c.propagate(1.0, 20, 5)["pops"] - o["pops"]).max() < 1e-5


@pytest.mark.parametrize("complex_h,terminator,keep_blocks,node_threads", [
    (True, 0, None, 8), (False, 0, None, 2), (True, 1, None, 2), (True, 0, 152, 2), (True, 0, 153, 8),
    (True, 0, 228, 8), (True, 0, 229, 2)])
def test_eight_sites_fp64_just_above_one_block_per_sm(complex_h, terminator, keep_blocks, node_threads):
    """Depth 7 (6435 nodes, 202 blocks of 32 on 152 SMs) and first nodes of depth 8, at the edges of the range in
    which the load views are the default."""
    K = 7 if keep_blocks is None else 8
    w = workloads.random_instance(8, K, seed=21, complex_h=complex_h, terminator=terminator)
    M, p, keep = heom.num_nodes(8, K), w["params"], None
    if keep_blocks is not None:
        keep = (np.arange(M) < 32 * keep_blocks - 5).astype(np.uint8)
        multi, _, _ = heom.build_index(8, K)
        pos = {tuple(m): i for i, m in enumerate(oracle.multi_indices(8, K).tolist())}
        okeep = np.zeros(M, np.uint8)
        okeep[[pos[tuple(m)] for m in multi[keep > 0].tolist()]] = 1
        p = dict(p, keep=okeep)
    o = oracle.propagate(p, w["rho0"], 1.0, 4, 2)
    with heom.Context(w["params"], "fp64", keep=keep) as c:
        assert c.get_launch()["mode"] == 1 and c.get_launch()["node_threads"] == node_threads
        c.set_rho0(w["rho0"])
        r = c.propagate(1.0, 4, 2)
    assert np.abs(r["pops"] - o["pops"]).max() < 1e-10
    assert np.abs(r["eta"] - o["eta"]).max() < 1e-10
