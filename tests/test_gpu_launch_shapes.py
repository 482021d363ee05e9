"""heom_set_launch on a small hierarchy that still has its default shape."""
import pytest

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
