"""What a workspace remembers of a relation that a route did not suit does not keep the next relation off
the route: layers after relations without any and after refused calls, walks after wide closures."""
import numpy as np
import pytest

import oracle
from paper_1608_00139_gb300 import dl, inputs

pytestmark = pytest.mark.gpu


def check_sg(c, p, want):
    bits, st = c.sg_least_model(p)
    assert np.array_equal(bits, want)
    return st


@pytest.mark.parametrize("n", [700, 6200])
def test_layers_after_relations_without(n):
    forest, other = inputs.forest_dag(n, 3), inputs.forest_dag(n, 4)
    cyclic = inputs.er_digraph(n, 2.0 / n, 5)
    want = [oracle.sg_model(p) for p in (forest, other, cyclic)]
    with dl.Context(0) as c:  # by layers: their number, and the launches of that route
        layers = [check_sg(c, p, w) for p, w in zip((forest, other), want)]
    assert all(st["path_used"] == dl.PATHS["auto"] for st in layers)
    with dl.Context(0) as c:
        plain = check_sg(c, cyclic, want[2])
        for _ in range(3):
            for p, w, st in zip((forest, other), want, layers):
                now = check_sg(c, p, w)
                assert (now["path_used"], now["iters"], now["gpu_launches"]) == (
                    st["path_used"], st["iters"], st["gpu_launches"])
                now = check_sg(c, cyclic, want[2])
                assert now["path_used"] == plain["path_used"] and now["iters"] == plain["iters"]
        for _ in range(10):  # of one shape: looked for again after a while
            now = check_sg(c, cyclic, want[2])
            assert now["path_used"] == plain["path_used"] and now["iters"] == plain["iters"]
        bad = forest.copy()
        bad[n // 2, 3] = 7
        for call in (lambda: c.sg_least_model(bad), lambda: c.sg_least_model(forest, eps=3.0)):
            with pytest.raises(dl.DLError) as err:
                call()
            assert err.value.status == dl.DL_EINVAL
        assert check_sg(c, forest, want[0])["gpu_launches"] == layers[0]["gpu_launches"]


def test_walks_after_a_wide_closure():
    n = 3000
    dag = inputs.pa_dag(n, n)
    wide = dag | dag.T
    assert dag.sum(axis=1).max() > 256
    want, want_wide = oracle.tc_model(dag), oracle.tc_model(wide)
    with dl.Context(0) as c:
        c.tc_closure(dag)  # (the next call knows of heavy rows)
        bits, walks = c.tc_closure(dag)
        assert np.array_equal(bits, want)
        for _ in range(3):
            assert np.array_equal(c.tc_closure(wide)[0], want_wide)
        bits, now = c.tc_closure(dag)
        assert np.array_equal(bits, want)
        assert now["gpu_launches"] == walks["gpu_launches"] and now["recheck_sweeps"] == walks["recheck_sweeps"]
