"""Long runs replay graphs of several steps: the state after any sequence of step counts, odd ones and both
read parities among them, equals that of plain launches, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("calls", [(130,), (65, 3, 5, 4, 9, 1, 8), (1,) * 66 + (4, 7, 12)])
def test_multi_step_graphs_equal_plain_launches(calls):
    from paper_2305_12071_gb300 import duwp, workloads as W

    p = W.shock(3.0, n_cells=24, ppc_ref=25.0, precision="fp64", seed=3)
    a, b = duwp.Solver(p), duwp.Solver(p, graphs=False)
    for n in calls:
        a.step(n)
        b.step(n)
    assert a.info()["steps_done"] == b.info()["steps_done"] == sum(calls)
    pa, pb = a.particles(), b.particles()
    for k in pa:
        assert np.array_equal(pa[k], pb[k]), k
    assert np.array_equal(a.fields()[0], b.fields()[0])
    assert np.array_equal(a.fields(which=duwp.AVERAGED)[0], b.fields(which=duwp.AVERAGED)[0])
    a.close()
    b.close()
