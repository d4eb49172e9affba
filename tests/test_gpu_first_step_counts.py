"""First steps of wave-regime cells with many candidates: nothing has arrived, so the absorption passes no
barrier between the two rounding draws of a cell (two threads) and the thread that forms the re-sampled and
the candidate count from them.  More such cells than the block kernel has blocks, so a block takes several
one after the other and a draw left over from the one before would change the counts: every count, and the
particles of the first step, equal the oracle's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_first_step_counts_of_empty_heavy_cells(precision):
    import oracle as O
    import torch
    from paper_2305_12071_gb300 import duwp, workloads as W

    plist = [W.sod(n_cells=500, Kn=kn, ppc_ref=ppc, precision=precision, seed=50 + i)
             for i, (kn, ppc) in enumerate([(2e-4, 300.0), (1e-4, 260.0), (1.5e-4, 310.0), (1.8e-4, 350.0), (1.2e-4, 280.0)])]
    orc = [O.Oracle(p) for p in plist]
    heavy = 0
    for o in orc:
        absorbs = o.prim()["P"] > 0
        assert len(o.particles()["cell"]) == 0
        o.step(1)
        heavy += int((absorbs & (o.counters()["ncand"] >= 96)).sum())
    # five blocks of the block kernel per SM: most of them take a second cell
    assert heavy > 1.5 * 5 * torch.cuda.get_device_properties(0).multi_processor_count
    g = duwp.Solver(plist)
    g.step(1)
    for i, o in enumerate(orc):
        for k, v in g.counters(i).items():
            assert np.array_equal(v, o.counters()[k]), (i, k)
        assert np.array_equal(g.particles(i)["cell"], o.particles()["cell"]), i
    g.close()
