"""Streaming with one warp per cell and with blocks of 2, 4 and 8 warps per cell: an instance stepped alone
(a pool so small that a block streams each cell) and inside pools of growing size (which take fewer warps
per cell, then the warp-per-cell kernel) ends in the same state, bit for bit.  The cells' lists lie around
the edges of a chunk (512 records with 2 or 4 warps, 768 with eight) and of a group of 32, in both
precisions, with walls, reservoirs, far movers (vacuum, large dt) and staged lists (wave regime)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (problem, extra keywords): list lengths near 1, 32, 256, 512 and 768 records per cell
SMALL = [
    ("shock", dict(mach=3.0, n_cells=7, ppc_ref=31.0)),
    ("shock", dict(mach=8.0, n_cells=33, ppc_ref=256.0)),
    ("sod", dict(n_cells=21, Kn=3e-4, ppc_ref=512.0)),
    ("sod", dict(n_cells=9, Kn=1.0, ppc_ref=769.0, cfl=2.5)),
    ("uniform", dict(n_cells=5, Kn=1.0, ppc_ref=3.0, bc="vacuum")),
]


def _make(W, kind, kw, precision):
    kw = dict(kw, precision=precision)
    if kind == "uniform":
        return W.uniform(seed=5, **kw)
    return getattr(W, kind)(seed=5, **kw)


def _state(g, i):
    return g.particles(i), g.fields(i)[0], g.counters(i), g.cmax(i)


# fillers: cells and particles per cell of the instance added to the pool
@pytest.mark.parametrize("fill_cells,fill_ppc", [(1200, 40.0), (2600, 30.0), (20000, 20.0)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_same_state_for_every_warp_count(precision, fill_cells, fill_ppc):
    from paper_2305_12071_gb300 import duwp, workloads as W

    small = [_make(W, k, kw, precision) for k, kw in SMALL]
    filler = W.shock(2.0, n_cells=fill_cells, ppc_ref=fill_ppc, precision=precision, seed=9)
    pool = duwp.Solver(small + [filler])
    pool.step(6)
    for i, p in enumerate(small):
        alone = duwp.Solver(p)
        alone.step(6)
        a, b = _state(alone, 0), _state(pool, i)
        for k in a[0]:
            assert np.array_equal(a[0][k], b[0][k]), (i, k)
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[3], b[3]), i
        for k in a[2]:
            assert np.array_equal(a[2][k], b[2][k]), (i, k)
        alone.close()
    pool.close()


# pools with the QMC split mark the survivors of the absorption instead of copying them: instances stepped
# alone (Eq. p: copied; QMC: marked, streamed by a block) against the same in a pool with a QMC instance
# (marked, streamed by a warp in the larger pool), with lists past the survivor index's 2048 single words
@pytest.mark.parametrize("fill_cells,fill_ppc", [(40, 20.0), (20000, 20.0)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_same_state_with_marked_survivors(precision, fill_cells, fill_ppc):
    from paper_2305_12071_gb300 import duwp, workloads as W

    small = [W.sod(n_cells=21, Kn=3e-3, ppc_ref=90.0, precision=precision, seed=5),
             W.sod(n_cells=4, Kn=2e-3, ppc_ref=4500.0, precision=precision, seed=6),
             W.sod(n_cells=17, Kn=1e-2, ppc_ref=120.0, precision=precision, seed=7, split_mode="qmc", resample_mode="ce"),
             W.shock(3.0, n_cells=5, ppc_ref=3000.0, precision=precision, seed=8, split_mode="qmc")]
    filler = W.shock(2.0, n_cells=fill_cells, ppc_ref=fill_ppc, precision=precision, seed=9, split_mode="qmc")
    pool = duwp.Solver(small + [filler])
    pool.step(5)
    for i, p in enumerate(small):
        alone = duwp.Solver(p)
        alone.step(5)
        a, b = _state(alone, 0), _state(pool, i)
        assert a[2]["nabs"].sum() > 0, i
        for k in a[0]:
            assert np.array_equal(a[0][k], b[0][k]), (i, k)
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[3], b[3]), i
        for k in a[2]:
            assert np.array_equal(a[2][k], b[2][k]), (i, k)
        alone.close()
    pool.close()
