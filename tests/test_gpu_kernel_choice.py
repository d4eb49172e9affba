"""Every kernel that the launch rules choose from is run by a pool shown to choose it (Solver.launch): the streaming
kernel with 1, 2, 4 and 8 warps per cell, its launch shapes, its form for cells that mark their survivors,
its periodic ends, specular walls and phantom ends with a warp per cell, and the collision kernel's reruns of
a batch on one warp.  Small instances in such pools end bit for bit as they do alone (a block per cell), where
the oracle tests hold them; the reruns are compared with the oracle itself."""
import numpy as np
import pytest

import oracle as O
from paper_2305_12071_gb300 import workloads as W
from parity_util import compare_counters, compare_fields, compare_particles, solver

pytestmark = pytest.mark.gpu


def _state(g, i=0):
    return {**g.particles(i), "psi": g.fields(i)[0], "cmax": g.cmax(i), **g.counters(i)}


def _equal(a, b, what):
    for k in a:
        assert np.array_equal(a[k], b[k]), (what, k)


def _periodic(precision):
    # 1.6 cells per step at the thermal speed: many far movers, and wraps across the whole domain
    return W.uniform(n_cells=37, Kn=0.05, ppc_ref=80, state=(1.0, 0.7, 0.0, 0.0, 1.0), bc="periodic", x_max=1.0,
                     dt=0.02, precision=precision, seed=11)


def _walls(precision):
    return W.sod(n_cells=40, Kn=3e-4, ppc_ref=150, precision=precision, seed=8)


# the pool's filler: its cells and particles per cell decide the warps per cell (fp32, fp64)
@pytest.mark.parametrize("fill,warps", [((20000, 20.0), (1, 1)), ((2600, 20.0), (1, 2)), ((1200, 20.0), (2, 4)),
                                        ((300, 20.0), (4, 4))])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_same_state_for_every_chosen_warp_count(precision, fill, warps):
    small = [_periodic(precision), _walls(precision), W.shock(8.0, n_cells=33, ppc_ref=60.0, precision=precision, seed=5)]
    pool = solver(small + [W.shock(2.0, n_cells=fill[0], ppc_ref=fill[1], precision=precision, seed=9)])
    info = pool.launch()
    assert info["stream_warps"] == warps[precision == "fp64"] and info["masked"] == 0
    assert info["ordered"] == (info["stream_warps"] == 1)
    pool.step(6)
    for i, p in enumerate(small):
        alone = solver(p)
        assert alone.launch()["stream_warps"] == 8
        alone.step(6)
        _equal(_state(alone), _state(pool, i), i)
        alone.close()
    pool.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_two_warps_per_cell_match_one(precision):
    # a pool that takes two warps per cell by itself, and one warp per cell beside a filler
    p = W.large_shock(n_cells=1500, ppc_ref=60.0, precision=precision, seed=4)
    a, b = solver(p), solver([p, W.shock(2.0, n_cells=20000, ppc_ref=20.0, precision=precision, seed=9)])
    assert a.launch()["stream_warps"] == 2 and b.launch()["stream_warps"] == 1
    a.step(6)
    b.step(6)
    _equal(_state(a), _state(b), "")
    a.close()
    b.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_every_launch_shape_on_a_warp_per_cell(precision):
    # all threads per block, register budgets and record groups the autotuner tries
    from paper_2305_12071_gb300 import autotune
    small = [_walls(precision), _periodic(precision), W.shock(8.0, n_cells=33, ppc_ref=200.0, precision=precision, seed=5)]
    plist = small + [W.shock(2.0, n_cells=20000, ppc_ref=20.0, precision=precision, seed=9)]
    ref = None
    for shape in autotune.CANDIDATES_FP32 + [(32, 0, 2)]:
        s = solver(plist)
        s.set_launch(*shape)
        info = s.launch()
        assert info["stream_warps"] == 1 and (info["threads"], info["reg_capped"], info["groups"]) == shape
        s.step(4)
        got = [_state(s, i) for i in range(len(plist))]
        s.close()
        ref = ref or got
        for i in range(len(plist)):
            _equal(ref[i], got[i], (shape, i))


@pytest.mark.parametrize("shape", [(128, 1, 2), (64, 0, 3)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_marked_survivors_on_a_warp_per_cell(precision, shape):
    # a pool with QMC instances: the warp-per-cell kernel skips the absorbed particles by their bits (lists
    # around 32 and 64 records, Eq. (p) cells that copy when alone, NS-corrected sampling)
    small = [W.sod(n_cells=21, Kn=3e-3, ppc_ref=90.0, precision=precision, seed=5),
             W.sod(n_cells=17, Kn=1e-2, ppc_ref=120.0, precision=precision, seed=7, split_mode="qmc", resample_mode="ce"),
             W.shock(3.0, n_cells=25, ppc_ref=32.0, precision=precision, seed=8, split_mode="qmc"),
             W.shock(6.0, n_cells=9, ppc_ref=100.0, precision=precision, seed=6, split_mode="qmc")]
    pool = solver(small + [W.shock(2.0, n_cells=20000, ppc_ref=20.0, precision=precision, seed=9, split_mode="qmc")])
    pool.set_launch(*shape)
    info = pool.launch()
    assert info["stream_warps"] == 1 and info["masked"] == 1
    pool.step(6)
    for i, p in enumerate(small):
        alone = solver(p)
        assert alone.launch()["stream_warps"] == 8
        alone.step(6)
        a = _state(alone)
        assert a["nabs"].sum() > 0, i
        _equal(a, _state(pool, i), i)
        alone.close()
    pool.close()


@pytest.mark.parametrize("make", [lambda pr: W.shock(3.0, n_cells=24000, ppc_ref=10.0, precision=pr, seed=2),
                                  lambda pr: W.sod(n_cells=24000, Kn=1e-5, ppc_ref=10.0, precision=pr, seed=4)],
                         ids=["shock", "sod"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_split_parts_on_a_warp_per_cell(precision, make):
    # phantom ends (the runs crossing into a neighbouring part) in the warp-per-cell kernel
    from paper_2305_12071_gb300 import duwp
    p = make(precision)
    whole, split = solver(p), duwp.Split(p, 2)
    assert whole.launch()["stream_warps"] == 1 and all(q.launch()["stream_warps"] == 1 for q in split.parts)
    whole.step(6)
    split.step(6)
    a = _state(whole)
    b = {**split.particles(), "psi": split.fields(), "cmax": split.cmax(), **split.counters()}
    _equal(a, b, "")
    split.close()
    whole.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_raises_of_cmax_in_batches_on_one_warp(precision):
    # a Mach-8 shock at small Kn, every cell absorbing, in a pool of more than seven cells per SM: cells with 8 to
    # 95 candidates are collided by one warp each, and particles meeting cold cells raise c_max inside a
    # batch, which reruns up to the raising candidate
    p = W.shock(8.0, omega=0.81, n_cells=80, ppc_ref=60.0, precision=precision, seed=3)
    p["Kn"] = 0.01
    o = O.Oracle(p)
    g = solver([p, W.shock(2.0, n_cells=1200, ppc_ref=20.0, precision=precision, seed=9)])
    assert g.launch()["heavy_min"] == 96
    raised = 0
    for step in range(10 if precision == "fp64" else 5):
        cm0, P = o.cmax().copy(), o.prim()["P"].copy()
        o.step(1)
        g.step(1)
        n = o.counters()["ncand"]
        raised += int(((o.cmax() > cm0) & (P > 0) & (n >= 8) & (n < 96)).sum())
        compare_counters(g.counters(0), o.counters(), f"step {step + 1}")
        compare_particles(g.particles(0), o.particles(), 1e-9 if precision == "fp64" else 1e-5, f"step {step + 1}")
        compare_fields(g.fields(0)[0], o.psi(), 1e-9, f"step {step + 1}")
    assert raised > 0
    g.close()
