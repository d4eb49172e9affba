"""The order in which the warp-per-cell passes of a large pool take its cells needs no memory beyond the handle's
own slab: a caller's arena that holds the slab and nothing else still creates and steps such a pool.  The
order shares its place with a work list, so a checkpoint (which keeps that list, not the order) restores
bit for bit into a fresh handle."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _pool(W, precision):
    # 80 cells with 33 to 95 collision candidates (a warp each) and a pool large enough for a warp per cell
    return [W.shock(8.0, n_cells=80, ppc_ref=200.0, half_width=10.0, precision=precision, seed=3),
            W.shock(2.0, n_cells=20000, ppc_ref=20.0, precision=precision, seed=9)]


def _same(a, b):
    for i in range(a.n):
        pa, pb = a.particles(i), b.particles(i)
        for k in pa:
            assert np.array_equal(pa[k], pb[k]), (i, k)
        assert np.array_equal(a.fields(i)[0], b.fields(i)[0]) and np.array_equal(a.cmax(i), b.cmax(i)), i
        ca, cb = a.counters(i), b.counters(i)
        for k in ca:
            assert np.array_equal(ca[k], cb[k]), (i, k)


def test_one_allocation_creates_and_steps_a_large_pool():
    import torch
    from paper_2305_12071_gb300 import duwp, workloads as W

    plist = _pool(W, "fp32")
    a = duwp.Solver(plist)
    assert a._alloc.calls == 1
    L = duwp.load()
    stream = torch.cuda.Stream()
    blocks = []

    def alloc(nbytes, s, ctx):
        if blocks:
            return None                       # the arena is used up
        blocks.append(torch.empty(int(nbytes), dtype=torch.uint8, device="cuda"))
        return blocks[0].data_ptr()

    fa, ff = duwp.ALLOC_FN(alloc), duwp.FREE_FN(lambda p, n, s, c: None)
    arr = (duwp.Params * len(plist))(*[duwp.make_params(p) for p in plist])
    h = C.c_void_p()
    torch.cuda.synchronize()
    assert L.duwp_init_batch(arr, len(plist), C.c_void_p(stream.cuda_stream), fa, ff, None, C.byref(h)) == duwp.OK
    assert L.duwp_step(h, 3) == duwp.OK
    a.step(3)
    for i, p in enumerate(plist):
        out, navg = np.empty((p["n_cells"], 5)), C.c_int64()
        assert L.duwp_fields(h, i, duwp.INSTANT, out.ctypes.data_as(C.POINTER(C.c_double)), p["n_cells"], C.byref(navg)) == duwp.OK
        assert np.array_equal(out, a.fields(i)[0])
    assert L.duwp_destroy(h) == duwp.OK
    a.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_checkpoint_of_an_ordered_pool(precision):
    from paper_2305_12071_gb300 import duwp, workloads as W

    plist = _pool(W, precision)
    a = duwp.Solver(plist)
    a.step(5)
    blob = a.checkpoint()
    a.step(4)
    n = a.counters(0)["ncand"]
    assert ((n > 32) & (n < 96)).sum() > 10
    b = duwp.Solver(plist)
    b.restore(blob)
    assert b.checkpoint() == blob
    b.step(4)
    _same(a, b)
    a.close()
    b.close()
