"""The acceptance test by bounds of u^(2/e) at every exponent e = 1 - 2 upsilon: hard spheres (e = 1), the usual
VHS gases, nearly and exactly Maxwell molecules (e small and 0), on cells with few candidates (collision
kernel) and many (block kernel): candidates, accepted pairs and cell order equal the oracle's exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("omega", [0.5, 0.68, 0.81, 0.95, 0.9999, 1.0])
def test_accepted_pairs_equal_the_oracle(omega, precision):
    import oracle as O
    from paper_2305_12071_gb300 import duwp, workloads as W

    # cells of about 15, 60 and 250 particles; Kn sets about 2 to 200 candidates per cell and step
    probs = [W.shock(3.0, omega=omega, n_cells=12, ppc_ref=15.0, half_width=6.0, precision=precision, seed=21),
             W.shock(6.0, omega=omega, n_cells=10, ppc_ref=60.0, half_width=10.0, precision=precision, seed=22),
             W.sod(n_cells=8, Kn=2e-2, ppc_ref=250.0, omega=omega, precision=precision, seed=23)]
    steps = 8 if precision == "fp64" else 4
    for p in probs:
        g, o = duwp.Solver(p), O.Oracle(p)
        g.step(steps)
        o.step(steps)
        for k, v in g.counters().items():
            assert np.array_equal(v, o.counters()[k]), (p["n_cells"], k)
        assert g.counters()["nacc"].sum() > 0
        assert np.array_equal(g.particles()["cell"], o.particles()["cell"])
        g.close()
