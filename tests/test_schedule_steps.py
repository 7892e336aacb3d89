"""The level-scheduled micro sweeps at their edges: schedules shorter than the
prefetch, steps with one cell, ragged last velocity tiles, and one, two and
four velocities per thread.  With one velocity per thread in float32 a step's
coefficients are formed a step ahead; the arithmetic of a (cell, velocity) is
the same in every shape, so the states must agree bit for bit (the per-iteration
comparison with the oracle is test_unstructured's)."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {
    "triangles_2": I.tri_cavity(2, nv=10, cfl_imp=10.0),
    "triangles_7": I.tri_cavity(7, nv=13, cfl_imp=10.0),
    "triangles_40": I.tri_cavity(40, nv=8, cfl_imp=10.0),
    "hybrid_ring": I.hybrid_cylinder(ntheta=16, nr=6, nr_quad=3, nv=11, Ma=2.0, cfl_imp=10.0),
}


def state(prob, precision, tv, vpt):
    from paper_1709_01819_gb300.solver import Solver

    s = Solver(prob, precision)
    s.set_tuning(sweep_tv=tv, sweep_vpt=vpt)
    s.init_uniform()
    s.iterate(5)
    return s.get_state()


@pytest.mark.parametrize("name", sorted(CASES))
def test_every_launch_shape_gives_the_same_state(name):
    prob = CASES[name]
    ref = state(prob, "mixed", 1, 1)
    for tv, vpt in ((4, 1), (2, 2), (1, 4), (2, 4)):
        for a, b in zip(ref, state(prob, "mixed", tv, vpt)):
            assert np.array_equal(a, b), (tv, vpt)
    r64 = state(prob, "fp64", 4, 1)
    for a, b in zip(r64, state(prob, "fp64", 2, 2)):
        assert np.array_equal(a, b)
