"""The adjoint's transposed sweeps along lines of cells, where a block holds
more than one strip of lines and where a periodic seam lies along or across
the lines: the adjoint's first two passes against central differences of the
forward iteration (the second pass runs the transposed micro and macroscopic
sweeps over every cell).

Tolerances: with a step of 1e-5 on the relative perturbation the differences'
truncation is of order 1e-10 relative and their rounding of order
1e-16 / 1e-5 = 1e-11 of the state, a few orders below the 1e-6 (objective) and
1e-5 (one iteration's increments, summed against the multipliers) held here.
"""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LID = 1 << I.JMAX


def channel(ni, nj, nv):
    """Walls below and above, periodic in x, the upper wall moving."""
    X, Y = I.uniform_nodes(ni, nj)
    bc = [(I.BC_PERIODIC, 0, 0, 0, 0), (I.BC_PERIODIC, 0, 0, 0, 0),
          (I.BC_WALL, 1.0, -0.1, 0.0, 1.0), (I.BC_WALL, 1.0, 0.1, 0.0, 1.0)]
    return I.Problem(X, Y, bc, I.NC_TRAP, nv, nv, (-4.0, 4.0, -4.0, 4.0), K=1, Pr=1.0, omega=0.5,
                     Kn=0.1, shakhov=0, cfl_imp=100.0, init=(1.0, 0.0, 0.0, 1.0),
                     name=f"channel_{ni}x{nj}_v{nv}")


CASES = {
    "two_velocities_a_warp_two_strips": I.cavity(n=20, nv=18, Kn=0.075, name="cavity_20_v18"),
    "one_velocity_a_warp_two_strips": I.cavity(n=35, nv=8, Kn=0.075, name="cavity_35_v8"),
    "seam_along_rows": channel(36, 34, 8),
    "seam_across_columns": channel(34, 36, 8),
}


@pytest.mark.parametrize("name", list(CASES))
def test_transposed_sweeps_match_forward_differences(name):
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver

    s = Solver(CASES[name], "fp64")
    s.init_uniform()
    ok, n, r = s.iterate(40000, 1e-12)
    assert ok, (n, r)
    G, H, W = s.get_state()
    rng = np.random.default_rng(20)
    v = [u * rng.standard_normal(u.shape) for u in (G, H, W)]
    s.adjoint(B.IDG_OBJ_FORCE_X, LID, [], 1, 0.0, keep_state=True)
    l1 = s.adjoint_state(1)
    s.adjoint(B.IDG_OBJ_FORCE_X, LID, [], 2, 0.0, keep_state=True)
    l2 = s.adjoint_state(1)
    eps, J, u = 1e-5, {}, {}
    for sign in (1, -1):
        s.set_state(*[a + sign * eps * b for a, b in zip((G, H, W), v)])
        s.iterate(1)
        J[sign], u[sign] = s.wall_force(LID)[0], s.get_state()
    dot = lambda lam, w: sum(float(np.sum(a * b)) for a, b in zip(lam, w))  # noqa: E731
    fd1 = (J[1] - J[-1]) / (2 * eps)
    ad1 = dot(l1, v)
    fd2 = dot(l1, [(a - b) / (2 * eps) for a, b in zip(u[1], u[-1])])
    ad2 = dot([a - b for a, b in zip(l2, l1)], v)
    print(name, ad1, fd1, ad2, fd2)
    assert abs(ad1 - fd1) <= 1e-6 * abs(fd1), (ad1, fd1)
    assert abs(ad2 - fd2) <= 1e-5 * abs(fd2), (ad2, fd2)
