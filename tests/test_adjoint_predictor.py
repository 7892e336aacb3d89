"""The transposed macroscopic sweep of blocks whose increments do not fit shared
memory (more than 7168 cells), of up to 128 lines and of more: the adjoint's
first two passes against central differences of the forward iteration about the
gas at rest (steady from the first iteration up to the quadrature's error, which
a few remove, where a driven flow on so many cells takes tens of thousands),
held to the bounds of the smaller blocks' test (1e-6 of the objective's
derivative, 1e-5 of one iteration's increments summed against the multipliers:
with a relative step of 1e-5 the differences' truncation is of order 1e-10 and
their rounding 1e-11 of the state)."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LID = 1 << I.JMAX


@pytest.mark.parametrize("ni,nj", [(90, 80), (129, 131)])
def test_transposed_predictor_from_global_memory(ni, nj):
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver

    p = I.cavity(ni, Kn=0.1, U=0.0, nv=8)
    p.nodes_x, p.nodes_y = I.uniform_nodes(ni, nj)
    s = Solver(p, "fp64")
    s.init_uniform()
    s.iterate(300)
    G, H, W = s.get_state()
    rng = np.random.default_rng(21)
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
    print(ni, nj, ad1, fd1, ad2, fd2)
    assert abs(ad1 - fd1) <= 1e-6 * abs(fd1), (ad1, fd1)
    assert abs(ad2 - fd2) <= 1e-5 * abs(fd2), (ad2, fd2)
