"""The line micro sweeps of a structured block at the edges of their shapes:
lines short of a warp, one over it, one cell wide, periodic across and along
the lines, every split of a warp between lines and velocities.  FP64 against
the oracle after three iterations at the parity suite's per-iteration bound
(1e-12 of the largest value), mixed precision bitwise the same for every shape
(the arithmetic of a cell does not depend on the launch)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

PER = (I.BC_PERIODIC, 0, 0, 0, 0)
WALL = (I.BC_WALL, 1.0, 0.1, 0.0, 1.1)
STILL = (I.BC_WALL, 1.0, 0.0, 0.0, 1.0)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


def _block(ni, nj, per_i, per_j, nv=7):
    X, Y = I.uniform_nodes(ni, nj, 0.0, 1.0, 0.0, 1.0)
    if not per_i and not per_j:  # slanted cells: every normal differs
        X, Y = X + 0.05 * Y * X, Y + 0.03 * X * Y
    bc = [PER, PER] if per_i else [STILL, STILL]
    bc += [PER, PER] if per_j else [STILL, WALL]
    p = I.cavity(2, Kn=0.2, nv=nv, cfl_imp=50.0)
    p.nodes_x, p.nodes_y, p.bc = np.ascontiguousarray(X), np.ascontiguousarray(Y), bc
    return p


BLOCKS = [(1, 7, True, False), (7, 1, False, True), (2, 5, False, False), (2, 9, True, False), (9, 2, True, True),
          (3, 3, True, True), (4, 37, False, False), (33, 9, False, True), (32, 35, True, False), (65, 33, False, False),
          (17, 66, False, True)]


@pytest.mark.parametrize("ni,nj,per_i,per_j", BLOCKS)
def test_line_sweeps_at_the_edges_of_their_shapes(ni, nj, per_i, per_j):
    from paper_1709_01819_gb300.solver import Solver
    prob = _block(ni, nj, per_i, per_j)
    G0, H0, W0 = I.random_state(prob, 5)
    o = O.Oracle(prob)
    o.set_state(G0, H0, W0)
    o.iterate(3)
    Go, Ho, Wo = o.get_state()
    shapes = [None] + [(tv, vpt, st) for tv in (1, 2, 8, 32) for vpt in (1, 2, 4) for st in (2, 8)
                       if tv * min(ni, nj) <= 512]
    ref = None
    for shape in shapes:
        for prec in ("fp64", "mixed"):
            if prec == "fp64" and shape not in (None, (1, 1, 2), (2, 4, 8), (8, 2, 2)):
                continue
            s = Solver(prob, prec)
            s.init_uniform()
            if shape:
                s.set_tuning(sweep_tv=shape[0], sweep_vpt=shape[1], sweep_stages=shape[2])
            s.set_state(G0, H0, W0)
            s.iterate(3)
            got = s.get_state()
            if prec == "fp64":
                for a, b in zip(got, (Go, Ho, Wo)):
                    assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), shape
            elif ref is None:
                ref = got
            else:
                for a, b in zip(got, ref):
                    np.testing.assert_array_equal(a, b, err_msg=str(shape))
