"""fb at the faces from the cells' side (k_cell_recon): velocities along a face
(both sides count half), on axis-aligned and diagonal faces, interior and
boundary, across a direction one cell wide and on triangles; limiter on and
off, alone and in one batch; cell counts that do not fill a block's cells.
FP64 against the oracle at the parity suite's bound (1e-12 of the largest
value per iteration)."""
import dataclasses
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


def _rotated(prob, angle):
    c, s = math.cos(angle), math.sin(angle)
    X, Y = prob.nodes_x, prob.nodes_y
    return dataclasses.replace(prob, nodes_x=np.ascontiguousarray(c * X - s * Y),
                               nodes_y=np.ascontiguousarray(s * X + c * Y))


def _cases():
    odd = I.cavity(6, Kn=0.1, nv=9, cfl_imp=50.0)
    c = {"axis_ties": odd,
         "diagonal_ties": _rotated(I.cavity(5, Kn=0.1, nv=8, cfl_imp=50.0), 0.25 * math.pi),
         "axis_ties_limited": dataclasses.replace(odd, limiter=1),
         "one_wide_periodic": I.couette(7, nv=9),
         "triangles": I.tri_cavity(4, Kn=0.1, nv=9, cfl_imp=10.0),
         "triangles_limited": dataclasses.replace(I.tri_cavity(4, Kn=0.1, nv=9, cfl_imp=10.0), limiter=1),
         # four cells a block from 4864 blocks of 256 velocities on, two from 2432
         "cells_4_per_block_ragged": I.cavity(71, Kn=0.1, nv=16, cfl_imp=50.0),
         # a row of velocities shared by two and by four warps (2116, 4225 velocities)
         "rows_2_warps": dataclasses.replace(I.cavity(4, Kn=0.1, nv=46, cfl_imp=50.0), implicit_wall=1),
         "rows_4_warps": dataclasses.replace(I.cavity(4, Kn=0.1, nv=65, cfl_imp=50.0), implicit_wall=1),
         "cells_2_per_block_ragged": I.cavity(51, Kn=0.1, nv=16, cfl_imp=50.0)}
    p = c["axis_ties"]
    c["unequal_rows_and_columns"] = dataclasses.replace(p, nvx=11, nvy=7)
    return c


CASES = _cases()


@pytest.mark.parametrize("name", sorted(CASES))
def test_faces_match_the_oracle(name):
    from paper_1709_01819_gb300.solver import Solver
    prob = CASES[name]
    G, H, W = I.random_state(prob, 3, amp=0.02)
    o = O.Oracle(prob)
    o.set_state(G, H, W)
    s = Solver(prob, "fp64")
    s.init_uniform()
    s.set_state(G, H, W)
    o.iterate(2)
    s.iterate(2)
    for a, b in zip(s.get_state(), o.get_state()):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max(), name


def test_limited_and_unlimited_instances_share_a_batch():
    from paper_1709_01819_gb300.solver import BatchSolver, Solver
    probs = [CASES["axis_ties"], CASES["axis_ties_limited"]]
    b = BatchSolver(probs, "mixed")
    b.iterate(3)
    for prob, s in zip(probs, b.solvers):
        one = Solver(prob, "mixed")
        one.init_uniform()
        one.iterate(3)
        for x, y in zip(one.get_state(), s.get_state()):
            np.testing.assert_array_equal(x, y)
