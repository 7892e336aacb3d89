"""A wait between the warps of a sweep kernel that runs out (idg_set_wait_limit
with no poll beyond the first: a strip of lines gives up on the strip before it)
is reported as IDG_ERR_TIMEOUT by every call that launches such a kernel, also
where the stale values make the residual NaN; no wait is endless and no access
depends on what was read, so the kernels end by themselves.  A restart with the
default limit gives the bits of a solver that never timed out."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

POLLS = 1 << 22


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


def _timeout(call):
    from paper_1709_01819_gb300 import binding as B
    with pytest.raises(B.IdgError) as e:
        call()
    assert e.value.status == B.IDG_ERR_TIMEOUT, e.value
    assert "ran out" in str(e.value)


def _solver(prec, n=64):
    from paper_1709_01819_gb300.solver import Solver
    s = Solver(I.cavity(n, Kn=0.1, U=0.15, nv=8), prec)
    s.init_uniform()
    return s


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_iterations_report_a_wait_that_ran_out(prec):
    from paper_1709_01819_gb300 import binding as B
    ref = _solver(prec)
    ref.iterate(3)
    s = _solver(prec)
    B.idg_set_wait_limit(s.ctx, 0)
    _timeout(lambda: s.iterate(1))
    _timeout(lambda: s.iterate(16))  # sticky until the restart
    s.init_uniform()
    _timeout(s.iterate_profiled)
    B.idg_set_wait_limit(s.ctx, POLLS)
    s.init_uniform()
    s.iterate(3)
    for a, b in zip(s.get_state(), ref.get_state()):
        assert np.array_equal(a, b)
    with pytest.raises(B.IdgError) as e:
        B.idg_set_wait_limit(s.ctx, -1)
    assert e.value.status == B.IDG_ERR_ARG


def test_a_batch_reports_the_instance_whose_wait_ran_out():
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import BatchSolver
    bs = BatchSolver([I.cavity(64, Kn=0.1, U=0.15, nv=8), I.cavity(6, Kn=0.5, U=0.1, nv=8)], "mixed")
    B.idg_set_wait_limit(bs.solvers[0].ctx, 0)
    _timeout(lambda: bs.iterate(2))
    assert "ran out" in B.idg_last_error(bs.solvers[0].ctx)
    assert len(bs.solvers[1].residual_history()) == 2
    bs.solvers[1].iterate(2)  # the other instance is untouched


def test_the_adjoint_reports_its_own_waits_and_leaves_the_iteration_alone():
    from paper_1709_01819_gb300 import binding as B
    s = _solver("fp64", 35)  # two strips of lines
    s.iterate(5)
    ok, J, g, n, r = s.adjoint(B.IDG_OBJ_FORCE_X, 1 << I.JMAX, [], 2, 0.0)
    B.idg_set_wait_limit(s.ctx, 0)
    _timeout(lambda: s.adjoint(B.IDG_OBJ_FORCE_X, 1 << I.JMAX, [], 2, 0.0))
    B.idg_set_wait_limit(s.ctx, POLLS)
    s.iterate(1)  # nothing of the adjoint's is blamed on the iteration
    s.iterate(0)
    s.adjoint(B.IDG_OBJ_FORCE_X, 1 << I.JMAX, [], 2, 0.0)


def test_the_gmres_adjoint_reports_its_waits():
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver
    s = Solver(I.cylinder(36, 34, 0.1, 2.0, 9, vmax=9.0, cfl_imp=10.0), "fp64")
    s.init_uniform()
    s.iterate(3)
    B.idg_set_wait_limit(s.ctx, 0)
    _timeout(lambda: s.adjoint(B.IDG_OBJ_FORCE_X, 1 << I.JMIN, [], 8, 1e-8, solver="gmres", restart=4))
