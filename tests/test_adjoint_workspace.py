"""The adjoint's workspace: nothing of what it held before reaches the result,
and the smaller layout gives what the full one gives: a buffer of the size a
far-field problem needed before the Maxwellians and couplings were kept
(201708288 bytes for 48 x 32 cells with 21 x 21 velocities) is taken.  Both
layouts form the same numbers by the same functions; only the rounding of
contracted multiply-adds may differ, 1e-12 of the largest multiplier after the
passes made here.  A closed domain's two solves share their scratch; what holds
neither layout is refused."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

OLD = 201708288
WALL = 1 << I.JMIN


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


def _run(s, buf, nbytes, method):
    from paper_1709_01819_gb300 import binding as B
    B.idg_set_adjoint_solver(s.ctx, method, 4)
    p = [B.IDG_PARAM(B.IDG_PAR_KN), B.IDG_PARAM(B.IDG_PAR_WALL_T, WALL)]
    st, J, g, n, r = B.idg_adjoint(s.ctx, B.IDG_OBJ_FORCE_X, WALL, p, buf, nbytes, 12, 0.0, s.stream)
    return J, g, B.idg_adjoint_state(s.ctx, buf, 0, s.N, s.Nv, s.stream)


@pytest.mark.parametrize("method", [0, 1])
def test_a_workspace_full_of_nan_gives_the_same_bits(method):
    import torch
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver
    s = Solver(I.cylinder(24, 16, nv=11, Ma=2.0, vmax=9.0, cfl_imp=10.0), "fp64")
    s.init_uniform()
    s.iterate(20)
    B.idg_set_adjoint_solver(s.ctx, method, 4)
    nbytes = B.idg_adjoint_workspace_size(s.ctx)
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    buf = (ws.data_ptr() + 255) & ~255
    out = []
    for fill in (0, 255):
        ws.fill_(fill)
        out.append(_run(s, buf, nbytes, method))
    assert out[0][0] == out[1][0] and np.array_equal(out[0][1], out[1][1])
    for a, b in zip(out[0][2], out[1][2]):
        assert np.isfinite(a).all() and np.array_equal(a, b)


@pytest.mark.parametrize("method", [0, 1])
def test_a_far_field_problem_runs_in_the_smaller_layout(method):
    import torch
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver
    s = Solver(I.cylinder(48, 32, nv=21, Ma=2.0, vmax=9.0, cfl_imp=10.0), "fp64")
    s.init_uniform()
    s.iterate(20)
    B.idg_set_adjoint_solver(s.ctx, method, 4)
    full = B.idg_adjoint_workspace_size(s.ctx)
    krylov = full
    B.idg_set_adjoint_solver(s.ctx, 0, 4)
    krylov -= B.idg_adjoint_workspace_size(s.ctx)  # the Krylov vectors come on top of either layout
    old = OLD + krylov
    assert old < full
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    buf = (ws.data_ptr() + 255) & ~255
    J, g, lam = _run(s, buf, full, method)
    for nbytes in (full - 1, old):
        ws.fill_(255)  # nothing of the run before is left
        J2, g2, lam2 = _run(s, buf, nbytes, method)
        assert J2 == J
        np.testing.assert_allclose(g2, g, rtol=1e-11)
        for a, b in zip(lam2, lam):
            assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
    with pytest.raises(B.IdgError) as e:
        _run(s, buf, old - full // 4, method)
    assert e.value.status == B.IDG_ERR_OOM
    # a full workspace afterwards is laid out in full again
    J3, g3, lam3 = _run(s, buf, full, method)
    assert J3 == J and np.array_equal(g3, g) and all(np.array_equal(a, b) for a, b in zip(lam3, lam))


def test_a_closed_domain_runs_both_solves_in_either_layout():
    import torch
    from paper_1709_01819_gb300 import binding as B
    from paper_1709_01819_gb300.solver import Solver
    s = Solver(I.cavity(14, Kn=0.1, U=0.15, nv=12), "fp64")
    s.init_uniform()
    s.iterate(50)
    full = B.idg_adjoint_workspace_size(s.ctx)
    ws = torch.empty(full + 256, dtype=torch.uint8, device="cuda")
    buf = (ws.data_ptr() + 255) & ~255
    lid = 1 << I.JMAX
    p = [B.IDG_PAR_KN, B.IDG_PARAM(B.IDG_PAR_WALL_U, lid)]
    out = []
    for nbytes in (full, full - 1):
        st, J, g, n, r = B.idg_adjoint(s.ctx, B.IDG_OBJ_FORCE_X, lid, p, buf, nbytes, 40, 0.0, s.stream)
        out.append((J, g, [B.idg_adjoint_state(s.ctx, buf, q, s.N, s.Nv, s.stream) for q in range(3)]))
    assert out[0][0] == out[1][0]
    np.testing.assert_allclose(out[1][1], out[0][1], rtol=1e-11)
    for x, y in zip(out[1][2], out[0][2]):
        for a, b in zip(x, y):
            assert np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 1e-300)
