"""The adjoint's workspace: nothing of what it held before reaches the result."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

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
