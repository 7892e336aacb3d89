"""Launch-shape tuning: what is read back is what runs.  Setting what was read
leaves the shape as it is; a tile that is accepted is the one that runs; a
request that shared memory does not hold is refused and changes nothing; lines
padded to whole warps may cost a step of the prefetch depth, which is read back;
an unstructured mesh has one depth.  The widest tiles, whose border rings or
lines per warp give way, give the bits of the default shape."""
import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu

LIMIT = 227 * 1024  # bytes of shared memory a block can have


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


def _block(ni, nj, nv=8):
    p = I.cavity(2, Kn=0.2, nv=nv, cfl_imp=50.0)
    p.nodes_x, p.nodes_y = I.uniform_nodes(ni, nj, 0.0, 1.0, 0.0, 1.0)
    return p


def _solver(prob, prec):
    from paper_1709_01819_gb300.solver import Solver
    return Solver(prob, prec)


def _request_bytes(lines, tv, vpt, stages, prec):
    """stages steps of `lines` cells (R or Delta* and f~ of the tile, a record),
    and two steps' borders."""
    T = 8 if prec == "fp64" else 4
    tile = tv * vpt * 2 * T
    return lines * (stages * (2 * tile + 9 * T + 16) + 2 * tile)


PROBLEMS = {"square": _block(20, 20), "lines128": _block(128, 128), "narrow": I.couette(40, U=0.1, Kn=0.1, nv=8), "three": _block(3, 9), "wide": _block(100, 130),
            "many_velocities": _block(65, 66, nv=40), "widest": _block(256, 256, nv=4),
            "triangles": I.tri_cavity(6, nv=8, cfl_imp=10.0)}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_setting_what_was_read_leaves_the_shape(name, prec):
    s = _solver(PROBLEMS[name], prec)
    own = s.tuning()
    s.set_tuning(**own)
    assert s.tuning() == own
    other = 1 if own["sweep_tv"] > 1 else 2
    s.set_tuning(sweep_tv=other)
    assert s.tuning()["sweep_tv"] == other
    s.set_tuning(**own)
    assert s.tuning() == own


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("lines", [2, 5, 9, 12, 16, 17, 21, 25, 32, 37, 43, 46, 58, 64, 81, 85, 128])
def test_a_tile_runs_as_asked_or_is_refused(lines, prec):
    from paper_1709_01819_gb300 import binding as B
    s = _solver(_block(lines, lines + 1), prec)
    for tv in (1, 2, 4, 8, 16, 32):
        for vpt in (1, 2, 4):
            for st in (2, 4, 8):
                if tv * lines > 512:
                    continue
                s.set_tuning(sweep_stages=2, sweep_tv=1, sweep_vpt=1)
                ask = dict(sweep_tv=tv, sweep_vpt=vpt, sweep_stages=st)
                need = _request_bytes(lines, tv, vpt, st, prec)
                try:
                    s.set_tuning(**ask)
                except B.IdgError as e:
                    assert e.status == B.IDG_ERR_ARG and need > LIMIT
                    continue
                got = s.tuning()
                assert (got["sweep_tv"], got["sweep_vpt"]) == (tv, vpt)
                if got["sweep_stages"] != st:  # only the padding and the rings stand in the way
                    assert got["sweep_stages"] < st and need <= LIMIT < 1.6 * need


def test_a_refused_call_changes_nothing_and_one_key_leaves_the_others():
    from paper_1709_01819_gb300 import binding as B
    s = _solver(_block(16, 16), "fp64")
    s.set_tuning(sweep_tv=8)
    before = s.tuning()
    s.set_tuning(sweep_vpt=2)
    assert s.tuning() == dict(before, sweep_vpt=2)
    s.set_tuning(sweep_tv=32, sweep_vpt=4, sweep_stages=2)
    before = s.tuning()
    with pytest.raises(B.IdgError):
        B.idg_set_tuning(s.ctx, B.IDG_TUNE_SWEEP_STAGES, 8)
    assert s.tuning() == before
    m = _solver(PROBLEMS["many_velocities"], "mixed")
    auto = m.tuning()["sweep_vpt"]
    assert auto > 1
    m.set_tuning(sweep_tv=2)
    assert m.tuning()["sweep_vpt"] == auto


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["lines128", "wide", "widest"])
def test_one_key_is_taken_by_an_untouched_solver(name, prec):
    """The depth a solver starts with is one its tile can have: nothing has to be
    set first."""
    for key in ("sweep_tv", "sweep_vpt"):
        s = _solver(PROBLEMS[name], prec)
        s.set_tuning(**{key: 1})
        assert s.tuning()[key] == 1


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_an_unstructured_mesh_prefetches_four_steps(prec):
    from paper_1709_01819_gb300 import binding as B
    s = _solver(PROBLEMS["triangles"], prec)
    assert s.tuning()["sweep_stages"] == 4
    s.set_tuning(sweep_stages=4)
    for st in (2, 8):
        with pytest.raises(B.IdgError) as e:
            s.set_tuning(sweep_stages=st)
        assert e.value.status == B.IDG_ERR_ARG
    assert s.tuning()["sweep_stages"] == 4


@pytest.mark.parametrize("lines,tile", [(57, (8, 4, 2)), (29, (16, 4, 2)), (14, (32, 4, 2)), (20, (16, 4, 4)),
                                        (11, (32, 4, 4)), (6, (32, 4, 8)), (42, (8, 2, 8))])
def test_the_widest_tiles_give_the_bits_of_the_default_shape(lines, tile):
    prob = _block(lines, lines + 2, nv=11)
    G, H, W = I.random_state(prob, 5)
    out = []
    for shape in (None, tile):
        s = _solver(prob, "fp64")
        s.init_uniform()
        if shape:
            s.set_tuning(sweep_tv=tile[0], sweep_vpt=tile[1], sweep_stages=tile[2])
            assert s.tuning()["sweep_tv"] == tile[0] and s.tuning()["sweep_vpt"] == tile[1]
        s.set_state(G, H, W)
        s.iterate(3)
        out.append(s.get_state())
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


def test_the_autotuner_times_the_librarys_own_shape():
    from paper_1709_01819_gb300.solver import Autotuner
    s = _solver(PROBLEMS["narrow"], "mixed")
    s.init_uniform()
    own = s.tuning()
    assert own["sweep_tv"] == 32
    best = Autotuner(candidates_tv=(), repeats=1).tune(s)
    assert s.tuning() == own and best["sweep_tv"] == 32
