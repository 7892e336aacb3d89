"""Workspace sizes (no GPU work): a buffer that held a problem when the
increments, or each adjoint solve's scratch, had memory of their own still holds
it."""
import json

import pytest

from paper_1709_01819_gb300 import binding as B
from paper_1709_01819_gb300 import build as BUILD
from paper_1709_01819_gb300 import inputs as I
from paper_1709_01819_gb300.solver import configure


@pytest.fixture(scope="module", autouse=True)
def _built():
    BUILD.build()


def _relaxed(p):
    p.relax_sweeps = 9
    return p


# bytes: float64, mixed, as they were
SIZES = json.loads("""{
  "couette64": [6031384, 3335192],
  "couette64_v8": [993304, 793112],
  "cavity64": [346565144, 175536664],
  "cavity64_v8": [29918744, 17190424],
  "cavity128_v28": [1064448536, 540340248],
  "cavity64_relax": [346696216, 175602200],
  "long": [29049880, 16695320],
  "cylinder": [8734767640, 4372522264],
  "cylinder48x32_v21": [80405784, 41214232],
  "triangles64": [621458200, 346948376],
  "triangles8_v8": [1377048, 1033496]
}""")

PROBLEMS = {"couette64": lambda: I.couette(64), "couette64_v8": lambda: I.couette(64, nv=8),
            "cavity64": lambda: I.cavity(64, nv=32), "cavity64_v8": lambda: I.cavity(64, nv=8),
            "cavity128_v28": lambda: I.cavity(128, nv=28), "cavity64_relax": lambda: _relaxed(I.cavity(64, nv=32)),
            "long": lambda: I.couette(4000, nv=8), "cylinder": I.cylinder_c5,
            "cylinder48x32_v21": lambda: I.cylinder(48, 32, nv=21), "triangles64": lambda: I.tri_cavity(64, nv=32),
            "triangles8_v8": lambda: I.tri_cavity(8, nv=8)}


@pytest.mark.parametrize("name", sorted(SIZES))
def test_no_workspace_has_grown(name):
    for prec, size in ((B.IDG_FP64, SIZES[name][0]), (B.IDG_MIXED, SIZES[name][1])):
        ctx = B.idg_create(prec, 0)
        configure(ctx, PROBLEMS[name]())
        assert B.idg_workspace_size(ctx) <= size
        B.idg_destroy(ctx)


# closed domains: two solves
ADJOINT = {"couette64": 29743616, "couette64_v8": 2909696, "cavity64": 1840644352, "cavity64_v8": 120324352,
           "cavity128_v28": 5629411584, "long": 117116672}


@pytest.mark.parametrize("name", sorted(ADJOINT))
def test_no_closed_domains_adjoint_workspace_has_grown(name):
    ctx = B.idg_create(B.IDG_FP64, 0)
    configure(ctx, PROBLEMS[name]())
    assert B.idg_adjoint_workspace_size(ctx) <= ADJOINT[name]
    B.idg_destroy(ctx)
