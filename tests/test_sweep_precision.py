"""Rounding of the float32 micro sweeps on a structured block.

The diagonal D of a cell enters every step of a line, so an error that is the
same in all its cells adds up along the line: on the mixed solver's 90 x 70
block G was 0.96e-9 (LU-SGS predictor) and 1.05e-9 (point relaxation) off the
float64 solver's, rms after 16 iterations, with the fluxes' sum rounded by
itself, and is 0.42e-9 and 0.43e-9 with them added to the cell's base, as it was
when a hyperplane was swept at a time; 0.6e-9 lies between.

The reciprocal of D is the correctly rounded one for every float whose
reciprocal is normal."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1709_01819_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_01819_gb300 import build
    build.build()


@pytest.mark.parametrize("relax", [0, 9])
def test_the_diagonals_rounding_does_not_add_up_along_the_lines(relax):
    from paper_1709_01819_gb300.solver import Solver
    p = I.cavity(90, 0.5, 0.15, 27, 4.0, 1000.0)
    p.vrule = I.NC_SIMPSON
    p.nodes_x, p.nodes_y = I.uniform_nodes(90, 70, 0.0, 1.0, 0.0, 70 / 90)
    west = list(p.bc[I.IMIN])
    west[4] = 1.03
    p.bc[I.IMIN] = tuple(west)
    p.relax_sweeps = relax
    G = {}
    for prec in ("fp64", "mixed"):
        s = Solver(p, prec)
        s.init_uniform()
        s.iterate(16)
        G[prec] = s.get_state()[0]
    err = float(np.sqrt(np.mean((G["mixed"] - G["fp64"]) ** 2)))
    assert err < 0.6e-9, err


RECIPROCALS = r"""
#include "wavefront.cuh"
__global__ void check(unsigned long long *off)
{
    const unsigned long long n = 253ull << 23;  // the normal floats of one sign but the largest exponent
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((unsigned)(i + (1u << 23))), r = __frcp_rn(x);
        if (r >= 1.17549435e-38f && idg::rcp_nr(x) != r) atomicAdd(off, 1ull);
    }
}
extern "C" int reciprocals_off(unsigned long long *count)
{
    unsigned long long *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 8);
    if (e == cudaSuccess) e = cudaMemset(d, 0, 8);
    if (e == cudaSuccess) check<<<4096, 256>>>(d);
    if (e == cudaSuccess) e = cudaMemcpy(count, d, 8, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""


def test_the_sweeps_reciprocal_is_correctly_rounded(tmp_path):
    from paper_1709_01819_gb300 import build
    src, lib = tmp_path / "reciprocals.cu", tmp_path / "reciprocals.so"
    src.write_text(RECIPROCALS)
    subprocess.run([build.NVCC, *build.ARCH, "-O3", "-std=c++17", "-I" + build.CSRC, "-shared", "-Xcompiler", "-fPIC",
                    str(src), "-o", str(lib)], check=True, capture_output=True)
    off = ctypes.c_ulonglong(1)
    assert ctypes.CDLL(os.fspath(lib)).reciprocals_off(ctypes.byref(off)) == 0
    assert off.value == 0
