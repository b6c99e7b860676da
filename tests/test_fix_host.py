"""The fixed-point form of the FP64 operator (fix_core.cuh), compiled for the
host with overflow checks and run tile by tile against the oracle's assembled
matrix: ragged tiles, every boundary kind, k = 1..5, element magnitudes that
differ by 1e12 and viscosities by 1e6."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import sip
from paper_1607_03777_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
TOL64 = 1e-10
KIND = {"navier": 0, "neumann": 1, "dirichlet": 2}
BCS = [("navier",) * 4, synth.SINKER_BC, ("dirichlet",) * 4, ("neumann", "dirichlet", "navier", "neumann")]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    so = str(tmp_path_factory.mktemp("fix") / "fix_host.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ftrapv", "-shared", "-fPIC", "-o", so,
                    os.path.join(HERE, "fix_host_check.cpp")], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("mesh", [(1, 1), (17, 3), (4, 19)])
def test_fixed_point_apply(lib, k, mesh):
    """Entry errors against the magnitude of the terms they sum, |A| |x| over
    the element, to the tolerance of the FP64 operators (the oracle's quadrature
    points carry coordinates of the whole domain, which leaves it about 1e-13)."""
    nx, ny = mesh
    n = k + 1
    g = np.random.default_rng(100 * k + nx)
    for i, bc in enumerate(BCS):
        eta = synth.random_eta(nx * ny, 7 + i, (0.0, 6.0))
        A = sip.assemble_A(sip.Problem(nx, ny, k, eta, bc=bc, lx=1.0, ly=0.7))
        for spread in (0.0, 6.0):
            x = g.standard_normal((nx * ny, 2 * n * n)) * 10.0 ** g.uniform(-spread, spread, (nx * ny, 1))
            x = np.ascontiguousarray(x.reshape(-1))
            y = np.full_like(x, np.nan)
            kinds = np.array([KIND[b] for b in bc], dtype=np.int32)
            st = lib.fix_apply(n, nx, ny, ctypes.c_double(1.0), ctypes.c_double(0.7), ptr(kinds),
                               ctypes.c_double(2.0 * n * n), ptr(x), ptr(eta), ptr(y))
            assert st == 0
            size = (abs(A) @ np.abs(x)).reshape(nx * ny, -1).max(axis=1, keepdims=True)
            err = np.abs(y - A @ x).reshape(nx * ny, -1)
            assert (err <= TOL64 * size).all(), (bc, spread, (err / np.maximum(size, 1e-300)).max())


def test_out_of_range_factors_are_refused(lib):
    x = np.zeros(8)
    eta = np.ones(1)
    kinds = np.zeros(4, dtype=np.int32)
    for ly, ch in ((1e7, 8.0), (1.0, 1e10), (1.0, 0.0)):
        assert lib.fix_apply(2, 1, 1, ctypes.c_double(1.0), ctypes.c_double(ly), ptr(kinds),
                             ctypes.c_double(ch), ptr(x), ptr(eta), ptr(np.zeros(8))) == 1
