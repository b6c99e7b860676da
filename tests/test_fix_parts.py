"""Precision of the fixed-point form of the FP64 operator (fix_core.cuh), on the host
with overflow checks, against the operator in extended precision: a component, or the
modes beside the constant one, that are small next to the rest of the element keep their
bits, and inputs whose signs add up reach the largest sums without overflow."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import sip
from paper_1607_03777_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
KIND = {"navier": 0, "neumann": 1, "dirichlet": 2}
BCS = [("navier",) * 4, synth.SINKER_BC, ("dirichlet",) * 4, ("neumann", "dirichlet", "navier", "neumann")]
NEUMANN = ("neumann",) * 4
LD = np.longdouble
# Roundings between exact integer sums, each at most 2^-53 of what it rounds: the factors
# (mesh sizes, their ratio, 2 / (2 b + 1), penalty: 6), s_i s_j into the integers (4) and out
# of them (5), and the grid itself (2^-55 of the component's largest entry, summed over the
# entries of a row): 16, twice that here.
TOL = 32 * 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended precision")
    so = str(tmp_path_factory.mktemp("fix") / "fix_parts.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ftrapv", "-shared", "-fPIC", "-o", so,
                    os.path.join(HERE, "fix_parts_check.cpp")], check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def fixed(lib, k, nx, ny, x, eta, bc):
    n = k + 1
    y = np.full(x.size, np.nan)
    x = np.ascontiguousarray(x.reshape(-1))
    kinds = np.array([KIND[b] for b in bc], dtype=np.int32)
    assert lib.fix_apply_parts(n, nx, ny, ctypes.c_double(1.0), ctypes.c_double(1.0), ptr(kinds),
                               ctypes.c_double(2.0 * n * n), ptr(x), ptr(eta), ptr(y)) == 0
    return y.reshape(ny, nx, 2, n, n)


def exact(k, nx, ny, x, eta, bc):
    """A x in extended precision, x[ey, ex, c, j, i] on the unit square."""
    n = k + 1
    i = np.arange(n)
    s = np.sqrt((2 * i + 1).astype(LD) / 2)
    m = np.minimum(i[:, None], i[None, :])
    even = (i[:, None] + i[None, :]) % 2 == 0
    G = np.where(even, s[:, None] * s[None, :] * (m * (m + 1)), LD(0))
    D = np.where((i[None, :] > i[:, None]) & ~even, 2 * s[:, None] * s[None, :], LD(0))
    sign = (-1.0) ** i
    V, S = [sign * s, s], [-sign * s * i * (i + 1) / 2, s * i * (i + 1) / 2]
    hx, hy = LD(1) / nx, LD(1) / ny
    u = x.reshape(ny, nx, 2, n, n).astype(LD)
    e2 = eta.reshape(ny, nx).astype(LD)
    e4 = e2[..., None, None]
    ux, uy = u[:, :, 0], u[:, :, 1]
    y = np.stack([e4 * (2 * hy / hx * ux @ G + hx / hy * G @ ux + D.T @ (uy @ D.T)),
                  e4 * (hy / hx * uy @ G + 2 * hx / hy * G @ uy + D @ (ux @ D))], axis=2)
    pen = 4 * (k + 1) ** 2
    for nc, hn, ht in ((0, hx, hy), (1, hy, hx)):
        w, e, out = (u, e2, y) if nc == 0 else (np.transpose(a, t) for a, t in (
            (u, (1, 0, 2, 4, 3)), (e2, (1, 0)), (y, (1, 0, 2, 4, 3))))   # views: [line, along, c, m, q]
        tc = 1 - nc
        e = e[..., None]
        val = [w @ V[s] for s in (0, 1)]
        der = [w @ S[s] * (2 / hn) for s in (0, 1)]
        shear = [v[:, :, nc] @ D.T * (2 / ht) for v in val]

        def add(at, s, wn, wt, tn, tt, sigma, own, half):
            sg = 1 if s else -1
            Pn = -ht * sg * tn / 2 - half * own * sg * (wt @ D) + ht * sigma * wn / 2
            Pt = -ht * sg * tt / 2 + ht * sigma * wt / 2
            for comp, P, Q in ((nc, Pn, -2 * half * own * sg * ht / hn * wn), (tc, Pt, -half * own * sg * ht / hn * wt)):
                out[:, at, comp] += P[..., None] * V[s] + Q[..., None] * S[s]

        L, R = slice(None, -1), slice(1, None)
        if w.shape[1] > 1:
            eL, eR = e[:, L], e[:, R]
            sigma = pen / hn * np.maximum(eL, eR)
            jump = val[1][:, L] - val[0][:, R]
            tn = eL * der[1][:, L, nc] + eR * der[0][:, R, nc]
            tt = (eL * (der[1][:, L, tc] + shear[1][:, L]) + eR * (der[0][:, R, tc] + shear[0][:, R])) / 2
            add(L, 1, jump[:, :, nc], jump[:, :, tc], tn, tt, sigma, eL, LD(0.5))
            add(R, 0, -jump[:, :, nc], -jump[:, :, tc], tn, tt, sigma, eR, LD(0.5))
        for s, at in ((0, slice(0, 1)), (1, slice(-1, None))):
            kind = bc[2 * nc + s]
            if kind == "neumann":
                continue
            own, vn, vt = e[:, at], val[s][:, at, nc], val[s][:, at, tc]
            full = kind == "dirichlet"
            tt = own * (der[s][:, at, tc] + shear[s][:, at])
            add(at, s, vn, vt * full, 2 * own * der[s][:, at, nc], tt * full, 2 * pen / hn * own, own, LD(1))
    return y


def magnitudes(k, nx, ny, eta, bc):
    return abs(sip.assemble_A(sip.Problem(nx, ny, k, eta, bc=bc)))


def check(lib, k, nx, ny, x, eta, bc, absA, part=None):
    """Rows of each component against the largest |A| |part| among them (part: x without
    what A maps to zero)."""
    n = k + 1
    part = x if part is None else part
    y, ref = fixed(lib, k, nx, ny, x, eta, bc), exact(k, nx, ny, part, eta, bc)
    size = (absA @ np.abs(part).reshape(-1)).reshape(ny, nx, 2, n, n).max(axis=(3, 4), keepdims=True)
    err = np.abs(y - ref)
    assert (err <= TOL * size).all(), (k, bc, float((err / size).max() / TOL))


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("mesh", [(1, 1), (17, 2), (5, 9)])
def test_small_parts(lib, k, mesh):
    nx, ny = mesh
    n = k + 1
    g = np.random.default_rng(10 * k + nx)
    for bc in BCS:
        eta = 10.0 ** g.uniform(0.0, 6.0, nx * ny)
        absA = magnitudes(k, nx, ny, eta, bc)
        for spread in (0.0, 6.0):   # of an element's components and of their constant modes
            x = g.standard_normal((ny, nx, 2, n, n)) * 10.0 ** g.uniform(-spread, spread, (ny, nx, 2, 1, 1))
            x[..., 0, 0] *= 10.0 ** g.uniform(-spread, spread, (ny, nx, 2))
            check(lib, k, nx, ny, x, eta, bc, absA)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_translation(lib, k):
    """A translation is in the null space where no boundary holds it: what lies on top of it
    is all that remains, to its own precision."""
    nx, ny, n = 17, 6, k + 1
    g = np.random.default_rng(k)
    eta = 10.0 ** g.uniform(0.0, 6.0, nx * ny)
    absA = magnitudes(k, nx, ny, eta, NEUMANN)
    for size, moves in ((1e-4, (1.0, 0.0)), (1e-8, (1.0, 0.0)), (1e-12, (0.7, -1.3)), (1e-30, (0.7, -1.3))):
        for still in ((), (0,), (1,)):   # components without modes of their own
            part = size * g.standard_normal((ny, nx, 2, n, n))
            part[..., 0, 0] = 0.0
            part[:, :, list(still)] = 0.0
            x = part.copy()
            x[..., 0, 0] = moves
            check(lib, k, nx, ny, x, eta, NEUMANN, absA, part)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_aligned_signs(lib, k):
    """Entries just below a power of two whose signs make every trace, jump and
    derivative sum as large as it gets (an overflow aborts)."""
    nx, ny, n = 9, 5, k + 1
    g = np.random.default_rng(k)
    eta = 10.0 ** g.uniform(0.0, 6.0, nx * ny)
    i = np.arange(n)
    checker = (-1.0) ** (np.arange(ny)[:, None] + np.arange(nx)[None, :])
    for bc in (BCS[0], BCS[2]):
        absA = magnitudes(k, nx, ny, eta, bc)
        for pat in range(16):
            x = np.full((ny, nx, 2, n, n), 1.0 - 2.0 ** -53)
            if pat & 1:
                x = x * (-1.0) ** i
            if pat & 2:
                x = x * ((-1.0) ** i)[:, None]
            if pat & 4:
                x = x * checker[:, :, None, None, None]
            if pat & 8:
                x[:, :, 1] *= -1.0
            check(lib, k, nx, ny, x, eta, bc, absA)
