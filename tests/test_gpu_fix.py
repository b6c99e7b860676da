"""GPU parity of the fixed-point FP64 apply (schedule codes 4 and 5, the
default): tile edges and both tile shapes against the oracle, its error against
the double-double operator beside the FP64 kernel's, and values outside its
range (infinities, NaN, magnitudes near the ends of FP64), which take the FP64
formulas and reach the same entries as in the FP64 kernel."""
import numpy as np
import pytest
import torch

from oracle import sip
from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu

BCS = [("navier",) * 4, synth.SINKER_BC, ("dirichlet",) * 4, ("neumann", "dirichlet", "navier", "neumann")]
FP64, FIX = 1, 4
TOL64 = 1e-10   # of the FP64 operators against the oracle


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=torch.float64)


def apply(prob, x, code):
    prob.set_schedule(apply=[code, 0])
    y = torch.full_like(x, float("nan"))
    prob.apply_A(x, y)
    return y


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("mesh", [(1, 1), (9, 5), (37, 3), (4, 35)])
def test_apply_fix(ctx, k, mesh):
    nx, ny = mesh
    for i, bc in enumerate(BCS):
        eta = synth.random_eta(nx * ny, 40 + i, (0.0, 6.0))
        prob = api.Problem(ctx, nx, ny, k, eta, bc=bc, lx=1.0, ly=0.7)
        A = sip.assemble_A(sip.Problem(nx, ny, k, eta, bc=bc, lx=1.0, ly=0.7))
        x = synth.random_vector(prob.n_u, 50 + i)
        y = apply(prob, dev(x), FIX).cpu().numpy()
        size = (abs(A) @ np.abs(x)).reshape(nx * ny, -1).max(axis=1, keepdims=True)
        assert (np.abs(y - A @ x).reshape(nx * ny, -1) <= TOL64 * size).all(), bc


@pytest.mark.parametrize("k,n", [(2, 131), (3, 129), (4, 131), (5, 99)])
def test_apply_fix_error_not_above_fp64(ctx, k, n):
    """2-norm error against the double-double operator: at most that of the
    FP64 kernel (both are a few 2^-53)."""
    eta = synth.random_eta(n * n, 3, (0.0, 4.0))
    prob = api.Problem(ctx, n, n, k, eta, bc=synth.SINKER_BC)
    x = dev(synth.random_vector(prob.n_u, 4))
    xu = torch.zeros(2 * prob.n_u, dtype=torch.float64, device="cuda")
    xu[0::2] = x
    xp = torch.zeros(2 * prob.n_p, dtype=torch.float64, device="cuda")
    ru, rp = torch.empty_like(xu), torch.empty_like(xp)
    prob.residual_dd(torch.zeros_like(x), xu, xp, ru, rp)
    err = {c: float(((apply(prob, x, c) + ru[0::2]) + ru[1::2]).norm() / ru[0::2].norm()) for c in (FP64, FIX)}
    assert err[FIX] <= err[FP64] < 1e-15, err


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_apply_fix_out_of_range(ctx, k):
    nx, ny = 21, 11
    eta = synth.random_eta(nx * ny, 5, (0.0, 3.0))
    prob = api.Problem(ctx, nx, ny, k, eta, bc=BCS[3])
    g = np.random.default_rng(k)
    base = synth.random_vector(prob.n_u, 6)
    for value in (np.nan, np.inf, -np.inf, 1e300, 1e-310):
        x = base.copy()
        x[g.integers(0, x.size, 3)] = value
        a, b = (apply(prob, dev(x), c).cpu().numpy() for c in (FP64, FIX))
        assert (np.isnan(a) == np.isnan(b)).all() and (np.isinf(a) == np.isinf(b)).all(), value
        fine = np.isfinite(a)
        assert np.abs(a - b)[fine].max() <= 1e-13 * np.abs(a[fine]).max(), value
    for scale in (1e-300, 1e250):
        a, b = (apply(prob, dev(base * scale), c).cpu().numpy() for c in (FP64, FIX))
        assert np.abs(a - b).max() <= 1e-13 * np.abs(a).max(), scale
