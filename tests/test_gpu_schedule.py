"""What the FP64 schedule codes run: 4 the fixed-point kernel, 1, 2, 3 and 5 kernels of FP64
arithmetic, with B and B^T one thread per mode as in Stokes solves of high contrast; each
of these against the double-double operators, every degree and boundary kind."""
import numpy as np
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu

BCS = [("navier",) * 4, synth.SINKER_BC, ("dirichlet",) * 4, ("neumann", "dirichlet", "navier", "neumann")]
# at most 100 roundings of 2^-53 on the chain of any entry, each of at most the largest result
# or (B, B^T: pressures in the null space leave nothing) the terms, h / 4 times the input
TOL = 100 * 2.0 ** -53


def widened(x):
    y = torch.zeros(2 * x.numel(), dtype=torch.float64, device="cuda")
    y[0::2] = x
    return y


def double_double(prob, u, p):
    """(A u, B p, B^T u) by the double-double operators, rounded."""
    zu, zp = torch.zeros(2 * prob.n_u, dtype=torch.float64, device="cuda"), \
        torch.zeros(2 * prob.n_p, dtype=torch.float64, device="cuda")
    f = torch.zeros(prob.n_u, dtype=torch.float64, device="cuda")
    ru, rp = torch.empty_like(zu), torch.empty_like(zp)
    prob.residual_dd(f, widened(u), zp, ru, rp)
    Au, Btu = -ru[0::2], -rp[0::2]
    prob.residual_dd(f, zu, widened(p), ru, rp)
    return Au.clone(), -ru[0::2], Btu.clone()


def operators(prob, u, p):
    y = [torch.full((n,), float("nan"), dtype=torch.float64, device="cuda") for n in (prob.n_u, prob.n_u, prob.n_p)]
    prob.apply_A(u, y[0])
    prob.apply_B(p, y[1])
    prob.apply_Bt(u, y[2])
    return y


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("mesh", [(1, 1), (33, 5), (70, 67)])
def test_operators_of_each_code(ctx, k, mesh):
    nx, ny = mesh
    for i, bc in enumerate(BCS):
        prob = api.Problem(ctx, nx, ny, k, synth.random_eta(nx * ny, 3 + i, (0.0, 4.0)), bc=bc, lx=1.0, ly=0.7)
        u = torch.from_numpy(synth.random_vector(prob.n_u, 4 + i)).cuda()
        p = torch.from_numpy(synth.random_vector(prob.n_p, 5 + i)).cuda()
        ref = double_double(prob, u, p)
        got = {}
        for code in (1, 2, 3, 4, 5) if k <= 5 else (3,):
            prob.set_schedule(apply=[code, 0])
            assert prob.schedule()["apply"][0] == code
            got[code] = operators(prob, u, p)
            h = 0.25 * min(1.0 / nx, 0.7 / ny)
            for y, r, term in zip(got[code], ref, (0.0, h * float(p.abs().max()), h * float(u.abs().max()))):
                assert float((y - r).abs().max()) <= TOL * max(float(r.abs().max()), term), (bc, code)
        if nx * ny > 1000 and k <= 5:   # roundings of another arithmetic fall differently somewhere
            assert all(not torch.equal(got[4][0], got[c][0]) for c in (1, 2, 3, 5)), bc
            assert all(torch.equal(a, b) for c in (2, 3, 5) for a, b in zip(got[1][1:], got[c][1:])), bc
            assert not torch.equal(got[4][1], got[1][1]) and not torch.equal(got[4][2], got[1][2]), bc


def test_unpinned_runs_the_default_again(ctx):
    """A pin of an FP64 kernel, taken back, leaves nothing of it after the next set-up."""
    n, k = 32, 3
    a, b = (api.Problem(ctx, n, n, k, np.ones(n * n), bc=synth.SINKER_BC, n_hlevels=1, seed=1) for _ in range(2))
    p = torch.from_numpy(synth.random_vector(a.n_p, 5)).cuda()
    y = [torch.empty(a.n_u, dtype=torch.float64, device="cuda") for _ in range(3)]
    b.set_schedule(apply=[1, 0])
    b.apply_B(p, y[0])
    b.set_schedule(apply=[0, 0])
    for q, out in ((a, y[1]), (b, y[2])):
        q.setup()
        q.apply_B(p, out)
    assert a.schedule() == b.schedule()
    assert torch.equal(y[1], y[2]) and not torch.equal(y[0], y[1])


@pytest.mark.parametrize("k,n,code", [(1, 32, 1), (1, 109, 1), (1, 110, 4), (1, 128, 4), (2, 8, 4), (5, 3, 4)])
def test_default_before_setup(ctx, k, n, code):
    """A problem that was not set up reports and runs the default: fixed point, but at degree
    1 on small meshes the component-split kernel."""
    prob = api.Problem(ctx, n, n, k, synth.random_eta(n * n, 3, (0.0, 3.0)), bc=synth.SINKER_BC)
    u = torch.from_numpy(synth.random_vector(prob.n_u, 4)).cuda()
    y = [torch.empty_like(u) for _ in range(2)]
    prob.apply_A(u, y[0])
    assert prob.schedule()["apply"][0] == code
    prob.set_schedule(apply=[code, 0])
    prob.apply_A(u, y[1])
    assert torch.equal(*y)
