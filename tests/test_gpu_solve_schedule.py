"""Stokes solves of viscosity contrast above 128 keep the kernels of FP64 arithmetic
whatever ran before them and however they are solved."""
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu


def problem(ctx, n, k, contrast, precision="fp64", code=0):
    """(problem, load vector) of a box inclusion of this contrast."""
    wl = synth.single_box_inclusion(n=n, k=k, eta_in=contrast, n_hlevels=synth.levels_to_17(n))
    eta, rho = ctx.rasterise_inclusions(n, n, wl.shapes)
    P = api.Problem(ctx, n, n, k, eta.cpu().numpy(), bc=wl.bc, n_hlevels=wl.n_hlevels, seed=1,
                    precision=precision)
    if code:
        P.set_schedule(apply=[code, 0])
    f = torch.empty(P.n_u, dtype=torch.float64, device="cuda")
    P.rhs_body_force(rho, synth.GRAVITY, f)
    return P, f


def solve(P, f, **kw):
    u, p = torch.empty_like(f), torch.empty(P.n_p, dtype=torch.float64, device="cuda")
    rep = P.solve(f, u, p, rtol=1e-8, **kw)
    assert rep["rel_residual"] <= 1e-8
    return torch.cat([u, p])


@pytest.mark.parametrize("n,k", [(32, 1), (32, 2), (64, 2), (128, 2), (32, 3), (64, 3)])
def test_fp32_setup_keeps_the_choice(ctx, n, k):
    """A set-up of the FP32 cycle between set-up and solve changes no bit: the fused or
    split smoother of the solve's schedule is the FP64 set-up's choice."""
    P, f = problem(ctx, n, k, 1e3)
    Q, _ = problem(ctx, n, k, 1e3)
    Q.setup()
    x = torch.as_tensor(synth.random_vector(Q.n_u, 3)).float().cuda()
    Q.vcycle_f32(x, torch.empty_like(x))
    assert torch.equal(solve(P, f), solve(Q, f))


def grouped(ctx, members):
    """Grouped batch of (problem, load vector) pairs; the solutions."""
    fs = [f for _, f in members]
    us = [torch.empty_like(f) for f in fs]
    ps = [torch.empty(P.n_p, dtype=torch.float64, device="cuda") for P, _ in members]
    st, reps = api.solve_batch(ctx, [P for P, _ in members], fs, us, ps, n_streams=len(members), rtol=1e-8,
                               grouped=True)
    assert st == 0 and all(r["rel_residual"] <= 1e-8 for r in reps)
    return [torch.cat([u, p]) for u, p in zip(us, ps)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("k", [2, 3])
def test_grouped_stiff_members(ctx, precision, k):
    """Stiff members of a grouped batch run the FP64 kernels: their bits are those of one of
    the pinned kernels (outer operator and set-up follow the pin, the inner loop is the
    same).  Members of low contrast do not depend on them."""
    contrasts = (1e3, 1e4, 1e2)

    def run(code, which=contrasts):
        return grouped(ctx, [problem(ctx, 32, k, c, precision, code) for c in which])

    got, pinned = run(0), [run(code) for code in (1, 2, 3, 5)]
    for m in (0, 1):
        assert any(torch.equal(got[m], p[m]) for p in pinned), contrasts[m]
    assert torch.equal(got[2], run(0, (1e2, 50.0))[0])
