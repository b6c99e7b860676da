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


@pytest.mark.parametrize("inner_loop", ["device", "host"])
@pytest.mark.parametrize("k", [2, 3])
def test_marked_tiles_of_the_fp32_cycle(ctx, k, inner_loop):
    """Mixed form, contrast 1e5: the solve's FP32 cycle runs its marked tiles in FP64
    arithmetic, so a run with pinned FP64 kernels has its bits; outside a solve they run in
    fixed point unless an FP64 kernel is pinned."""
    n = 32
    P, f = problem(ctx, n, k, 1e5, "mixed")
    got = solve(P, f, inner_loop=inner_loop)
    pinned = []
    for code in (1, 2, 3, 5):
        Q, g = problem(ctx, n, k, 1e5, "mixed", code)
        pinned.append(solve(Q, g, inner_loop=inner_loop))
    assert any(torch.equal(got, p) for p in pinned)
    # a linear field without strain: what remains inside is rounding, another in either form
    m, h = k + 1, 1.0 / n
    x = torch.zeros(n, n, 2, m, m, dtype=torch.float64)
    at = (torch.arange(n, dtype=torch.float64) + 0.5) * h - 0.5
    x[:, :, 0, 0, 0], x[:, :, 1, 0, 0] = -2.0 * at[:, None], 2.0 * at[None, :]
    x[:, :, 0, 1, 0], x[:, :, 1, 0, 1] = -h / 3.0 ** 0.5, h / 3.0 ** 0.5
    x = x.reshape(-1).float().cuda()
    y = [torch.empty_like(x) for _ in range(3)]
    for q, out in ((P, y[0]), (Q, y[1])):
        q.apply_A_f32(x, out)
    assert P.schedule()["apply"][1] == 4   # marked tiles
    assert not torch.equal(y[0], y[1])
    Q.set_schedule(apply=[4, 0])
    Q.setup()
    Q.apply_A_f32(x, y[2])
    assert torch.equal(y[0], y[2])


@pytest.mark.parametrize("contrast", [1e2, 1e3])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_fixed_point_and_fp64_do_not_mix(ctx, contrast, precision):
    """With the fixed-point kernel pinned a stiff problem's viscous solves run it and its
    Stokes solves FP64 kernels: neither leaves its schedule behind for the other."""
    def fresh():
        P, f = problem(ctx, 32, 2, contrast, precision, code=4)
        P.set_schedule(fused=[0, 0])   # bits do not depend on the autotuner
        return P, f

    def viscous(P, f):
        x = torch.as_tensor(synth.random_vector(P.n_u, 5)).cuda()
        y = torch.empty_like(x)
        P.inner_solve(x, y, rtol=1e-3)
        return y

    s0, v0 = solve(*fresh()), viscous(*fresh())
    P, Q = fresh(), fresh()
    for _ in range(2):
        assert torch.equal(solve(*P), s0) and torch.equal(viscous(*Q), v0)
        assert torch.equal(viscous(*P), v0) and torch.equal(solve(*Q), s0)
