"""Stokes solves of stiff problems (viscosity contrast above 128) run their operators in
FP64 arithmetic, viscous solves and V-cycles of the same problem in fixed point: neither
may leave its schedule behind for the other."""
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("contrast", [1e2, 1e3])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_schedules_do_not_mix(contrast, precision):
    n, k = 32, 2
    ctx = api.Context(0)
    wl = synth.single_box_inclusion(n=n, k=k, eta_in=contrast, n_hlevels=1)
    eta, rho = ctx.rasterise_inclusions(n, n, wl.shapes)

    def fresh():
        P = api.Problem(ctx, n, n, k, eta.cpu().numpy(), bc=wl.bc, n_hlevels=1, seed=1, precision=precision)
        P.set_schedule(apply=[5, 5], fused=[0, 0])   # bits do not depend on the autotuner
        return P

    def stokes(P):
        f, u = (torch.empty(P.n_u, dtype=torch.float64, device="cuda") for _ in range(2))
        p = torch.empty(P.n_p, dtype=torch.float64, device="cuda")
        P.rhs_body_force(rho, 10.0, f)
        rep = P.solve(f, u, p, rtol=1e-8)
        assert rep["status"] == 0 and rep["rel_residual"] <= 1e-8
        return torch.cat([u, p])

    def viscous(P):
        x = torch.as_tensor(synth.random_vector(P.n_u, 5)).cuda()
        y = torch.empty_like(x)
        P.inner_solve(x, y, rtol=1e-3)
        return y

    s0, v0 = stokes(fresh()), viscous(fresh())
    P, Q = fresh(), fresh()
    for a, b in ((stokes, viscous), (viscous, stokes)) * 2:
        assert torch.equal(a(P), s0 if a is stokes else v0)
        assert torch.equal(b(Q), s0 if b is stokes else v0)
    # a problem that turns stiff, and back
    P.update_eta(torch.ones_like(eta))
    stokes(P)
    P.update_eta(eta)
    assert torch.equal(stokes(P), s0) and torch.equal(viscous(P), v0)
