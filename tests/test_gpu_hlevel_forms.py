"""Continuous levels in two launches or one per step, by the number of FP64 vertices that
share the launch: a hierarchy that changes form on the way down against the oracle's
V-cycle, and members of a grouped batch in either form, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import multigrid, sip
from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nh", [(144, 120, 3), (136, 124, 2), (132, 124, 2)])
def test_vcycle_changes_form(ctx, nx, ny, nh):
    k = 1
    eta = synth.random_eta(nx * ny, nx + ny, (0.0, 1.0))
    ref = sip.Problem(nx, ny, k, eta, bc=synth.SINKER_BC)
    r = synth.random_vector(8 * nx * ny, 5)
    z_ref = multigrid.HPMultigrid(ref, sip.assemble_A(ref), nh, seed=1)(r)
    prob = api.Problem(ctx, nx, ny, k, eta, bc=synth.SINKER_BC, n_hlevels=nh, seed=1)
    z = torch.empty(prob.n_u, dtype=torch.float64, device="cuda")
    prob.vcycle(torch.from_numpy(r).cuda(), z)
    # tolerance of the V-cycle tests
    assert np.linalg.norm(z.cpu().numpy() - z_ref) < 1e-9 * np.linalg.norm(z_ref)


@pytest.mark.parametrize("contrast", [50.0, 1e4])
def test_batch_members_in_either_form(ctx, contrast):
    """Six members of 64^2 share more vertices than the limit, two share fewer."""
    def grouped(count):
        args = ([], [], [], [])
        for i in range(count):
            wl = synth.single_box_inclusion(n=64, k=1, eta_in=contrast + i, n_hlevels=synth.levels_to_17(64))
            eta, rho = ctx.rasterise_inclusions(64, 64, wl.shapes)
            P = api.Problem(ctx, 64, 64, 1, eta.cpu().numpy(), bc=wl.bc, n_hlevels=wl.n_hlevels, seed=1)
            f = torch.empty(P.n_u, dtype=torch.float64, device="cuda")
            P.rhs_body_force(rho, synth.GRAVITY, f)
            for a, v in zip(args, (P, f, torch.empty_like(f), torch.empty(P.n_p, dtype=torch.float64, device="cuda"))):
                a.append(v)
        st, reps = api.solve_batch(ctx, *args, n_streams=count, rtol=1e-8, grouped=True)
        assert st == 0 and all(r["rel_residual"] <= 1e-8 for r in reps)
        return args[2:]

    many, few = grouped(6), grouped(2)
    for a, b in zip(many, few):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
