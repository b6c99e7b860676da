"""The V-cycle with its continuous levels in two launches each, against the
oracle's: tiles of 2 to 6 coarse vertices with cut edges, one to four steps (and
five, which takes one launch per step), FP64 and FP32 (tolerances of the
V-cycle tests)."""
import numpy as np
import pytest
import torch

from oracle import multigrid, sip
from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nh,steps", [(20, 12, 2, 3), (24, 16, 1, 1), (24, 16, 3, 2), (36, 20, 2, 4),
                                            (20, 12, 2, 5), (64, 60, 2, 3), (660, 12, 2, 3)])
def test_vcycle_levels(ctx, nx, ny, nh, steps):
    k = 1
    eta = synth.random_eta(nx * ny, nx + ny, (0.0, 1.0))
    ref = sip.Problem(nx, ny, k, eta, bc=synth.SINKER_BC)
    r = synth.random_vector(8 * nx * ny, 5).astype(np.float32).astype(np.float64)
    z_ref = multigrid.HPMultigrid(ref, sip.assemble_A(ref), nh, seed=1, h_steps=steps)(r)
    for precision, dtype, tol in (("fp64", torch.float64, 1e-9), ("mixed", torch.float32, 2e-4)):
        prob = api.Problem(ctx, nx, ny, k, eta, bc=synth.SINKER_BC, n_hlevels=nh, cheb_steps_h=steps,
                           seed=1, precision=precision)
        z = torch.empty(prob.n_u, dtype=dtype, device="cuda")
        x = torch.from_numpy(r).to("cuda", dtype)
        (prob.vcycle if precision == "fp64" else prob.vcycle_f32)(x, z)
        err = np.linalg.norm(z.double().cpu().numpy() - z_ref) / np.linalg.norm(z_ref)
        assert err < tol, (precision, err)
