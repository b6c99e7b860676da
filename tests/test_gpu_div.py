"""B and B^T in FP64 where their CTAs of 32 elements end: full, cut and single
columns, every boundary kind and degree, against the oracle (tolerance of the
FP64 operators), and <B p, u> = <p, B^T u> to rounding."""
import numpy as np
import pytest
import torch

from oracle import sip
from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu

TOL64 = 1e-10
BCS = [("navier",) * 4, synth.SINKER_BC, ("neumann", "dirichlet", "navier", "neumann")]


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("mesh", [(32, 2), (33, 1), (31, 3), (65, 2)])
def test_B_and_Bt_tiles(ctx, k, mesh):
    nx, ny = mesh
    for i, bc in enumerate(BCS):
        prob = api.Problem(ctx, nx, ny, k, np.ones(nx * ny), bc=bc, lx=0.8, ly=1.3)
        p, u = synth.random_vector(prob.n_p, 3 + i), synth.random_vector(prob.n_u, 4 + i)
        yu = torch.full((prob.n_u,), float("nan"), dtype=torch.float64, device="cuda")
        yp = torch.full((prob.n_p,), float("nan"), dtype=torch.float64, device="cuda")
        prob.apply_B(torch.from_numpy(p).cuda(), yu)
        prob.apply_Bt(torch.from_numpy(u).cuda(), yp)
        yu, yp = yu.cpu().numpy(), yp.cpu().numpy()
        # both are sums of terms of this size: a few hundred roundings of 2^-53 of it
        assert abs(yu @ u - yp @ p) <= 1e-13 * np.linalg.norm(yu) * np.linalg.norm(u), bc
        if i == 0 or k <= 3:
            B = sip.assemble_B(sip.Problem(nx, ny, k, np.ones(nx * ny), bc=bc, lx=0.8, ly=1.3))
            assert np.abs(yu - B @ p).max() <= TOL64 * np.abs(yu).max(), bc
            assert np.abs(yp - B.T @ u).max() <= TOL64 * np.abs(yp).max(), bc
