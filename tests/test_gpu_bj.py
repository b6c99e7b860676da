"""The block-Jacobi apply where its CTAs serve more than one group of elements.

M_K z_K = r_K is checked with the operator itself: on a checkerboard colour no two
elements share a face, so A of a vector supported there gives M_K z_K on each."""
import numpy as np
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,nx,ny", [(1, 216, 208), (2, 144, 136), (2, 160, 128), (3, 8, 24), (5, 8, 8)])
def test_inverse_blocks(k, nx, ny):
    ctx = api.Context(0)
    # all interior, side and corner classes, and a ring of unique blocks
    ex, ey = np.arange(nx * ny) % nx, np.arange(nx * ny) // nx
    eta = np.where((ex > nx // 3) & (ex < 2 * nx // 3) & (ey > ny // 3) & (ey < 2 * ny // 3), 1e2, 1.0)
    P = api.Problem(ctx, nx, ny, k, eta, bc=synth.SINKER_BC, n_hlevels=3)
    r = torch.as_tensor(np.random.default_rng(3).uniform(-1.0, 1.0, P.n_u)).cuda()
    z, t = torch.empty_like(r), torch.empty_like(r)
    P.block_jacobi(r, z)
    colour = torch.as_tensor((ex + ey) % 2).cuda().repeat_interleave(2 * (k + 1) ** 2)
    got = torch.zeros_like(r)
    for c in (0, 1):
        P.apply_A(torch.where(colour == c, z, torch.zeros_like(z)), t)
        got = torch.where(colour == c, t, got)
    # FP64 rounding times the blocks' condition (below 1e6 at k = 5, contrast 1e2)
    assert float((got - r).norm() / r.norm()) <= 1e-8


@pytest.mark.parametrize("k,nx,ny", [(2, 184, 184), (3, 144, 128), (4, 104, 96), (5, 72, 64), (6, 56, 56)])
def test_inverse_blocks_in_fp32_cycle(k, nx, ny):
    """The FP32 V-cycle, whose smoother takes the kernel above, against the FP64 one."""
    ctx = api.Context(0)
    ex, ey = np.arange(nx * ny) % nx, np.arange(nx * ny) // nx
    eta = np.where((ex > nx // 3) & (ex < 2 * nx // 3) & (ey > ny // 3) & (ey < 2 * ny // 3), 10.0, 1.0)
    r = torch.as_tensor(np.random.default_rng(4).uniform(-1.0, 1.0, 2 * (k + 1) ** 2 * nx * ny)).cuda().float()
    z = []
    for precision in ("fp64", "mixed"):
        P = api.Problem(ctx, nx, ny, k, eta, bc=synth.SINKER_BC, n_hlevels=3, seed=1, precision=precision)
        x = r.double() if precision == "fp64" else r
        z.append(torch.empty_like(x))
        (P.vcycle if precision == "fp64" else P.vcycle_f32)(x, z[-1])
    # the tolerance of the FP32 V-cycle tests
    assert float((z[1].double() - z[0]).norm() / z[0].norm()) <= 2e-4
