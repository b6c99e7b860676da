"""The fixed-point operator on the GPU where one component, or the modes beside the
constant one, are small next to the rest of the element: a translation, which no Neumann
boundary holds, with something small on top, against the FP64 kernel on the small part
alone; both tile shapes, cut tiles, and the marked tiles of the FP32 operator."""
import numpy as np
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu

FP64, FIX = 1, 4
NEUMANN = ("neumann",) * 4


def apply(prob, x, code):
    prob.set_schedule(apply=[code, 0])
    y = torch.full_like(x, float("nan"))
    prob.apply_A(x, y)
    return y


def translated(n_e, n, size, g):
    """(small part, small part on a translation); exact in FP32 and FP64."""
    part = (size * g.standard_normal((n_e, 2, n, n))).astype(np.float32).astype(np.float64)
    part[:, 0] = 0.0
    part[:, 1, 0, 0] = 0.0
    x = part.copy()
    x[:, 0, 0, 0], x[:, 1, 0, 0] = 1.0, -1.5
    return [torch.from_numpy(a.reshape(-1)).cuda() for a in (part, x)]


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("mesh", [(9, 5), (37, 3), (133, 101)])
@pytest.mark.parametrize("size", [1e-4, 1e-8, 1e-12])
def test_translation(ctx, k, mesh, size):
    nx, ny = mesh
    prob = api.Problem(ctx, nx, ny, k, synth.random_eta(nx * ny, 5, (0.0, 6.0)), bc=NEUMANN)
    part, x = translated(nx * ny, k + 1, size, np.random.default_rng(k))
    ref, y = apply(prob, part, FP64), apply(prob, x, FIX)
    # both errors: a few dozen roundings of the terms, which are at most 100 times the result
    assert float((y - ref).norm() / ref.norm()) < 1e-13


@pytest.mark.parametrize("k", [2, 3, 4, 5])
def test_translation_marked_tiles(ctx, k):
    """FP32 vectors, FP64-accurate tiles next to stiff elements: inside the mesh, where no
    boundary holds the translation, the result is the small part's, rounded to FP32 (2^-24)."""
    n = 64
    eta = np.ones(n * n)
    eta[::7] = 1e5
    prob = api.Problem(ctx, n, n, k, eta, bc=synth.SINKER_BC, n_hlevels=2, seed=1, precision="mixed")
    part, x = translated(n * n, k + 1, 1e-12, np.random.default_rng(k))
    prob.setup()
    assert prob.schedule()["apply"][1] == 4   # marked tiles
    y = torch.full_like(x, float("nan")).float()
    prob.apply_A_f32(x.float(), y)
    ref = apply(prob, part, FP64)
    inside = lambda v: v.reshape(n, n, -1)[1:-1, 1:-1].double()   # noqa: E731
    assert float((inside(y) - inside(ref)).norm() / inside(ref).norm()) < 2.0 ** -23
