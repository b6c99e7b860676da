"""B and B^T by even and odd sums: 2-norm error against extended precision at most that of
the kernels that take one thread per mode (any pinned FP64 schedule code)."""
import numpy as np
import pytest
import torch

from paper_1607_03777_gb300 import api, synth

pytestmark = pytest.mark.gpu

LD = np.longdouble


def exact(k, nx, ny, bc, p, u):
    """B p and B^T u in extended precision on the unit square, with FP64 mesh sizes."""
    n = k + 1
    s = np.sqrt((2 * np.arange(n) + 1).astype(LD) / 2)
    i = np.arange(n)
    D = np.where((i[None, :] > i[:, None]) & ((i[:, None] + i[None, :]) % 2 == 1), 2 * s[:, None] * s[None, :], LD(0))
    V = [(-1.0) ** i * s, s]
    hx, hy = LD(1.0 / nx), LD(1.0 / ny)
    p, u = p.reshape(ny, nx, k, k).astype(LD), u.reshape(ny, nx, 2, n, n).astype(LD)
    Bp, Btu = np.zeros((ny, nx, 2, n, n), dtype=LD), np.zeros((ny, nx, k, k), dtype=LD)
    for c, h in ((0, hy), (1, hx)):
        # views [line, along, m, q], q along the normal
        turn = lambda a: a if c == 0 else np.swapaxes(np.swapaxes(a, -1, -2), 0, 1)   # noqa: E731
        P, U, out, outt = turn(p), turn(u[:, :, c]), turn(Bp[:, :, c]), turn(Btu)
        out[:, :, :k] -= h / 2 * (P @ D[:k])
        outt -= h / 2 * (U[:, :, :k] @ D[:k].T)
        pv, uv = [P @ V[e][:k] for e in (0, 1)], [U[:, :, :k] @ V[e] for e in (0, 1)]
        avg, jump = (pv[1][:, :-1] + pv[0][:, 1:]) * h / 4, (uv[1][:, :-1] - uv[0][:, 1:]) * h / 4
        out[:, :-1, :k] += avg[..., None] * V[1]
        out[:, 1:, :k] -= avg[..., None] * V[0]
        outt[:, :-1] += jump[..., None] * V[1][:k]
        outt[:, 1:] += jump[..., None] * V[0][:k]
        for e, at in ((0, slice(0, 1)), (1, slice(-1, None))):
            if bc[2 * c + e] != "neumann":
                sg = 1 if e else -1
                out[:, at, :k] += sg * h / 2 * pv[e][:, at][..., None] * V[e]
                outt[:, at] += sg * h / 2 * uv[e][:, at][..., None] * V[e][:k]
    return Bp.reshape(-1), Btu.reshape(-1)


@pytest.mark.parametrize("k,mesh", [(1, (129, 67)), (2, (67, 97)), (3, (64, 96)), (4, (70, 50)), (5, (65, 40)),
                                    (6, (45, 30))])
@pytest.mark.parametrize("bc", [("navier",) * 4, synth.SINKER_BC])
def test_error_not_above_one_thread_per_mode(ctx, k, mesh, bc):
    if np.finfo(LD).nmant < 63:
        pytest.skip("no extended precision")
    nx, ny = mesh
    prob = api.Problem(ctx, nx, ny, k, np.ones(nx * ny), bc=bc)
    p, u = synth.random_vector(prob.n_p, 3), synth.random_vector(prob.n_u, 4)
    ref = exact(k, nx, ny, bc, p, u)

    def errors():
        y = [torch.empty(n, dtype=torch.float64, device="cuda") for n in (prob.n_u, prob.n_p)]
        prob.apply_B(torch.from_numpy(p).cuda(), y[0])
        prob.apply_Bt(torch.from_numpy(u).cuda(), y[1])
        return [float(np.sqrt(((a.cpu().numpy() - r) ** 2).sum() / (r ** 2).sum())) for a, r in zip(y, ref)]

    sums = errors()
    prob.set_schedule(apply=[1 if k <= 5 else 3, 0])
    modes = errors()
    assert all(s <= m for s, m in zip(sums, modes)), (modes, sums)
