"""The work whose speed matters to a user of this library, as cases that can be timed and checked.

A case names an entry point (``op``), a mesh, a velocity degree ``k``, a viscosity field with its
contrast, the boundary condition of the left, right, bottom and top side (v Navier, n Neumann,
d Dirichlet) and the problem's precision.  Sizes and fields are those of the benchmark and the tests:
the 128 x 128, k = 3 box inclusion, the 512 x 512, k = 4 many-disc field, the six sedimenting
inclusions on 32 ... 256 elements per side with k = 2 ... 5, ragged meshes with random viscosities.
``Reference`` restates the method in plain torch (64 bits) for ``exact``.
"""
import math

import numpy as np
import torch

from paper_1607_03777_gb300 import api, synth

BC = {"v": "navier", "n": "neumann", "d": "dirichlet"}
GRAVITY = 10.0
SEED = 2            # of the eigenvalue estimate's start vector
RTOL = 1e-8         # of the Stokes solves
INNER_RTOL = 1e-3   # of the viscous solves


def case(op, nx, ny, k, field, contrast, bc="vvvn", precision="fp64", count=1):
    return {"op": op, "nx": nx, "ny": ny, "k": k, "field": field, "contrast": contrast, "bc": bc,
            "precision": precision, "count": count}


def named(name, *args, **kw):
    return {"name": name, **case(*args, **kw)}


def listed():
    return [
        # one operator apply on a small ragged mesh without a multigrid set-up: latency
        named("apply_f64_37x35_k2", "apply", 37, 35, 2, "random", 1e3, "dvnv"),
        # the operator of the headline solve, once per Krylov step and several times per V-cycle
        named("apply_f64_128_k3", "apply", 128, 128, 3, "box", 1e4),
        # the same on the largest mesh of the benchmark (residuals, smoother), contrast up to 1e6
        named("apply_f64_512_k4", "apply", 512, 512, 4, "discs", 1e6),
        # the single-precision operator of the mixed form, no element far stiffer than the rest
        named("apply_f32_512_k4", "apply_f32", 512, 512, 4, "sinkers", 1e2, precision="mixed"),
        # ... and next to stiff inclusions, where the mixed form keeps 64-bit arithmetic
        named("apply_f32_stiff_256_k3", "apply_f32", 256, 256, 3, "sinkers", 1e5, precision="mixed"),
        # pressure gradient and divergence, once each per outer iteration, on a ragged mesh
        named("gradient_divergence_250x190_k4", "grad_div", 250, 190, 4, "random", 1e3, "vvvv"),
        # the element-block smoother alone
        named("block_jacobi_128_k3", "block_jacobi", 128, 128, 3, "sinkers", 1e4),
        # the preconditioner of the headline solve
        named("vcycle_f64_128_k3", "vcycle", 128, 128, 3, "box", 1e4),
        # the single-precision preconditioner of the mixed, batched and served solves
        named("vcycle_f32_256_k4", "vcycle_f32", 256, 256, 4, "sinkers", 1e3, precision="mixed"),
        # one viscous solve of a middle-sized instance of the batched list
        named("viscous_solve_64_k2", "viscous", 64, 64, 2, "sinkers", 1e3),
        # the headline: a step with new viscosities (upload, set-up, load vector, Stokes solve)
        named("stokes_step_128_k3", "step", 128, 128, 3, "box", 1e4),
        # many small instances in one call
        named("stokes_batch_16x32_k2", "batch", 32, 32, 2, "sinkers", 1e2, count=16),
    ]


def draw(rng):
    def side(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["apply", "apply", "apply_f32", "apply_f32", "grad_div", "block_jacobi", "vcycle",
                     "vcycle_f32", "viscous", "step"])
    k = rng.choice([2, 3, 4, 5])
    precision = "mixed" if op.endswith("_f32") else "fp64"
    if op in ("apply", "apply_f32", "grad_div"):       # any mesh, any boundary
        field, contrast = rng.choice(["random", "box", "sinkers", "discs"]), 10.0 ** rng.uniform(1.0, 6.0)
        bc = "".join(rng.choice("vvnd") for _ in range(4))
        return case(op, side(24, 400), side(24, 400), k, field, contrast, bc, precision)
    bc = rng.choice(["vvvn", "vvvv"])
    field = rng.choice(["box", "sinkers"])
    if op in ("viscous", "step"):                      # meshes that can be coarsened
        nx, ny = 8 * side(4, 10), 8 * side(4, 10)
        return case(op, nx, ny, min(k, 4), field, 10.0 ** rng.uniform(1.0, 3.0), "vvvn", precision)
    nx, ny = 8 * side(4, 28), 8 * side(4, 28)
    return case(op, nx, ny, k, field, 10.0 ** rng.uniform(1.0, 4.0 if op != "vcycle_f32" else 3.0), bc,
                precision)


# ---------------------------------------------------------------- inputs
def levels(c):
    """h-coarsenings down to about 16 elements a side (0: the mesh cannot be coarsened)."""
    nx, ny, n = c["nx"], c["ny"], 0
    while nx % 2 == 0 and ny % 2 == 0 and min(nx, ny) > 16:
        nx, ny, n = nx // 2, ny // 2, n + 1
    return n if nx * ny <= 2048 else 0


def materials(c, seed):
    """(viscosity, density) of every element, element ey * nx + ex."""
    nx, ny = c["nx"], c["ny"]
    lc = math.log10(c["contrast"])
    g = np.random.Generator(np.random.PCG64(seed))
    if c["field"] == "random":
        return 10.0 ** g.uniform(0.0, lc, nx * ny), g.uniform(1.0, 1.2, nx * ny)
    if c["field"] == "box":
        shapes = [synth.box(0.25, 0.75, 0.25, 0.75, 10.0 ** (lc + g.uniform(-0.05, 0.05)), g.uniform(1.15, 1.25))]
    elif c["field"] == "sinkers":
        shapes = synth.jittered_sinkers(seed, (lc, lc))
    else:
        shapes = synth.random_discs(64, 0.02, (0.0, lc), seed)
    x = np.tile((np.arange(nx) + 0.5) / nx, ny)
    y = np.repeat((np.arange(ny) + 0.5) / ny, nx)
    eta, rho = np.ones(nx * ny), np.ones(nx * ny)
    for kind, a, b, cc, d, e, r in shapes:
        inside = (x - a) ** 2 + (y - b) ** 2 <= cc * cc if kind == 0 else (x > a) & (x < b) & (y > cc) & (y < d)
        eta[inside], rho[inside] = np.maximum(eta[inside], e), r
    return eta, rho


def vectors(c, seed, *sizes):
    """Normally distributed vectors."""
    g = np.random.Generator(np.random.PCG64(seed + 1))
    return [torch.from_numpy(g.standard_normal(n, dtype=np.float32).astype(np.float64)) for n in sizes]


_context = None


def context():
    global _context
    if _context is None:
        _context = api.Context(0)
    return _context


def problem(c, eta):
    return api.Problem(context(), c["nx"], c["ny"], c["k"], eta, bc=tuple(BC[b] for b in c["bc"]),
                       n_hlevels=levels(c), seed=SEED, precision=c["precision"])


def prepare(c, seed):
    op = c["op"]
    s = {"op": op}

    def put(v, dtype=torch.float64):
        return (torch.from_numpy(v) if isinstance(v, np.ndarray) else v).to("cuda", dtype)

    def empty(n, dtype=torch.float64):
        return torch.empty(n, dtype=dtype, device="cuda")

    if op == "batch":
        s["P"], s["f"], s["u"], s["p"] = [], [], [], []
        for i in range(c["count"]):
            one = dict(c, k=c["k"] + i % 2)     # degrees k and k + 1 in turn
            eta, rho = materials(one, 1000 * seed + i)
            P = problem(one, eta)
            P.setup()
            f = empty(P.n_u)
            P.rhs_body_force(put(rho), GRAVITY, f)
            s["P"].append(P)
            s["f"].append(f)
            s["u"].append(empty(P.n_u))
            s["p"].append(empty(P.n_p))
        return s
    eta, rho = materials(c, seed)
    P = s["P"] = problem(c, eta)
    if levels(c) > 0:
        P.setup()
    x, p = vectors(c, seed, P.n_u, P.n_p)
    t = torch.float32 if op.endswith("_f32") else torch.float64
    s["x"], s["y"] = put(x, t), empty(P.n_u, t)
    if op == "grad_div":
        s["p"], s["q"] = put(p), empty(P.n_p)
    if op == "step":
        s["eta"], s["rho"], s["p"] = put(eta), put(rho), empty(P.n_p)
    return s


def run(s):
    op, P = s["op"], s["P"]
    if op == "batch":
        api.solve_batch(context(), P, s["f"], s["u"], s["p"], n_streams=len(P), grouped=True, rtol=RTOL)
        return {"u": s["u"], "p": s["p"]}
    x, y = s["x"], s["y"]
    if op == "apply":
        P.apply_A(x, y)
    elif op == "apply_f32":
        P.apply_A_f32(x, y)
    elif op == "grad_div":
        P.apply_B(s["p"], y)
        P.apply_Bt(x, s["q"])
        return {"gradient": y, "divergence": s["q"]}
    elif op == "block_jacobi":
        P.block_jacobi(x, y)
    elif op == "vcycle":
        P.vcycle(x, y)
    elif op == "vcycle_f32":
        P.vcycle_f32(x, y)
    elif op == "viscous":
        P.inner_solve(x, y, rtol=INNER_RTOL)
    elif op == "step":
        P.update_eta(s["eta"])
        P.rhs_body_force(s["rho"], GRAVITY, x)
        P.solve(x, y, s["p"], rtol=RTOL, check=False)
        return {"u": y, "p": s["p"]}
    return y


def work(c):
    n, ne = c["k"] + 1, c["nx"] * c["ny"]
    n_u, n_p, word = 2 * n * n * ne, c["k"] ** 2 * ne, 4 if c["op"].endswith("_f32") else 8
    apply = ne * (16 * n ** 3 + 128 * n * n)            # sum-factorised volume terms, face terms
    jacobi = ne * 2 * (2 * n * n) ** 2 // 4             # block inverses by reflection parity
    cycle = 4 * apply + 4 * jacobi                      # 2 + 2 smoother steps and the residual
    if c["op"] == "grad_div":
        return {"bytes": word * 2 * (n_u + n_p), "flops": 4 * ne * 2 * n * c["k"] * (n + c["k"] + 4)}
    if c["op"] == "batch":     # about 25 outer x 9 inner iterations
        return {"bytes": c["count"] * 8 * (2 * n_u + n_p + ne), "flops": c["count"] * 225 * (cycle + apply)}
    if c["op"] == "step":      # about 26 outer x 12 inner iterations
        return {"bytes": 8 * (2 * n_u + n_p + 2 * ne), "flops": 312 * (cycle + apply)}
    flops = {"apply": apply, "apply_f32": apply, "block_jacobi": jacobi, "vcycle": cycle, "vcycle_f32": cycle,
             "viscous": 10 * (cycle + apply)}[c["op"]]
    return {"bytes": word * (2 * n_u + ne), "flops": flops}


# ---------------------------------------------------------------- the method in plain torch, 64 bits
class Reference:
    """SIP operator A, B, B^T, element-block Jacobi and the hp V-cycle on element arrays
    u[ey, ex, c, j, i] (x-degree i), p[ey, ex, j, i]; unit square."""

    def __init__(self, c, eta, device):
        self.nx, self.ny, self.k, self.bc, self.dev = c["nx"], c["ny"], c["k"], c["bc"], device
        self.eta = torch.as_tensor(eta, dtype=torch.float64, device=device).reshape(self.ny, self.nx)
        self.pen = 4.0 * (self.k + 1) ** 2
        self.levels = levels(c)

    def tables(self, n):
        i = np.arange(n)
        s = np.sqrt((2.0 * i + 1.0) / 2.0)
        m = np.minimum(i[:, None], i[None, :])
        even = (i[:, None] + i[None, :]) % 2 == 0
        G = np.where(even, s[:, None] * s[None, :] * m * (m + 1), 0.0)        # int l_a' l_b'
        D = np.where((i[None, :] > i[:, None]) & ~even, 2.0 * s[:, None] * s[None, :], 0.0)  # int l_p l_q'
        sign = (-1.0) ** i
        value = np.stack([sign * s, s])                                        # l_i(-1), l_i(+1)
        slope = np.stack([-sign * s * i * (i + 1) / 2, s * i * (i + 1) / 2])
        return [torch.from_numpy(np.ascontiguousarray(a)).to(self.dev) for a in (G, D, value, slope)]

    def apply(self, u):
        """A u for modes u[..., c, j, i] of any degree; the penalty is that of degree k."""
        n = u.shape[-1]
        G, D, V, S = self.tables(n)
        hx, hy = 1.0 / self.nx, 1.0 / self.ny
        eta = self.eta[..., None, None]
        ux, uy = u[..., 0, :, :], u[..., 1, :, :]
        yx = eta * (2 * hy / hx * ux @ G + hx / hy * G @ ux + D.T @ (uy @ D.T))
        yy = eta * (hy / hx * uy @ G + 2 * hx / hy * G @ uy + D @ (ux @ D))
        out = torch.stack([yx, yy], dim=-3)
        for normal, (hn, ht) in enumerate(((hx, hy), (hy, hx))):
            w = u if normal == 0 else u.transpose(-1, -2).transpose(0, 1)      # [line, along, c, m, q]
            e = self.eta if normal == 0 else self.eta.T
            y = torch.zeros_like(w)
            self.faces(w, e, y, normal, hn, ht, D, V, S)
            out = out + (y if normal == 0 else y.transpose(0, 1).transpose(-1, -2))
        return out

    def faces(self, w, eta, y, nc, hn, ht, D, V, S):
        """Adds the face terms of one normal direction: w[line, along, c, m, q], q along the normal."""
        tc = 1 - nc
        eta = eta[..., None]
        val = [w @ V[s] for s in (0, 1)]                      # [line, along, c, m] at the low / high end
        der = [w @ S[s] * (2.0 / hn) for s in (0, 1)]
        shear = [v[..., nc, :] @ D.T * (2.0 / ht) for v in val]   # tangential derivative, tested

        def add(at, s, wn, wt, traction_n, traction_t, sigma, own, half):
            """Test functions of the elements `at`, end s: consistency, symmetry and penalty terms."""
            sg = 1.0 if s else -1.0
            Pn = -0.5 * ht * sg * traction_n - half * own * sg * (wt @ D) + 0.5 * ht * sigma * wn
            Pt = -0.5 * ht * sg * traction_t + 0.5 * ht * sigma * wt
            Qn = -2.0 * half * own * sg * ht / hn * wn
            Qt = -half * own * sg * ht / hn * wt
            for comp, P, Q in ((nc, Pn, Qn), (tc, Pt, Qt)):
                y[:, at, comp] += P[..., None] * V[s] + Q[..., None] * S[s]

        L, R = slice(None, -1), slice(1, None)
        if w.shape[1] > 1:
            eL, eR = eta[:, L], eta[:, R]
            sigma = self.pen / hn * torch.maximum(eL, eR)
            jump = val[1][:, L] - val[0][:, R]
            tn = eL * der[1][:, L, nc] + eR * der[0][:, R, nc]                 # average of 2 eta d_n u_n
            tt = 0.5 * (eL * (der[1][:, L, tc] + shear[1][:, L]) + eR * (der[0][:, R, tc] + shear[0][:, R]))
            add(L, 1, jump[..., nc, :], jump[..., tc, :], tn, tt, sigma, eL, 0.5)
            add(R, 0, -jump[..., nc, :], -jump[..., tc, :], tn, tt, sigma, eR, 0.5)
        for s, at in ((0, slice(0, 1)), (1, slice(-1, None))):
            kind = self.bc[2 * nc + s]
            if kind == "n":
                continue
            own, vn, vt = eta[:, at], val[s][:, at, nc], val[s][:, at, tc]
            sigma = 2.0 * self.pen / hn * own
            tn = 2.0 * own * der[s][:, at, nc]
            if kind == "v":      # normal component only
                zero = torch.zeros_like(vt)
                add(at, s, vn, zero, tn, zero, sigma, own, 1.0)
            else:
                add(at, s, vn, vt, tn, own * (der[s][:, at, tc] + shear[s][:, at]), sigma, own, 1.0)

    def divergence_form(self):
        """b(v, p) per element pair as functions p -> B p and u -> B^T u."""
        n, k = self.k + 1, self.k
        _, D, V, _ = self.tables(n)
        hx, hy = 1.0 / self.nx, 1.0 / self.ny

        def jump_terms(p_like, comp, h_t):
            """Face part of B for velocity component comp (normal direction comp)."""
            p = p_like if comp == 0 else p_like.transpose(-1, -2).transpose(0, 1)   # [line, along, m, q]
            pv = [p @ V[s][:k] for s in (0, 1)]
            f = torch.zeros(*p.shape[:2], n, n, dtype=torch.float64, device=self.dev)
            if p.shape[1] > 1:
                avg = 0.25 * h_t * (pv[1][:, :-1] + pv[0][:, 1:])
                f[:, :-1, :k] += avg[..., None] * V[1]
                f[:, 1:, :k] -= avg[..., None] * V[0]
            for s, at in ((0, slice(0, 1)), (1, slice(-1, None))):
                if self.bc[2 * comp + s] != "n":
                    f[:, at, :k] += (1.0 if s else -1.0) * 0.5 * h_t * pv[s][:, at][..., None] * V[s]
            return f if comp == 0 else f.transpose(0, 1).transpose(-1, -2)

        def B(p):
            out = torch.zeros(self.ny, self.nx, 2, n, n, dtype=torch.float64, device=self.dev)
            out[:, :, 0, :k, :] -= 0.5 * hy * p @ D[:k, :]
            out[:, :, 1, :, :k] -= 0.5 * hx * D[:k, :].T @ p
            out[:, :, 0] += jump_terms(p, 0, hy)
            out[:, :, 1] += jump_terms(p, 1, hx)
            return out

        def Bt(u):     # the transpose of B, by automatic differentiation of <u, B p>
            p = torch.zeros(self.ny, self.nx, k, k, dtype=torch.float64, device=self.dev, requires_grad=True)
            return torch.autograd.grad((B(p) * u).sum(), p)[0]

        return B, Bt

    # -- smoother and hierarchy
    def setup(self):
        n = self.k + 1
        nb = 2 * n * n
        blocks = torch.zeros(self.ny, self.nx, nb, nb, dtype=torch.float64, device=self.dev)
        ey, ex = torch.arange(self.ny, device=self.dev), torch.arange(self.nx, device=self.dev)
        colour = (ey[:, None] + ex[None, :]) % 2
        for col in (0, 1):
            at = (colour == col).to(torch.float64)[..., None]
            for q in range(nb):
                e = torch.zeros(self.ny, self.nx, nb, dtype=torch.float64, device=self.dev)
                e[..., q] = at[..., 0]
                blocks[..., q] += self.apply(e.reshape(self.ny, self.nx, 2, n, n)).reshape(e.shape) * at
        self.inv = torch.linalg.inv(blocks)

    def jacobi(self, r):
        return (self.inv @ r.reshape(self.ny, self.nx, -1, 1)).reshape(r.shape)

    @staticmethod
    def start_vector(seed, n, device):
        with np.errstate(over="ignore"):
            z = np.uint64(seed) + np.arange(1, n + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            z = z ^ (z >> np.uint64(31))
        return torch.from_numpy((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0).to(device)

    def estimate(self, A, M, shape, seed):
        """Largest Ritz value of ten Arnoldi steps on M A."""
        v = M(self.start_vector(seed, math.prod(shape), self.dev).reshape(shape))
        V, H = [v / v.norm()], np.zeros((11, 10))
        for j in range(10):
            w = M(A(V[j]))
            for _ in range(2):
                for i in range(j + 1):
                    h = torch.sum(V[i] * w)
                    H[i, j] += float(h)
                    w = w - h * V[i]
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
        return float(np.linalg.eigvals(H[:10]).real.max())

    @staticmethod
    def chebyshev(A, M, b, x, steps, lmax):
        lo, hi = 0.1 * lmax, 1.1 * lmax
        theta, delta = 0.5 * (hi + lo), 0.5 * (hi - lo)
        r = b if x is None else b - A(x)
        d = M(r) / theta
        x = d if x is None else x + d
        rho = delta / theta
        for _ in range(steps - 1):
            r = r - A(d)
            new = 1.0 / (2.0 * theta / delta - rho)
            d = new * rho * d + 2.0 * new / delta * M(r)
            x = x + d
            rho = new
        return x

    def to_elements(self, v):
        """Continuous bilinears v[vy, vx, c] -> modes of degree 1."""
        a, b = math.sqrt(0.5), math.sqrt(1.0 / 6.0)
        W = torch.tensor([[a, a], [-b, b]], dtype=torch.float64, device=self.dev)
        t = torch.stack([v[:, :-1], v[:, 1:]], dim=-1)
        t = torch.stack([t[:-1], t[1:]], dim=-2)              # [ey, ex, c, q, p]
        return W @ t @ W.T

    def to_vertices(self, u):
        a, b = math.sqrt(0.5), math.sqrt(1.0 / 6.0)
        W = torch.tensor([[a, a], [-b, b]], dtype=torch.float64, device=self.dev)
        t = W.T @ u @ W
        v = torch.zeros(self.ny + 1, self.nx + 1, 2, dtype=torch.float64, device=self.dev)
        for q in (0, 1):
            for p in (0, 1):
                v[q:self.ny + q, p:self.nx + p] += t[..., q, p]
        return v

    @staticmethod
    def interpolate(v):
        f = torch.zeros(2 * v.shape[0] - 1, 2 * v.shape[1] - 1, 2, dtype=v.dtype, device=v.device)
        f[::2, ::2] = v
        f[::2, 1::2] = 0.5 * (v[:, :-1] + v[:, 1:])
        f[1::2] = 0.5 * (f[:-1:2] + f[2::2])
        return f

    @staticmethod
    def restrict(f):
        g = f[::2].clone()
        g[:-1] += 0.5 * f[1::2]
        g[1:] += 0.5 * f[1::2]
        v = g[:, ::2].clone()
        v[:, :-1] += 0.5 * g[:, 1::2]
        v[:, 1:] += 0.5 * g[:, 1::2]
        return v

    def hierarchy(self):
        self.lmax = self.estimate(self.apply, self.jacobi, (self.ny, self.nx, 2, self.k + 1, self.k + 1), SEED)
        self.grids = []
        operator = lambda v: self.to_vertices(self.apply(self.to_elements(v)))  # noqa: E731
        shape = (self.ny + 1, self.nx + 1, 2)
        for level in range(self.levels + 1):
            S = self.stencil(operator, shape)
            A = lambda v, S=S: self.stencil_apply(S, v)  # noqa: E731
            if level == self.levels:
                eye = torch.eye(math.prod(shape), dtype=torch.float64, device=self.dev)
                self.coarsest = torch.linalg.inv(torch.stack([A(e.reshape(shape)).reshape(-1) for e in eye]))
                break
            diagonal = torch.stack([S[1][1][..., 0, 0], S[1][1][..., 1, 1]], dim=-1)
            M = lambda r, d=diagonal: r / d  # noqa: E731
            self.grids.append((A, M, self.estimate(A, M, shape, SEED + 1 + level)))
            operator = lambda v, A=A: self.restrict(A(self.interpolate(v)))  # noqa: E731
            shape = ((shape[0] + 1) // 2, (shape[1] + 1) // 2, 2)

    def stencil(self, operator, shape):
        """The 3 x 3 blocks of a nearest-neighbour operator, by probing with 9 colours."""
        vy = torch.arange(shape[0], device=self.dev)[:, None]
        vx = torch.arange(shape[1], device=self.dev)[None, :]
        S = [[torch.zeros(*shape, 2, dtype=torch.float64, device=self.dev) for _ in range(3)] for _ in range(3)]
        for col in range(9):
            on = ((vy % 3 == col // 3) & (vx % 3 == col % 3)).to(torch.float64)
            for comp in (0, 1):
                e = torch.zeros(shape, dtype=torch.float64, device=self.dev)
                e[..., comp] = on
                y = operator(e)
                for a in range(3):
                    for b in range(3):      # rows whose neighbour (a - 1, b - 1) has this colour
                        hit = ((vy + a - 1) % 3 == col // 3) & ((vx + b - 1) % 3 == col % 3)
                        S[a][b][..., comp] += y * hit[..., None]
        return S

    @staticmethod
    def stencil_apply(S, v):
        pad = torch.nn.functional.pad(v, (0, 0, 1, 1, 1, 1))
        ny, nx = v.shape[:2]
        return sum((S[a][b] @ pad[a:a + ny, b:b + nx, :, None])[..., 0] for a in range(3) for b in range(3))

    def coarse_cycle(self, b, level=0):
        if level == self.levels:
            return (self.coarsest @ b.reshape(-1)).reshape(b.shape)
        A, M, lmax = self.grids[level]
        x = self.chebyshev(A, M, b, None, 3, lmax)
        x = x + self.interpolate(self.coarse_cycle(self.restrict(b - A(x)), level + 1))
        return self.chebyshev(A, M, b, x, 3, lmax)

    def vcycle(self, b):
        y = self.chebyshev(self.apply, self.jacobi, b, None, 2, self.lmax)
        r = b - self.apply(y)
        y = y.clone()
        y[..., :2, :2] += self.to_elements(self.coarse_cycle(self.to_vertices(r[..., :2, :2])))
        return self.chebyshev(self.apply, self.jacobi, b, y, 2, self.lmax)

    def viscous_solve(self, t, rtol=INNER_RTOL):
        """Conjugate gradients preconditioned with the V-cycle."""
        y, r, limit = torch.zeros_like(t), t, rtol * float(t.norm())
        d = z = self.vcycle(r)
        rz = torch.sum(r * z)
        for _ in range(200):
            q = self.apply(d)
            a = rz / torch.sum(d * q)
            y, r = y + a * d, r - a * q
            if float(r.norm()) < limit:
                break
            z = self.vcycle(r)
            old, rz = rz, torch.sum(r * z)
            d = z + rz / old * d
        return y

    def stokes_solve(self, f, rtol):
        """Right-preconditioned flexible GMRES from zero; returns u, p."""
        B, Bt = self.divergence_form()
        n_u = f.numel()
        mass = self.eta[..., None, None] * (4.0 * self.nx * self.ny)      # inverse of the scaled pressure mass
        closed = "n" not in self.bc
        shape_p = (self.ny, self.nx, self.k, self.k)

        def split(x):
            return x[:n_u].reshape(f.shape), x[n_u:].reshape(shape_p)

        def join(u, p):
            if closed:
                p = p.clone()
                p[..., 0, 0] -= p[..., 0, 0].mean()
            return torch.cat([u.reshape(-1), p.reshape(-1)])

        def K(x):
            u, p = split(x)
            return join(self.apply(u) + B(p), Bt(u))

        def precondition(x):
            u, p = split(x)
            p = split(join(u, -mass * p))[1]
            return join(self.viscous_solve(u - B(p)), p)

        b = join(f, torch.zeros(shape_p, dtype=torch.float64, device=self.dev))
        V, Z, H = [b / b.norm()], [], np.zeros((101, 100))
        for j in range(100):
            Z.append(precondition(V[j]))
            w = K(Z[j])
            Q = torch.stack(V)
            for _ in range(2):
                h = Q @ w
                H[:j + 1, j] += h.cpu().numpy()
                w = w - h @ Q
            H[j + 1, j] = float(w.norm())
            V.append(w / H[j + 1, j])
            e = np.zeros(j + 2)
            e[0] = float(b.norm())
            y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(e - H[:j + 2, :j + 1] @ y) < rtol * e[0]:
                break
        return split(torch.from_numpy(y).to(self.dev) @ torch.stack(Z))


def exact(c, seed):
    op = c["op"]
    if op == "batch":
        return None     # 16 solves: over the time that this may take
    device = "cuda" if torch.cuda.is_available() else "cpu"
    eta, rho = materials(c, seed)
    n, ne = c["k"] + 1, c["nx"] * c["ny"]
    if 2 * n * n * ne > 8_000_000 and not op.startswith("apply"):
        return None     # the blocks alone would take tens of gigabytes
    R = Reference(c, eta, device)
    x, p = vectors(c, seed, 2 * n * n * ne, c["k"] ** 2 * ne)
    x = x.to(device).reshape(c["ny"], c["nx"], 2, n, n)
    if op.startswith("apply"):
        return R.apply(x).reshape(-1)
    if op == "grad_div":
        B, Bt = R.divergence_form()
        p = p.to(device).reshape(c["ny"], c["nx"], c["k"], c["k"])
        return {"gradient": B(p).reshape(-1), "divergence": Bt(x).reshape(-1)}
    R.setup()
    if op == "block_jacobi":
        return R.jacobi(x).reshape(-1)
    R.hierarchy()
    if op.startswith("vcycle"):
        return R.vcycle(x).reshape(-1)
    if op == "viscous":
        return R.viscous_solve(x).reshape(-1)
    load = torch.zeros_like(x)
    load[..., 1, 0, 0] = -GRAVITY / (2.0 * ne) * torch.as_tensor(rho, device=device).reshape(c["ny"], c["nx"])
    u, q = R.stokes_solve(load, 0.1 * RTOL)
    return {"u": u.reshape(-1), "p": q.reshape(-1)}
