"""The calls whose time counts: brackets, operator applications, Poisson solves, time steps,
batched steps and diagnostics of the dG solver, each through the package's public binding
(paper_1311_7477_gb300.dg), over the sizes, orders and options that users run.

A case is a dict with a "kind":
  bracket, laplace, invariants   one operator call on a grid of Nx x Ny cells, n nodes
  poisson                        one Poisson solve from a zero guess
  step                           `steps` time steps of one simulation, then its fields
  batch                          `steps` batched steps of an ensemble, then every member's fields
exact() recomputes a case in float64 with torch alone: Lagrange bases on Gauss nodes, cell-wise
block products, and the Poisson solve by a Fourier transform over the cells (periodic) or an
eigen-decomposition of the 1D matrices (Dirichlet).
"""
import math

import numpy as np
import torch

from paper_1311_7477_gb300 import dg

L = 2.0 * math.pi
PRECISION = {"fp64": dg.DG_FP64, "mixed": dg.DG_MIXED, "mixed64": dg.DG_MIXED64, "fp64pc32": dg.DG_FP64_PC32}


def listed():
    return [
        # one bracket of the paper's Table 1 grid: a call so small that its latency shows
        {"name": "bracket_100_n4", "kind": "bracket", "Nx": 100, "Ny": 100, "n": 4, "arith": "fp64"},
        # one float64 bracket on a large grid: the right-hand side of a production run
        {"name": "bracket_1000_n4", "kind": "bracket", "Nx": 1000, "Ny": 1000, "n": 4, "arith": "fp64"},
        # the double-float bracket of the mixed mode on a rectangular grid with ragged tiles
        {"name": "bracket_mixed_501x373_n3", "kind": "bracket", "Nx": 501, "Ny": 373, "n": 3, "arith": "mixed"},
        # the LDG Laplacian of a field on a ragged grid, as an implicit or diagnostic code applies it
        {"name": "laplace_500x300_n5", "kind": "laplace", "Nx": 500, "Ny": 300, "n": 5, "mode": 1},
        # a bounded box: the only preconditioner there is W^-1, many short CG iterations
        {"name": "poisson_dirichlet_48_n3", "kind": "poisson", "Nx": 48, "Ny": 48, "n": 3, "bc": "dirichlet",
         "precond": "jacobi", "tol": 1e-12},
        # a solve with the two-level preconditioner, which takes any periodic grid
        {"name": "poisson_twolevel_256_n3", "kind": "poisson", "Nx": 256, "Ny": 256, "n": 3, "precond": "twolevel",
         "tol": 1e-12},
        # a cold solve with the spectral preconditioner, as at the start of a run
        {"name": "poisson_spectral_512_n4", "kind": "poisson", "Nx": 512, "Ny": 512, "n": 4, "precond": "spectral",
         "tol": 1e-10},
        # ten steps of a small interactive run
        {"name": "step_32_n3", "kind": "step", "Nx": 32, "Ny": 32, "n": 3, "precision": "fp64", "precond": "spectral",
         "field": "sinsin", "D": 0.0, "dt": 1e-3, "tol": 1e-12, "steps": 10},
        # the double shear layer with viscosity, float64
        {"name": "step_512_n4", "kind": "step", "Nx": 512, "Ny": 512, "n": 4, "precision": "fp64",
         "precond": "spectral", "field": "shear", "D": 1e-4, "dt": 1e-4, "tol": 1e-10, "steps": 1},
        # the largest single run: decaying turbulence, inviscid, float64 and mixed precision
        {"name": "step_1024_n5", "kind": "step", "Nx": 1024, "Ny": 1024, "n": 5, "precision": "fp64",
         "precond": "spectral", "field": "random", "D": 0.0, "dt": 2e-4, "tol": 1e-10, "steps": 1},
        {"name": "step_1024_n5_mixed", "kind": "step", "Nx": 1024, "Ny": 1024, "n": 5, "precision": "mixed",
         "precond": "spectral", "field": "random", "D": 0.0, "dt": 2e-4, "tol": 1e-10, "steps": 1},
        # an uneven ensemble advanced together, the way a parameter study or the server runs
        {"name": "batch_16", "kind": "batch", "members": 16, "precision": "mixed", "tol": 1e-10, "steps": 2},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bracket", "bracket", "laplace", "poisson", "poisson", "step", "step", "step", "batch", "invariants"])
    n = rng.randint(1, 5)
    if kind == "batch":
        return {"kind": kind, "members": rng.randint(2, 16), "precision": rng.choice(["fp64", "mixed"]), "tol": 1e-10,
                "steps": rng.randint(1, 3)}
    if kind in ("bracket", "laplace", "invariants"):
        c = {"kind": kind, "Nx": _side(rng, 24, 1024), "Ny": _side(rng, 24, 1024), "n": n}
        if kind == "bracket":
            c["arith"] = rng.choice(["fp64", "fp64", "mixed"])
        if kind == "laplace":
            c["mode"] = rng.randint(0, 1)
        if kind != "invariants":
            c["bc"] = rng.choice(["periodic", "periodic", "dirichlet"])
        return c
    precond = rng.choice(["spectral", "spectral", "spectral", "twolevel"])
    if precond == "twolevel":
        N = (2 ** rng.randint(5, 8), 2 ** rng.randint(5, 8))
    elif rng.random() < 0.6:
        N = (2 ** rng.randint(5, 10), 2 ** rng.randint(5, 10))
    else:
        N = (_side(rng, 24, 160), _side(rng, 24, 160))
    if kind == "poisson":
        if rng.random() < 0.2:
            return {"kind": kind, "Nx": rng.randint(12, 48), "Ny": rng.randint(12, 48), "n": rng.randint(1, 4),
                    "bc": rng.choice(["periodic", "dirichlet"]), "precond": "jacobi", "tol": 1e-12}
        return {"kind": kind, "Nx": N[0], "Ny": N[1], "n": n, "precond": precond,
                "tol": 1e-10 if precond == "spectral" else 1e-12}
    D = rng.choice([0.0, math.exp(rng.uniform(math.log(1e-5), math.log(1e-3)))])
    N = (min(N[0], 512), min(N[1], 512)) if n == 5 else N
    dt = _stable_dt(max(N), n, D)
    return {"kind": "step", "Nx": N[0], "Ny": N[1], "n": n, "precision": rng.choice(["fp64", "fp64", "mixed", "mixed64", "fp64pc32"]),
            "precond": precond, "field": rng.choice(["random", "shear", "sinsin"]), "D": D, "dt": dt, "tol": 1e-10,
            "steps": rng.randint(1, 2)}


def _stable_dt(N, n, D):
    """A time step within the explicit scheme's limits for |u| + |v| <= 2."""
    h = L / N
    dt = min(2e-4, 0.1 * h / (n * n))
    return min(dt, 0.02 * h * h / (D * n ** 4)) if D > 0 else dt


def _ensemble(case, seed):
    """Members of the uneven ensemble: cells per side, nodes and viscosity drawn by member, so
    that a case of m members always holds the same sizes; the seed makes their fields."""
    out = []
    for i in range(case["members"]):
        r = np.random.default_rng(100 + i)
        N, n = int(r.choice((32, 64, 128, 256))), int(r.choice((2, 3, 4, 5)))
        D = float(np.exp(r.uniform(np.log(1e-5), np.log(1e-3))))
        out.append({"Nx": N, "Ny": N, "n": n, "D": D, "dt": _stable_dt(N, n, D), "field": "random", "seed": 1000 * seed + i,
                    "steps": case["steps"], "tol": case["tol"], "precision": case["precision"], "precond": "spectral"})
    return out


# ---- inputs -------------------------------------------------------------------------------

def _nodes(N, n):
    x = np.polynomial.legendre.leggauss(n)[0]
    h = L / N
    return torch.from_numpy(((np.arange(N)[:, None] + 0.5) * h + 0.5 * h * x[None, :]).reshape(-1)).cuda()


def _blocked(G, Ny, Nx, n):
    """Node array [Y][X] -> the library's cell-blocked order (cy, cx, a, b)."""
    return G.reshape(Ny, n, Nx, n).permute(0, 2, 1, 3).contiguous()


def _random_phase(Nx, Ny, n, seed, kmax=32, k0=6.0):
    """Random-phase field with spectrum k^4 exp(-(k/k0)^2) and unit enstrophy."""
    kmax = min(kmax, max(4, min(Nx, Ny) * n // 4))
    rng = np.random.default_rng(seed)
    kx, ky = np.meshgrid(np.arange(-kmax, kmax + 1), np.arange(0, kmax + 1))
    kk = np.hypot(kx, ky)
    keep = (kk > 0) & (kk <= kmax) & ((ky > 0) | (kx > 0))
    A = np.where(keep, np.sqrt(kk ** 5 * np.exp(-(kk / k0) ** 2)), 0.0)
    A /= np.sqrt(np.pi ** 2 * np.sum(A ** 2))
    C = torch.from_numpy(A * np.exp(1j * rng.uniform(0, 2 * np.pi, A.shape))).cuda()
    xs, ys = _nodes(Nx, n), _nodes(Ny, n)
    ph = torch.outer(torch.arange(-kmax, kmax + 1, device="cuda", dtype=torch.float64), xs)
    py = torch.outer(ys, torch.arange(0, kmax + 1, device="cuda", dtype=torch.float64))
    P = torch.polar(torch.ones_like(py), py) @ C
    return _blocked(P.real @ torch.cos(ph) - P.imag @ torch.sin(ph), Ny, Nx, n)


def _field(case, seed):
    Nx, Ny, n = case["Nx"], case["Ny"], case["n"]
    kind = case.get("field", "random")
    w = _random_phase(Nx, Ny, n, seed)
    if kind == "random":
        return w
    X, Y = _nodes(Nx, n)[None, :], _nodes(Ny, n)[:, None]
    if kind == "shear":  # double shear layer, and a small seeded perturbation
        rho = 0.05
        s = torch.where(Y <= math.pi, -1.0 / (rho * torch.cosh((Y - math.pi / 2) / rho) ** 2),
                        1.0 / (rho * torch.cosh((1.5 * math.pi - Y) / rho) ** 2))
        return _blocked(0.05 * torch.cos(X) + s, Ny, Nx, n) + 0.05 * w
    g = torch.Generator(device="cuda").manual_seed(seed)  # a steady state and noise on every node
    noise = torch.rand((Ny, Nx, n, n), generator=g, device="cuda", dtype=torch.float64) * 2e-3 - 1e-3
    return _blocked(2.0 * torch.sin(X) * torch.sin(Y), Ny, Nx, n) + noise


def _grid(case):
    g = dg.Grid(case["Nx"], case["Ny"], case["n"], bc=case.get("bc", "periodic"))
    if case.get("precond", "jacobi") != "jacobi":
        g.set_precond(case["precond"])
    return g


def _sim(case, seed):
    g = _grid(case)
    s = dg.Sim(g, _field(case, seed), D=case["D"], dt=case["dt"], precision=PRECISION[case["precision"]],
               cg_tol=case["tol"])
    s.step(2)  # the multistep method's start-up
    return s, torch.empty(g.shape, dtype=torch.float64, device="cuda"), torch.empty(g.shape, dtype=torch.float64, device="cuda")


def _correlate(psi, omega):
    """A field with a mean, and a stream function correlated with it: no integral cancels."""
    omega += 0.1
    psi += 0.5 * omega


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        s, om, ps = _sim(case, seed)
        return {"case": case, "sim": s, "omega": om, "psi": ps}
    if kind == "batch":
        members = [_sim(m, m["seed"]) for m in _ensemble(case, seed)]
        b = dg.Batch(len(members))
        for s, _, _ in members:
            b.admit(s)
        return {"case": case, "batch": b, "members": members}
    st = {"case": case, "grid": _grid(case), "omega": _field(case, 2 * seed)}
    st["out"] = torch.empty_like(st["omega"])
    if kind in ("bracket", "invariants"):
        st["psi"] = _field(case, 2 * seed + 1)
    if kind == "invariants":
        _correlate(st["psi"], st["omega"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "bracket":
        f = dg.dg_bracket_mixed if case["arith"] == "mixed" else dg.dg_bracket
        f(state["grid"], state["psi"], state["omega"], state["out"])
        return state["out"]
    if kind == "laplace":
        dg.dg_laplace_apply(state["grid"], state["omega"], state["out"], mode=case["mode"])
        return state["out"]
    if kind == "invariants":
        return list(dg.dg_invariants(state["grid"], state["psi"], state["omega"]))
    if kind == "poisson":
        state["out"].zero_()
        dg.dg_poisson_solve(state["grid"], state["omega"], state["out"], tol=case["tol"])
        return state["out"]
    if kind == "step":
        state["sim"].step(case["steps"])
        state["sim"].get(state["omega"], state["psi"])
        return [state["omega"], state["psi"]]
    state["batch"].step(case["steps"])
    for s, om, ps in state["members"]:
        s.get(om, ps)
    return [t for _, om, ps in state["members"] for t in (om, ps)]


# ---- work ---------------------------------------------------------------------------------

def work(case):
    """Bytes and operations the method cannot do without: every input read once, every output
    written once; 1D operators as one own-block product and two rank-one neighbour terms."""
    kind = case["kind"]
    if kind == "batch":
        w = [work(dict(m, kind="step")) for m in _ensemble(case, 0)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    Nx, Ny, n = case["Nx"], case["Ny"], case["n"]
    dof = Nx * Ny * n * n
    op = 4.0 * (n + 4)                  # a 1D operator along x and along y
    bracket = 3 * op + 12               # six first derivatives, the products
    # a direct solve by transforms: 2D real FFT over the cells both ways, n x n transforms
    solve = 2 * 2.5 * math.log2(Nx * Ny) + 2 * 2 * 4.0 * n + 6 + op
    if kind == "bracket":
        return {"bytes": 24.0 * dof, "flops": bracket * dof}
    if kind == "laplace":
        return {"bytes": 16.0 * dof, "flops": op * dof}
    if kind == "invariants":
        return {"bytes": 16.0 * dof, "flops": 6.0 * dof}
    if kind == "poisson":
        return {"bytes": 16.0 * dof, "flops": solve * dof}
    step = bracket + (op if case["D"] > 0 else 0) + 6 + solve
    # omega, psi, two psi and two history fields in; omega, psi and R out; the two fields returned
    return {"bytes": (case["steps"] * 64.0 + 32.0) * dof, "flops": case["steps"] * step * dof}


# ---- the same in float64 with torch alone ---------------------------------------------------

def _basis(n):
    x, w = np.polynomial.legendre.leggauss(n)
    d = np.zeros((n, n))
    lL, lR = np.ones(n), np.ones(n)
    for j in range(n):
        others = [m for m in range(n) if m != j]
        den = np.prod([x[j] - x[m] for m in others]) if others else 1.0
        lL[j] = np.prod([-1.0 - x[m] for m in others]) / den if others else 1.0
        lR[j] = np.prod([1.0 - x[m] for m in others]) / den if others else 1.0
        for i in range(n):
            d[i, j] = sum(np.prod([x[i] - x[m] for m in others if m != k]) for k in others) / den
    return x, w, d, lL, lR


class _Line:
    """The 1D blocks of one direction: N cells, own block, right and left neighbour blocks."""

    def __init__(self, N, n, dirichlet):
        x, w, d, lL, lR = _basis(n)
        h = L / N
        iw = 1.0 / w[:, None]
        self.N, self.n, self.dirichlet, self.w = N, n, dirichlet, 0.5 * h * w
        s = 2.0 / h
        up, lo = iw * lR[:, None], iw * lL[:, None]          # lifts of the right and left face
        # central flux: the mean of the two traces on an inner face, 0 on a Dirichlet boundary face
        self.c = (s * (d - 0.5 * up * lR + 0.5 * lo * lL), s * 0.5 * up * lL, -s * 0.5 * lo * lR)
        self.c_first, self.c_last = s * 0.5 * lo * lL, -s * 0.5 * up * lR
        # flux from the right cell
        self.f = (s * (d - up * lR), s * up * lL, None)
        self.f_first = s * lo * lL                          # the left boundary face's own trace drops out
        self.pen = np.outer(lL, lL) / h

    def dense(self, blocks, first, last):
        N, n = self.N, self.n
        A = np.zeros((N, n, N, n))
        for c in range(N):
            A[c, :, c, :] += blocks[0]
            if blocks[1] is not None and (c + 1 < N or not self.dirichlet):
                A[c, :, (c + 1) % N, :] += blocks[1]
            if blocks[2] is not None and (c > 0 or not self.dirichlet):
                A[c, :, (c - 1) % N, :] += blocks[2]
        if self.dirichlet:
            A[0, :, 0, :] += first
            A[N - 1, :, N - 1, :] += last
        return A.reshape(N * n, N * n)

    def ldg_scaled(self):
        """Dense W^-1/2 A1 W^-1/2 (Dirichlet grids)."""
        F = self.dense(self.f, self.f_first, np.zeros((self.n, self.n)))
        W = np.tile(self.w, self.N)
        G = np.sqrt(W)[:, None] * F / np.sqrt(W)[None, :]
        K = G.T @ G
        K[:self.n, :self.n] += self.pen / np.sqrt(np.outer(self.w, self.w))
        return K

    def symbols(self):
        """Singular values squared and right singular vectors of the scaled forward derivative
        at every wave number of a periodic line."""
        sw = np.sqrt(self.w)
        th = 2 * np.pi * np.arange(self.N) / self.N
        G = self.f[0][None] + np.exp(1j * th)[:, None, None] * self.f[1][None]
        G = sw[None, :, None] * G / sw[None, None, :]
        _, s, vh = np.linalg.svd(G)
        s = s ** 2
        s[0, -1] = 0.0                                       # the constant
        return torch.from_numpy(s).cuda(), torch.from_numpy(vh).cuda()


class _Exact:
    def __init__(self, case):
        self.Nx, self.Ny, self.n = case["Nx"], case["Ny"], case["n"]
        self.dirichlet = case.get("bc", "periodic") == "dirichlet"
        self.x, self.y = _Line(self.Nx, self.n, self.dirichlet), _Line(self.Ny, self.n, self.dirichlet)
        self.W = torch.from_numpy(np.outer(self.y.w, self.x.w)).cuda()
        self.sym = None

    def _blocks(self, u, line, blocks, first, last, dim):
        """dim 1: along x (cell axis 1, node axis 3); dim 0: along y (axes 0 and 2)."""
        t = lambda B: torch.from_numpy(np.ascontiguousarray(B)).cuda()  # noqa: E731
        mul = (lambda B, v: v @ t(B).T) if dim == 1 else (lambda B, v: t(B) @ v)
        out = mul(blocks[0], u)
        cut = lambda v, i: v.narrow(dim, i, 1)  # noqa: E731
        for B, s, edge in ((blocks[1], -1, line.N - 1), (blocks[2], 1, 0)):
            if B is not None:
                v = torch.roll(u, s, dim)
                if self.dirichlet:
                    cut(v, edge).zero_()
                out += mul(B, v)
        if self.dirichlet:
            cut(out, 0).add_(mul(first, cut(u, 0)))
            if last is not None:
                cut(out, line.N - 1).add_(mul(last, cut(u, line.N - 1)))
        return out

    def d(self, u, dim):
        line = self.x if dim == 1 else self.y
        return self._blocks(u, line, line.c, line.c_first, line.c_last, dim)

    def minus_laplace(self, u):
        out = torch.zeros_like(u)
        for dim, line in ((1, self.x), (0, self.y)):
            q = self._blocks(u, line, line.f, line.f_first, None, dim)
            # W^-1 D^T W: transposed blocks, the neighbours swapped
            w = line.w
            tr = lambda B: (B * w[:, None]).T / w[:, None]  # noqa: E731
            out += self._blocks(q, line, (tr(line.f[0]), None, tr(line.f[1])), tr(line.f_first), None, dim)
            if self.dirichlet:
                B = torch.from_numpy(line.pen / w[:, None]).cuda()
                e = u.narrow(dim, 0, 1)
                out.narrow(dim, 0, 1).add_(e @ B.T if dim == 1 else B @ e)
        return out

    def bracket(self, f, g):
        fx, fy, gx, gy = self.d(f, 1), self.d(f, 0), self.d(g, 1), self.d(g, 0)
        return (fx * gy - fy * gx + self.d(f * gy - fy * g, 1) + self.d(fx * g - f * gx, 0)) / 3.0

    def solve(self, w):
        sw = self.W.sqrt()
        if self.dirichlet:
            if self.sym is None:
                self.sym = [torch.linalg.eigh(torch.from_numpy(ln.ldg_scaled()).cuda()) for ln in (self.x, self.y)]
            (lx, vx), (ly, vy) = self.sym
            b = (w * sw).permute(0, 2, 1, 3).reshape(self.Ny * self.n, self.Nx * self.n)
            y = vy @ ((vy.T @ b @ vx) / (ly[:, None] + lx[None, :])) @ vx.T
            return _blocked(y, self.Ny, self.Nx, self.n) / sw
        if self.sym is None:
            self.sym = self.x.symbols(), self.y.symbols()
        (lx, vx), (ly, vy) = self.sym
        mean = (w * self.W).sum() / (L * L)
        h = torch.fft.fft2((w - mean) * sw, dim=(0, 1))
        # t[ky, kx, i, j] = sum vy[ky, i, a] vx[kx, j, b] h[ky, kx, a, b]
        h = vy[:, None] @ (h @ vx.transpose(1, 2)[None])
        lam = ly[:, None, :, None] + lx[None, :, None, :]
        h /= torch.where(lam == 0, torch.ones_like(lam), lam)
        h *= lam != 0
        del lam
        h = vy.conj().transpose(1, 2)[:, None] @ (h @ vx.conj()[None])
        y = torch.fft.ifft2(h, dim=(0, 1)).real / sw
        return y - (y * self.W).sum() / (L * L)

    def advance(self, case, w):
        D, dt = case["D"], case["dt"]
        rhs = lambda w: -self.bracket(self.solve(w), w) - (D * self.minus_laplace(w) if D > 0 else 0.0)  # noqa: E731
        hist = []
        for _ in range(2):  # classical Runge-Kutta start-up
            k1 = rhs(w)
            k2 = rhs(w + 0.5 * dt * k1)
            k3 = rhs(w + 0.5 * dt * k2)
            k4 = rhs(w + dt * k3)
            hist.append(k1)
            w = w + dt * (k1 + 2 * k2 + 2 * k3 + k4) / 6.0
        for _ in range(case["steps"]):
            hist = hist[-2:] + [rhs(w)]
            w = w + dt * (23 * hist[2] - 16 * hist[1] + 5 * hist[0]) / 12.0
        return [w, self.solve(w)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [t for m in _ensemble(case, seed) for t in _Exact(m).advance(m, _field(m, m["seed"]))]
    E = _Exact(case)
    if kind == "step":
        return E.advance(case, _field(case, seed))
    w = _field(case, 2 * seed)
    if kind == "poisson":
        return E.solve(w)
    if kind == "laplace":
        v = E.minus_laplace(w)
        return -v if case["mode"] == 1 else v * E.W
    p = _field(case, 2 * seed + 1)
    if kind == "bracket":
        return E.bracket(p, w)
    _correlate(p, w)
    return [(E.W * w).sum(), 0.5 * (E.W * w * p).sum(), 0.5 * (E.W * w * w).sum()]
