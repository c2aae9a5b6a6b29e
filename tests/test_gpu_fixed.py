"""The fixed-point kernels where they can go wrong: tile edges and remainders for every n,
anisotropic cells, the parts the tables do not cover (a jump penalty), values outside the
fixed-point range, which the float64 tile takes; and the spectral solve on the shortest, the
unequal and the odd-power lines of its integer DFTs.

Bars: 1e-12 in relative L2 against the float64 oracle, as for the float64 evaluation: one rounding of
2^-60 of a tile's largest value per term against the oracle's own 2^-53.  Fields are i.i.d. normal,
so no value is more than a few bits below its tile's largest.  The spectral solve is held to the bar of
two backward-stable solutions (test_gpu_spectral.solve_bar) and, scaled by a power of two, to the
same bits.
"""
import numpy as np
import pytest

from oracle.operators import Operators
from oracle.solver import Spectral, poisson_rhs, rounding_floor2
from oracle.tables import Grid as OGrid
from tests.test_gpu_parity import RHO_D, bracket_scale, dev, host, rel_l2
from tests.test_gpu_spectral import solve_bar

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# default tiles are 16 x 16 (n = 1, 2), 8 x 16 (n = 3), 8 x 8 (n = 4, 5), smaller on small grids
SHAPES = [(33, 17, 1), (17, 35, 2), (40, 41, 3), (9, 70, 4), (41, 33, 5), (2, 3, 5)]


@pytest.fixture(scope="module")
def dg(native):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return native


@pytest.mark.parametrize("Nx,Ny,n", SHAPES)
@pytest.mark.parametrize("bc,tau", [("periodic", 0.0), ("periodic", 0.3), ("dirichlet", 0.0)])
def test_rhs(dg, Nx, Ny, n, bc, tau):
    """R = -J(psi, omega) + D Delta_h omega of one Adams-Bashforth step, read back from the state."""
    Lx, Ly, D = 1.5, 2.0, 0.05
    g = dg.Grid(Nx, Ny, n, Lx, Ly, tau, bc=bc)
    o = Operators(OGrid(Nx, Ny, n, Lx, Ly), tau=tau, bc=bc)
    psi, w, z = np.random.default_rng(Nx + n).standard_normal((3, Ny, Nx, n, n))
    s = dg.Sim(g, dev(np.zeros(g.shape)), D=D, dt=1e-6)
    s.set_state(5, dev(w), dev(psi), dev(psi), dev(z), dev(z))
    s.set_cg(1e-30, 10, fixed_iters=1)
    s.step(1)
    b = [torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(5)]
    s.get_state(*b)
    R = host(b[3])
    lap = D * o.laplacian(w)
    ref = -o.bracket(psi, w) + lap
    assert rel_l2(R, ref, bracket_scale(o, psi, w) + np.linalg.norm(lap.ravel())) < 1e-12
    assert rel_l2(host(b[0]), w + 1e-6 * (23 * ref - 16 * z + 5 * z) / 12) < 1e-12


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_bracket_outside_the_fixed_point_range(dg, n):
    Nx, Ny = 21, 19
    g = dg.Grid(Nx, Ny, n)
    o = Operators(OGrid(Nx, Ny, n))
    f, h = np.random.default_rng(n).standard_normal((2, Ny, Nx, n, n))
    J = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    ref = o.bracket(f, h)
    scale = bracket_scale(o, f, h)
    for a, b in ((1e250, 1e-80), (1e-150, 1e-150), (1e150, 1e150), (0.0, 1e200)):
        dg.dg_bracket(g, dev(a * f), dev(b * h), J)
        assert rel_l2(host(J) / a / b if a else host(J), ref if a else 0.0 * ref, scale) < 1e-12, (a, b)
    # a value that is not finite spoils exactly the nodes whose stencils reach it
    for bad in (np.nan, np.inf):
        f2 = f.copy()
        f2[9, 10, n // 2, 0] = bad
        dg.dg_bracket(g, dev(f2), dev(h), J)
        with np.errstate(invalid="ignore"):
            want = o.bracket(f2, h)
        got = host(J)
        assert np.array_equal(np.isfinite(got), np.isfinite(want))
        ok = np.isfinite(want)
        assert rel_l2(got[ok], ref[ok], scale) < 1e-12


@pytest.mark.parametrize("Nx,Ny,n", [(1, 1, 4), (1, 4, 3), (2, 1, 5), (2, 2, 1), (8, 4, 2), (16, 8, 3), (32, 64, 4),
                                     (128, 2, 5), (4, 256, 2), (64, 32, 5)])
@pytest.mark.parametrize("field", ["noise", "point", "mode"])
def test_spectral_solve(dg, Nx, Ny, n, field):
    Lx, Ly = 1.5, 2.0
    g = dg.Grid(Nx, Ny, n, Lx, Ly)
    g.set_precond("spectral")
    og = OGrid(Nx, Ny, n, Lx, Ly)
    o = Operators(og)
    w = np.random.default_rng(Nx + n).standard_normal(g.shape)
    if field == "point":
        w = np.zeros(g.shape)
        w[Ny // 2, Nx // 2, 0, n - 1] = 1.0
    if field == "mode":
        X, Y = og.mesh()
        w = np.cos(2 * np.pi * X / Lx) * np.cos(2 * np.pi * Y / Ly) + 1e-9 * w
    ref = Spectral(o)(poisson_rhs(o, w))
    out = []
    for k in (0, 300, -300):
        psi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        rc, it, relres = dg.dg_poisson_solve(g, dev(np.ldexp(w, k)), psi, 1e-10, 50)
        assert it <= 2 and relres <= 1e-10
        out.append(np.ldexp(host(psi), -k))
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    assert rel_l2(out[0], ref) < solve_bar(o, Lx, Ly)


def test_spectral_solve_batched(dg):
    """Float64 members with the spectral preconditioner: batched steps against the same steps alone
    (the sums run over other block counts)."""
    def make():
        out = []
        for Nx, Ny, n in ((32, 16, 3), (16, 64, 5), (8, 8, 2)):
            g = dg.Grid(Nx, Ny, n)
            g.set_precond("spectral")
            X, Y = OGrid(Nx, Ny, n).mesh()
            w = np.sin(X) * np.cos(2 * Y) + 0.3 * np.cos(X + Y)
            out.append((g, dg.Sim(g, dev(w), D=1e-3, dt=1e-3, cg_tol=1e-11)))
        return out
    alone, members = make(), make()
    b = dg.Batch(3)
    for _, s in members:
        b.admit(s)
    b.step(4)
    assert b.status()["rc"] == 0
    for (g, s), (_, t) in zip(alone, members):
        s.step(6)  # two start-up steps on admission, four batched
        f = [torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(4)]
        s.get(f[0], f[1])
        t.get(f[2], f[3])
        assert rel_l2(host(f[2]), host(f[0])) < 1e-11 and rel_l2(host(f[3]), host(f[1])) < 1e-10


def _steady(Nx, Ny, n):
    X, Y = OGrid(Nx, Ny, n).mesh()
    return 2 * np.sin(X) * np.sin(Y)


@pytest.mark.parametrize("maxit", [0, 50])
def test_spectral_solve_of_an_accepted_guess(dg, maxit):
    """A guess that meets the tolerance, plus a constant: no application, and the constant goes.  The
    mean left is that of one rounding (2^-53) of each value, here held to ten times that."""
    Nx, Ny, n = 32, 16, 4
    g = dg.Grid(Nx, Ny, n)
    g.set_precond("spectral")
    W = OGrid(Nx, Ny, n).weights()
    w = _steady(Nx, Ny, n)
    psi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    dg.dg_poisson_solve(g, dev(w), psi, 1e-11)
    good = host(psi).copy()
    psi += 3.0
    rc, it, relres = dg.dg_poisson_solve(g, dev(w), psi, 1e-7, maxit=maxit)
    assert it == 0 and relres <= 1e-7
    got = host(psi)
    assert abs(np.sum(W * got) / np.sum(W * np.ones(g.shape))) < 10 * 2.0 ** -53 * 4
    assert rel_l2(got, good) < 1e-14
    # not converged and no application allowed: the guess without its mean, and the error
    psi = dev(0.5 * good + 3.0)
    rc, it, relres = dg.dg_poisson_solve(g, dev(w), psi, 1e-7, maxit=0, check=False)
    assert rc == dg.DG_ERR_NOCONV and it == 0 and abs(relres - 0.5) < 1e-6
    assert rel_l2(host(psi), 0.5 * good) < 1e-14


def test_accepted_guess_leaves_its_operator_product(dg):
    """Solves that accept their guess, after a state was set over unrelated fields: the next solve
    starts from the products that these left, so one application is enough."""
    Nx, Ny, n = 32, 32, 3
    g = dg.Grid(Nx, Ny, n)
    g.set_precond("spectral")
    noise = np.random.default_rng(5).standard_normal(g.shape)
    s = dg.Sim(g, dev(1e3 * noise), D=0.0, dt=1e-7, cg_tol=1e-10)
    s.step(4)
    w = _steady(Nx, Ny, n)
    psi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
    dg.dg_poisson_solve(g, dev(w), psi, 1e-12)
    z = dev(np.zeros(g.shape))
    s.set_state(4, dev(w), psi, psi, z, z)
    s.set_cg(1e-4, 100)
    s.step(3)
    assert s.status().cg_iters_last == 0
    s.set_cg(1e-10, 100)
    s.step(1)
    assert s.status().cg_iters_last <= 1


@pytest.mark.parametrize("Nx,Ny,n", [(4096, 2, 4), (1, 4096, 5)])
@pytest.mark.parametrize("mode", ["mixed", "mixed64"])
def test_mixed_steps_on_lines_too_long_for_the_fixed_point_solve(dg, Nx, Ny, n, mode):
    """The mixed modes on a side whose 16-byte lines exceed shared memory: their float32 sweeps.  The
    residual of the initial solve and of a step is measured with the oracle's operator; the bar is
    the tolerance and the float64 rounding floor of the residual."""
    g = dg.Grid(Nx, Ny, n)
    g.set_precond("spectral")
    og = OGrid(Nx, Ny, n)
    o = Operators(og)
    X, Y = og.mesh()
    w = np.sin(3 * X) * np.cos(Y) + 0.3 * np.cos(5 * X + 2 * Y) + 0.2 * np.sin(7 * Y) + 0.2 * np.sin(4 * X)
    s = dg.Sim(g, dev(w), D=0.0, dt=1e-6, precision={"mixed": dg.DG_MIXED, "mixed64": dg.DG_MIXED64}[mode], cg_tol=1e-8)
    om, ps = (torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(2))
    for k in range(2):
        s.step(k)
        assert s.status().status == 0
        s.get(om, ps)
        p, b = host(ps), poisson_rhs(o, host(om))
        r = b - o.A(p)
        norm = lambda v: np.sqrt(np.sum(v * v / o.W2))
        floor = np.sqrt(rounding_floor2(o) * np.sum(o.W2 * p * p))
        assert norm(r) <= 1e-8 * norm(b) + 2 * floor


def _line_mode(dg, N, n, L, k, branch):
    """A real eigenvector of the scaled 1D operator of a line as node values (N, n) of the field (the
    scaled one over sqrt(w)), and its eigenvalue."""
    lam, V = dg.spectral_symbol(N, n, L, k)
    u = np.real(np.exp(2j * np.pi * (k * np.arange(N) % N) / N)[:, None] * V[None, :, branch])
    return u / np.sqrt(np.polynomial.legendre.leggauss(n)[1]), lam[branch]


@pytest.mark.parametrize("Nx,Ny,n", [(4, 1024, 5), (4, 2048, 5), (2, 4096, 3), (1024, 4, 5), (2, 16, 4)])
def test_spectral_solve_of_high_modes(dg, Nx, Ny, n):
    """Single eigenmodes of the highest branch along the long side, with quotients up to 2^27 below those
    of the line's smooth modes: solved in one application or two."""
    Lx, Ly = 1.5, 2.0
    g = dg.Grid(Nx, Ny, n, Lx, Ly)
    g.set_precond("spectral")
    bar = solve_bar(Operators(OGrid(Nx, Ny, n, Lx, Ly)), Lx, Ly)
    N, L = max((Nx, Lx), (Ny, Ly))
    for k in sorted({0, 1, 3, N // 4, N // 2 - 1, N // 2}):
        u, lam = _line_mode(dg, N, n, L, k, n - 1)
        u /= np.abs(u).max()
        w = np.empty(g.shape)
        w[:] = u[None, :, None, :] if Nx > Ny else u[:, None, :, None]
        psi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        rc, it, relres = dg.dg_poisson_solve(g, dev(w), psi, 1e-10, 50)
        assert it <= 2 and relres <= 1e-10, k
        assert rel_l2(host(psi), w / lam) < bar, k


def test_spectral_solve_of_a_high_and_a_small_smooth_mode(dg):
    """A mode of the highest branch along the long lines, and a smooth one across them that is small in
    the right-hand side and larger in the solution."""
    Nx, Ny, n, Lx = 1024, 16, 5, 1.0
    g = dg.Grid(Nx, Ny, n, Lx, 16 * Lx)
    g.set_precond("spectral")
    hi, lam = _line_mode(dg, Nx, n, Lx, 1, n - 1)
    lo, mu = _line_mode(dg, Ny, n, 16 * Lx, 1, 0)
    hi, lo = hi / np.abs(hi).max(), lo / np.abs(lo).max()
    for s in (-28, -29, -30):
        w = hi[None, :, None, :] + 2.0 ** s * lo[:, None, :, None]
        ref = hi[None, :, None, :] / lam + 2.0 ** s / mu * lo[:, None, :, None]
        psi = torch.zeros(g.shape, dtype=torch.float64, device="cuda")
        rc, it, relres = dg.dg_poisson_solve(g, dev(w), psi, 1e-12, 50)
        assert it <= 2 and relres <= 1e-12, s
        assert rel_l2(host(psi), ref) < 1e-5, s


@pytest.mark.parametrize("n,tile", [(4, (26, 25)), (5, (20, 21))])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("precond", ["jacobi", "twolevel"])
def test_batch_with_large_solve_tiles(dg, n, tile, prec, precond):
    """Solve tiles that fit shared memory with their face traces, but not with the fixed-point results
    beside the box: accepted, and the steps agree with those on the built-in tiles to the bar of the
    batched tests for solves stopped by a tolerance (1e-8)."""
    out = []
    for t in (tile, (0, 0)):
        g = dg.Grid(30, 28, n)
        g.set_precond(precond)
        X, Y = OGrid(30, 28, n).mesh()
        s = dg.Sim(g, dev(np.sin(X) * np.cos(2 * Y) + 0.3 * np.cos(X + Y)), D=1e-3, dt=1e-3, cg_tol=1e-12,
                   precision=dg.DG_FP64 if prec == "fp64" else dg.DG_MIXED)
        b = dg.Batch(1)
        b.set_tiles(n, cg=t)
        b.admit(s)
        b.step(2)
        assert b.status()["rc"] == 0
        f = [torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(2)]
        s.get(*f)
        out.append([host(x) for x in f])
    for a, c in zip(*out):
        assert rel_l2(a, c) < 1e-8


def test_batch_refuses_tiles_that_never_fitted(dg):
    g = dg.Grid(32, 32, 5)
    s = dg.Sim(g, dev(np.random.default_rng(0).standard_normal(g.shape)), dt=1e-6)
    b = dg.Batch(1)
    b.set_tiles(5, cg=(28, 28))
    b.admit(s)
    with pytest.raises(dg.DGError) as e:
        b.step(1)
    assert e.value.code == dg.DG_ERR_ARG


@pytest.mark.parametrize("N,n", [(640, 4), (512, 5)])
def test_pointwise_bracket_of_resolved_fields(dg, N, n):
    """J++ alone on fields whose derivatives are far below the range of their rows.  The bar is the
    float64 rounding of the two factors: each derivative is off by about 2^-53 rho_D / h |f|, and
    |f| ~ |f_x| here; four times that."""
    g = dg.Grid(N, N, n)
    og = OGrid(N, N, n)
    o = Operators(og)
    X, Y = og.mesh()
    f, h = np.sin(X) * np.cos(Y) + 0.2 * np.cos(2 * Y), np.cos(X - Y) + 0.3 * np.sin(2 * X)
    J = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    dg.dg_bracket_parts(g, dev(f), dev(h), J, 1)
    assert rel_l2(host(J), o.bracket_parts(f, h)[0]) < 4 * 2.0 ** -53 * RHO_D[n] / og.hx


@pytest.mark.parametrize("Nx,Ny,n", SHAPES)
@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
def test_pointwise_bracket(dg, Nx, Ny, n, bc):
    """J++ alone, in a bracket and in a step with viscosity; it changes sign with its arguments' order
    and vanishes on equal ones, bitwise; its result scales with powers of two."""
    Lx, Ly, D = 1.5, 2.0, 0.05
    g = dg.Grid(Nx, Ny, n, Lx, Ly, bc=bc)
    o = Operators(OGrid(Nx, Ny, n, Lx, Ly), bc=bc)
    psi, w, z = np.random.default_rng(Nx + n).standard_normal((3, Ny, Nx, n, n))
    scale = bracket_scale(o, psi, w)
    J = torch.empty(g.shape, dtype=torch.float64, device="cuda")

    def jpp(a, b):
        dg.dg_bracket_parts(g, dev(a), dev(b), J, 1)
        return host(J).copy()
    a = jpp(psi, w)
    assert rel_l2(a, o.bracket_parts(psi, w)[0], scale) < 1e-12
    assert np.array_equal(jpp(w, psi), -a) and not jpp(psi, psi).any()
    assert np.array_equal(jpp(np.ldexp(psi, 200), np.ldexp(w, -100)), np.ldexp(a, 100))
    s = dg.Sim(g, dev(np.zeros(g.shape)), D=D, dt=1e-6)
    s.set_bracket("naive")
    s.set_state(5, dev(w), dev(psi), dev(psi), dev(z), dev(z))
    s.set_cg(1e-30, 10, fixed_iters=1)
    s.step(1)
    b = [torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(5)]
    s.get_state(*b)
    lap = D * o.laplacian(w)
    assert rel_l2(host(b[3]), lap - o.bracket_parts(psi, w)[0], scale + np.linalg.norm(lap.ravel())) < 1e-12


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("bc", ["periodic", "dirichlet"])
@pytest.mark.parametrize("bits", [5, 8, 9, 20, 45, 70, 300])
def test_cells_far_below_their_tile(dg, n, bc, bits):
    """A cell 2^bits times the others, or others that are that much smaller: away from it the operators'
    results are those without it, to the bar of the other fields, 1e-12 of the local scale (2^12 times
    2^-53 where the fixed-point range ends)."""
    Nx, Ny, Lx, Ly, D = 19, 17, 1.5, 2.0, 0.05
    g = dg.Grid(Nx, Ny, n, Lx, Ly, bc=bc)
    g.set_tiles(16 if n < 3 else 8, 16 if n < 3 else 8)  # (not the small tiles of a small grid)
    o = Operators(OGrid(Nx, Ny, n, Lx, Ly), bc=bc)
    f, h = np.random.default_rng(n).standard_normal((2, Ny, Nx, n, n))
    out = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    cy, cx = 6, 9
    dy, dx = np.abs(np.arange(Ny) - cy), np.abs(np.arange(Nx) - cx)
    away = np.maximum(dy[:, None], dx[None, :]) >= 2
    lap = o.laplacian(h)
    J, scale = o.bracket(f, h), bracket_scale(o, f, h)
    Jp = o.bracket_parts(f, h)[0]

    def check(got, want, k, scale=0.0):
        assert rel_l2(np.ldexp(host(got), k)[away], want[away], scale) < 1e-12

    for up in (True, False):  # the cell raised, or the rest lowered (into subnormal products at 300)
        def spiked(u):
            v = u.copy() if up else np.ldexp(u, -bits)
            v[cy, cx] = np.ldexp(u[cy, cx], bits) if up else u[cy, cx]
            return dev(v), 0 if up else bits
        F, k = spiked(f)
        H, _ = spiked(h)
        for a, b, m in ((F, dev(h), k), (dev(f), H, k), (F, H, 2 * k)):
            dg.dg_bracket(g, a, b, out)
            check(out, J, m, scale)
            dg.dg_bracket_parts(g, a, b, out, 1)
            check(out, Jp, m, scale)
        for mode, want in ((0, o.A(h)), (1, lap)):
            dg.dg_laplace_apply(g, H, out, mode=mode)
            check(out, want, k)
        # a step's right-hand side, J and the viscous term, from the spiked vorticity
        s = dg.Sim(g, dev(np.zeros(g.shape)), D=D, dt=1e-6)
        z = dev(np.zeros(g.shape))
        s.set_state(5, H, dev(f), dev(f), z, z)
        s.set_cg(1e-30, 10, fixed_iters=1)
        s.step(1)
        b = [torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(5)]
        s.get_state(*b)
        check(b[3], D * lap - J, k, scale)


def test_zero_far_from_a_compact_field(dg):
    """A field of a few cells: exactly zero where its stencils do not reach."""
    Nx, Ny, n = 40, 24, 4
    g = dg.Grid(Nx, Ny, n)
    f, h = np.random.default_rng(1).standard_normal((2, Ny, Nx, n, n))
    h[:10], h[13:], h[:, :20], h[:, 23:] = 0, 0, 0, 0
    out = torch.empty(g.shape, dtype=torch.float64, device="cuda")
    dg.dg_bracket(g, dev(f), dev(h), out)
    J = host(out).copy()
    assert np.abs(J[9:14, 19:24]).max() > 0
    J[8:15, 18:25] = 0
    assert not J.any()
    dg.dg_laplace_apply(g, dev(h), out, mode=1)
    q = host(out).copy()
    q[8:15, 18:25] = 0
    assert not q.any()


@pytest.mark.parametrize("mode", ["mixed", "mixed64"])
def test_mixed_caps_on_the_fixed_point_solve(dg, mode):
    """The inner iteration cap of a mixed simulation is no cap on the solve's applications (several are
    needed here, to the rounding floor below an unreachable tolerance); its sweep cap is."""
    g = dg.Grid(32, 32, 4)
    g.set_precond("spectral")
    w = np.random.default_rng(3).standard_normal(g.shape)
    s = dg.Sim(g, dev(w), D=0.0, dt=1e-7, precision={"mixed": dg.DG_MIXED, "mixed64": dg.DG_MIXED64}[mode], cg_tol=1e-10)
    s.set_cg(1e-18, 1)
    s.step(2)
    info = s.status()
    assert info.status == 0 and info.cg_iters_last > 1
    s.set_refinement(1e-4, 1)
    s.step(1)
    info = s.status(check=False)
    assert info.status == dg.DG_ERR_NOCONV and info.cg_iters_last == 1
