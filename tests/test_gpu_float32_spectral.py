"""The float32 spectral transforms on power-of-two lines (radix-4 passes with and without a radix-2
one), which a single simulation's tolerance-stopped solves leave to the fixed-point solve: batched
members of the mixed modes, and the float32 preconditioner of DG_FP64_PC32 with a fixed iteration
count."""
import numpy as np
import pytest

from oracle.operators import Operators
from oracle.solver import Spectral, poisson_rhs
from oracle.stepper import Simulation
from oracle.tables import Grid as OGrid
from paper_1311_7477_gb300 import fields
from tests.test_gpu_spectral import dev, host, rel, solve_bar

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# even and odd powers of two, equal and unequal sides, every n
GRIDS = [(16, 16, 1), (32, 8, 2), (16, 64, 3), (32, 32, 4), (8, 16, 5), (128, 4, 3)]


@pytest.fixture(scope="module")
def dg(native):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return native


@pytest.mark.parametrize("mode", ["mixed", "mixed64"])
def test_batched_mixed_members(dg, mode):
    """One batched AB3 step from the oracle's state: omega and psi within 1e-10 of the oracle's and the
    true residual on its operator within the tolerance, the bars of the mixed modes alone."""
    D, dt = 1e-3, 5e-4
    b = dg.Batch(len(GRIDS))
    members = []
    for i, (Nx, Ny, n) in enumerate(GRIDS):
        og = OGrid(Nx, Ny, n)
        X, Y = og.mesh()
        osim = Simulation(Operators(og), fields.random_phase(X, Y, seed=20 + i, kmax=3), D, dt, tol=1e-13, K=3,
                          precond="spectral")
        osim.step(3)
        g = dg.Grid(Nx, Ny, n)
        g.set_precond("spectral")
        s = dg.Sim(g, dev(osim.omega), D=D, dt=dt, precision={"mixed": dg.DG_MIXED, "mixed64": dg.DG_MIXED64}[mode],
                   cg_tol=1e-12)
        s.set_state(3, dev(osim.omega), dev(osim.psi), dev(osim.psi_prev), dev(osim.R_hist[0]), dev(osim.R_hist[1]))
        b.admit(s)
        members.append((g, s, osim))
    b.step(1)
    assert b.status()["rc"] == 0
    for g, s, osim in members:
        osim.step(1)
        om, ps = (torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(2))
        s.get(om, ps)
        o, p = osim.ops, host(ps)
        assert rel(host(om), osim.omega) < 1e-10 and rel(p, osim.psi) < 1e-10, g.shape
        rhs = poisson_rhs(o, host(om))
        r = rhs - o.A(p)
        assert np.sqrt(np.sum(r * r / o.W2) / np.sum(rhs * rhs / o.W2)) < 1.5e-12, g.shape
        assert s.status().refine_sweeps_last >= 1, g.shape


@pytest.mark.parametrize("Nx,Ny,n", GRIDS)
def test_float32_preconditioner_with_fixed_iterations(dg, Nx, Ny, n):
    """DG_FP64_PC32, three fixed iterations from zero: each leaves the float32 rounding of its correction
    (1e-5 or better), so the solution is the direct solve's to its bar."""
    Lx, Ly = 2 * np.pi, 2 * np.pi
    og = OGrid(Nx, Ny, n)
    o = Operators(og)
    X, Y = og.mesh()
    g = dg.Grid(Nx, Ny, n)
    g.set_precond("spectral")
    w = fields.random_phase(X, Y, seed=Nx + n, kmax=3)
    z = dev(np.zeros(g.shape))
    s = dg.Sim(g, z, D=0.0, dt=1e-3, precision=dg.DG_FP64_PC32)
    s.set_cg(1e-30, 1000, fixed_iters=3)
    s.set_state(5, dev(w), z, z, z, z)  # psi = 0 and no history: omega stays, the solve starts from zero
    s.step(1)
    om, ps = (torch.empty(g.shape, dtype=torch.float64, device="cuda") for _ in range(2))
    s.get(om, ps)
    assert np.array_equal(host(om), w)
    assert rel(host(ps), Spectral(o)(poisson_rhs(o, w))) < solve_bar(o, Lx, Ly)
