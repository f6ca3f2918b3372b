"""The tiled FP64 passes of the finest 3D level at the edges of their tiles (32 x 8 nodes; 43 x 5 where that leaves fewer
idle lanes) and of their z runs, with Dirichlet nodes anywhere, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg, solvers  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

EDGES = [(31, 7, 4), (30, 6, 5), (32, 8, 3), (63, 15, 2), (42, 4, 6), (42, 9, 7), (43, 5, 8), (85, 9, 3), (4, 4, 40),
         (9, 33, 10)]


def problem(dims, seed):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    rng = np.random.default_rng(seed)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = (rng.uniform(size=g.n_nodes) < 0.03).astype(np.uint8)
    # (a coarse node whose fine nodes are all fixed has no equation)
    grid = fixed.reshape(nz + 1, ny + 1, nx + 1)
    grid[-2:] = grid[:, -2:] = grid[:, :, -2:] = 0
    fixed[0] = 1
    return g, rho, fixed, workloads.nodal_load(fixed), rng


@pytest.mark.parametrize("dims", EDGES)
def test_product_and_vcycle(dims):
    nx, ny, nz = dims
    g, rho, fixed, q, rng = problem(dims, 31)
    A = fem.system_matrix(g, rho, fixed)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2)
    with mgar.Solver(p, fixed, q) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        x = rng.standard_normal(g.n_nodes)
        y = torch.empty(g.n_nodes, dtype=torch.float64, device=DEV)
        s.apply_K(torch.tensor(x, device=DEV), y)
        ref = A @ x
        np.testing.assert_allclose(y.cpu().numpy(), ref, rtol=0, atol=1e-13 * np.abs(ref).max())
        s.build_hierarchy()
        b = rng.standard_normal(g.n_nodes) * (fixed == 0)
        x0 = rng.standard_normal(g.n_nodes) * (fixed == 0)
        ref = mg.vcycle(mg.build_hierarchy(A, fixed, (nx, ny, nz), 2), b, x0.copy())
        xg = torch.tensor(x0, device=DEV)
        s.vcycle(torch.tensor(b, device=DEV), xg)
        np.testing.assert_allclose(xg.cpu().numpy(), ref, rtol=0, atol=1e-10 * np.abs(ref).max())


@pytest.mark.parametrize("dims", EDGES)
@pytest.mark.parametrize("guess", [mgar.MGAR_GUESS_ZERO, mgar.MGAR_GUESS_PREVIOUS])
def test_solves(dims, guess):
    # MGCG from a warm start with values on fixed nodes, then a reanalysis of a
    # changed design against the oracle's on the same hierarchy
    nx, ny, nz = dims
    g, rho, fixed, q, rng = problem(dims, 37)
    A = fem.system_matrix(g, rho, fixed)
    ref = solvers.exact_solve(A, q)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, eps2=1e-12, m=2, basis_guess=guess)
    with mgar.Solver(p, fixed, q) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        T = torch.tensor(rng.standard_normal(g.n_nodes) * np.abs(ref).max(), device=DEV)
        _, _, ok = s.solve_mgcg(T)
        assert ok
        np.testing.assert_allclose(T.cpu().numpy(), ref, rtol=0, atol=1e-9 * np.abs(ref).max())
        rho2 = np.clip(rho + rng.uniform(-0.05, 0.05, g.n_elems), 0.05, 1.0)
        A2 = fem.system_matrix(g, rho2, fixed)
        levels = mg.build_hierarchy(A, fixed, (nx, ny, nz), 2)
        t_o, res_o = solvers.mgar(A2, A, levels, q, ref, m=2,
                                  basis_guess="zero" if guess == mgar.MGAR_GUESS_ZERO else "previous")
        s.set_density(torch.tensor(rho2, device=DEV), physical=True)
        out = torch.empty_like(T)
        res, _ = s.solve_mgar(torch.tensor(ref, device=DEV), out)
        np.testing.assert_allclose(out.cpu().numpy(), t_o, rtol=0, atol=1e-9 * np.abs(t_o).max())
        assert abs(res - res_o) < 1e-8 * max(1.0, res_o)
