"""The tiled 2D passes at the edges of their tiles: grids one short of, at and one past the own nodes of a tile (60 x 20
going down, 62 x 22 going up and in the product), their coarse levels (30 x 6 and 30 x 8), odd axes, and Dirichlet nodes
anywhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg, solvers  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def problem(nx, ny, seed):
    g = fem.Grid(nx, ny, 0)
    rng = np.random.default_rng(seed)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = (rng.uniform(size=g.n_nodes) < 0.03).astype(np.uint8)
    # a coarse node whose fine nodes are all fixed has no equation: on an odd axis
    # the last one hangs on the last fine node alone
    grid = fixed.reshape(ny + 1, nx + 1)
    grid[-2:, :] = grid[:, -2:] = 0
    fixed[0] = 1
    return g, rho, fixed, workloads.nodal_load(fixed), rng


EDGES = [(59, 19), (60, 20), (61, 21), (62, 22), (63, 44), (119, 43), (121, 41), (124, 63), (7, 130), (130, 5)]


@pytest.mark.parametrize("nx,ny", EDGES)
@pytest.mark.parametrize("precision,tol", [(mgar.MGAR_FP64, 1e-10), (mgar.MGAR_MIXED, 5e-4)])
def test_vcycle(nx, ny, precision, tol):
    g, rho, fixed, q, rng = problem(nx, ny, 11)
    levels = mg.build_hierarchy(fem.system_matrix(g, rho, fixed), fixed, (nx, ny), 3)
    b = rng.standard_normal(g.n_nodes) * (fixed == 0)
    x0 = rng.standard_normal(g.n_nodes) * (fixed == 0)
    ref = mg.vcycle(levels, b, x0.copy())
    p = mgar.default_params(nx=nx, ny=ny, nz=0, nl=3, precision=precision)
    with mgar.Solver(p, fixed, q) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        s.build_hierarchy()
        x = torch.tensor(x0, device=DEV)
        s.vcycle(torch.tensor(b, device=DEV), x)
        np.testing.assert_allclose(x.cpu().numpy(), ref, rtol=0, atol=tol * np.abs(ref).max())


@pytest.mark.parametrize("nx,ny", EDGES)
@pytest.mark.parametrize("precision", [mgar.MGAR_FP64, mgar.MGAR_MIXED])
@pytest.mark.parametrize("graph", [True, False])
def test_mgcg(nx, ny, precision, graph, monkeypatch):
    # a warm start with values on fixed nodes (which their identity rows remove)
    if not graph:
        monkeypatch.setenv("MGAR_NO_GRAPHS", "1")
    g, rho, fixed, q, rng = problem(nx, ny, 13)
    ref = solvers.exact_solve(fem.system_matrix(g, rho, fixed), q)
    p = mgar.default_params(nx=nx, ny=ny, nz=0, nl=3, eps2=1e-12, precision=precision)
    with mgar.Solver(p, fixed, q) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        T = torch.tensor(rng.standard_normal(g.n_nodes) * np.abs(ref).max(), device=DEV)
        _, _, ok = s.solve_mgcg(T)
    assert ok
    np.testing.assert_allclose(T.cpu().numpy(), ref, rtol=0, atol=1e-9 * np.abs(ref).max())
