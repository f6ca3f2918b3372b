"""The FP32 passes of the finest 3D level on linear segments of the node planes: rows from a few nodes to the longest that
are staged (1151) and one more (the tiled passes), planes shorter and longer than a segment, Dirichlet nodes anywhere,
against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg, solvers  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

EDGES = [(4, 4, 40), (31, 31, 5), (31, 32, 6), (9, 113, 3), (250, 9, 4), (506, 6, 4), (762, 5, 4), (1150, 4, 3),
         (1151, 4, 3)]


@pytest.mark.parametrize("dims", EDGES)
def test_vcycle_and_solve(dims):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    rng = np.random.default_rng(41)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = (rng.uniform(size=g.n_nodes) < 0.03).astype(np.uint8)
    # (a coarse node whose fine nodes are all fixed has no equation)
    grid = fixed.reshape(nz + 1, ny + 1, nx + 1)
    grid[-2:] = grid[:, -2:] = grid[:, :, -2:] = 0
    fixed[0] = 1
    q = workloads.nodal_load(fixed)
    A = fem.system_matrix(g, rho, fixed)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, eps2=1e-12, precision=mgar.MGAR_MIXED)
    with mgar.Solver(p, fixed, q) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        s.build_hierarchy()
        b = rng.standard_normal(g.n_nodes) * (fixed == 0)
        x0 = rng.standard_normal(g.n_nodes) * (fixed == 0)
        ref = mg.vcycle(mg.build_hierarchy(A, fixed, (nx, ny, nz), 2), b, x0.copy())
        xg = torch.tensor(x0, device=DEV)
        s.vcycle(torch.tensor(b, device=DEV), xg)
        # ~30 FP32 roundings per row and pass, times the coarse level's conditioning (1e3 at most here)
        np.testing.assert_allclose(xg.cpu().numpy(), ref, rtol=0, atol=1e-4 * np.abs(ref).max())
        ref = solvers.exact_solve(A, q)
        T = torch.tensor(rng.standard_normal(g.n_nodes) * np.abs(ref).max(), device=DEV)
        _, _, ok = s.solve_mgcg(T)
        assert ok
        np.testing.assert_allclose(T.cpu().numpy(), ref, rtol=0, atol=1e-9 * np.abs(ref).max())
