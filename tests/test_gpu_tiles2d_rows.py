"""The tiled 2D passes with two and three rows per warp, which large and long grids take (the rule: as few rounds of tiles
over the SMs as possible), at the edges of their tiles and against the oracle, with Dirichlet nodes anywhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg, solvers  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
UP = {1: 6, 2: 14, 3: 22}    # own rows of a tile going up and in the product, by rows per warp
DOWN = {1: 2, 2: 6, 3: 10}   # coarse rows of a tile going down


def rows(width, height, per_x, per_y):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    best = None
    for r in (3, 2, 1):
        cost = r * -(-(-(-width // per_x) * -(-height // per_y[r])) // sms)
        if best is None or cost < best[1]:
            best = (r, cost)
    return best[0]


def grids(r, down):
    """(nx, ny) one tile wide whose tiles have r rows per warp: as many rows as fill whole tiles, one less and one more."""
    per = DOWN[r] if down else UP[r]
    for count in range(1, 2000):
        tall = [count * per + d for d in (-1, 0, 1)]
        if down:
            found = [rows(31, h, 30, DOWN) == r for h in tall]
            dims = [(60, 2 * (h - 1)) for h in tall]
        else:
            found = [rows(62, h, 62, UP) == r for h in tall]
            dims = [(61, h - 1) for h in tall]
        if all(found):
            return dims
    raise AssertionError("no such grid")


def problem(nx, ny, seed):
    g = fem.Grid(nx, ny, 0)
    rng = np.random.default_rng(seed)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = (rng.uniform(size=g.n_nodes) < 0.03).astype(np.uint8)
    grid = fixed.reshape(ny + 1, nx + 1)
    grid[-2:, :] = grid[:, -2:] = 0
    fixed[0] = 1
    return g, rho, fixed, workloads.nodal_load(fixed), rng


@pytest.mark.parametrize("down", [False, True])
@pytest.mark.parametrize("r", [2, 3])
@pytest.mark.parametrize("precision,tol", [(mgar.MGAR_FP64, 1e-10), (mgar.MGAR_MIXED, 5e-4)])
def test_vcycle_and_solve(r, down, precision, tol):
    for nx, ny in grids(r, down):
        g, rho, fixed, q, rng = problem(nx, ny, 17)
        A = fem.system_matrix(g, rho, fixed)
        levels = mg.build_hierarchy(A, fixed, (nx, ny), 5)
        b = rng.standard_normal(g.n_nodes) * (fixed == 0)
        ref_t = solvers.exact_solve(A, q)
        p = mgar.default_params(nx=nx, ny=ny, nz=0, nl=5, eps2=1e-12, precision=precision)
        with mgar.Solver(p, fixed, q) as s:
            s.set_density(torch.tensor(rho, device=DEV), physical=True)
            s.build_hierarchy()
            for x0 in (np.zeros(g.n_nodes), rng.standard_normal(g.n_nodes) * (fixed == 0)):
                ref = mg.vcycle(levels, b, x0.copy())
                x = torch.tensor(x0, device=DEV)
                s.vcycle(torch.tensor(b, device=DEV), x)
                np.testing.assert_allclose(x.cpu().numpy(), ref, rtol=0, atol=tol * np.abs(ref).max())
            T = torch.zeros(g.n_nodes, dtype=torch.float64, device=DEV)
            _, _, ok = s.solve_mgcg(T)
        assert ok
        np.testing.assert_allclose(T.cpu().numpy(), ref_t, rtol=0, atol=1e-9 * np.abs(ref_t).max())
