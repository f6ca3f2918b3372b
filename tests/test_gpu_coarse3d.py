"""FP32 coarse levels in 3D: the restriction by columns, the rows by flat offsets (large levels) and the residual with its
restriction in one launch (small levels), at odd and even sizes and at the edges of their tiles, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# (elements per axis, levels): level 1 of 3 to 29 nodes per axis, every parity
SIZES = [((12, 12, 12), 3), ((13, 14, 15), 3), ((16, 31, 33), 4), ((57, 21, 18), 3), ((30, 47, 29), 4), ((7, 40, 25), 3)]


@pytest.mark.parametrize("split", ["1", "100000"])  # every coarse level by flat offsets, or by the fused launch
@pytest.mark.parametrize("dims,nl", SIZES)
def test_vcycle(dims, nl, split, monkeypatch):
    monkeypatch.setenv("MGAR_SPLIT_COARSE", split)
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    rng = np.random.default_rng(43)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = (rng.uniform(size=g.n_nodes) < 0.02).astype(np.uint8)
    # (a coarse node whose fine nodes are all fixed has no equation)
    grid = fixed.reshape(nz + 1, ny + 1, nx + 1)
    grid[-6:] = grid[:, -6:] = grid[:, :, -6:] = 0
    fixed[0] = 1
    A = fem.system_matrix(g, rho, fixed)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=nl, precision=mgar.MGAR_MIXED)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        s.build_hierarchy()
        b = rng.standard_normal(g.n_nodes) * (fixed == 0)
        ref = mg.vcycle(mg.build_hierarchy(A, fixed, (nx, ny, nz), nl), b, np.zeros(g.n_nodes))
        x = torch.zeros(g.n_nodes, dtype=torch.float64, device=DEV)
        s.vcycle(torch.tensor(b, device=DEV), x)
        # ~30 FP32 roundings per row and pass, times the coarsest level's conditioning (1e3 at most here)
        np.testing.assert_allclose(x.cpu().numpy(), ref, rtol=0, atol=1e-4 * np.abs(ref).max())
