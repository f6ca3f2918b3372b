"""The coarsest factor and inverse on both sides of each change of kernel: band widths 31 and 32 (one and two unknowns per
lane), 63 and 64 (LDL^T and Cholesky form in shared memory), and a band too large for shared memory; FP64, and double-float
or FP64 (MGAR_FP64_COARSE=1) under the FP32 V-cycle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import fem, multigrid as mg  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

# elements of the finest grid; the coarsest (nl = 2) has nx / 2 + 1 nodes per row and that band width plus one
WIDTHS = {31: (58, 10), 32: (60, 10), 62: (120, 6), 63: (122, 6), 64: (124, 6), 65: (126, 6), 90: (176, 44)}


@pytest.mark.parametrize("width", sorted(WIDTHS))
@pytest.mark.parametrize("precision,fp64_coarse,tol", [(mgar.MGAR_FP64, False, 1e-10), (mgar.MGAR_MIXED, False, 5e-4),
                                                       (mgar.MGAR_MIXED, True, 5e-4)])
def test_vcycle(width, precision, fp64_coarse, tol, monkeypatch):
    if fp64_coarse:
        monkeypatch.setenv("MGAR_FP64_COARSE", "1")
    nx, ny = WIDTHS[width]
    assert nx // 2 + 2 == width
    g = fem.Grid(nx, ny, 0)
    rng = np.random.default_rng(23)
    rho = rng.uniform(0.1, 1.0, g.n_elems)
    fixed = workloads.heat_sink_mask(nx, ny, 0)
    levels = mg.build_hierarchy(fem.system_matrix(g, rho, fixed), fixed, (nx, ny), 2)
    b = rng.standard_normal(g.n_nodes) * (fixed == 0)
    ref = mg.vcycle(levels, b, np.zeros(g.n_nodes))
    p = mgar.default_params(nx=nx, ny=ny, nz=0, nl=2, precision=precision)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        s.build_hierarchy()
        x = torch.zeros(g.n_nodes, dtype=torch.float64, device=DEV)
        s.vcycle(torch.tensor(b, device=DEV), x)
    np.testing.assert_allclose(x.cpu().numpy(), ref, rtol=0, atol=tol * np.abs(ref).max())
