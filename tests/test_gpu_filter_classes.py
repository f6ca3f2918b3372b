"""1/Hs and dv, formed per class of distances to the faces, on grids around the size where the classes begin to
repeat (4 ceil(r) + 1 elements per axis)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import design, fem  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("precision", [mgar.MGAR_FP64, mgar.MGAR_MIXED])
@pytest.mark.parametrize("dims,r", [
    ((9, 8, 0), 1.5), ((10, 9, 0), 2.0), ((12, 40, 0), 3.0), ((13, 14, 0), 3.0), ((60, 33, 0), 6.4),
    ((9, 10, 8), 1.5), ((13, 6, 20), 2.5), ((30, 13, 14), 3.0)])
def test_filter_sums_and_volume_gradient(dims, r, precision):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    H, Hs = design.filter_matrix(g, r)
    ne = g.n_elems
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, rmin=r, precision=precision)
    x = np.random.default_rng(5).uniform(0.1, 1.0, ne)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as sv:
        out = torch.empty(ne, dtype=torch.float64, device=DEV)
        sv.filter(torch.tensor(x, device=DEV), out)
        fwd = out.cpu().numpy()
        sv.filter(torch.tensor(x, device=DEV), out, transpose=True)
        adj = out.cpu().numpy()
        dv = torch.empty(ne, dtype=torch.float64, device=DEV)
        T = torch.zeros(sv.n_nodes, dtype=torch.float64, device=DEV)
        sv.set_density(torch.tensor(x, device=DEV))
        sv.sensitivity(T, None, dv)
        dv = dv.cpu().numpy()
    # sums of at most 500 positive terms in FP64
    np.testing.assert_allclose(fwd, (H @ x) / Hs, rtol=1e-13)
    np.testing.assert_allclose(adj, H.T @ (x / Hs), rtol=1e-13)
    np.testing.assert_allclose(dv, H.T @ (np.full(ne, 1.0 / ne) / Hs), rtol=1e-13)
