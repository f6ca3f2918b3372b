"""The 3D filter by classes of equal weight (radii above 2, mixed path) against the oracle: every reach, grids smaller
than the filter, ragged tiles of 32 x 8, and several runs along z."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

from oracle import design, fem  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def filter_matrix(g, r):
    """The oracle's, or on a grid smaller than the filter (which the oracle's shifted slices do not cover) Eq. 7 pair by
    pair."""
    if min(g.nx, g.ny, g.nz) > r:
        return design.filter_matrix(g, r)
    e = np.arange(g.n_elems)
    c = np.stack([e % g.nx, (e // g.nx) % g.ny, e // (g.nx * g.ny)], axis=1)
    w = np.maximum(0.0, r - np.sqrt(((c[:, None] - c[None]) ** 2).sum(-1).astype(float)))
    H = sp.csr_matrix(w)
    return H, np.asarray(H.sum(axis=1)).reshape(-1)


@pytest.mark.parametrize("dims,r", [
    ((13, 11, 9), 2.001), ((33, 9, 40), 2.5), ((32, 8, 12), 3.0), ((13, 11, 9), 3.7), ((35, 17, 20), 4.2),
    ((20, 18, 16), 5.0), ((13, 11, 9), 6.27), ((40, 20, 33), 6.27), ((6, 5, 4), 7.5), ((20, 12, 16), 8.9)])
def test_filter_and_transpose(dims, r):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    rng = np.random.default_rng(21)
    rho = rng.uniform(0.05, 1.0, g.n_elems)
    t = rng.uniform(0.0, 1.0, g.n_nodes)
    x = rng.standard_normal(g.n_nodes)
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    H, Hs = filter_matrix(g, r)
    rho_phys = design.filter_forward(H, Hs, rho)
    dc_ref, _ = design.sensitivities(g, H, Hs, rho_phys, t)
    y_ref = fem.system_matrix(g, rho_phys, fixed) @ x
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, rmin=r, precision=mgar.MGAR_MIXED)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as s:
        s.set_density(torch.tensor(rho, device=DEV))
        y = torch.empty(g.n_nodes, dtype=torch.float64, device=DEV)
        s.apply_K(torch.tensor(x, device=DEV), y)
        dc = torch.empty(g.n_elems, dtype=torch.float64, device=DEV)
        s.sensitivity(torch.tensor(t, device=DEV), dc, None)
    # pairs: about 2^-46 per operation, all terms of a filter sum of one sign;
    # k_e carries three times rho's relative error and the row cancels at most
    # 27 terms; an element's energy is a sum of squares of differences of order 1
    np.testing.assert_allclose(y.cpu().numpy(), y_ref, rtol=0, atol=1e-12 * np.abs(y_ref).max())
    np.testing.assert_allclose(dc.cpu().numpy(), dc_ref, rtol=1e-11)
