"""The df64 filters where a thread takes one or two elements (the line lies near 0.62 M elements on 152 SMs), with an
incomplete last block, and the OC update whose ambiguous elements are few, more than the bisection keeps in shared
memory, or more than it lists at all (the plain bisection then), against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import design, fem  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def solver(dims, precision):
    nx, ny, nz = dims
    fixed = np.zeros((nx + 1) * (ny + 1) * ((nz + 1) if nz else 1), dtype=np.uint8)
    fixed[0] = 1
    nl = 2 + int(np.log2(max(dims) / 8))  # a coarsest level of some 16 elements per axis
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=max(nl, 2), precision=precision)
    return mgar.Solver(p, fixed, workloads.nodal_load(fixed))


@pytest.mark.parametrize("dims", [(787, 789, 0), (797, 789, 0), (91, 87, 83), (7, 5, 3)])
def test_filters(dims):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz) if nz else fem.Grid(nx, ny)
    rng = np.random.default_rng(47)
    rho = rng.uniform(0.05, 1.0, g.n_elems)
    t = rng.uniform(0.0, 1.0, g.n_nodes)
    H, Hs = design.filter_matrix(g, 1.5)
    rho_phys = design.filter_forward(H, Hs, rho)
    dc_ref, _ = design.sensitivities(g, H, Hs, rho_phys, t)
    with solver(dims, mgar.MGAR_MIXED) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=False)
        dc = torch.empty(g.n_elems, dtype=torch.float64, device=DEV)
        s.sensitivity(torch.tensor(t, device=DEV), dc, None)
        # pairs hold 2^-46 relative per operation; 19 terms and two filters
        np.testing.assert_allclose(dc.cpu().numpy(), dc_ref, rtol=1e-11, atol=0)


@pytest.mark.parametrize("equal", [3, 300, 5000])
def test_oc_at_a_breakpoint(equal):
    # equal elements that reach their upper limit at the very multiplier that
    # meets the volume: all of them stay ambiguous to the end
    dims = (120, 90, 0)
    g = fem.Grid(120, 90)
    rng = np.random.default_rng(53)
    rho = rng.uniform(0.1, 0.7, g.n_elems)
    dc = -(10.0 ** rng.uniform(-2, 2, g.n_elems))
    at = 2000 + np.arange(equal)  # away from the faces: dv is the same there
    at = at[(at % 120 > 2) & (at % 120 < 117)]
    rho[at], dc[at] = 0.4, -1.0
    H, Hs = design.filter_matrix(g, 1.5)
    dv = design.filter_transpose(H, Hs, np.full(g.n_elems, 1.0 / g.n_elems))
    s_e = rho * np.sqrt(-dc / dv)
    mu = 0.6 / s_e[at[0]]
    volfrac = float(dv @ np.clip(s_e * mu, np.maximum(0.0, rho - 0.2), np.minimum(1.0, rho + 0.2)))
    ref, lam_ref = design.oc_update(rho, dc, dv, volfrac, 0.2)
    with solver(dims, mgar.MGAR_FP64) as s:
        r = torch.tensor(rho, device=DEV)
        lam, _ = s.oc_update(r, torch.tensor(dc, device=DEV), volfrac, 0.2)
        assert abs(lam - lam_ref) / lam_ref < 1e-12
        np.testing.assert_allclose(r.cpu().numpy(), ref, rtol=1e-11, atol=1e-12)
