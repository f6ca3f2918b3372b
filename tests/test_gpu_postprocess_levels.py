"""The level search of the post-processing against the oracle's bisection: sizes at the edges of its passes, volume
fractions whose target is a whole number of lattice points (the count can meet it exactly), and fields whose values
coincide."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import design, fem, postprocess as pp  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def fields(nx, ny, nz, seed, spread):
    rng = np.random.default_rng(seed)
    ne, n = workloads.num_elements(nx, ny, nz), workloads.num_nodes(nx, ny, nz)
    rho = rng.uniform(0.05, 1.0, ne)
    t = rng.uniform(0.0, 1.0, n) * 10.0 ** rng.uniform(-spread, 0.0, n)
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    return rho, t * (fixed == 0), fixed


@pytest.mark.parametrize("dims,r,vf,spread", [
    ((2, 2, 0), 1.5, 0.4, 0.0), ((33, 17, 0), 1.5, 0.3, 0.0), ((64, 64, 0), 2.3, 0.5, 4.0),
    ((150, 131, 0), 3.0, 0.2, 2.0), ((2, 2, 2), 1.5, 0.5, 0.0), ((9, 8, 7), 1.5, 0.3, 0.0),
    ((16, 16, 16), 2.3, 0.4, 3.0), ((31, 20, 25), 1.5, 0.25, 1.0)])
def test_level_matches_bisection(dims, r, vf, spread):
    nx, ny, nz = dims
    rho, t, fixed = fields(nx, ny, nz, 7, spread)
    g = fem.Grid(nx, ny, nz)
    H, Hs = design.filter_matrix(g, r)
    rho_phys = design.filter_forward(H, Hs, rho)
    rho_o, ns_o, level_o = pp.postprocess(g, rho_phys, t, vf, r)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, rmin=r)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as sv:
        out = torch.empty(rho.size, dtype=torch.float64, device=DEV)
        level, vol = sv.postprocess(torch.tensor(rho, device=DEV), torch.tensor(t, device=DEV), vf, out)
        rho_g = out.cpu().numpy()
    assert abs(level - level_o) <= 1e-9 * abs(level_o)
    assert vol <= vf and abs(vol - rho_g.mean()) < 1e-12
    vals = ns_o[g.element_nodes()] @ pp.lattice_shape_values(g.dim).T
    near = np.any(np.abs(vals - level_o) <= 1e-9 * abs(level_o), axis=1)
    assert near.sum() <= 2 ** (g.dim + 1)
    np.testing.assert_array_equal(rho_g[~near], rho_o[~near])


@pytest.mark.parametrize("dims", [(24, 16, 0), (8, 6, 5)])
def test_level_of_coinciding_values(dims):
    # constant temperatures: every nodal value is 0, the level 0, no element above it
    nx, ny, nz = dims
    rho, t, fixed = fields(nx, ny, nz, 3, 0.0)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as sv:
        out = torch.empty(rho.size, dtype=torch.float64, device=DEV)
        level, vol = sv.postprocess(torch.tensor(rho, device=DEV), torch.ones(t.size, dtype=torch.float64, device=DEV),
                                    0.4, out)
    assert level == 0.0 and vol == 0.0 and float(out.abs().max()) == 0.0
