"""The post-processing's level where the target volume is a whole number of lattice points, so that the count can meet it
exactly and the floating-point sum of the densities decides: the volume stays at or below the fraction, and the next lower
level's exceeds it (the level is the smallest that does not)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import design, fem, postprocess as pp  # noqa: E402
from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def mean_as_summed(values):
    """The mean of up to 256 densities in the kernel's order: a tree per warp, the warps in turn."""
    v = np.zeros(256)
    v[: values.size] = values
    v = v.reshape(8, 32)
    for o in (16, 8, 4, 2, 1):
        v = v[:, :o] + v[:, o: 2 * o]
    total = 0.0
    for w in v[:, 0]:
        total += w
    return total / values.size


@pytest.mark.parametrize("dims,vf", [((16, 16, 0), 0.2), ((16, 16, 0), 0.4), ((10, 10, 0), 0.4), ((10, 10, 0), 0.3),
                                     ((8, 8, 0), 0.35), ((4, 4, 4), 0.2), ((6, 6, 6), 0.3), ((5, 4, 3), 0.6)])
def test_target_of_whole_points(dims, vf):
    nx, ny, nz = dims
    g = fem.Grid(nx, ny, nz)
    r = 1.5
    H, Hs = design.filter_matrix(g, r)
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    points = 5 ** g.dim
    assert abs(vf * points * g.n_elems - round(vf * points * g.n_elems)) < 1e-9
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, rmin=r)
    out = torch.empty(g.n_elems, dtype=torch.float64, device=DEV)
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as sv:
        for seed in range(60):
            rng = np.random.default_rng(1000 + seed)
            rho = rng.uniform(0.05, 1.0, g.n_elems)
            t = rng.uniform(0.0, 1.0, g.n_nodes) * (fixed == 0)
            level, vol = sv.postprocess(torch.tensor(rho, device=DEV), torch.tensor(t, device=DEV), vf, out)
            rho_g = out.cpu().numpy()
            assert vol == mean_as_summed(rho_g), seed
            assert vol <= vf, (seed, vol)
            ns = pp.nodal_projection(g, pp.element_signal(g, design.filter_forward(H, Hs, rho), t), r)
            below = pp.densities(g, ns, level * (1 - 1e-9))
            assert mean_as_summed(below) > vf, (seed, level)
