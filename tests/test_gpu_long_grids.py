"""Grids so long that a launch with the tiles' rows (or the restriction's planes) along its second dimension alone would pass
the limit of 65535 there: the tiled passes against the general ones (MGAR_UNTILED=1)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2210_00947_gb300 import mgar  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def problem(nx, ny, nz):
    n = (nx + 1) * (ny + 1) * (nz + 1 if nz else 1)
    fixed = np.zeros(n, dtype=np.uint8)
    fixed[:: 4099] = 1
    q = np.full(n, 0.01)
    rng = np.random.default_rng(3)
    return fixed, q, rng.uniform(0.1, 1.0, nx * ny * max(nz, 1)), rng.standard_normal(n) * (fixed == 0)


def handle(nx, ny, nz, fixed, q, **kw):
    nl, rows = 2, max(ny, nz) // 2
    while (rows + 1) * 4 > 8192:
        nl, rows = nl + 1, (rows + 1) // 2
    return mgar.Solver(mgar.default_params(nx=nx, ny=ny, nz=nz, nl=nl, **kw), fixed, q)


@pytest.mark.parametrize("dims,precision,tol", [((1, 800001, 0), mgar.MGAR_FP64, 1e-10),
                                                ((1, 800001, 0), mgar.MGAR_MIXED, 5e-4),
                                                ((1, 530001, 1), mgar.MGAR_FP64, 1e-10),
                                                ((1, 1, 270001), mgar.MGAR_MIXED, 5e-4)])
def test_vcycle_and_product(dims, precision, tol, monkeypatch):
    fixed, q, rho, b = problem(*dims)

    def go():
        with handle(*dims, fixed, q, precision=precision) as s:
            s.set_density(torch.tensor(rho, device=DEV), physical=True)
            s.build_hierarchy()
            bd = torch.tensor(b, device=DEV)
            x, y = torch.zeros_like(bd), torch.empty_like(bd)
            s.vcycle(bd, x)
            s.apply_K(bd, y)
            return x.cpu().numpy(), y.cpu().numpy()

    x, y = go()
    monkeypatch.setenv("MGAR_UNTILED", "1")
    xr, yr = go()
    np.testing.assert_allclose(x, xr, rtol=0, atol=tol * np.abs(xr).max())
    np.testing.assert_allclose(y, yr, rtol=0, atol=1e-13 * np.abs(yr).max())


@pytest.mark.parametrize("dims,precision", [((1, 800001, 0), mgar.MGAR_FP64), ((1, 800001, 0), mgar.MGAR_MIXED),
                                            ((1, 1450001, 0), mgar.MGAR_FP64), ((1, 1450001, 0), mgar.MGAR_MIXED),
                                            ((1, 530001, 1), mgar.MGAR_FP64), ((1, 1, 270001), mgar.MGAR_MIXED)])
def test_cg_iterations(dims, precision):
    # the residual that a dozen iterations carry along is that of their solution, converged or not
    fixed, q, rho, _ = problem(*dims)
    with handle(*dims, fixed, q, precision=precision, eps2=1e-13, cg_max=12) as s:
        s.set_density(torch.tensor(rho, device=DEV), physical=True)
        T = torch.zeros(s.n_nodes, dtype=torch.float64, device=DEV)
        it, rel, _ = s.solve_mgcg(T)
        y = torch.empty_like(T)
        s.apply_K(T, y)
    qf = q * (fixed == 0)
    true = np.linalg.norm(y.cpu().numpy() - qf) / np.linalg.norm(qf)
    assert it == 12
    assert abs(rel - true) <= 1e-8 * max(true, 1.0)


def test_filter_of_a_larger_radius():
    nx, ny, nz = 2, 530001, 2
    fixed, q, rho, _ = problem(nx, ny, nz)
    out = {}
    for precision in (mgar.MGAR_MIXED, mgar.MGAR_FP64):
        with handle(nx, ny, nz, fixed, q, precision=precision, rmin=2.5) as s:
            s.set_density(torch.tensor(rho, device=DEV))
            x = torch.tensor(np.random.default_rng(4).standard_normal(s.n_nodes), device=DEV)
            y = torch.empty_like(x)
            s.apply_K(x, y)
            out[precision] = y.cpu().numpy()
    ref = out[mgar.MGAR_FP64]
    np.testing.assert_allclose(out[mgar.MGAR_MIXED], ref, rtol=0, atol=1e-12 * np.abs(ref).max())
