"""Kernels that start while their predecessor runs read its results only after the wait: every solve, whole cycle and
batched cycle gives the same bits with ordinary launches (MGAR_NO_PDL=1), whether the launches are captured or not."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2210_00947_gb300 import batch, mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

CASES = [((40, 32, 0), "fp64"), ((361, 122, 0), "fp64"), ((40, 32, 0), "mixed"), ((250, 251, 0), "mixed"),
         ((24, 17, 13), "fp64"), ((24, 17, 13), "mixed"), ((75, 53, 41), "mixed"), ((48, 48, 48), "fp64")]


def results(dims, precision):
    nx, ny, nz = dims
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    nl = workloads.levels_for_direct_coarsest(nx, ny, nz, max_nodes=300)
    prec = mgar.MGAR_MIXED if precision == "mixed" else mgar.MGAR_FP64
    out = []
    for guess in (mgar.MGAR_GUESS_ZERO, mgar.MGAR_GUESS_PREVIOUS):
        p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=nl, precision=prec, volfrac=0.3, m=2, basis_guess=guess,
                                eps2=1e-9, n_on=1, eps1=0.9)
        rng = np.random.default_rng(2)
        with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as s:
            rho = torch.tensor(rng.uniform(0.1, 0.5, s.n_elems), device=DEV)
            T = torch.zeros(s.n_nodes, dtype=torch.float64, device=DEV)
            for k in range(1, 5):
                info = s.step(rho, T, k)
                out += [T.cpu().numpy().copy(), rho.cpu().numpy().copy(),
                        np.array([info["compliance"], info["lam"]])]
            x = torch.zeros_like(T)
            s.vcycle(T, x)
            out.append(x.cpu().numpy())
    return out


@pytest.mark.parametrize("dims,precision", CASES)
@pytest.mark.parametrize("graphs", [True, False])
def test_same_bits(dims, precision, graphs, monkeypatch):
    if not graphs:
        monkeypatch.setenv("MGAR_NO_GRAPHS", "1")
    a = results(dims, precision)
    monkeypatch.setenv("MGAR_NO_PDL", "1")
    b = results(dims, precision)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)


def test_same_bits_batched(monkeypatch):
    designs = [batch.Design(**d) for d in workloads.batched_designs(7, 5)]

    def go():
        solvers = [mgar.Solver(d.params(30, mgar.MGAR_MIXED, n_on=1000, eps2=1e-10), d.fixed(), d.q()) for d in designs]
        rhos = [torch.full((d.nx * d.ny,), 0.4, dtype=torch.float64, device=DEV) for d in designs]
        Ts = [torch.zeros((d.nx + 1) * (d.ny + 1), dtype=torch.float64, device=DEV) for d in designs]
        b = mgar.BatchSolver(solvers)
        for _ in range(3):
            b.cycle(rhos, Ts, [d.volfrac for d in designs], 0.2)
        out = [t.cpu().numpy() for t in rhos + Ts]
        b.close()
        for s in solvers:
            s.close()
        return out

    a = go()
    monkeypatch.setenv("MGAR_NO_PDL", "1")
    for x, y in zip(a, go()):
        np.testing.assert_array_equal(x, y)
