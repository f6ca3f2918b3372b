"""The post-processing at nodal values of any size: scaling the temperatures by a power of two scales the energies without
rounding, so it scales the level and changes no density, also where the values leave FP32's normal range."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2210_00947_gb300 import mgar, workloads  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dims", [(96, 80, 0), (20, 16, 18)])
@pytest.mark.parametrize("power", [30, 64, 65, 66, 67, 70, 73, 80])
def test_scaled_temperatures(dims, power):
    nx, ny, nz = dims
    fixed = workloads.heat_sink_mask(nx, ny, nz)
    ne, n = workloads.num_elements(nx, ny, nz), workloads.num_nodes(nx, ny, nz)
    p = mgar.default_params(nx=nx, ny=ny, nz=nz, nl=2, rmin=1.5)
    a, b = (torch.empty(ne, dtype=torch.float64, device=DEV) for _ in range(2))
    with mgar.Solver(p, fixed, workloads.nodal_load(fixed)) as sv:
        for seed in range(20):
            rng = np.random.default_rng(seed)
            rho = torch.tensor(rng.uniform(0.05, 1.0, ne), device=DEV)
            t = torch.tensor(rng.uniform(0.0, 1.0, n) * (fixed == 0), device=DEV)
            level, vol = sv.postprocess(rho, t, 0.3, a)
            level_s, vol_s = sv.postprocess(rho, t * 2.0 ** -power, 0.3, b)
            # (the bracket starts at -1 whatever the values: its last steps leave an absolute 1e-60)
            assert abs(level_s * 4.0 ** power - level) <= 1e-9 * level
            assert vol_s == vol, seed
            np.testing.assert_array_equal(b.cpu().numpy(), a.cpu().numpy())
