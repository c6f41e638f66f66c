"""z slabs in FP32 with an even nx take the kernel with two nodes per thread: slabs exchanging halos through
device buffers reproduce the single-domain run to the bit, small ones and ones large enough (more than half
of L2 each) for their odd steps to walk the grid backwards."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import Solver, inputs  # noqa: E402
from paper_1905_10182_gb300.slabs import LocalRing, SolverSlab  # noqa: E402


@pytest.mark.parametrize("heights,nx,ny,force", [
    ((12,), 20, 10, "uniform"), ((5, 7), 66, 10, "uniform"), ((3, 3, 4, 2), 2, 7, "uniform"), ((2, 3), 128, 9, "kolmogorov"),
    ((88, 90), 128, 64, "uniform"), ((180, 170), 60, 66, "kolmogorov")])
def test_slabs_match_single_domain(heights, nx, ny, force):
    nz = sum(heights)
    if nz > 100:
        half = torch.cuda.get_device_properties(0).L2_cache_size / 2
        assert all(4 * 27 * nx * ny * (h + 2) > half for h in heights)
    args = ("uniform", (1e-4, 0.0, -5e-5)) if force == "uniform" else ("kolmogorov", (1e-4,))
    g = inputs.random_deviations(nx, ny, nz, seed=52)
    ref = Solver(nx, ny, nz, nu=0.04)
    ref.set_force(*args)
    ref.set_populations(g)
    ref.step(8)
    slabs, z = [], 0
    for h in heights:
        s = Solver(nx, ny, h, nu=0.04, slab_z=True)
        s.set_force(*args)
        s.set_populations(g[:, z:z + h])
        slabs.append(s)
        z += h
    LocalRing([SolverSlab(s) for s in slabs]).step(8)
    got = np.concatenate([s.get_populations() for s in slabs], axis=1)
    assert np.array_equal(got, ref.get_populations())
