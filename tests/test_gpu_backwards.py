"""Odd steps of a store larger than half of L2 walk the grid backwards.  A small box (walked forwards) and
the same state repeated along z until the store is beyond half of L2, and beyond L2 where the prefetch joins
in, hold the same flow; every node runs the same arithmetic, so the fields agree to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import Solver, inputs  # noqa: E402

NY, NZ = 11, 5


def _run(nx, kind, storage, reps):
    rng = np.random.default_rng(4)

    def rep(a):
        return np.tile(a.astype(np.float32), (reps, 1, 1))
    shape = (NZ, NY, nx)
    rho = rep(1 + 0.02 * rng.random(shape))
    u = [rep(0.02 * rng.standard_normal(shape)) for _ in range(3)]
    kw = dict(mask=np.tile(inputs.random_mask(nx, NY, NZ, seed=5, fraction=0.15), (reps, 1, 1)), walls_y=True) if kind == "mask" else {}
    s = Solver(nx, NY, NZ * reps, nu=0.05, storage=storage, **kw)
    s.set_state(rho, *u)
    s.set_force("uniform", (1e-4, 0.0, 2e-5))
    if kind == "mhd":
        s.set_magnetic(0.02, [rep(0.02 * rng.standard_normal(shape)) for _ in range(3)])
    s.step(5)
    return np.stack(s.macroscopic())


@pytest.mark.parametrize("beyond", [0.5, 1.0], ids=["half_l2", "l2"])
@pytest.mark.parametrize("nx,kind,storage", [(60, "plain", "fp32"), (61, "plain", "fp32"), (128, "plain", "fp32"), (60, "plain", "fp16"),
                                             (61, "plain", "bf16"), (93, "mask", "fp32"), (128, "mask", "fp16"), (61, "mhd", "fp32")])
def test_backwards_equals_forwards(nx, kind, storage, beyond):
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    box = 27 * nx * NY * NZ * (4 if storage == "fp32" else 2)
    reps = int(beyond * l2 / box) + 2
    one, many = _run(nx, kind, storage, 1), _run(nx, kind, storage, reps)
    assert np.abs(one[1:]).max() > 1e-6  # a flow to compare
    assert np.array_equal(np.tile(one, (1, reps, 1, 1)), many)
