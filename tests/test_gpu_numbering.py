"""The two node numberings of the kernels with one thread per node: a domain of nx = 60 (nodes numbered
through) and the same state twice side by side, nx = 120 (a row of blocks per grid row), hold the same
flow; every node runs the same arithmetic, so the fields agree to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import Solver, inputs  # noqa: E402

NX, NY, NZ = 60, 7, 5


def _run(kind, reps):
    rng = np.random.default_rng(3)

    def twice(a):
        return np.concatenate([a] * reps, axis=-1)
    rho = twice((1 + 0.02 * rng.random((NZ, NY, NX))).astype(np.float32))
    u = [twice((0.02 * rng.standard_normal((NZ, NY, NX))).astype(np.float32)) for _ in range(3)]
    kw = dict(walls_y=True)
    if kind.startswith("mask"):
        kw.update(mask=twice(inputs.random_mask(NX, NY, NZ, seed=5, fraction=0.15)), storage=kind[4:])
    s = Solver(NX * reps, NY, NZ, nu=0.05, **kw)
    if kind == "cg":
        s.set_colour_gradient(twice(rng.random((NZ, NY, NX))) + 0.5, twice(rng.random((NZ, NY, NX))) + 0.5, 3.0, 1.0, 0.05, 0.02,
                              g=(0.0, -1e-5, 0.0))
    else:
        s.set_state(rho, *u)
        s.set_force("uniform", (1e-4, 0.0, 2e-5))
    if kind == "mhd":
        s.set_magnetic(0.02, [twice((0.02 * rng.standard_normal((NZ, NY, NX))).astype(np.float32)) for _ in range(3)])
    s.step(5)
    return np.stack(s.macroscopic())


@pytest.mark.parametrize("kind", ["maskfp32", "maskfp16", "mhd", "cg"])
def test_numberings_agree(kind):
    one, two = _run(kind, 1), _run(kind, 2)
    assert np.abs(one[1:]).max() > 1e-6  # a flow to compare
    assert np.array_equal(np.concatenate([one, one], axis=-1), two)
