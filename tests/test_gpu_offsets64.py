"""Domains with links whose element offsets need 64 bits (27 N >= 2^32) against the 32-bit form.  A small box
with walls and a mask (32-bit offsets, walked forwards) and the same box repeated along z until it is beyond
the limit (64-bit offsets) hold the same flow; every node runs the same arithmetic, so
the fields of every repetition agree to the bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import Solver, inputs  # noqa: E402

NY, NZ = 120, 40


def _run(nx, storage, walls, model, reps, steps):
    rng = np.random.default_rng(12)

    def rep(a):
        return torch.from_numpy(a).cuda().repeat(reps, 1, 1)
    shape = (NZ, NY, nx)
    mask = rep(inputs.random_mask(nx, NY, NZ, seed=7, fraction=0.15).astype(np.uint8))
    s = Solver(nx, NY, NZ * reps, nu=0.05, storage=storage, walls_y=walls, mask=mask)
    s.set_model(model)
    s.set_force("uniform", (1e-4, 0.0, 2e-5))
    s.set_state(rep((1 + 0.02 * rng.random(shape)).astype(np.float32)),
                *(rep((0.02 * rng.standard_normal(shape)).astype(np.float32)) for _ in range(3)))
    s.step(steps)
    out = torch.empty((4, NZ * reps, NY, nx), device="cuda")
    s.macroscopic(*out)
    s.close()
    return out


# nx = 93, 61: nodes numbered through; 128, 250: a row of blocks per grid row
@pytest.mark.parametrize("nx,storage,walls,model,steps", [
    (93, "fp32", True, "M1", 4), (128, "fp32", False, "M1", 5), (93, "fp16", False, "M1", 5), (128, "fp16", True, "M1", 4),
    (250, "bf16", True, "M1", 5), (61, "bf16", False, "M5", 4), (128, "fp32", True, "M4", 5)])
def test_64_bit_offsets(nx, storage, walls, model, steps):
    box = nx * NY * NZ
    reps = 2 ** 32 // (27 * box) + 1
    assert 27 * box < 2 ** 32 <= 27 * box * reps
    one = _run(nx, storage, walls, model, 1, steps)
    many = _run(nx, storage, walls, model, reps, steps).view(4, reps, NZ, NY, nx)
    assert float(one[1:].abs().max()) > 1e-6  # a flow to compare
    assert all(torch.equal(many[:, r], one) for r in range(reps))
    del many
    torch.cuda.empty_cache()
