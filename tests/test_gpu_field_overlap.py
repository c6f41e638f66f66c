"""Field arrays that lie in the caller's population store, or over one another, give what separate arrays
give, the later output counting where two share memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import BatchSolver, Solver  # noqa: E402
from paper_1905_10182_gb300 import _native as nat  # noqa: E402

SHAPE = (70, 33, 24)


def _fields():
    rng = np.random.default_rng(8)
    nx, ny, nz = SHAPE
    return [torch.from_numpy(f.astype(np.float32)).cuda()
            for f in (1 + 0.02 * rng.random((nz, ny, nx)), *(0.03 * rng.standard_normal((3, nz, ny, nx))))]


@pytest.mark.parametrize("storage,planes", [("fp32", (0, 1, 13, 26)), ("fp32", (2, 1, 4, 3)), ("fp16", (0, 1, 7, 12))])
def test_fields_in_the_store(storage, planes):
    n, f = int(np.prod(SHAPE)), _fields()
    store = torch.zeros(27 * n * (4 if storage == "fp32" else 2), dtype=torch.uint8, device="cuda")
    s, ref = Solver(*SHAPE, nu=0.04, storage=storage, store=store), Solver(*SHAPE, nu=0.04, storage=storage)
    held = [store.view(torch.float32)[p * n:(p + 1) * n].view(f[0].shape) for p in planes]
    for h, a in zip(held, f):
        h.copy_(a)
    s.set_state(*held)
    ref.set_state(*f)
    s.step(3)
    ref.step(3)
    want = np.stack(ref.macroscopic())
    assert np.array_equal(s.get_populations(), ref.get_populations())
    s.macroscopic(*held)  # overwrites the populations
    assert np.array_equal(torch.stack(held).cpu().numpy(), want)


@pytest.mark.parametrize("batch", [False, True])
def test_outputs_over_one_another(batch):
    n, f = int(np.prod(SHAPE)), _fields()
    if batch:
        s = BatchSolver([dict(nx=SHAPE[0], ny=SHAPE[1], nz=SHAPE[2], nu=0.04)])
        s.set_state(0, *f)
        want = np.stack(s.macroscopic(0)).reshape(4, n)
    else:
        s = Solver(*SHAPE, nu=0.04)
        s.set_state(*f)
        want = np.stack(s.macroscopic()).reshape(4, n)
    for at in ((0, 0, 1, 2), (0, n // 2, 3 * n, 4 * n), (2 * n, n, n + 1, 0), (0, n - 1, 2 * n - 1, 3 * n)):
        at = [a if a > 3 else a * n for a in at]
        buf, ref = torch.zeros(5 * n, device="cuda"), np.zeros(5 * n, dtype=np.float32)
        for a, w in zip(at, want):
            ref[a:a + n] = w
        ptrs = [buf.data_ptr() + 4 * a for a in at]
        L = nat.lib()
        assert (L.lbm_batch_macroscopic(s._h, 0, *ptrs) if batch else L.lbm_macroscopic(s._h, *ptrs)) == 0
        assert np.array_equal(buf.cpu().numpy(), ref)
