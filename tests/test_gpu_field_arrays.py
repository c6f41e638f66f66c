"""Fields handed over in device memory (read and written where they lie) and in host memory (through a
copy) give the same bits, mixed and with outputs left out, for a single domain and for a batch."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1905_10182_gb300 import BatchSolver, Solver  # noqa: E402
from paper_1905_10182_gb300 import _native as nat  # noqa: E402

SHAPES = [(13, 9, 7), (34, 5, 3)]


def _fields(nx, ny, nz):
    rng = np.random.default_rng(nx)
    u = 0.03 * rng.standard_normal((3, nz, ny, nx))
    return [f.astype(np.float32) for f in (1 + 0.02 * rng.random((nz, ny, nx)), *u)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("walls", [False, True])
def test_single_domain(shape, walls):
    host = _fields(*shape)
    dev = [torch.from_numpy(f).cuda() for f in host]
    got = []
    for src in (host, dev, [host[0], dev[1], host[2], dev[3]]):
        s = Solver(*shape, nu=0.04, walls_y=walls)
        s.set_state(*src)
        s.step(3)
        got.append(np.stack(s.macroscopic()))
        out = [torch.empty_like(d) for d in dev]
        s.macroscopic(*out)
        assert np.array_equal(np.stack([o.cpu().numpy() for o in out]), got[-1])
        part = torch.empty_like(dev[0])
        s.macroscopic(None, None, part, np.empty_like(host[0]))
        assert np.array_equal(part.cpu().numpy(), got[-1][2])
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])


def test_batch():
    L = nat.lib()
    got = []
    for dev in (False, True):
        b = BatchSolver([dict(nx=s[0], ny=s[1], nz=s[2], nu=0.04, walls_y=True) for s in SHAPES])
        for k, s in enumerate(SHAPES):
            f = _fields(*s)
            b.set_state(k, *([torch.from_numpy(a).cuda() for a in f] if dev else f))
        b.step(5)
        fields = []
        for k, s in enumerate(SHAPES):
            host = np.stack(b.macroscopic(k))
            out = torch.zeros((4,) + host.shape[1:], device="cuda")
            assert L.lbm_batch_macroscopic(b._h, k, out[0].data_ptr(), None, out[2].data_ptr(), ctypes.c_void_p(out[3].data_ptr())) == 0
            assert np.array_equal(out.cpu().numpy()[[0, 2, 3]], host[[0, 2, 3]]) and not out[1].any()
            fields.append(host)
        got.append(fields)
    assert all(np.array_equal(a, c) for a, c in zip(*got))


def test_unaligned_device_arrays():
    """Device pointers off the 4-byte alignment are copied."""
    L, (nx, ny, nz) = nat.lib(), SHAPES[0]
    N, host = nx * ny * nz, _fields(*SHAPES[0])
    raw = torch.zeros(4, 4 * N + 4, dtype=torch.uint8, device="cuda")
    raw[:, 2:-2] = torch.stack([torch.from_numpy(f.reshape(-1).view(np.uint8)) for f in host]).cuda()
    s, ref = Solver(nx, ny, nz, nu=0.04), Solver(nx, ny, nz, nu=0.04)
    b = BatchSolver([dict(nx=nx, ny=ny, nz=nz, nu=0.04)])
    ref.set_state(*host)
    for put, get, h in ((L.lbm_set_state, L.lbm_macroscopic, (s._h,)), (L.lbm_batch_set_state, L.lbm_batch_macroscopic, (b._h, 0))):
        assert put(*h, *(raw[k].data_ptr() + 2 for k in range(4))) == 0
        out = torch.zeros_like(raw)
        assert get(*h, *(out[k].data_ptr() + 2 for k in range(4))) == 0
        out = out.cpu().numpy()
        assert np.array_equal(out[:, 2:-2].copy().view(np.float32).reshape(4, nz, ny, nx), np.stack(ref.macroscopic()))
        assert not out[:, :2].any() and not out[:, -2:].any()
