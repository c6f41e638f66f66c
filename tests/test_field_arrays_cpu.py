"""Field arrays handed to the C ABI, on a host CUDA runtime (fake_runtime.py): what the calls do when a copy
fails, memory is short, an array is too short or arrays lie over one another."""
import ctypes

import numpy as np
import pytest

import fake_runtime
from paper_1905_10182_gb300 import _native as nat

SHAPES = [(13, 9, 7), (20, 11, 6)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_runtime.build(tmp_path_factory.mktemp("host"))


@pytest.fixture
def batch(lib):
    lib.fake_reset()
    arr = (nat.LbmDomain * len(SHAPES))()
    for a, s in zip(arr, SHAPES):
        a.nx, a.ny, a.nz, a.nu, a.walls_y = *s, 0.05, 1
    h = ctypes.c_void_p()
    assert lib.lbm_batch_create(arr, len(SHAPES), 1.0, None, ctypes.byref(h)) == nat.LBM_OK
    yield h
    lib.lbm_batch_destroy(h)


def host(n):
    return [np.zeros(n, dtype=np.float32) for _ in range(4)]


def ptrs(arrays):
    return [a.ctypes.data if isinstance(a, np.ndarray) else a for a in arrays]


@pytest.fixture
def domain(lib):
    lib.fake_reset()
    d = nat.LbmDesc()
    d.nx, d.ny, d.nz, d.nu, d.rho0 = *SHAPES[0], 0.05, 1.0
    h = ctypes.c_void_p()
    assert lib.lbm_create(ctypes.byref(d), ctypes.byref(h)) == nat.LBM_OK
    yield h
    lib.lbm_destroy(h)


@pytest.fixture
def alloc(lib):
    made = []

    def f(n):
        made.append(lib.fake_alloc(n))
        return made[-1]
    yield f
    for p in made:
        lib.cudaFree(p)


def call(lib, kind, which, handle, arrays):
    if kind == "batch":
        return getattr(lib, "lbm_batch_" + which)(handle, 0, *ptrs(arrays))
    return getattr(lib, "lbm_" + which)(handle, *ptrs(arrays))


@pytest.mark.parametrize("which", ["set_state", "macroscopic"])
@pytest.mark.parametrize("kind", ["batch", "domain"])
@pytest.mark.parametrize("fails,nth", [("cudaMemcpyAsync", 1), ("cudaMemcpyAsync", 2), ("cudaMemcpyAsync", 3), ("launch", 1)])
def test_nothing_runs_after_an_error(lib, request, kind, which, fails, nth, alloc):
    """The arrays are the caller's again when the call returns, with an error too: no copy and no kernel may
    still be reading or writing them.  The first array lies in device memory, the others need copies."""
    handle = request.getfixturevalue(kind)
    n = int(np.prod(SHAPES[0]))
    arrays = [alloc(4 * n)] + host(n)[1:]
    lib.fake_fail(fails.encode(), nth)
    assert call(lib, kind, which, handle, arrays) == nat.LBM_ERR_CUDA
    assert lib.fake_pending() == 0


def test_batch_scratch_where_memory_is_short(lib, batch):
    """A call on host arrays needs four planes of its own domain, not of the largest one."""
    small, large = (int(np.prod(s)) for s in SHAPES)
    free = 16 * small + 64
    assert free < 16 * large
    lib.fake_limit(lib.fake_used() + free)
    a, b = host(small), host(large)
    for _ in range(2):
        assert lib.lbm_batch_set_state(batch, 0, *ptrs(a)) == nat.LBM_OK
        assert lib.lbm_batch_macroscopic(batch, 0, *ptrs(a)) == nat.LBM_OK
    assert lib.lbm_batch_set_state(batch, 1, *ptrs(b)) == nat.LBM_ERR_OOM
    assert lib.lbm_batch_set_state(batch, 0, *ptrs(a)) == nat.LBM_OK
    lib.fake_limit(1 << 40)
    assert lib.lbm_batch_macroscopic(batch, 1, *ptrs(b)) == nat.LBM_OK
    made = lib.fake_calls(b"cudaMalloc")
    for k, f in ((0, a), (1, b)):  # then kept
        assert lib.lbm_batch_set_state(batch, k, *ptrs(f)) == nat.LBM_OK
    assert lib.fake_calls(b"cudaMalloc") == made


KERNEL = {"set_state": b"k_init_equilibrium", "macroscopic": b"k_macroscopic"}


def given(lib, which):
    """The arrays that the kernel got."""
    return [lib.fake_pointer(KERNEL[which], k) for k in range(4)]


@pytest.mark.parametrize("which", ["set_state", "macroscopic"])
@pytest.mark.parametrize("kind", ["batch", "domain"])
def test_device_arrays_that_end_early_are_refused(lib, request, kind, which, alloc):
    """A device array with fewer bytes than the domain needs is refused by the copy's range check; no kernel
    gets it.  One that fits to the byte is used where it lies."""
    handle = request.getfixturevalue(kind)
    n = int(np.prod(SHAPES[0]))
    fit = [alloc(4 * n) for _ in range(4)]
    assert call(lib, kind, which, handle, fit) == nat.LBM_OK and given(lib, which) == fit
    for k in range(4):
        for short, off in ((4 * n - 4, 0), (4 * n, 4)):
            arrays = fit[:k] + [alloc(short) + off] + fit[k + 1:]
            assert call(lib, kind, which, handle, arrays) == nat.LBM_ERR_CUDA
            assert arrays[k] not in given(lib, which)


@pytest.mark.parametrize("kind", ["batch", "domain"])
def test_outputs_over_one_another_are_copied(lib, request, kind, alloc):
    """Outputs that share memory are written one after the other, so that the later one counts."""
    handle = request.getfixturevalue(kind)
    n = int(np.prod(SHAPES[0]))
    a = alloc(40 * n)
    for rel, direct in (((0, 0, 2, 3), (0, 0, 1, 1)), ((0, 0.5, 2, 3), (0, 0, 1, 1)), ((3, 2, 1, 0), (1, 1, 1, 1)), ((0, 2, 1, 1.5), (1, 0, 0, 0))):
        arrays = [a + 4 * int(r * n) for r in rel]
        assert call(lib, kind, "macroscopic", handle, arrays) == nat.LBM_OK
        assert tuple(int(g == p) for g, p in zip(given(lib, "macroscopic"), arrays)) == direct


def test_arrays_in_the_callers_store_are_copied(lib, alloc):
    """A store of the caller's may hold the fields that are to fill it."""
    lib.fake_reset()
    d = nat.LbmDesc()
    d.nx, d.ny, d.nz, d.nu, d.rho0 = *SHAPES[0], 0.05, 1.0
    n = int(np.prod(SHAPES[0]))
    d.store = alloc(27 * 4 * n)
    h = ctypes.c_void_p()
    assert lib.lbm_create(ctypes.byref(d), ctypes.byref(h)) == nat.LBM_OK
    other = alloc(16 * n)
    for which in ("set_state", "macroscopic"):
        arrays = [d.store, d.store + 26 * 4 * n, other, other + 4 * n]
        assert call(lib, "domain", which, h, arrays) == nat.LBM_OK
        assert [g == p for g, p in zip(given(lib, which), arrays)] == [False, False, True, True]
    lib.lbm_destroy(h)
