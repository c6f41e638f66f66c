"""The neural operator on more than one device of a process, and after a failed first call, on a host CUDA
runtime (fake_runtime.py) that refuses a launch beyond 48 KB of dynamic shared memory until the kernel is
allowed it on that device."""
import ctypes

import pytest

import fake_runtime
from paper_1905_10182_gb300 import _native as nat

D, W, M, L, B, CH = 16, 32, 4, 2, 8, 4


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_runtime.build(tmp_path_factory.mktemp("host"))


def operator(lib):
    h = ctypes.c_void_p()
    assert lib.lbm_no_create(D, W, M, L, CH, CH, B, 1, None, ctypes.byref(h)) == nat.LBM_OK
    n = 4 * B * CH * D ** 3
    return h, lib.fake_alloc(n), lib.fake_alloc(n)


def passes(lib, h, a, o):
    return [lib.lbm_no_forward(h, B, a, o), lib.lbm_no_backward(h, o)]


def test_each_device_is_prepared(lib):
    lib.fake_reset()
    made = [None, None]
    for d in (0, 1):
        lib.fake_device(d)
        made[d] = operator(lib)
        assert passes(lib, *made[d]) == [nat.LBM_OK] * 2
        assert lib.fake_launches(b"k_map_act") == (d + 1) * (L - 1)
        # the copy-engine kernels cover the device's own multiprocessors (100 + d of them)
        assert lib.fake_blocks(b"k_map_act") == min(B * 8, 2 * (100 + d))
        assert lib.fake_blocks(b"k_gemm_bf16_tma") in (2 * (100 + d), 100 + d)
    lib.fake_device(0)
    assert passes(lib, *made[0]) == [nat.LBM_OK] * 2


def test_a_failed_first_call_is_tried_again(lib):
    lib.fake_reset()
    lib.fake_device(2)
    made = operator(lib)
    lib.fake_fail(b"cudaFuncSetAttribute", 1)
    assert lib.lbm_no_forward(made[0], B, made[1], made[2]) == nat.LBM_ERR_CUDA
    done = lib.fake_calls(b"cudaFuncSetAttribute")
    assert passes(lib, *made) == [nat.LBM_OK] * 2 and lib.fake_calls(b"cudaFuncSetAttribute") > done
    for nth in range(2, 12):  # each of the kernels in turn
        lib.fake_device(nth + 1)
        made = operator(lib)
        lib.fake_fail(b"cudaFuncSetAttribute", nth)
        passes(lib, *made)
        assert passes(lib, *made) == [nat.LBM_OK] * 2
