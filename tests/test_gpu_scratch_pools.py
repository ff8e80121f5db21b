"""The scratch pool of the library: what it keeps is bounded and given back, and
calls made in turn in two contexts of one device do not make a new pool (and
leave the last one's memory behind) at every change."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_is_bounded_and_released(api):
    """2000 x 2000: working copies of 128 MB and more, above the 256 MB that are kept."""
    G = torch.randn((2000, 2000), dtype=torch.float64, device="cuda").t()
    J = torch.ones(2000, dtype=torch.int8, device="cuda")
    o = api.make_opts(max_sweeps=1)
    r = api.hsvd_solve_ex(G, J, o, check=False)
    torch.cuda.synchronize()
    api.hsvd_release_scratch()
    base = _free()
    api.hsvd_solve_ex(G, J, o, check=False, out=(r.sigma, r.U, r.V))
    held = base - _free()
    # reserved in blocks of at least 2 MB, in whole blocks
    assert 0 < held <= (256 + 64) * MB
    api.hsvd_release_scratch()
    assert base - _free() <= 2 * MB


def test_two_contexts_in_turn(api):
    L = api.lib()
    torch.zeros(1, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    p = ctypes.c_void_p
    dev, first, second = ctypes.c_int(-1), p(), p()
    assert cu.cuDeviceGet(ctypes.byref(dev), 0) == 0
    assert cu.cuCtxGetCurrent(ctypes.byref(first)) == 0 and first.value
    assert cu.cuCtxCreate_v2(ctypes.byref(second), 0, dev) == 0

    def in_turn(count):
        for _ in range(count):
            for ctx in (second, first):
                assert cu.cuCtxSetCurrent(ctx) == 0
                assert L.hsvd_diag_wait_timeout(None) == 0  # takes 4 bytes of scratch

    try:
        in_turn(2)  # modules loaded, pools made
        before = _free()
        in_turn(20)
        assert before - _free() <= 2 * MB
    finally:
        cu.cuCtxSetCurrent(second)
        cu.cuCtxDestroy_v2(second)
        cu.cuCtxSetCurrent(first)
    assert L.hsvd_diag_wait_timeout(None) == 0
