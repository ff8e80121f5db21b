"""Calls on a stream that may use part of the SMs only (a green context of 16):
the kernels whose CTAs wait for each other take their size from the stream, so
the symmetric factorisation (a CTA per SM elsewhere), the pointwise method (a
16-CTA cluster elsewhere) and a batch of few factors give the bits they give on
the whole device."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1008_1371_gb300 import workloads as W

pytestmark = pytest.mark.gpu
RESOURCE_BYTES = 144  # sizeof(CUdevResource): type, 92 bytes, 48 bytes
SM = 1                # CU_DEV_RESOURCE_TYPE_SM


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


@pytest.fixture(scope="module")
def confined(api):
    """(torch stream of a green context, its SMs)."""
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    names = ["cuDeviceGet", "cuDeviceGetDevResource", "cuDevSmResourceSplitByCount", "cuDevResourceGenerateDesc",
             "cuGreenCtxCreate", "cuGreenCtxStreamCreate", "cuGreenCtxDestroy", "cuStreamDestroy_v2", "cuStreamGetCtx_v2"]
    if not all(hasattr(cu, n) for n in names):
        pytest.skip("this driver has no green contexts")

    def ck(st):
        assert st == 0, st

    p = ctypes.c_void_p
    dev = ctypes.c_int(-1)
    ck(cu.cuDeviceGet(ctypes.byref(dev), 0))
    whole, part, rest = (ctypes.create_string_buffer(RESOURCE_BYTES) for _ in range(3))
    ck(cu.cuDeviceGetDevResource(dev, whole, SM))
    groups = ctypes.c_uint(1)
    ck(cu.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), whole, rest, 0, 16))
    sms = int(np.frombuffer(part.raw, dtype=np.uint32)[24])  # byte 96: sm.smCount
    assert groups.value == 1 and 16 <= sms < 152
    desc, ctx, st = p(), p(), p()
    ck(cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1))
    ck(cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, 1))       # CU_GREEN_CTX_DEFAULT_STREAM
    ck(cu.cuGreenCtxStreamCreate(ctypes.byref(st), ctx, 1, 0))     # CU_STREAM_NON_BLOCKING
    yield torch.cuda.ExternalStream(st.value), sms
    torch.cuda.synchronize()
    ck(cu.cuStreamDestroy_v2(st))
    ck(cu.cuGreenCtxDestroy(ctx))


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("n", [40, 97, 600, 1001])
def test_sym_factor(api, confined, n):
    A = torch.randn((n, n), dtype=torch.float64, generator=torch.Generator().manual_seed(n)).cuda()
    M = (A + A.t()) / 2
    want = api.hsvd_sym_factor(M)
    torch.cuda.synchronize()
    got = api.hsvd_sym_factor(M, stream=confined[0])
    confined[0].synchronize()
    assert _same(got, want)


@pytest.mark.parametrize("n", [12, 64, 128])
def test_pointwise_and_batch(api, confined, n):
    G, J = W.gaussian(n, m=n, seed=n)
    G, J = torch.from_numpy(np.asfortranarray(G)).cuda().t().contiguous().t(), torch.from_numpy(J).cuda()
    o = api.make_opts(method=api.HSVD_METHOD_POINTWISE)
    bo = api.make_batch_opts()
    one, few = api.hsvd_solve_ex(G, J, o), api.hsvd_solve_batched([G] * 5, [J] * 5, bo)
    torch.cuda.synchronize()
    st, sms = confined
    a = api.hsvd_solve_ex(G, J, o, stream=st)
    b = api.hsvd_solve_batched([G] * 5, [J] * 5, bo, stream=st)
    st.synchronize()
    assert a.status == 0 and b.rc == 0
    assert _same((a.sigma, a.U, a.V), (one.sigma, one.U, one.V))
    assert _same((*b.sigma, *b.U, *b.V), (*few.sigma, *few.U, *few.V))
