"""The symmetric factorisation with G in M's own memory: M is read whole before G
is written, so the result is that of separate arrays, bit for bit (one
cooperative launch up to n = 4096, three kernels a step beyond; a singular M's
zero columns too).  Rows between n and the leading dimension stay as they are."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


def _sym(n, kind):
    g = torch.Generator().manual_seed(n)
    if kind == "singular":  # integers: the trailing matrix ends at zero exactly
        x = torch.zeros((n, n), dtype=torch.float64)
        x[0, 0], x[n - 1, n - 1], x[0, n - 1], x[n - 1, 0] = 4.0, -8.0, 2.0, 2.0
        return x.cuda()
    A = torch.randn((n, n), dtype=torch.float64, generator=g).cuda()
    M = (A + A.t()) / 2
    if kind == "saddle":
        M[:n // 2, :n // 2] = 0.0
    return M


@pytest.mark.parametrize("n,kind", [(1, "plain"), (5, "saddle"), (130, "plain"), (130, "singular"), (600, "saddle"),
                                    (1000, "plain"), (4097, "plain"), (4097, "singular")])
def test_in_place_equals_separate(api, n, kind):
    M = _sym(n, kind)
    want_G, want_J, want_r = api.hsvd_sym_factor(M, want_rank=True)
    assert want_r == (2 if kind == "singular" else n)
    ld = n + 3
    buf = torch.full((n, ld), 7.0, dtype=torch.float64, device="cuda")  # row j: column j
    buf[:, :n] = M
    J = torch.empty(n, dtype=torch.int8, device="cuda")
    rank = ctypes.c_int64(-1)
    st = api.lib().hsvd_sym_factor(buf.data_ptr(), n, ld, buf.data_ptr(), ld, J.data_ptr(), ctypes.byref(rank),
                                   torch.cuda.current_stream().cuda_stream)
    assert st == api.HSVD_OK and rank.value == want_r
    assert torch.equal(J, want_J) and torch.equal(buf[:, :n].t(), want_G)
    assert bool((buf[:, n:] == 7.0).all())
