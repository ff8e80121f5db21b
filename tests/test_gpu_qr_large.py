"""The shortening QR past its limits: more than 64 splits' worth of rows (a split
then has more than 256), and more than 2048 columns (taken in chunks, with the
identity's columns before a panel skipped in the second chunk too).  R and Q to
the bound of Householder QR, c m u of a column's norm (c = 8)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
U64 = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


@pytest.mark.parametrize("m,n", [(17000, 33), (20000, 64), (2100, 2081)])
def test_qr_beyond_the_limits(api, m, n):
    g = torch.Generator(device="cuda").manual_seed(m)
    scale = 10.0 ** (6 * torch.rand(n, generator=g, dtype=torch.float64, device="cuda") - 3)
    G = (torch.randn((n, m), generator=g, dtype=torch.float64, device="cuda") * scale[:, None]).t()
    R, Q = api.hsvd_shorten_qr(G)
    nrm = torch.linalg.vector_norm(G, dim=0)
    eps = 8 * m * U64
    assert not bool(torch.tril(R, -1).any())
    assert float((torch.linalg.vector_norm(Q @ R - G, dim=0) / nrm).max()) <= eps
    assert float((Q.t() @ Q - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max()) <= eps
    R2, none = api.hsvd_shorten_qr(G, want_q=False)
    assert none is None and torch.equal(R, R2)
