"""The split-precision products under power-of-two scales: digits are relative
to each row's or column's exponent and the recombination rounds the same
integers, in 64-bit words in the middle of the exponent range and in 128-bit
ones beyond 2^900, so scaled inputs give exactly scaled outputs.  Inputs with
small, zero and cancelling entries, so that sums of every size occur."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


def _matrix(rows, cols, seed):
    g = torch.Generator().manual_seed(seed)
    X = torch.randn(rows, cols, dtype=torch.float64, generator=g)
    X *= 2.0 ** torch.randint(-30, 1, (rows, cols), generator=g).double()
    X[:, 3] = 0.0
    X[::2, 7] = X[1::2, 7]
    X[::2, 8] = X[1::2, 9]
    X[1::2, 8] = -X[::2, 9]
    return X.t().contiguous().cuda().t()


@pytest.mark.parametrize("k", [-440, -100, 100, 460])
def test_gram_scaled(api, k):
    G = _matrix(320, 128, 1)
    c0 = torch.tensor([[0, 64]], dtype=torch.int32, device="cuda")
    A = api.hsvd_pivot_gram_x(G, c0)
    assert torch.equal(api.hsvd_pivot_gram_x(G * 2.0 ** k, c0), A * 2.0 ** (2 * k))


@pytest.mark.parametrize("k", [-880, -100, 100, 950])
def test_update_scaled(api, k):
    X = _matrix(192, 128, 2)
    W = torch.linalg.qr(torch.randn(1, 128, 128, dtype=torch.float64, generator=torch.Generator().manual_seed(3)))[0]
    c0 = torch.tensor([[0, 64]], dtype=torch.int32, device="cuda")
    rot = torch.ones(1, dtype=torch.int32, device="cuda")
    out = []
    for s in (1.0, 2.0 ** k):
        Y = (X * s).t().contiguous().t()
        api.hsvd_pivot_update_x(Y, c0, W.cuda(), rot)
        out.append(Y)
    assert torch.equal(out[1], out[0] * 2.0 ** k)
