"""The Gram kernel's two forms (every full block; one of two mirrored entries of
the diagonal blocks) give the same bits: 64 rows, two splits, few pairs take the
first, many the second.  Against FP64 matrix products: an entry is a sum of
`rows` products, so within rows * u of the norms' product."""
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


@pytest.mark.parametrize("b,npairs,rows", [(16, 100, 64), (32, 27, 64), (64, 8, 64), (16, 7, 1088), (32, 9, 704),
                                           (64, 3, 320)])
def test_gram_forms(api, b, npairs, rows):
    g = torch.Generator().manual_seed(b + rows)
    n = 2 * b * npairs
    G = torch.randn(n, rows, dtype=torch.float64, generator=g).cuda().t()
    blocks = torch.randperm(2 * npairs, generator=g).reshape(npairs, 2).to(torch.int32).cuda() * b
    A = api.hsvd_pivot_gram(G, b, blocks)
    assert torch.equal(A, A.transpose(1, 2))
    for k in (0, npairs - 1):
        cols = torch.cat([torch.arange(int(c), int(c) + b) for c in blocks[k]])
        X = G[:, cols.cuda()]
        nrm = torch.linalg.vector_norm(X, dim=0)
        assert float(((A[k] - X.t() @ X).abs() / (nrm[:, None] * nrm[None, :])).max()) <= 2 * rows * U64
        if rows == 64:
            assert torch.equal(api.hsvd_pivot_gram(G, b, blocks[k:k + 1])[0], A[k])
