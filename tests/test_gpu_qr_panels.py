"""The shortening QR at the sizes where its split changes: panels of fewer than 32
columns, fewer rows than a cluster's CTAs take, one warp's rows just filled or
one over, more rows than the cluster keeps in shared memory (in place), more
than 64 row splits' worth of rows.  R and Q against LAPACK (the same sign
convention), each column to c m u of its norm (Householder QR's column-wise
bound; c = 8), and the thin Q orthonormal to c m u."""
import numpy as np
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


@pytest.mark.parametrize("m,n", [(31, 31), (32, 32), (33, 32), (40, 33), (64, 64), (513, 31), (2049, 65), (4097, 96),
                                 (13312, 33), (13400, 40), (9000, 1)])
def test_shorten_qr_edges(api, m, n):
    rng = np.random.default_rng(m + n)
    G = np.asfortranarray(rng.standard_normal((m, n)) * 10.0 ** rng.uniform(-3, 3, n)[None, :])
    R, Q = api.hsvd_shorten_qr(torch.from_numpy(G).cuda())
    R, Q = R.cpu().numpy(), Q.cpu().numpy()
    Rl = np.linalg.qr(G, mode="r")
    nrm = np.linalg.norm(G, axis=0)
    assert np.max(np.abs(R - Rl).max(axis=0) / nrm) <= 8 * m * U64
    assert np.max(np.linalg.norm(Q @ R - G, axis=0) / nrm) <= 8 * m * U64
    assert np.max(np.abs(Q.T @ Q - np.eye(n))) <= 8 * m * U64
    assert not np.any(np.tril(R, -1))
