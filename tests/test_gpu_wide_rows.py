"""The hyperbolic QR of the wide case at its kernels' edges: more rows than the
selection's 1024 threads, than one warp's or one CTA's columns, and on both
sides of the row count up to which V's columns are held in shared memory.
Gaussian factors with three positive signs to one negative, so that G J G^T is
well conditioned and row interchanges still occur.  Checked by the invariants
of Eq. 1.1 and LAPACK's eigenvalues of G J G^T, within the bounds that the
wide tests use (16 n u relative to the largest eigenvalue for values computed
from sums of n terms, 1e-12 n for the residuals)."""
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


@pytest.mark.parametrize("m,n", [(1, 2), (2, 33), (33, 1024), (33, 1057), (257, 300), (9, 11377), (9, 11378),
                                 (40, 14001)])
def test_wide_rows(api, m, n):
    rng = np.random.default_rng(100 * m + n)
    G = np.asfortranarray(rng.standard_normal((m, n)))
    J = np.where(rng.permutation(n) < n - n // 4, 1, -1).astype(np.int8)
    dev = torch.device("cuda:0")
    r = api.hsvd_solve_ex(torch.from_numpy(G).to(dev), torch.from_numpy(J).to(dev), api.make_opts(max_sweeps=40))
    s, U, V, jo = r.sigma.cpu().numpy(), r.U.cpu().numpy(), r.V.cpu().numpy(), r.jout.cpu().numpy()
    assert r.status == api.HSVD_OK and r.shortened == 2
    ev = np.linalg.eigvalsh((G * J[None, :]) @ G.T)
    assert np.max(np.abs(ev - np.sort(s ** 2 * jo))) <= 16 * n * U64 * np.max(np.abs(ev))
    assert np.max(np.abs(U.T @ U - np.eye(m))) <= 1e-12 * m
    res = np.linalg.norm(G @ V - U * s[None, :], axis=0) / (np.linalg.norm(G) * np.linalg.norm(V, axis=0))
    assert np.max(res) <= 1e-12 * n
    jv = np.max(np.abs((V.T * J[None, :]) @ V - np.diag(jo.astype(float)))) / max(1.0, np.max(np.abs(V)) ** 2)
    assert jv <= 1e-12 * n, jv
