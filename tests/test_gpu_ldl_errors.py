"""The one-launch symmetric factorisation ends with a status where it cannot go
on, with one CTA and with many: a NaN or an infinity in M, and a 2 x 2 pivot
block without an inverse, as the oracle."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    oracle.build()
    assert torch.cuda.is_available()
    return api


def _status(api, M):
    try:
        api.hsvd_sym_factor(torch.from_numpy(np.asfortranarray(M)).cuda())
        return api.HSVD_OK
    except api.HsvdError as e:
        return e.status


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,at", [(1, (0, 0)), (7, (6, 6)), (130, (0, 0)), (130, (129, 3)), (600, (599, 599))])
def test_non_finite(api, n, at, value):
    A = np.random.default_rng(n).standard_normal((n, n))
    M = (A + A.T) / 2
    M[at] = M[at[::-1]] = value
    assert _status(api, M) == api.HSVD_ERR_RANK
    # and the next call is not affected
    assert _status(api, (A + A.T) / 2) == api.HSVD_OK


@pytest.mark.parametrize("n", [2, 12, 130, 511])
def test_oracle_status_on_underflow(api, n):
    """det of a 2 x 2 block underflows to zero (entries of 2^-600): no inverse."""
    M = np.zeros((n, n))
    for i in range(0, n - 1, 2):
        M[i, i + 1] = M[i + 1, i] = 2.0 ** -600
    if n % 2:
        M[n - 1, n - 1] = 2.0 ** -600
    st = oracle.sym_factor(M)[3]
    assert _status(api, M) == (api.HSVD_ERR_RANK if st else api.HSVD_OK)
