"""The symmetric factorisation in one cooperative launch (n <= 4096) against the
CPU oracle, bit for bit, at the sizes where its split changes (one CTA, fewer
CTAs than SMs, one per SM; fewer rows than threads, just more), with forced
2 x 2 pivots, ties and rank deficiency; and against the three-kernel form that
larger n take."""
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


def _sym(n, kind, seed):
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((n, n))
    M = (A + A.T) / 2
    if kind == "saddle":  # a zero diagonal block forces 2 x 2 pivots
        M[:n // 2, :n // 2] = 0.0
    if kind == "ties":  # small integers: equal magnitudes everywhere
        M = np.round(2.0 * M)
    if kind == "singular":
        B = np.round(rng.standard_normal((n, max(1, n // 3))) * 4)
        s = np.sign(rng.standard_normal(B.shape[1]))
        M = (B * s[None, :]) @ B.T
    return np.asfortranarray(M)


@pytest.mark.parametrize("kind", ["plain", "saddle", "ties", "singular"])
@pytest.mark.parametrize("n", [1, 2, 3, 11, 12, 13, 65, 130, 511, 513, 520])
def test_one_launch_equals_oracle_bitwise(api, n, kind):
    M = _sym(n, kind, 7 * n)
    Go, Jo, _, st, ro = oracle.sym_factor(M, want_rank=True)
    if st != 0:
        pytest.skip("singular 2 x 2 block in the oracle too")
    G, J, r = api.hsvd_sym_factor(torch.from_numpy(M).cuda(), want_rank=True)
    assert r == ro and np.array_equal(J.cpu().numpy(), Jo) and np.array_equal(G.cpu().numpy(), Go)


def test_one_per_sm_equals_oracle_bitwise(api):
    M = _sym(1000, "plain", 3)
    Go, Jo, _, st = oracle.sym_factor(M)
    G, J = api.hsvd_sym_factor(torch.from_numpy(M).cuda())
    assert st == 0 and np.array_equal(J.cpu().numpy(), Jo) and np.array_equal(G.cpu().numpy(), Go)


def test_three_kernel_form_agrees_bitwise(api):
    """n = 4097 takes the three kernels a step, n = 4096 the one launch.  A last
    row and column of zeros with a tiny diagonal entry is pivoted last and
    leaves every other operation as it was."""
    n = 4096
    g = torch.Generator(device="cuda").manual_seed(11)
    M = torch.zeros((n + 1, n + 1), dtype=torch.float64, device="cuda")
    A = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda")
    M[:n, :n] = (A + A.t()) / 2
    M[n, n] = 2.0 ** -400
    G1, J1 = api.hsvd_sym_factor(M)
    G0, J0 = api.hsvd_sym_factor(M[:n, :n].contiguous())
    assert torch.equal(J1[:n], J0) and int(J1[n]) == 1
    assert torch.equal(G1[:n, :n], G0)
    assert float(G1[n, n]) == 2.0 ** -200 and not bool(G1[n, :n].any()) and not bool(G1[:n, n].any())
