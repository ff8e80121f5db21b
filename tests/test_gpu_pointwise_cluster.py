"""The single-factor pointwise kernel (one cluster, a warp per pair, columns
moving between slots) against the batched kernel (one group of an SM, columns
in place): the same arithmetic in the same order, so the results are compared
bit for bit, at the sizes where the cluster's split changes (one, two, four,
eight and sixteen CTAs, four and five pairs a CTA, a last CTA with fewer
pairs), for odd n (bordered), tall factors, with and without V, with and
without sorting and the tangent threshold."""
import numpy as np
import pytest
import torch

from paper_1008_1371_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


def _factor(m, n, seed):
    rng = np.random.default_rng(seed)
    G = torch.from_numpy(np.asfortranarray(rng.standard_normal((m, n)))).cuda().t().contiguous().t()
    return G, torch.from_numpy(W.signs_random(rng, n, int(rng.integers(0, n + 1)))).cuda()


SHAPES = [(1, 1), (2, 2), (5, 3), (40, 2), (8, 8), (9, 9), (16, 16), (300, 18), (33, 33), (64, 64), (66, 65),
          (127, 127), (128, 128), (129, 129), (400, 50), (156, 156)]


@pytest.mark.parametrize("m,n", SHAPES)
def test_cluster_equals_batched_bitwise(api, m, n):
    G, J = _factor(m, n, 1000 * m + n)
    # group_width: the queue of groups, whatever the batch
    for sort, tstop, want_v in ((True, 0.0, True), (False, 0.0, True), (True, -1.0, True), (True, 0.0, False)):
        tol = n * 2.0 ** -53
        one = api.hsvd_solve_ex(G, J, api.make_opts(method=api.HSVD_METHOD_POINTWISE, sort=sort, tstop=tstop, tol=tol,
                                                    shorten=api.HSVD_SHORTEN_NEVER), compute_v=want_v)
        b = api.hsvd_solve_batched([G], [J], api.make_batch_opts(sort=sort, tstop=tstop, tol=tol, group_width=512),
                                   compute_v=want_v)
        assert one.status == b.status[0] == 0 and one.sweeps == b.sweeps[0]
        assert one.rotations == b.info.rotations
        assert torch.equal(one.sigma, b.sigma[0]) and torch.equal(one.U, b.U[0])
        assert not want_v or torch.equal(one.V, b.V[0])


def test_two_long_columns_take_the_one_cta_kernel(api):
    """Two columns of 12,000 rows fit no cluster slot pair (four columns with
    their V rows are past an SM's shared memory); J = I, so the values are the
    singular values of the n = 2 factor, each to a few units in the last place
    of the dot products over m rows (sqrt(m) u, with a factor 8 of slack)."""
    G, _ = _factor(12000, 2, 5)
    r = api.hsvd_solve_ex(G, torch.ones(2, dtype=torch.int8, device="cuda"),
                          api.make_opts(method=api.HSVD_METHOD_POINTWISE, shorten=api.HSVD_SHORTEN_NEVER))
    ref = np.sort(np.linalg.svd(G.cpu().numpy(), compute_uv=False))
    assert r.status == 0
    assert np.max(np.abs(np.sort(r.sigma.cpu().numpy()) - ref) / ref) <= 8 * np.sqrt(12000) * 2.0 ** -53


@pytest.mark.parametrize("sizes", [[256, 40, 17, 3], [64] * 30, [200, 131, 90, 16, 5] * 8])
def test_few_factors_take_clusters_bitwise(api, sizes):
    """A batch too short for the SMs runs one cluster per factor: the same bits
    as the queue of 1024-thread groups."""
    facs = [_factor(n, n, 31 * k + n) for k, n in enumerate(sizes)]
    Gs, Js = [f[0] for f in facs], [f[1] for f in facs]
    a = api.hsvd_solve_batched(Gs, Js, api.make_batch_opts())
    b = api.hsvd_solve_batched(Gs, Js, api.make_batch_opts(group_width=1024))
    assert a.info.kernel_launches == b.info.kernel_launches == 1 and a.info.grid > len(sizes) >= b.info.grid
    assert a.sweeps == b.sweeps and a.status == b.status and a.info.rotations == b.info.rotations
    for k in range(len(sizes)):
        assert torch.equal(a.sigma[k], b.sigma[k]) and torch.equal(a.U[k], b.U[k]) and torch.equal(a.V[k], b.V[k])
