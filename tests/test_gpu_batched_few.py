"""Batches of few small or tall factors: which of them take a cluster per factor
(the queue of groups has fewer barriers to wait for only where a factor fills an
SM), and every split of the dots over a group's warps (one to four pairs a
warp, a last warp with fewer) gives the bits of the single-factor solve."""
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


def _factors(m, n, count):
    out = []
    for k in range(count):
        rng = np.random.default_rng(1000 * m + 10 * n + k)
        G = torch.from_numpy(np.asfortranarray(rng.standard_normal((m, n)))).cuda().t().contiguous().t()
        out.append((G, torch.from_numpy(W.signs_random(rng, n, n // 2)).cuda()))
    return [f[0] for f in out], [f[1] for f in out]


def _equal(a, b, count):
    return a.sweeps == b.sweeps and all(torch.equal(a.sigma[k], b.sigma[k]) and torch.equal(a.U[k], b.U[k]) and
                                        torch.equal(a.V[k], b.V[k]) for k in range(count))


@pytest.mark.parametrize("m,n,count,clusters", [(1, 1, 3, True), (4, 4, 150, True), (8, 8, 1, True), (8, 8, 150, True),
                                                (9, 9, 40, True), (16, 16, 11, True), (17, 13, 40, True),
                                                (256, 8, 60, True), (40, 40, 114, False), (300, 100, 110, False)])
def test_form_by_size(api, m, n, count, clusters):
    Gs, Js = _factors(m, n, count)
    a = api.hsvd_solve_batched(Gs, Js, api.make_batch_opts(), check=False)
    b = api.hsvd_solve_batched(Gs, Js, api.make_batch_opts(group_width=1024), check=False)
    assert a.rc == b.rc == 0
    assert (a.info.tuned == 0) == clusters  # 0 without a width: a cluster per factor
    assert a.info.kernel_launches == 1 and _equal(a, b, count)


@pytest.mark.parametrize("m,n", [(2, 2), (6, 6), (300, 14), (260, 18), (40, 32), (33, 33), (50, 50), (70, 66),
                                 (130, 64)])
def test_dots_split_over_the_warps(api, m, n):
    G, J = (x[0] for x in _factors(m, n, 1))
    one = api.hsvd_solve_ex(G, J, api.make_opts(method=api.HSVD_METHOD_POINTWISE, sort=True,
                                                shorten=api.HSVD_SHORTEN_NEVER))
    for w in (256, 512, 1024):
        b = api.hsvd_solve_batched([G], [J], api.make_batch_opts(group_width=w))
        assert b.sweeps[0] == one.sweeps and b.info.rotations == one.rotations
        assert torch.equal(b.sigma[0], one.sigma) and torch.equal(b.U[0], one.U) and torch.equal(b.V[0], one.V)


@pytest.mark.parametrize("n,count", [(8, 160), (8, 700), (24, 305), (33, 700), (64, 161), (64, 460)])
def test_queue_dealt_out(api, n, count):
    """Queues of one width: the first factor of every group by its index (fewer
    factors than groups, a last round with some), the rest from the counter."""
    Gs, Js = _factors(n + 1, n, count)
    a = api.hsvd_solve_batched(Gs, Js, api.make_batch_opts(group_width=1024))
    for kw in (dict(), dict(group_width=512), dict(group_width=256), dict(cta_threads=512),
               dict(group_width=256, cta_threads=512)):
        assert _equal(a, api.hsvd_solve_batched(Gs, Js, api.make_batch_opts(**kw)), count)
