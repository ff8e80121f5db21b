"""The pair schedule's groups of visits (a whole step in one, half the nodes,
one visit each; on both sides of the sizes where they change) and its order of
updates (V's columns after G's, beside the next visits) change no visit's
arithmetic: the same bits as the step schedule, with V and without."""
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


@pytest.mark.parametrize("b,n,prec,sort", [(16, 40, 0, False), (16, 416, 0, False), (16, 420, 0, True),
                                           (16, 512, 0, False), (32, 96, 0, True), (32, 520, 0, False),
                                           (64, 640, 1, True), (64, 200, 1, False)])
def test_groups_agree_with_steps(api, b, n, prec, sort):
    G, J = W.graded(n, m=n + 7, decades=4.0, seed=n)
    Gd, Jd = torch.from_numpy(np.asfortranarray(G)).cuda(), torch.from_numpy(J).cuda()
    kw = dict(method=api.HSVD_METHOD_BLOCKED, block_w=b, precision=prec, sort=sort, max_sweeps=40,
              shorten=api.HSVD_SHORTEN_NEVER)
    a = api.hsvd_solve_ex(Gd, Jd, api.make_opts(schedule=api.HSVD_SCHEDULE_STEPS, **kw))
    p = api.hsvd_solve_ex(Gd, Jd, api.make_opts(schedule=api.HSVD_SCHEDULE_PAIRS, **kw))
    assert a.sweeps == p.sweeps and a.rotations == p.rotations and a.pair_updates == p.pair_updates
    assert torch.equal(a.sigma, p.sigma) and torch.equal(a.U, p.U) and torch.equal(a.V, p.V)
    q = api.hsvd_solve_ex(Gd, Jd, api.make_opts(schedule=api.HSVD_SCHEDULE_PAIRS, **kw), compute_v=False)
    assert torch.equal(a.sigma, q.sigma) and torch.equal(a.U, q.U)
