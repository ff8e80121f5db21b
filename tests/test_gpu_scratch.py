"""The calls' scratch: the same results with the pool empty and filled, from
several threads on streams of their own, and the memory given back on request."""
import threading

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


def _inputs(m, n, seed):
    G, J = W.gaussian(n, m=m, seed=seed)
    return torch.from_numpy(np.asfortranarray(G)).cuda().t().contiguous().t(), torch.from_numpy(J).cuda()


def test_release_and_reuse(api):
    Gd, Jd = _inputs(700, 300, 1)
    first = api.hsvd_solve_ex(Gd, Jd, api.make_opts())
    again = api.hsvd_solve_ex(Gd, Jd, api.make_opts())
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    assert api.lib().hsvd_release_scratch() == api.HSVD_OK
    assert torch.cuda.mem_get_info()[0] >= before
    after = api.hsvd_solve_ex(Gd, Jd, api.make_opts())
    for r in (again, after):
        assert torch.equal(first.sigma, r.sigma) and torch.equal(first.U, r.U) and torch.equal(first.V, r.V)


def test_threads_and_streams(api):
    shapes = [(24, 24), (333, 301), (130, 64), (600, 90)]
    data = [_inputs(m, n, 10 + i) for i, (m, n) in enumerate(shapes)]
    want = [api.hsvd_solve_ex(G, J, api.make_opts()) for G, J in data]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(5):
                r = api.hsvd_solve_ex(*data[i], api.make_opts())
                st.synchronize()
                if not (torch.equal(r.sigma, want[i].sigma) and torch.equal(r.V, want[i].V)):
                    bad.append(i)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(shapes))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
