"""Host threads on streams of their own, in the same entry point with very
different sizes: what a launch needs of a kernel (its limit of dynamic shared
memory) must not be taken back by another thread's smaller call.  Every call
succeeds and gives the bits it gives alone."""
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


def _factor(m, n, seed):
    rng = np.random.default_rng(seed)
    G = torch.from_numpy(np.asfortranarray(rng.standard_normal((m, n)))).cuda().t().contiguous().t()
    return G, torch.from_numpy(W.signs_random(rng, n, n // 2)).cuda()


def _sym_factor(api, n):
    A = torch.randn((n, n), dtype=torch.float64, generator=torch.Generator().manual_seed(n)).cuda()
    M = (A + A.t()) / 2
    return lambda: api.hsvd_sym_factor(M)


def _pointwise(api, n):
    G, J = _factor(n, n, n)
    # two sweeps are enough to compare
    o = api.make_opts(method=api.HSVD_METHOD_POINTWISE, max_sweeps=2)

    def go():
        r = api.hsvd_solve_ex(G, J, o, check=False)
        return r.sigma, r.U, r.V

    return go


def _batch(api, n):
    f = [_factor(n, n, 10 * n + k) for k in range(3)]
    Gs, Js = [x[0] for x in f], [x[1] for x in f]
    o = api.make_batch_opts(max_sweeps=2)

    def go():
        r = api.hsvd_solve_batched(Gs, Js, o, check=False)
        assert r.rc >= 0
        return (*r.sigma, *r.U, *r.V)

    return go


def _qr(api, m):
    G, _ = _factor(m, 64, m)
    return lambda: api.hsvd_shorten_qr(G)


@pytest.mark.parametrize("make,small,big,calls", [(_sym_factor, 3, 2100, 100), (_pointwise, 4, 150, 300),
                                                  (_batch, 4, 200, 300), (_qr, 100, 13000, 150)])
def test_threads_of_different_sizes(api, make, small, big, calls):
    """One thread makes `calls` large calls (more than 48 KB of shared memory, what
    every kernel has without asking) while six repeat small ones."""
    fns = [make(api, big)] + [make(api, small) for _ in range(6)]
    want = [fn() for fn in fns]
    torch.cuda.synchronize()
    wrong, done = [], threading.Event()

    def work(k):
        st = torch.cuda.Stream()
        count = 0
        with torch.cuda.stream(st):
            while count < calls if k == 0 else not done.is_set():
                count += 1
                try:
                    got = fns[k]()
                    st.synchronize()
                    if not all(torch.equal(a, b) for a, b in zip(got, want[k])):
                        wrong.append("bits")
                except Exception as e:
                    wrong.append(repr(e))
        if k == 0:
            done.set()

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(fns))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not wrong, (len(wrong), sorted(set(wrong)))
