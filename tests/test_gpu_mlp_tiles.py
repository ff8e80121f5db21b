"""The skip network's kernels at the edges of their tiles: 32 samples a tile in
the forward pass and a grid that wraps past 608 tiles, 64 samples a partial
gradient and 128 partials a stage of their sum.  Against the float64 oracle,
with the bounds of the other network tests (a logit is a sum of 64 products
after BF16 rounding of the weights: 2e-5 relative; the gradient's sums over
samples in FP32: 1e-4 of the largest entry)."""
import numpy as np
import pytest
import torch

from oracle import mlp as mlp_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1008_1371_gb300 import api, build_lib

    build_lib.build()
    assert torch.cuda.is_available()
    return api


def _inputs(n):
    rng = np.random.default_rng(n)
    p = (0.3 * rng.standard_normal(mlp_oracle.PARAMS)).astype(np.float32)
    X = rng.standard_normal((n, 8)).astype(np.float32)
    return p, X, (rng.random(n) < 0.4).astype(np.float32)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 608 * 32, 608 * 32 + 1, 2 * 608 * 32 + 17])
def test_forward_tiles(api, n):
    p, X, _ = _inputs(n)
    pd, Xd = torch.from_numpy(p).cuda(), torch.from_numpy(X).cuda()
    got = api.hsvd_mlp_forward(pd, Xd)
    want = mlp_oracle.forward(p.astype(np.float64), X.astype(np.float64))
    assert np.max(np.abs(got.cpu().numpy() - want) / (1.0 + np.abs(want))) <= 2e-5
    # a logit doesn't depend on its sample's place in a tile
    k = n // 2
    assert torch.equal(api.hsvd_mlp_forward(pd, Xd[k:].clone()), got[k:])


@pytest.mark.parametrize("n", [65, 127, 128 * 64, 128 * 64 + 1, 256 * 64 + 3])
def test_grad_stages(api, n):
    p, X, y = _inputs(n)
    g, loss = api.hsvd_mlp_grad(torch.from_numpy(p).cuda(), torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda())
    lw, gw = mlp_oracle.loss_grad(p.astype(np.float64), X.astype(np.float64), y.astype(np.float64))
    assert abs(float(loss.item()) - lw) <= 1e-5 * (1 + abs(lw))
    assert np.max(np.abs(g.cpu().numpy() - gw)) <= 1e-4 * np.max(np.abs(gw))
