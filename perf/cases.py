"""The measured workloads: what a user of the hyperbolic SVD library has it do.

A case is a dict of plain values; ``kind`` names the public call it goes through:

=============  =====================================================================
solve          ``api.hsvd_solve_ex`` of one factor, plain FP64: method and block width
               as given (0 = the library's choice), square, tall (shortened by QR) or
               wide (shortened by the hyperbolic QR), device or pinned host arrays
split          the same call with ``HSVD_PRECISION_BF16X8`` (tensor-core products)
learned        the same call with a skip network (masked sweeps, full judge sweeps)
batch          ``api.hsvd_solve_batched``: many factors of mixed sizes in one launch
sym_eig        ``api.hsvd_sym_eig``: a symmetric indefinite eigenproblem, M = G J G^T
               by Bunch-Parlett pivoting, then the HSVD of G
qr             ``api.hsvd_shorten_qr``: the shortening QR on its own, R and Q
mlp_train      one training step of the skip network: ``hsvd_mlp_forward``,
               ``hsvd_mlp_grad``, ``hsvd_mlp_adam``
=============  =====================================================================

``run`` returns every output of the call; where the outputs are a decomposition it
also returns the eigenvalues of G J G^T in ascending order (sigma^2 with the column
signs, sorted: the library leaves them in input column order), which is what
``exact`` can give in 64 bits.  The order of sigma, and the signs of the singular
vectors, are the method's own and have no value outside it.
"""
import math

import numpy as np
import torch

from paper_1008_1371_gb300 import api

DEV = "cuda:0"
EPS = 2.0 ** -53

# Sweeps a solve is counted with in work(): the runs take 6 (tall, graded) to 27
# (Haar, ungraded); the flops of a sweep are the paper's 2 n^2 (4 m + 2 n).
SWEEPS = 8


def listed():
    return [
        # a single small factor with every default: latency of one call (n < 32: one-CTA method)
        dict(name="solve_24", kind="solve", m=24, n=24, inputs="gaussian", method=0, block_w=0, host=False),
        # the plain scalar method at its standard size, N(0,1) 128 x 128, p = 64, tol = 128 2^-53
        dict(name="pointwise_128", kind="solve", m=128, n=128, inputs="gaussian", method=1, block_w=0, host=False),
        # an odd mid-size factor from pinned host memory, copies included, every default (bordered, blocked)
        dict(name="solve_odd_host", kind="solve", m=333, n=301, inputs="gaussian", method=0, block_w=0, host=True),
        # the plain blocked method at its standard size, graded over 6 decades, b = 32
        dict(name="graded_1024", kind="solve", m=1024, n=1024, inputs="graded", method=2, block_w=32, host=False),
        # a tall graded factor: Householder QR first, U = Q U_R after
        dict(name="tall_8192x512", kind="solve", m=8192, n=512, inputs="graded", method=0, block_w=0, host=False),
        # a wide factor: hyperbolic QR of the transpose first, V after
        dict(name="wide_400x900", kind="solve", m=400, n=900, inputs="gaussian", method=0, block_w=0, host=False),
        # the precision form at its standard size: Haar 4096, sigma log-uniform on [1e-6, 1]
        dict(name="split_haar_4096", kind="split", m=4096, n=4096, inputs="haar", method=2, block_w=64, host=False),
        # the learned form: visits skipped by the network, full sweeps as judge
        dict(name="learned_1024", kind="learned", m=1024, n=1024, inputs="graded", method=2, block_w=32, host=False),
        # the batched form's standard distribution of sizes
        dict(name="batch_600", kind="batch", count=600, nmin=16, nmax=256),
        # a symmetric indefinite eigenproblem, odd order
        dict(name="sym_eig_1001", kind="sym_eig", n=1001),
        # the shortening QR on its own, R and Q
        dict(name="qr_8192x1024", kind="qr", m=8192, n=1024),
        # one training step of the skip network at the trainer's minibatch
        dict(name="mlp_train_4096", kind="mlp_train", n=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "pointwise", "tall", "wide", "split", "learned", "batch", "sym_eig",
                       "qr", "mlp_train"])
    inputs = rng.choice(["gaussian", "graded"])
    host = rng.random() < 0.25
    if kind == "pointwise":
        n = _log(rng, 5, 140)
        return dict(kind="solve", m=n + rng.randrange(0, 8), n=n, inputs=inputs, method=1, block_w=0, host=host)
    if kind == "tall":
        n = _log(rng, 12, 700)
        return dict(kind="solve", m=_log(rng, 1.3 * n, 16 * n), n=n, inputs=inputs, method=0, block_w=0, host=host)
    if kind == "wide":
        m = _log(rng, 12, 600)
        return dict(kind="solve", m=m, n=_log(rng, 1.1 * m + 1, 4 * m), inputs="gaussian", method=0, block_w=0,
                    host=host)
    if kind == "split":
        n = _log(rng, 130, 3000)
        return dict(kind="split", m=n + rng.randrange(0, n // 8), n=n, inputs=rng.choice(["haar", "gaussian"]),
                    method=2, block_w=64, host=host)
    if kind == "learned":
        n = _log(rng, 256, 1300)
        return dict(kind="learned", m=n, n=n, inputs="graded", method=2, block_w=rng.choice([16, 32, 64]), host=False)
    if kind == "batch":
        lo = _log(rng, 8, 64)
        return dict(kind="batch", count=_log(rng, 4, 800), nmin=lo, nmax=min(256, _log(rng, lo + 1, 256)))
    if kind == "sym_eig":
        return dict(kind="sym_eig", n=_log(rng, 20, 1500))
    if kind == "qr":
        n = _log(rng, 16, 1100)
        return dict(kind="qr", m=_log(rng, n + 1, 12 * n), n=n)
    if kind == "mlp_train":
        return dict(kind="mlp_train", n=_log(rng, 100, 60000))
    n = _log(rng, 12, 1500)
    return dict(kind="solve", m=n + rng.randrange(0, n // 8 + 1), n=n, inputs=inputs, method=0,
                block_w=rng.choice([0, 0, 16, 32, 64]), host=host)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device=DEV)


def _signs(g, n, p):
    J = torch.full((n,), -1, dtype=torch.int8, device=DEV)
    J[torch.randperm(n, generator=g, device=DEV)[:p]] = 1
    return J


def _haar(g, n):
    Q, R = torch.linalg.qr(_randn(g, n, n))
    return Q * torch.sign(torch.diagonal(R))[None, :]


def _factor(case, g):
    """(G, J) as the standard workloads draw them, on the GPU; G column-major."""
    m, n, inputs = case["m"], case["n"], case["inputs"]
    if inputs == "haar" and m == n:
        sigma = 10.0 ** (6.0 * torch.rand(n, generator=g, dtype=torch.float64, device=DEV) - 6.0)
        G = (_haar(g, n) * sigma[None, :]) @ _haar(g, n)
        J = _signs(g, n, n // 2)
    else:
        G = _randn(g, n, m).t()
        if inputs == "graded":
            decades = 6.0
            G = G * (10.0 ** (-decades * torch.arange(n, dtype=torch.float64, device=DEV) / n))[None, :]
        J = torch.full((n,), -1, dtype=torch.int8, device=DEV)
        J[:n // 2] = 1
        if m < n:  # a wide factor's signs are mixed
            J = _signs(g, n, n // 2)
    return G.t().contiguous().t(), J


def _sym(n, g):
    """Symmetric indefinite M = Q diag(lambda) Q^T, lambda uniform on +-(20e-5, 20] (half of each sign)."""
    Q = _haar(g, n)
    lam = 20.0 * (1e-5 + (1 - 1e-5) * torch.rand(n, generator=g, dtype=torch.float64, device=DEV))
    lam[n // 2:] *= -1.0
    M = (Q * lam[None, :]) @ Q.t()
    return ((M + M.t()) / 2).contiguous()


def _skip_model():
    """A skip network with the rule that training finds, as plain weights: a visit whose largest
    scaled entry was below 2^16 tol at its last visit is predicted to pass (the first
    feature is log2 of that ratio / 64; logit = 64 relu(f0) - 16)."""
    p = torch.zeros(api.HSVD_MLP_PARAMS, dtype=torch.float32, device=DEV)
    w2 = 64 * 8 + 64
    w3 = w2 + 64 * 64 + 64
    p[0] = 1.0
    p[w2] = 1.0
    p[w3] = 64.0
    p[w3 + 64] = -16.0
    return p


def _pinned(t):
    """A pinned host copy with the same column-major layout."""
    return t.t().cpu().pin_memory().t() if t.dim() == 2 else t.cpu().pin_memory()


def _mlp_inputs(case, seed):
    g = _gen(seed)
    n = case["n"]
    X = torch.empty((n, api.HSVD_MLP_FEATURES), dtype=torch.float32, device=DEV)
    X.uniform_(-0.6, 0.7, generator=g)
    y = (X[:, 0] + 0.25 * torch.randn(n, generator=g, device=DEV) > 0.1).to(torch.float32)
    h, f = 64, api.HSVD_MLP_FEATURES
    parts = [torch.randn(h * f, generator=g, device=DEV) * (2.0 / f) ** 0.5, torch.zeros(h, device=DEV),
             torch.randn(h * h, generator=g, device=DEV) * (2.0 / h) ** 0.5, torch.zeros(h, device=DEV),
             torch.randn(h, generator=g, device=DEV) * (1.0 / h) ** 0.5, torch.full((1,), 2.0, device=DEV)]
    return X, y, torch.cat(parts).contiguous()


def _batch_sizes(case):
    rng = np.random.default_rng([case["count"], case["nmin"], case["nmax"]])
    ns = rng.integers(case["nmin"], case["nmax"] + 1, case["count"])
    ps = [int(rng.integers(0, n + 1)) for n in ns]
    return [int(n) for n in ns], ps


def _batch_factors(case, seed):
    g = _gen(seed)
    ns, ps = _batch_sizes(case)
    flat = _randn(g, sum(n * n for n in ns))
    Gs, Js, at = [], [], 0
    for n, p in zip(ns, ps):
        Gs.append(flat[at:at + n * n].view(n, n).t())
        Js.append(_signs(g, n, p))
        at += n * n
    return Gs, Js


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp_train":
        X, y, p = _mlp_inputs(case, seed)
        return dict(kind=kind, X=X, y=y, p0=p, p=p.clone(), m=torch.zeros_like(p), v=torch.zeros_like(p))
    if kind == "batch":
        # the outputs of a batch live in three buffers that the program keeps
        Gs, Js = _batch_factors(case, seed)
        ns = [G.shape[1] for G in Gs]
        s = torch.empty(sum(ns), dtype=torch.float64, device=DEV)
        U = torch.empty(sum(n * n for n in ns), dtype=torch.float64, device=DEV)
        V = torch.empty_like(U)
        sig, Us, Vs, a, b = [], [], [], 0, 0
        for n in ns:
            sig.append(s[a:a + n])
            Us.append(U[b:b + n * n].view(n, n).t())
            Vs.append(V[b:b + n * n].view(n, n).t())
            a += n
            b += n * n
        ids = torch.repeat_interleave(torch.arange(len(ns), device=DEV), torch.tensor(ns, device=DEV))
        return dict(kind=kind, Gs=Gs, Js=Js, out=(sig, Us, Vs), flat=(s, U, V), ids=ids,
                    signs=torch.cat(Js).to(torch.float64), opts=api.make_batch_opts())
    g = _gen(seed)
    if kind == "sym_eig":
        return dict(kind=kind, M=_sym(case["n"], g))
    if kind == "qr":
        G, _ = _factor(dict(case, inputs="gaussian"), g)
        return dict(kind=kind, G=G)
    G, J = _factor(case, g)
    if case["host"]:
        G, J = _pinned(G), _pinned(J)
    kw = dict(method=case["method"], block_w=case["block_w"])
    model = None
    if kind == "split":
        kw["precision"] = api.HSVD_PRECISION_BF16X8
    if kind == "learned":
        model = _skip_model()
        kw.update(sort=False, skip_model=model)
    if case["method"] == api.HSVD_METHOD_POINTWISE:
        kw["tol"] = case["n"] * EPS
    return dict(kind=kind, G=G, J=J, model=model, opts=api.make_opts(**kw))


def run(state):
    kind = state["kind"]
    if kind == "mlp_train":
        p, m, v = state["p"], state["m"], state["v"]
        p.copy_(state["p0"])
        m.zero_()
        v.zero_()
        z = api.hsvd_mlp_forward(p, state["X"])
        grad, loss = api.hsvd_mlp_grad(p, state["X"], state["y"])
        api.hsvd_mlp_adam(p, m, v, grad, 1, lr=3e-3)
        return dict(logits=z, grad=grad, loss=loss, params=p, m=m, v=v)
    if kind == "batch":
        api.hsvd_solve_batched(state["Gs"], state["Js"], state["opts"], out=state["out"])
        s, U, V = state["flat"]
        lam, at = torch.sort(s * s * state["signs"])
        order = torch.sort(state["ids"][at], stable=True).indices
        return dict(sigma=s, U=U, V=V, eigenvalues=lam[order])
    if kind == "sym_eig":
        lam, U, _ = api.hsvd_sym_eig(state["M"])
        return dict(lam=lam, U=U, eigenvalues=torch.sort(lam).values)
    if kind == "qr":
        R, Q = api.hsvd_shorten_qr(state["G"])
        return dict(R=R, Q=Q)
    r = api.hsvd_solve_ex(state["G"], state["J"], state["opts"])
    signs = r.jout if r.jout is not None else state["J"]
    return dict(sigma=r.sigma, U=r.U, V=r.V, eigenvalues=torch.sort(r.sigma * r.sigma * signs).values)


def work(case):
    kind = case["kind"]
    if kind == "mlp_train":
        n, w = case["n"], 64 * 8 + 64 * 64 + 64
        # read X twice (forward, gradient call), y, the parameters and moments; write logits, gradient and the update
        return dict(bytes=4 * (2 * n * 8 + 2 * n + 8 * api.HSVD_MLP_PARAMS), flops=2 * n * w + 6 * n * w)
    if kind == "batch":
        ns, _ = _batch_sizes(case)
        return dict(bytes=8 * 3 * sum(n * n for n in ns), flops=SWEEPS * sum(12 * n ** 3 for n in ns))
    if kind == "qr":
        m, n = case["m"], case["n"]
        f = 2 * m * n * n - 2 * n ** 3 / 3
        return dict(bytes=8 * (2 * m * n + n * n), flops=2 * f)
    if kind == "sym_eig":
        n = case["n"]
        return dict(bytes=8 * 2 * n * n, flops=n ** 3 / 3 + SWEEPS * 12 * n ** 3)
    m, n = case["m"], case["n"]
    nbytes = 8 * (m * n + m * min(m, n) + n * min(m, n))
    if m < n:  # hyperbolic QR of the transpose, a square solve, the reflectors applied
        return dict(bytes=nbytes, flops=4 * n * m * m + SWEEPS * 12 * m ** 3)
    if 4 * m >= 5 * n:  # QR, a square solve, Q applied
        return dict(bytes=nbytes, flops=4 * m * n * n + SWEEPS * 12 * n ** 3)
    return dict(bytes=nbytes, flops=SWEEPS * 2 * n * n * (4 * m + 2 * n))


def _eigenvalues(G, J):
    """Ascending eigenvalues of G J G^T that are not the m - n zeros of a tall factor: those of the
    square R J R^T (G = Q R)."""
    m, n = G.shape
    if m > n:
        G = torch.linalg.qr(G)[1]
    A = (G * J.to(torch.float64)[None, :]) @ G.t()
    return torch.linalg.eigvalsh((A + A.t()) / 2)


def _bf16(w):
    return w.to(torch.bfloat16).to(torch.float64)


def _exact_mlp(case, seed):
    """The network, its gradient and one Adam step in 64 bits; the weights rounded to BF16 where the network runs."""
    X32, y32, p32 = _mlp_inputs(case, seed)
    X, y, p = X32.double(), y32.double(), p32.double()
    f, h, n = 8, 64, case["n"]
    ends = np.cumsum([h * f, h, h * h, h, h, 1]).tolist()
    W1, b1, W2, b2, w3, b3 = (p32[a:b] for a, b in zip([0] + ends[:-1], ends))
    W1, W2, w3 = _bf16(W1).view(h, f), _bf16(W2).view(h, h), _bf16(w3)
    a1 = X @ W1.t() + b1.double()
    h1 = a1.clamp(min=0)
    a2 = h1 @ W2.t() + b2.double()
    h2 = a2.clamp(min=0)
    z = h2 @ w3 + b3.double()
    loss = (torch.nn.functional.softplus(z) - y * z).mean()
    dz = (torch.sigmoid(z) - y) / n
    d2 = (dz[:, None] * w3[None, :]) * (h2 > 0)
    d1 = (d2 @ W2) * (h1 > 0)
    grad = torch.cat([(d1.t() @ X).reshape(-1), d1.sum(0), (d2.t() @ h1).reshape(-1), d2.sum(0), h2.t() @ dz,
                      dz.sum().reshape(1)])
    m1, v1 = 0.1 * grad, 0.001 * grad * grad
    # the parameters move by lr g / (|g| + eps) in a first step: the sign of a gradient entry of
    # the size of its own rounding decides, so the updated parameters have no 64-bit value
    return dict(logits=z, grad=grad, loss=loss.reshape(1), params=None, m=m1, v=v1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_train":
        return _exact_mlp(case, seed)
    if kind == "batch":
        Gs, Js = _batch_factors(case, seed)
        lam = []
        for G, J in zip(Gs, Js):
            G, J = G.cpu().numpy(), J.cpu().numpy().astype(np.float64)
            A = (G * J[None, :]) @ G.T
            lam.append(np.linalg.eigvalsh((A + A.T) / 2))
        return dict(sigma=None, U=None, V=None, eigenvalues=np.concatenate(lam))
    g = _gen(seed)
    if kind == "sym_eig":
        return dict(lam=None, U=None, eigenvalues=torch.linalg.eigvalsh(_sym(case["n"], g)))
    if kind == "qr":
        G, _ = _factor(dict(case, inputs="gaussian"), g)
        Q, R = torch.linalg.qr(G)
        return dict(R=R, Q=Q)
    G, J = _factor(case, g)
    return dict(sigma=None, U=None, V=None, eigenvalues=_eigenvalues(G, J))
