"""The hyperparameter fit's evaluation by a cluster of eight CTAs at the edges of
its blocks and of its shared memory, and the kernel beyond it, against the log
marginal likelihood and its gradient in plain torch at 64 bits; and a matrix
that is not positive definite.

Bar: 1e-9 (1 + |value|), the rounding of two fp64 factorisations of matrices
whose condition numbers reach 1e6, as for the other evaluations."""
import math

import numpy as np
import pytest

from workloads import Stream

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PARAM = np.dtype([("kind", "<i4"), ("n_choices", "<i4"), ("lo", "<f4"), ("hi", "<f4")])
CATEGORICAL, CONTINUOUS = 2, 3


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_04323_gb300 as pkg
    pkg.build()
    from paper_2408_04323_gb300 import scoot
    return scoot


def inputs(n, d, M, starts):
    st = Stream(17 * n + d, "mle cluster")
    space = np.zeros(d, PARAM)
    space["kind"], space["hi"] = CONTINUOUS, 1.0
    space[1] = (CATEGORICAL, 3, 0, 0)
    u = st.uniform(d * n).reshape(d, n).astype(np.float32)
    words = u.view(np.int32).copy()
    words[1] = (u[1] * 3).astype(np.int32)
    y = st.normal(M * n).reshape(M, n).astype(np.float32)
    theta = 0.4 * st.normal(starts * M * (d + 2)).reshape(starts, M, d + 2)
    theta[..., d + 1] -= 3.0
    return space, words, u, y, theta


def reference(words, u, y, theta, kernel):
    d, n = words.shape
    th = torch.from_numpy(theta).cuda()
    x = torch.from_numpy(u.astype(np.float64)).cuda()
    parts = torch.stack([(torch.from_numpy((words[c][:, None] != words[c][None]).astype(np.float64)).cuda() if c == 1
                          else (x[c][:, None] - x[c][None]) ** 2) for c in range(d)])
    yy = torch.from_numpy(y.astype(np.float64)).cuda()
    il2, sf2, tau2 = torch.exp(-2 * th[..., :d]), th[..., d].exp(), th[..., d + 1].exp()
    r = torch.einsum("smc,cij->smij", il2, parts).sqrt()
    a = math.sqrt(3.0 if kernel else 5.0) * r
    k, dk = ((1 + a) * torch.exp(-a), -1.5 * torch.exp(-a)) if kernel else \
        ((1 + a + a * a / 3) * torch.exp(-a), -(5 / 6) * (1 + a) * torch.exp(-a))
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    L = torch.linalg.cholesky(sf2[..., None, None] * k + tau2[..., None, None] * eye)
    Ki = torch.cholesky_solve(eye.expand_as(L), L)
    al = torch.einsum("smij,mj->smi", Ki, yy)
    w = 0.5 * (al[..., :, None] * al[..., None, :] - Ki)
    g = torch.empty_like(th)
    g[..., :d] = -2 * sf2[..., None] * il2 * torch.einsum("smij,cij->smc", dk * w, parts)
    g[..., d] = sf2 * (w * k).sum((-1, -2))
    g[..., d + 1] = tau2 * torch.diagonal(w, dim1=-2, dim2=-1).sum(-1)
    logdet = 2 * torch.diagonal(L, dim1=-2, dim2=-1).log().sum(-1)
    return -0.5 * (al * yy).sum(-1) - 0.5 * logdet - 0.5 * n * math.log(2 * math.pi), g


def run(S, space, words, y, theta, kernel):
    starts, M, P = theta.shape
    th, g = (torch.full((starts, M, P), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
    lml = torch.zeros((starts, M), dtype=torch.float64, device="cuda")
    with S.Context(0) as ctx:
        S.scoot_gp_mle(ctx, space, torch.from_numpy(words).cuda(), words.shape[1], torch.from_numpy(y).cuda(),
                       torch.from_numpy(theta).cuda(), np.full(P, -100.0), np.full(P, 100.0), (1 << P) - 1, 0, 0.05, th,
                       lml, g, kernel=kernel)
        ctx.check()
    return th, lml, g


@pytest.mark.parametrize("n,d,M,starts,kernel", [
    (1, 2, 1, 1, 0), (2, 3, 2, 3, 1), (7, 4, 1, 2, 0), (8, 4, 2, 2, 1), (9, 16, 1, 2, 0), (63, 5, 2, 2, 0), (64, 5, 1, 3, 1),
    (65, 5, 1, 2, 0), (136, 8, 4, 5, 0), (199, 16, 1, 2, 1), (200, 3, 1, 2, 0), (288, 4, 1, 1, 0), (640, 4, 1, 1, 1),
    # the last and first n of each use of shared memory: two CTAs per SM, one that keeps the covariances, one that does
    # not, the kernel of one block per fit
    (212, 4, 1, 2, 1), (213, 4, 1, 1, 0), (317, 4, 1, 1, 0), (318, 4, 1, 1, 1), (325, 4, 1, 1, 0), (326, 4, 1, 1, 0),
    (506, 4, 1, 1, 1), (507, 4, 1, 1, 0), (264, 16, 1, 1, 0), (265, 16, 1, 1, 1), (300, 16, 1, 1, 0), (301, 16, 1, 1, 0),
    (442, 16, 1, 1, 0), (443, 16, 1, 1, 1),
    # enough fits of few observations for a block each, with the matrices in shared memory
    (1, 2, 2, 64, 0), (17, 5, 2, 64, 1), (64, 4, 1, 152, 0), (100, 16, 1, 152, 0), (110, 3, 1, 152, 1),
])
def test_evaluation(S, n, d, M, starts, kernel):
    space, words, u, y, theta = inputs(n, d, M, starts)
    th, lml, g = run(S, space, words, y, theta, kernel)
    want, wg = reference(words, u, y, theta, kernel)
    assert torch.equal(th.cpu(), torch.from_numpy(theta))
    worst = max(float(((lml - want).abs() / (1 + want.abs())).max()), float(((g - wg).abs() / (1 + wg.abs())).max()))
    print(f"mle n={n} d={d}: {worst:.2e}")
    assert worst <= 1e-9


@pytest.mark.parametrize("n", [24, 200])
def test_not_positive_definite(S, n):
    space, words, _, y, theta = inputs(n, 3, 1, 2)
    words[:, 10:14] = words[:, 9:10]      # equal observations ...
    theta[1, :, 4] = -90.0                # ... and no noise, in the second start alone
    _, lml, g = run(S, space, words, y, theta, 0)
    assert torch.isfinite(lml[0, 0]) and torch.isfinite(g[0]).all()
    assert lml[1, 0] == -math.inf and (g[1] == 0).all()


@pytest.mark.parametrize("n,d", [(16, 3), (100, 5), (200, 4)])
@pytest.mark.parametrize("noise", [1e-5, 1e-7])
def test_repeated_observations(S, n, d, noise):
    """Half of the observations repeat the other half and the noise is small: pivots of
    the noise's size.  Bar, relative to the largest value: 8 n u / noise (u = 2^-53), the
    rounding of a pivot of that size, twice, and of the n terms of each sum."""
    space, words, u, y, theta = inputs(n, d, 2, 2)
    order = np.argsort(Stream(n, "mle repeats").uniform(n))
    for a in (words, u):
        a[:, n // 2:] = a[:, :n - n // 2]
        a[:] = a[:, order]
    theta[..., d + 1] = math.log(noise)
    _, lml, g = run(S, space, words, y, theta, 0)
    want, wg = reference(words, u, y, theta, 0)
    worst = max(float(((lml - want).abs() / want.abs()).max()),
                float(((g - wg).abs() / wg.abs().amax(-1, keepdim=True)).max()))
    print(f"mle repeated n={n} noise={noise}: {worst:.2e}")
    assert worst <= 8 * n * 2.0 ** -53 / noise
