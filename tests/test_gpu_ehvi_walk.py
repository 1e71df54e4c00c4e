"""The Monte-Carlo EHVI over three objectives that visits only the boxes a
sample reaches, against the sum over all boxes in 64 bits from the same
moments: builder's boxes, boxes it has to refuse (another order, a floor that
rises, too few), odd pools and sample counts at the edges of its batches.

Bar: the terms are not negative, so the order and number of the additions
costs at most 2 u (B + S) of the sum (u = 2^-24); a sample's coordinate carries
4 u (|mu| + |eps| sigma + |edge|), whose effect is taken by moving each
objective by that much."""
import numpy as np
import pytest

from workloads import Stream, make_instance

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_04323_gb300 as pkg
    pkg.build()
    from paper_2408_04323_gb300 import scoot
    return scoot


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def all_boxes(mu, sd, eps, lo, hi, shift=None):
    y = [mu[m][:, None] + sd[m][:, None] * eps[None, :, m] for m in range(3)]
    if shift is not None:
        y[shift[0]] = y[shift[0]] + shift[1]
    total = torch.zeros_like(y[0])
    for b in range(len(lo)):
        p = 1.0
        for m in range(3):
            p = p * (torch.clamp(y[m], max=float(hi[b, m])) - float(lo[b, m])).clamp(min=0)
        total += p
    return total.mean(1)


@pytest.mark.parametrize("n_cand,n_mc,boxes,masked", [
    (9001, 128, "built", True), (4099, 1, "built", False), (4096, 33, "built", True), (3907, 1024, "built", False),
    (5000, 300, "built", True), (1, 128, "built", False), (8192, 64, "shuffled", True), (8192, 64, "risen", True),
    (8192, 64, "few", False),
])
def test_walk_equals_all_boxes(S, n_cand, n_mc, boxes, masked):
    inst = make_instance("d10-ehvi3", 1004, n_cand=n_cand)
    lo, hi, _ = S.scoot_boxes_build(inst.y_obs, inst.ref)
    assert len(lo) == 241
    if boxes == "shuffled":
        order = np.argsort(Stream(3, "order").uniform(len(lo)))
        lo, hi = lo[order], hi[order]
    elif boxes == "risen":
        lo = lo.copy()
        lo[len(lo) // 2, 2] = lo[:, 2].max()
    elif boxes == "few":
        lo, hi = lo[:90], hi[:90]
    lo, hi = np.ascontiguousarray(lo), np.ascontiguousarray(hi)
    eps = Stream(n_mc, "walk").normal(n_mc * 3).reshape(n_mc, 3).astype(np.float32)
    with S.Context(0) as ctx:
        layout = S.scoot_gp_layout_init(inst.space, inst.n_obs, 3)
        blob, _ = S.scoot_gp_prepare(inst.space, inst.x_obs, inst.y_obs, inst.lengthscale, inst.signal_var,
                                     inst.noise_var, layout)
        blob, cand = dev(blob), dev(inst.cand.view(np.int32))
        mask = dev((Stream(5, "mask").uniform(n_cand) < 0.6).astype(np.uint8)) if masked else None
        mean, var = (torch.zeros((3, n_cand), device="cuda") for _ in range(2))
        S.scoot_gp_posterior(ctx, layout, blob, cand, n_cand, mean, var)
        acq = torch.full((n_cand,), 7.0, device="cuda")
        S.scoot_score_ehvi(ctx, layout, blob, cand, n_cand, dev(lo), dev(hi), dev(eps), acq, mask)
        again = torch.zeros_like(acq)
        S.scoot_score_ehvi(ctx, layout, blob, cand, n_cand, dev(lo), dev(hi), dev(eps), again, mask)
        ctx.check()
    assert torch.equal(acq, again)
    live = torch.ones(n_cand, dtype=torch.bool, device="cuda") if mask is None else mask.bool()
    assert (acq[~live] == -np.inf).all()
    at = live.nonzero()[:, 0]
    at = at[torch.linspace(0, len(at) - 1, min(len(at), 400)).long().cuda()]
    mu, sd, e = mean[:, at].double(), var[:, at].double().sqrt(), dev(eps.astype(np.float64))
    want = all_boxes(mu, sd, e, lo, hi)
    edge = max(np.abs(lo).max(), np.abs(hi[np.isfinite(hi)]).max())
    tol = 2 * U32 * (len(lo) + n_mc) * want
    for m in range(3):
        d = 4 * U32 * (mu[m][:, None].abs() + sd[m][:, None] * e[None, :, m].abs() + float(edge))
        tol = tol + all_boxes(mu, sd, e, lo, hi, (m, d)) - want
    worst = float(((acq[at].double() - want).abs() / tol.clamp(min=1e-30)).max())
    print(f"{boxes} n={n_cand} S={n_mc}: {worst:.3f} of the tolerance")
    assert worst <= 1.0
