"""The Monte-Carlo EHVI over three objectives that visits only the boxes a
sample reaches, against the sum over all boxes in 64 bits from the oracle's
moments: builder's boxes, boxes it has to refuse (another order, a floor that
rises, too few), odd pools and sample counts at the edges of its batches.

Bar: the propagated posterior tolerance of the other acquisition tests; the
terms are not negative, so the order and number of the additions costs at most
2 u (B + S) of the sum more (u = 2^-24)."""
import numpy as np
import pytest

from workloads import Stream, make_instance

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from parity_tol import posterior_tols, propagated_tol  # noqa: E402

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


def all_boxes(mu, var, eps, lo, hi):
    """EHVI of moments [K][3] over every box, in 64 bits."""
    mu, sd = dev(mu), dev(np.sqrt(np.maximum(var, 0.0)))
    y = [mu[:, m, None] + sd[:, m, None] * eps[None, :, m] for m in range(3)]
    total = torch.zeros_like(y[0])
    for b in range(len(lo)):
        p = 1.0
        for m in range(3):
            p = p * (torch.clamp(y[m], max=float(hi[b, m])) - float(lo[b, m])).clamp(min=0)
        total += p
    return total.mean(1).cpu().numpy()


@pytest.mark.parametrize("n_cand,n_mc,boxes,masked", [
    (9001, 128, "built", True), (4099, 1, "built", False), (4096, 33, "built", True), (3907, 1024, "built", False),
    (5000, 300, "built", True), (1, 128, "built", False), (8192, 64, "shuffled", True), (8192, 64, "risen", True),
    (8192, 64, "few", False),
    # (the smallest pools that take the walk at their number of samples, and boxes refused there)
    (9600, 128, "built", True), (1203301, 1, "built", False), (36503, 33, "built", True), (4096, 1024, "built", False),
    (20001, 64, "shuffled", True), (20001, 64, "risen", False),
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
    gps = [O.GP(inst.space, inst.x_obs, inst.y_obs[m], inst.lengthscale[m], float(inst.signal_var[m]),
                float(inst.noise_var[m])) for m in range(3)]
    mu, v, e_mu, e_var = posterior_tols(gps, inst.cand[:, at.cpu().numpy()])
    e = dev(eps.astype(np.float64))
    want, tol = propagated_tol(lambda a, b: all_boxes(a, b, e, lo, hi), mu, v, e_mu, e_var)
    tol = tol + 2 * U32 * (len(lo) + n_mc) * want
    worst = float((np.abs(acq[at].cpu().numpy().astype(np.float64) - want) / tol).max())
    print(f"{boxes} n={n_cand} S={n_mc}: {worst:.3f} of the tolerance")
    assert worst <= 1.0
