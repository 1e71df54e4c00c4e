"""The tensor-core posterior of more than 256 observations, by groups of rows: its
moments against the oracle at the edges of the groups, with three objectives in
smaller groups (less shared memory left), and the masked calls and the
acquisitions built on it against the same moments.

Bars: the posterior's own; of the acquisitions of the same moments the roundings of
the two codes (u = 2^-24): EI moves by at most the change of mu and 0.4 that of
sigma, 8 u of what they are made of; the EHVI's terms are not negative, so its sums
may differ by 2 u (B + S), and a sample's rounding, 4 u R of values up to R, moves the
volume by at most that times the (2 R)^(M - 1) across it."""
import numpy as np
import pytest

import oracle as O  # noqa: F401
from test_gpu_gp_device import S, ctx, dev, host_blob, posterior_check, torch  # noqa: F401
from workloads import Stream, make_instance, seeds
from workloads.generate import draw_configs

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.mark.parametrize("name,n_obs,kernel", [("d8-ehvi2", 257, 0), ("d8-ehvi2", 320, 1), ("d8-ehvi2", 511, 0),
                                               ("d10-ehvi3", 513, 0), ("d10-ei", 640, 0), ("d12-fantasy", 640, 1)])
def test_long_histories(S, ctx, name, n_obs, kernel):  # noqa: F811
    base = make_instance(name, seeds(name)[0], n_cand=9729 + 128)
    w, st = base.workload, Stream(n_obs, "posterior-groups")

    class Inst:
        space, lengthscale, signal_var, cand, n_cand = (base.space, base.lengthscale, base.signal_var, base.cand,
                                                        base.n_cand)
        n_obj = w.n_obj
        x_obs = draw_configs(w, st, n_obs)
        y_obs = st.normal(w.n_obj * n_obs).reshape(w.n_obj, n_obs).astype(np.float32)
        noise_var = np.maximum(base.noise_var, np.float32(1e-3))
    n, M = Inst.n_cand, Inst.n_obj
    L = S.scoot_gp_layout_init(Inst.space, n_obs, M, kernel)
    state = dev(np.frombuffer(bytes(host_blob(S, Inst, L)), np.uint8).copy())
    posterior_check(S, ctx, Inst, L, state, f"{name} n={n_obs}", kernel, n_cand=n)
    cand = dev(Inst.cand.view(np.int32))
    mean, var, mean2, var2 = (torch.full((M, n), 7.0, device="cuda") for _ in range(4))
    mask = dev((st.uniform(n) < 0.4).astype(np.uint8))
    S.scoot_gp_posterior(ctx, L, state, cand, n, mean, var)
    S.scoot_gp_posterior(ctx, L, state, cand, n, mean2, var2, mask)
    live = mask.bool()
    for whole, part in ((mean, mean2), (var, var2)):
        assert torch.equal(part[:, live], whole[:, live]) and (part[:, ~live] == 7.0).all()
    got, want = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    S.scoot_score_ei(ctx, L, state, cand, n, 0.01, got, mask)
    S.scoot_acq_ei(ctx, mean[0], var[0], n, float(Inst.y_obs[0].max()), 0.01, want, mask)
    assert (got[~live] == -np.inf).all()
    sd0 = var[0].sqrt()
    assert ((got - want)[live].abs() <= (8 * U32 * (mean[0].abs() + abs(Inst.y_obs[0].max()) + 0.01 + sd0))[live]).all()
    if M > 1:
        lo, hi, _ = S.scoot_boxes_build(base.y_obs, base.ref)
        eps = dev(st.normal(64 * M).reshape(64, M).astype(np.float32))
        S.scoot_score_ehvi(ctx, L, state, cand, n, dev(lo), dev(hi), eps, got, mask)
        S.scoot_acq_ehvi(ctx, mean, var, n, dev(lo), dev(hi), eps, want, mask)
        assert (got[~live] == -np.inf).all()
        R = float(mean.abs().max() + var.max().sqrt() * eps.abs().max()) + np.abs(lo[np.isfinite(lo)]).max()
        bar = 2 * U32 * (len(lo) + 64) * want[live] + M * 4 * U32 * R * (2 * R) ** (M - 1)
        assert ((got - want)[live].abs() <= bar).all()
    ctx.check()


def test_refused_stays_refused(S, ctx):  # noqa: F811
    """A call whose boxes and samples do not fit beside a long history in the fused
    kernel is refused with the tensor cores on as with them off."""
    inst = make_instance("d8-ehvi2", seeds("d8-ehvi2")[0], n_cand=10000)
    n_obs, M = 640, inst.n_obj
    L = S.scoot_gp_layout_init(inst.space, n_obs, M, 0)
    state = torch.zeros(L.bytes, dtype=torch.uint8, device="cuda")
    cand, acq = dev(inst.cand.view(np.int32)), torch.empty(inst.n_cand, device="cuda")
    lo, hi, eps = (torch.zeros((k, M), device="cuda") for k in (4000, 4000, 1024))
    for on in (0, 1):
        S.scoot_ctx_set_tensor_cores(ctx, on)
        with pytest.raises(Exception, match="shared memory"):
            S.scoot_score_ehvi(ctx, L, state, cand, inst.n_cand, lo, hi, eps, acq)
