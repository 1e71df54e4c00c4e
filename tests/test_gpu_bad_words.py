"""Candidates whose covariance inputs are not finite (a NaN or infinite continuous
word, a zero or negative word of a log-uniform integer) on every route of the
posterior: the mean is NaN and the variance 0, which the acquisitions take for no
improvement, whether the tensor cores compute it (any number of observations, with
either square root and exponential) or the fp32 kernels do."""
import numpy as np
import pytest

from test_gpu_gp_device import S, ctx, dev, host_blob, torch  # noqa: F401
from workloads import CONTINUOUS, INT_LOG, Stream, make_instance, seeds
from workloads.generate import draw_configs

pytestmark = pytest.mark.gpu
N = 16384 + 5


def bad_pool(base):
    """The workload's pool with bad words in every 64th candidate, and which those are."""
    kinds = [int(k) for k in base.space["kind"]]
    real, log_int = kinds.index(CONTINUOUS), kinds.index(INT_LOG)
    cand = base.cand.copy()
    bad = np.arange(N) % 64 == 9
    for k, i in enumerate(np.nonzero(bad)[0]):
        if k % 5 < 3:
            cand[real, i] = np.float32((np.nan, np.inf, -np.inf)[k % 5]).view(np.uint32)
        else:
            cand[log_int, i] = np.int32((0, -7)[k % 5 - 3]).view(np.uint32)
    return cand, torch.from_numpy(bad).cuda()


@pytest.mark.parametrize("name,n_obs", [("d8-ehvi2", 100), ("d10-ehvi3", 200), ("d8-ehvi2", 256), ("d8-ehvi2", 257),
                                        ("d10-ei", 513)])
@pytest.mark.parametrize("tc", [1, 0], ids=["tensor", "fp32"])
def test_bad_words(S, ctx, name, n_obs, tc):  # noqa: F811
    base = make_instance(name, seeds(name)[0], n_cand=N)
    w, st = base.workload, Stream(n_obs, "bad words")

    class Inst:
        space, lengthscale, signal_var = base.space, base.lengthscale, base.signal_var
        x_obs = draw_configs(w, st, n_obs)
        y_obs = st.normal(w.n_obj * n_obs).reshape(w.n_obj, n_obs).astype(np.float32)
        noise_var = np.maximum(base.noise_var, np.float32(1e-3))
    M = w.n_obj
    L = S.scoot_gp_layout_init(Inst.space, n_obs, M, 0)
    state = dev(np.frombuffer(bytes(host_blob(S, Inst, L)), np.uint8).copy())
    words, bad = bad_pool(base)
    cand = dev(words.view(np.int32))
    mean, var = (torch.full((M, N), 7.0, device="cuda") for _ in range(2))
    acq = torch.full((N,), 7.0, device="cuda")
    S.scoot_ctx_set_tensor_cores(ctx, tc)
    try:
        S.scoot_gp_posterior(ctx, L, state, cand, N, mean, var)
        assert mean[:, bad].isnan().all() and (var[:, bad] == 0).all()
        assert mean[:, ~bad].isfinite().all() and var[:, ~bad].isfinite().all()
        S.scoot_score_ei(ctx, L, state, cand, N, 0.01, acq)
        assert (acq[bad] == 0).all() and acq[~bad].isfinite().all()
        three = torch.full((3, N), 7.0, device="cuda")
        S.scoot_score_mace(ctx, L, state, cand, N, 0.01, 2.0, three)
        assert three[0, bad].isnan().all() and (three[1:, bad] == 0).all() and three[:, ~bad].isfinite().all()
        if M > 1:
            lo, hi, _ = S.scoot_boxes_build(base.y_obs, base.ref)
            eps = dev(st.normal(128 * M).reshape(128, M).astype(np.float32))
            acq.fill_(7.0)
            S.scoot_score_ehvi(ctx, L, state, cand, N, dev(lo), dev(hi), eps, acq)
            assert (acq[bad] == 0).all() and acq[~bad].isfinite().all()
            grid, n_grid, corner = S.scoot_boxes_index(lo, hi)
            acq.fill_(7.0)
            S.scoot_score_ehvi_exact(ctx, L, state, cand, N, dev(grid), n_grid, dev(corner.view(np.int32)), acq)
            assert (acq[bad] == 0).all() and acq[~bad].isfinite().all()
    finally:
        S.scoot_ctx_set_tensor_cores(ctx, 1)
    ctx.check()
