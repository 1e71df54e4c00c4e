"""The closed-form EHVI of large pools on the tensor-core posterior, at the smallest
pools that take it, against the oracle.

Bar: that of the fused kernel's test (propagated posterior tolerance and the closed
form's own fp32 rounding)."""
import numpy as np
import pytest

import oracle as O
from parity_tol import posterior_tols, propagated_tol
from test_gpu_ehvi_exact import S, box_inputs, ctx, dev, np_, rounding_tol, torch  # noqa: F401
from workloads import Stream, make_instance, seeds

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n_cand,masked", [("d10-ehvi3", 16384, True), ("d10-ehvi3", 16385, False),
                                                ("d12-fantasy", 16384, False)])
def test_exact_on_tensor_cores(S, ctx, name, n_cand, masked):  # noqa: F811
    inst = make_instance(name, seeds(name)[1], n_cand=n_cand)
    n, M = inst.n_cand, inst.n_obj
    L = S.scoot_gp_layout_init(inst.space, inst.n_obs, M, 0)
    blob, _ = S.scoot_gp_prepare(inst.space, inst.x_obs, inst.y_obs, inst.lengthscale, inst.signal_var, inst.noise_var, L)
    lo, hi, grid, n_grid, corner = box_inputs(S, inst.y_obs, inst.ref)
    live = np.ones(n, bool) if not masked else Stream(5, "mask").uniform(n) < 0.4
    acq = torch.full((n,), 7.0, device="cuda")
    S.scoot_score_ehvi_exact(ctx, L, dev(blob), dev(inst.cand.view(np.int32)), n, grid, n_grid, corner, acq,
                             dev(live.astype(np.uint8)) if masked else None)
    ctx.check()
    g = np_(acq)
    assert (g[~live] == -np.inf).all() and np.isfinite(g[live]).all()
    idx = np.nonzero(live)[0]
    idx = idx[np.unique(np.linspace(0, len(idx) - 1, 150).astype(int))]
    gps = [O.GP(inst.space, inst.x_obs, inst.y_obs[m], inst.lengthscale[m], inst.signal_var[m], inst.noise_var[m], 0)
           for m in range(M)]
    mu, var, e_mu, e_var = posterior_tols(gps, np.ascontiguousarray(inst.cand[:, idx]))
    front = O.pareto_front(inst.y_obs.T, inst.ref)
    want, tol = propagated_tol(lambda a, b: O.ehvi_analytic(a, b, front, inst.ref), mu, var, e_mu, e_var)
    ratio = np.abs(g[idx] - want) / (tol + rounding_tol(mu, var, lo, hi))
    print(f"{name} n={n}: max|err|/tol={ratio.max():.3f}")
    assert ratio.max() <= 1.0
