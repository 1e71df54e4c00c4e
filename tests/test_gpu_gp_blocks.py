"""The blocked factorisation of the GP state at the edges of its blocks of eight
pivots and of its cluster (549 observations; 550 take the other kernel), against
the host-built state.

Bars: those of the device-built state's other tests (tables without a
factorisation one fp32 rounding, alpha and L^{-1} 1e-6 of the largest entry:
two fp64 orders at condition numbers up to 1e6 and one fp32 rounding)."""
import numpy as np
import pytest

from test_gpu_gp_device import S, compare_tables, ctx, device_blob, host_blob, torch  # noqa: F401
from workloads import Stream, make_instance, seeds
from workloads.generate import draw_configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_obs", [8, 9, 15, 16, 17, 191, 200, 385, 549, 550])
def test_device_state_blocks(S, ctx, n_obs):  # noqa: F811
    inst = make_instance("d8-ehvi2", seeds("d8-ehvi2")[0], n_cand=4096)
    w, st = inst.workload, Stream(n_obs, "gp-device-blocks")

    class Inst:
        space, lengthscale, signal_var = inst.space, inst.lengthscale, inst.signal_var
        x_obs = draw_configs(w, st, n_obs)
        y_obs = st.normal(w.n_obj * n_obs).reshape(w.n_obj, n_obs).astype(np.float32)
        noise_var = np.maximum(inst.noise_var, np.float32(1e-3))
    L = S.scoot_gp_layout_init(Inst.space, n_obs, w.n_obj, 0)
    db = device_blob(S, ctx, Inst, L)
    compare_tables(L, host_blob(S, Inst, L), db.cpu().numpy().tobytes(), f"n={n_obs}")
