"""The blocked factorisation of the GP state at the edges of its blocks of eight
pivots and of its cluster (549 observations; 550 take the other kernel), against
the host-built state.

Bars: those of the device-built state's other tests (tables without a
factorisation one fp32 rounding, alpha and L^{-1} 1e-6 of the largest entry:
two fp64 orders at condition numbers up to 1e6 and one fp32 rounding)."""
import numpy as np
import pytest

from test_gpu_gp_device import S, compare_tables, ctx, device_blob, host_blob, region, torch  # noqa: F401
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


@pytest.mark.parametrize("n_obs", [16, 100, 200])
@pytest.mark.parametrize("noise", [1e-6, 1e-8])
def test_repeated_observations(S, ctx, n_obs, noise):  # noqa: F811
    """Half of the observations repeat the other half with other results and little
    noise, so the pivots of the repeats are of the noise's size and the blocks that
    hold a pair are all but singular.  Bar: the same 1e-6.  The elimination's error is
    that of a pivot, u / noise of it (1e-8 at the smallest noise; against 80 bits 6e-11
    to 1e-8 measured on the CPU for eliminations pivot by pivot, and 1e-5 to 0.1 where
    blocks of eight were inverted)."""
    inst = make_instance("d8-ehvi2", seeds("d8-ehvi2")[0], n_cand=4096)
    w, st = inst.workload, Stream(n_obs, "gp-device-repeats")
    x = draw_configs(w, st, n_obs)
    x[:, n_obs // 2:] = x[:, :n_obs - n_obs // 2]

    class Inst:
        space, lengthscale, signal_var = inst.space, inst.lengthscale, inst.signal_var
        x_obs = np.ascontiguousarray(x[:, np.argsort(st.uniform(n_obs))])
        y_obs = st.normal(w.n_obj * n_obs).reshape(w.n_obj, n_obs).astype(np.float32)
        noise_var = np.full_like(inst.noise_var, noise)
    L = S.scoot_gp_layout_init(Inst.space, n_obs, w.n_obj, 0)
    db = device_blob(S, ctx, Inst, L).cpu().numpy().tobytes()
    hb = host_blob(S, Inst, L)
    # (no comparison of zeros: an entry between repeats may cancel to 0 in one order and to 1e-16 in the other)
    for off, count in ((L.off_alpha, L.n_obj * n_obs), (L.off_linv, L.n_obj * L.n_tiles * 2048)):
        host, got = (region(b, off, count).astype(np.float64) for b in (hb, db))
        worst = np.abs(got - host).max() / np.abs(host).max()
        print(f"repeated n={n_obs} noise={noise}: {worst:.2e}")
        assert worst <= 1e-6
