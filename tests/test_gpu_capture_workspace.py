"""Calls without a mask need no workspace on their fused kernels: captured as a
context's first call, when nothing may be allocated, they still run, and replay.
Captured on a context that has a workspace they use it, and replay after later calls
have taken a larger one."""
import numpy as np
import pytest

from workloads import Stream, make_instance, seeds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["ehvi", "exact"])
def test_first_call_captured(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_04323_gb300 as pkg
    pkg.build()
    from paper_2408_04323_gb300 import scoot as S
    inst = make_instance("d10-ehvi3", seeds("d10-ehvi3")[0], n_cand=16384)
    n, M = inst.n_cand, inst.n_obj
    L = S.scoot_gp_layout_init(inst.space, inst.n_obs, M, 0)
    blob, _ = S.scoot_gp_prepare(inst.space, inst.x_obs, inst.y_obs, inst.lengthscale, inst.signal_var, inst.noise_var, L)
    lo, hi, _ = S.scoot_boxes_build(inst.y_obs, inst.ref)
    grid, n_grid, corner = S.scoot_boxes_index(lo, hi)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()
    state, cand, lo, hi, grid = dev(blob), dev(inst.cand.view(np.int32)), dev(lo), dev(hi), dev(grid)
    corner, eps = dev(corner.view(np.int32)), dev(Stream(1, "eps").normal(32 * M).reshape(32, M).astype(np.float32))

    def run(ctx, acq):
        if call == "ehvi":
            S.scoot_score_ehvi(ctx, L, state, cand, n, lo, hi, eps, acq)
        else:
            S.scoot_score_ehvi_exact(ctx, L, state, cand, n, grid, n_grid, corner, acq)
    want, got = torch.empty(n, device="cuda"), torch.full((n,), 7.0, device="cuda")
    with S.Context(0) as fused:  # (also loads the kernels)
        S.scoot_ctx_set_tensor_cores(fused, 0)
        run(fused, want)
        fused.check()
    with S.Context(0) as ctx:
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            run(ctx, got)
        for _ in range(2):
            got.fill_(7.0)
            graph.replay()
            torch.cuda.synchronize()
            ctx.check()
            assert torch.equal(got, want)  # the fused kernel took the call


@pytest.mark.parametrize("call", ["posterior", "ehvi", "exact", "ehvi masked", "forest"])
def test_graph_outlives_growth(call):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_04323_gb300 as pkg
    pkg.build()
    from paper_2408_04323_gb300 import scoot as S
    inst = make_instance("d10-ehvi3", seeds("d10-ehvi3")[0], n_cand=1 << 18)
    small, M = 16384, inst.n_obj
    w = inst.workload
    L = S.scoot_gp_layout_init(inst.space, inst.n_obs, M, 0)
    blob, _ = S.scoot_gp_prepare(inst.space, inst.x_obs, inst.y_obs, inst.lengthscale, inst.signal_var, inst.noise_var, L)
    lo, hi, _ = S.scoot_boxes_build(inst.y_obs, inst.ref)
    grid, n_grid, corner = S.scoot_boxes_index(lo, hi)
    FL = S.scoot_forest_layout_init(inst.nodes, inst.tree_offset, inst.d, w.leaf_scale)
    forest = S.scoot_forest_pack(FL, inst.nodes, inst.tree_offset)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()
    state, cand, lo, hi, grid, forest = dev(blob), dev(inst.cand.view(np.int32)), dev(lo), dev(hi), dev(grid), dev(forest)
    corner, eps = dev(corner.view(np.int32)), dev(Stream(1, "eps").normal(32 * M).reshape(32, M).astype(np.float32))
    mask = dev((Stream(2, "mask").uniform(inst.n_cand) < 0.5).astype(np.uint8))
    outs = [torch.zeros((2 * M, inst.n_cand), device="cuda") for _ in range(3)]
    votes = [torch.zeros(inst.n_cand, dtype=torch.int32, device="cuda") for _ in range(3)]

    def run(ctx, n, k):
        out = outs[k]
        if call == "posterior":
            S.scoot_gp_posterior(ctx, L, state, cand, n, out[:M], out[M:])
        elif call == "exact":
            S.scoot_score_ehvi_exact(ctx, L, state, cand, n, grid, n_grid, corner, out[0])
        elif call == "forest":
            S.scoot_rf_predict(ctx, FL, forest, inst.space, cand, n, 10, 20, votes[k])
        else:
            S.scoot_score_ehvi(ctx, L, state, cand, n, lo, hi, eps, out[0], mask if "masked" in call else None)
    with S.Context(0) as ctx:
        n = inst.n_cand if call == "forest" else small  # (ranked from about 2^18 on)
        run(ctx, n, 0)
        run(ctx, n, 0)
        ctx.check()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph):
            run(ctx, n, 1)
        run(ctx, inst.n_cand, 2)      # takes a larger workspace
        S.scoot_score_ehvi(ctx, L, state, cand, inst.n_cand, lo, hi, eps, outs[2][0], mask)
        ballast = torch.full((64 << 20,), 1e30, device="cuda")  # where a freed one may have been
        for _ in range(2):
            outs[1].zero_()
            votes[1].zero_()
            graph.replay()
            torch.cuda.synchronize()
            ctx.check()
            assert torch.equal(outs[1], outs[0]) and torch.equal(votes[1], votes[0])
        assert (outs[1] != 0).any() or (votes[1] != 0).any()
        del ballast
