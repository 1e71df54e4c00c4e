"""The ranked forest walk (large pools, trees and depths together) against a plain
float walk of the same nodes: thresholds that repeat, meet the feature values
exactly or differ in the last bit, signed zeros, infinities and NaN among the
features, one-node trees, sixteen features, and forests on both sides of the
largest that is ranked.  Whole numbers: every vote and mask is the same."""
import numpy as np
import pytest

from workloads import Stream

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NODE = np.dtype([("val", "<f4"), ("left", "<u2"), ("feat", "u1"), ("flags", "u1")])
PARAM = np.dtype([("kind", "<i4"), ("n_choices", "<i4"), ("lo", "<f4"), ("hi", "<f4")])
CONTINUOUS = 3


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_04323_gb300 as pkg
    pkg.build()
    from paper_2408_04323_gb300 import scoot
    return scoot


def tree(st, d, size, grid, chain):
    """A random tree of `size` nodes (odd), children next to each other: breadth first, or one long path whose
    side alternates."""
    nodes = np.zeros(size, NODE)
    u = st.uniform(3 * size).reshape(3, size)
    nodes["val"], nodes["flags"] = np.floor(u[2] * 256), 1
    nxt, i = 1, 0
    while nxt < size:
        nodes[i] = (grid[int(u[0, i] * len(grid))], nxt, int(u[1, i] * d), 0)
        i = nxt + (nxt // 2) % 2 if chain else i + 1
        nxt += 2
    return nodes


@pytest.mark.parametrize("n,d,trees,size,distinct,chain", [
    (1 << 19, 16, 40, 81, 9, True), ((1 << 19) + 4465, 12, 320, 51, 600, False), ((1 << 19) + 1, 1, 6, 2729, 100000, True),
    ((1 << 19) + 35, 3, 6, 2727, 40, True), ((1 << 18) - 1, 5, 20, 63, 50, False),
])
def test_ranked_walk_equals_float_walk(S, n, d, trees, size, distinct, chain):
    st = Stream(1000 * d + trees, "ranked")
    grid = np.concatenate([[0.0, -0.0, 1.0, np.nextafter(np.float32(1), np.float32(2))], st.normal(distinct)]).astype(np.float32)
    parts = [tree(st, d, size, grid, chain) for _ in range(trees - 1)] + [tree(st, d, 1, grid, chain)]
    offs = np.zeros(trees + 1, np.int32)
    offs[1:] = np.cumsum([len(p) for p in parts])
    nodes = np.concatenate(parts)
    ld = (n + 3) // 4 * 4
    x = st.normal(d * ld).reshape(d, ld).astype(np.float32)
    x[:, ::3] = grid[(st.uniform(d * x[:, ::3].shape[1]) * len(grid)).astype(int)].reshape(d, -1)
    x[:, 7], x[:, 11], x[:, 13], x[:, 17] = np.nan, np.inf, -np.inf, -0.0
    space = np.zeros(d, PARAM)
    space["kind"], space["lo"], space["hi"] = CONTINUOUS, -10, 10
    L = S.scoot_forest_layout_init(nodes, offs, d, 255)
    blob = torch.from_numpy(S.scoot_forest_pack(L, nodes, offs)).cuda()
    cand = torch.from_numpy(x.view(np.int32)).cuda()
    mask0 = (st.uniform(n) < 0.7).astype(np.uint8)
    mask, votes = torch.from_numpy(mask0).cuda(), torch.full((n,), -1, dtype=torch.int32, device="cuda")
    free = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    with S.Context(0) as ctx:
        S.scoot_rf_predict(ctx, L, blob, space, cand, n, 1, 2, votes, mask, count)
        S.scoot_rf_predict(ctx, L, blob, space, cand, n, 1, 2, free)
        ctx.check()
    xs = torch.from_numpy(x[:, :n]).cuda()
    val, left, feat, leaf = (torch.from_numpy(nodes[f].astype(t)).cuda()
                             for f, t in (("val", np.float32), ("left", np.int64), ("feat", np.int64), ("flags", np.bool_)))
    want = torch.zeros(n, dtype=torch.int64, device="cuda")
    for t in range(trees):
        node = torch.full((n,), int(offs[t]), dtype=torch.int64, device="cuda")
        for _ in range(L.max_depth):
            go = ~(xs.gather(0, feat[node][None])[0] <= val[node])
            node = torch.where(leaf[node], node, int(offs[t]) + left[node] + go)
        want += val[node].long()
    live = torch.from_numpy(mask0).cuda().bool()
    assert torch.equal(free.long(), want)
    assert torch.equal(votes.long(), torch.where(live, want, 0))
    ok = live & (2 * want >= 255 * trees)
    assert torch.equal(mask.bool(), ok) and int(count.item()) == int(ok.sum())


@pytest.mark.parametrize("size,depth", [(255, 7), (13, 3)])
def test_both_sides_of_the_shortest_list(S, size, depth):
    """A masked call leaves the choice of the walk to the device: one live candidate
    fewer than the ranked walk takes, as many, none and all give the votes of the
    unmasked walk of a small pool."""
    n, d, trees = 1 << 20, 6, 180
    st = Stream(size, "ranked lists")
    grid = st.normal(50).astype(np.float32)
    parts = [tree(st, d, size, grid, False) for _ in range(trees)]
    offs = np.arange(trees + 1, dtype=np.int32) * size
    if size * trees > 16380:  # within the ranked walk's nodes
        keep = 16380 // size
        parts, offs, trees = parts[:keep], offs[:keep + 1], keep
    nodes = np.concatenate(parts)
    space = np.zeros(d, PARAM)
    space["kind"], space["lo"], space["hi"] = CONTINUOUS, -10, 10
    L = S.scoot_forest_layout_init(nodes, offs, d, 255)
    assert L.max_depth >= depth
    blob = torch.from_numpy(S.scoot_forest_pack(L, nodes, offs)).cuda()
    cand = torch.from_numpy(st.normal(d * n).reshape(d, n).astype(np.float32).view(np.int32)).cuda()
    edge = -(-400000000 // (trees * (L.max_depth + 1)))
    want = torch.empty(n, dtype=torch.int32, device="cuda")
    with S.Context(0) as ctx:
        for at in range(0, n, 1 << 16):  # pools that are not ranked
            S.scoot_rf_predict(ctx, L, blob, space, cand[:, at:at + (1 << 16)].contiguous(), 1 << 16, 1, 2,
                               want[at:at + (1 << 16)])
        order = torch.randperm(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        for live in (0, 1, edge - 1, edge, n):
            assert live <= n
            mask0 = torch.zeros(n, dtype=torch.uint8, device="cuda")
            mask0[order[:live]] = 1
            mask, votes = mask0.clone(), torch.full((n,), -1, dtype=torch.int32, device="cuda")
            count = torch.zeros(1, dtype=torch.int64, device="cuda")
            S.scoot_rf_predict(ctx, L, blob, space, cand, n, 1, 2, votes, mask, count)
            ctx.check()
            on = mask0.bool()
            assert torch.equal(votes, torch.where(on, want, 0))
            ok = on & (2 * want.long() >= 255 * trees)
            assert torch.equal(mask.bool(), ok) and int(count.item()) == int(ok.sum())
