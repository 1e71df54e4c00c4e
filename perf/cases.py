"""The work that a user of this library has it do, as cases that can be timed and compared.

A tuner that follows Algorithm 1 spends its device time on
  * suggestion rounds over a candidate pool (ScoringRound.run): prune, forest, posterior, acquisition, top-q, with the
    acquisitions a user can choose (EI, MACE, Monte-Carlo EHVI with two or three objectives, exact EHVI, sequential
    fantasised EHVI picks);
  * the posterior by itself (scoot_gp_posterior), for instance with a history longer than 256 observations;
  * fitting between rounds: GP hyperparameters (scoot_gp_mle), the feasibility forest (scoot_rf_train) and the GP state
    on the device (scoot_gp_prepare_device).

The sizes are those of the repository's workloads (4 to 12 parameters, 16 to 256 observations, pools of 2^12 to 2^22),
with odd ones between them.  Inputs follow the workloads' recipe: inference-engine parameters (integer, log-integer,
categorical, continuous), smooth conflicting surfaces with a little noise, a forest grown by CART on crash labels.
exact() is plain torch in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2408_04323_gb300 import scoot as S
from paper_2408_04323_gb300.pipeline import RoundInputs, ScoringRound

PARAM = np.dtype([("kind", "<i4"), ("n_choices", "<i4"), ("lo", "<f4"), ("hi", "<f4")])
CLAUSE = np.dtype([("n_guard", "<i4"), ("guard_param", "<i4", (2,)), ("guard_value", "<i4", (2,)), ("n_term", "<i4"),
                   ("term_param", "<i4", (4,)), ("coef", "<i8", (4,)), ("rhs", "<i8")])
NODE = np.dtype([("val", "<f4"), ("left", "<u2"), ("feat", "u1"), ("flags", "u1")])

# Engine parameters in the order in which a space of d of them takes them: (kind, lo, hi, choices, weight in the
# synthetic memory budget).  Every d from 4 to 12 holds all the kinds that matter to the path.
PARAMS = (
    (S.INT_LOG, 64, 8192, 0, 1.0),          # maximum number of sequences
    (S.INT_LOG, 1024, 65536, 0, 0.5),       # maximum number of batched tokens
    (S.CATEGORICAL, 0, 0, 3, 0.0),          # block size
    (S.CONTINUOUS, 0.5, 0.95, 0, 1.0),      # memory utilisation
    (S.INT_UNIFORM, 1, 4, 0, -0.5),         # tensor parallelism
    (S.CATEGORICAL, 0, 0, 2, 0.0),          # chunked prefill
    (S.CATEGORICAL, 0, 0, 2, 0.0),          # prefix caching
    (S.CONTINUOUS, 0.0, 2.0, 0, 0.0),       # scheduler delay
    (S.CATEGORICAL, 0, 0, 2, 0.0),          # custom all-reduce
    (S.CATEGORICAL, 0, 0, 2, 0.0),          # block manager
    (S.INT_LOG, 256, 8192, 0, 0.0),         # sequence length to capture
    (S.INT_UNIFORM, 0, 16, 0, 0.3),         # swap space
)
LEAF_SCALE, DELTA_NUM, DELTA_DEN = 255, 10, 20
ROUNDS = ("ei", "mace", "ehvi", "ehvi-exact", "fantasy")
MLE_LR, MLE_STEPS = 0.05, 60


def listed():
    return [
        # the first rounds of a small tuning session: latency and launches are what counts
        {"name": "round-ehvi2-small", "kind": "ehvi", "d": 4, "n": 16, "N": 4096, "M": 2, "S": 32, "T": 16, "depth": 6, "q": 1},
        # an ordinary two-objective round
        {"name": "round-ehvi2", "kind": "ehvi", "d": 8, "n": 64, "N": 1 << 18, "M": 2, "S": 64, "T": 100, "depth": 10, "q": 4},
        # a single-objective round over a large pool
        {"name": "round-ei", "kind": "ei", "d": 10, "n": 128, "N": 1 << 20, "M": 1, "S": 1, "T": 100, "depth": 12, "q": 1},
        # tail latencies against throughput: three objectives, many boxes
        {"name": "round-ehvi3", "kind": "ehvi", "d": 10, "n": 200, "N": 1 << 20, "M": 3, "S": 128, "T": 128, "depth": 12, "q": 8},
        # parallel suggestion over the largest pool: the benchmark's workload
        {"name": "round-fantasy", "kind": "fantasy", "d": 12, "n": 256, "N": 1 << 22, "M": 2, "S": 64, "T": 200, "depth": 14, "q": 16},
        # the same on a small odd pool, a few picks
        {"name": "round-fantasy-odd", "kind": "fantasy", "d": 9, "n": 97, "N": 50003, "M": 2, "S": 64, "T": 100, "depth": 10, "q": 5},
        # the paper's own single-objective suggestion (MACE), odd sizes
        {"name": "round-mace-odd", "kind": "mace", "d": 10, "n": 90, "N": 300007, "M": 1, "S": 1, "T": 100, "depth": 12, "q": 4},
        # the paper's own covariance (Matern-3/2, warped inputs) with the closed-form EHVI, odd sizes
        {"name": "round-exact-warped", "kind": "ehvi-exact", "d": 8, "n": 75, "N": 99991, "M": 2, "S": 1, "T": 100, "depth": 10, "q": 3, "kernel": 1, "warp": True},
        # mean and variance with a long history (beyond what the tensor cores' accumulators hold at once)
        {"name": "posterior-long", "kind": "posterior", "d": 12, "n": 400, "N": 1 << 17, "M": 2},
        # hyperparameter fits between rounds, at the tuning loop's defaults (8 starts, 60 steps)
        {"name": "fit-mle", "kind": "mle", "d": 8, "n": 128, "M": 2, "starts": 8},
        # the feasibility forest retrained between rounds
        {"name": "fit-forest", "kind": "forest", "d": 12, "n": 256, "T": 200, "depth": 14},
        # the GP state built on the device
        {"name": "gp-state", "kind": "gp-state", "d": 10, "n": 200, "M": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("ehvi", "ehvi", "ehvi", "fantasy", "fantasy", "ei", "mace", "ehvi-exact", "posterior", "mle",
                       "forest", "gp-state"))
    c = {"kind": kind, "d": rng.randint(4, 12), "n": _log_int(rng, 8, 256)}
    if kind in ROUNDS:
        c["M"] = 1 if kind in ("ei", "mace") else 2 if kind != "ehvi" else rng.choice((2, 2, 3))
        c["N"] = _log_int(rng, 1000, 1 << 18 if c["M"] == 3 else 1 << 20)
        c["S"] = rng.choice((32, 64, 100, 128)) if kind in ("ehvi", "fantasy") else 1
        c["T"], c["depth"], c["q"] = rng.randint(16, 200), rng.randint(6, 14), rng.randint(1, 16)
        c["kernel"] = rng.randint(0, 1)
        if kind != "fantasy":
            c["warp"] = rng.random() < 0.2
    elif kind == "posterior":
        c.update(n=_log_int(rng, 16, 512), N=_log_int(rng, 1000, 1 << 17), M=rng.randint(1, 2), kernel=rng.randint(0, 1),
                 warp=rng.random() < 0.2)
    elif kind == "mle":
        c.update(n=_log_int(rng, 12, 120), M=rng.randint(1, 2), starts=rng.randint(2, 10), kernel=rng.randint(0, 1))
    elif kind == "forest":
        c.update(T=rng.randint(16, 200), depth=rng.randint(4, 14))
    else:
        c.update(n=_log_int(rng, 16, 256), M=rng.randint(1, 3), kernel=rng.randint(0, 1), warp=rng.random() < 0.2)
    return c


# ---------------------------------------------------------------------------------------------- inputs

def _space(d):
    a = np.zeros(d, PARAM)
    for i, (kind, lo, hi, k, _) in enumerate(PARAMS[:d]):
        a[i] = (kind, k, lo, hi)
    return a


def _clauses(d):
    """Batched tokens >= sequences; chunked prefill and prefix caching not both; without chunked prefill the batched
    tokens cover the model length and the captured length; prefix caching wants a larger block."""
    rows = [((), ((1, 1), (0, -1)), 0)]
    if d > 5:
        rows.append((((5, 0),), ((1, 1),), 2560))
    if d > 6:
        rows += [(((5, 1),), ((6, -1),), 0), (((6, 1),), ((2, 1),), 1)]
    if d > 10:
        rows.append((((5, 0),), ((1, 1), (10, -1)), 0))
    a = np.zeros(len(rows), CLAUSE)
    for i, (guards, terms, rhs) in enumerate(rows):
        a[i]["n_guard"], a[i]["n_term"], a[i]["rhs"] = len(guards), len(terms), rhs
        for g, (p, v) in enumerate(guards):
            a[i]["guard_param"][g], a[i]["guard_value"][g] = p, v
        for t, (p, k) in enumerate(terms):
            a[i]["term_param"][t], a[i]["coef"][t] = p, k
    return a


def _pool(d, n, seed):
    """n configurations as words [d][ld] on the GPU, uniform over each range (log-uniform where the scale is)."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 16 + 1)
    ld = (n + 3) // 4 * 4
    words = torch.zeros((d, ld), dtype=torch.int32, device="cuda")
    for i, (kind, lo, hi, k, _) in enumerate(PARAMS[:d]):
        u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
        if kind == S.INT_LOG:
            v = torch.exp(math.log(lo) + u * (math.log(hi) - math.log(lo))).round_().clamp_(lo, hi).int()
        elif kind == S.INT_UNIFORM:
            v = (lo + (u * (hi - lo + 1)).floor_()).clamp_(max=hi).int()
        elif kind == S.CATEGORICAL:
            v = (u * k).floor_().clamp_(max=k - 1).int()
        else:
            v = (lo + u * (hi - lo)).float().clamp_(lo, hi).view(torch.int32)
        words[i, :n] = v
    return words


def _observations(d, n, rng):
    """n configurations: words uint32 [d][n], stored values [n][d], coordinates in [0, 1] [n][d]."""
    words, vals, unit = np.zeros((d, n), np.uint32), np.zeros((n, d)), np.zeros((n, d))
    for i, (kind, lo, hi, k, _) in enumerate(PARAMS[:d]):
        u = rng.random(n)
        if kind == S.INT_LOG:
            v = np.clip(np.rint(np.exp(np.log(lo) + u * (np.log(hi) - np.log(lo)))), lo, hi)
            unit[:, i] = (np.log(v) - np.log(lo)) / (np.log(hi) - np.log(lo))
        elif kind == S.INT_UNIFORM:
            v = rng.integers(lo, hi + 1, n).astype(float)
            unit[:, i] = (v - lo) / (hi - lo)
        elif kind == S.CATEGORICAL:
            v = rng.integers(0, k, n).astype(float)
            unit[:, i] = v / (k - 1)
        else:
            v = np.clip((lo + u * (hi - lo)).astype(np.float32), np.float32(lo), np.float32(hi)).astype(float)
            unit[:, i] = (v - lo) / (hi - lo)
        vals[:, i] = v
        words[i] = v.astype(np.float32).view(np.uint32) if kind == S.CONTINUOUS else v.astype(np.int32).view(np.uint32)
    return words, vals, unit


def _objectives(unit, M, rng):
    """M conflicting objectives with a little noise, standardised and to be maximised: float32 [M][n]; noise variances."""
    n, d = unit.shape
    w, c = 0.5 + 1.5 * rng.random((M, d)), rng.random((M, d))
    g = np.stack([np.sin(3.0 * w[m] * unit).sum(1) + 0.5 * ((unit - c[m]) ** 2).sum(1) for m in range(M)])
    if M > 1:
        trade = unit @ np.array([p[4] for p in PARAMS[:d]])
        g = (2.0 if M > 2 else 0.5) / math.sqrt(d) * g + np.outer([1.0, -1.0, 0.0][:M], trade)
    # latencies are minimised; the third objective is a throughput
    raw = np.array([[-1.0], [-1.0], [1.0]])[:M] * (g + 0.02 * rng.standard_normal(g.shape))
    sd = raw.std(1, keepdims=True)
    y = ((raw - raw.mean(1, keepdims=True)) / sd).astype(np.float32)
    return y, np.maximum(1e-6, (0.02 / sd[:, 0]) ** 2).astype(np.float32)


def _labels(unit, rng):
    """1 for a configuration that ran: a quarter exceeds the memory budget, and a tenth of the labels is flipped."""
    score = unit @ np.array([p[4] for p in PARAMS[:unit.shape[1]]])
    ran = score <= np.quantile(score, 0.75)
    return np.where(rng.random(len(ran)) < 0.1, ~ran, ran)


def _grow(x, y, max_depth):
    """A CART regression tree on (x, 0/1 labels y), breadth first, children next to each other, as node records."""
    nodes, queue, at = [None], [(np.arange(len(y)), 0)], 0
    while at < len(queue):
        idx, depth = queue[at]
        ys = y[idx]
        m, pos = len(idx), int(ys.sum())
        best = None
        if depth < max_depth and 0 < pos < m:
            xs = x[idx]
            order = xs.argsort(axis=0, kind="stable")
            srt = np.take_along_axis(xs, order, 0)
            left = np.cumsum(ys[order], axis=0)[:-1]
            k = np.arange(1, m)[:, None]
            cost = left * (k - left) / k + (pos - left) * ((m - k) - (pos - left)) / (m - k)
            cost[srt[1:] <= srt[:-1]] = np.inf
            f = int(cost.argmin())
            row, col = divmod(f, x.shape[1])
            if np.isfinite(cost[row, col]):
                best = (col, np.float32(0.5 * (srt[row, col] + srt[row + 1, col])))
                if not srt[row, col] <= best[1] < srt[row + 1, col]:
                    best = (col, np.float32(srt[row, col]))
        if best is None:
            nodes[at] = (math.floor(LEAF_SCALE * pos / m + 0.5), 0, 0, 1)
        else:
            go = x[idx, best[0]] <= best[1]
            nodes[at] = (best[1], len(queue), best[0], 0)
            queue += [(idx[go], depth + 1), (idx[~go], depth + 1)]
            nodes += [None, None]
        at += 1
    return np.array(nodes, NODE)


class _Inputs:
    """Everything a case's program has on the host, from the seed alone."""

    def __init__(self, case, seed):
        d, n, M = case["d"], case["n"], case.get("M", 1)
        rng = np.random.default_rng([seed, 7])
        self.space, self.clauses = _space(d), _clauses(d)
        self.words, vals, unit = _observations(d, n, rng)
        self.y, self.noise = _objectives(unit, M, rng)
        self.ref = self.y.min(axis=1).astype(np.float32)
        self.ls = np.exp(0.5 * rng.standard_normal((M, d))).astype(np.float32)
        self.sf2 = np.ones(M, np.float32)
        self.warp = np.exp(0.4 * rng.standard_normal((M, d, 2))).astype(np.float32) if case.get("warp") else None
        self.eps = rng.standard_normal((case.get("S", 1), M)).astype(np.float32)
        self.labels = _labels(unit, rng)
        if case["kind"] in ROUNDS:
            trees = []
            for _ in range(case["T"]):
                b = rng.integers(0, n, n)
                trees.append(_grow(vals[b], self.labels[b], case["depth"]))
            self.offsets = np.zeros(len(trees) + 1, np.int32)
            self.offsets[1:] = np.cumsum([len(t) for t in trees])
            self.nodes = np.concatenate(trees)
        if case["kind"] == "mle":
            P = d + 2
            self.lo = np.array([math.log(0.02)] * d + [math.log(0.05), math.log(1e-4)])
            self.hi = np.array([math.log(20.0)] * d + [math.log(20.0), math.log(1.0)])
            base = np.array([0.0] * d + [0.0, math.log(0.01)])
            self.theta0 = base + 0.5 * rng.standard_normal((case["starts"], M, P))
            self.theta0[0] = base
            self.theta0 = np.clip(self.theta0, self.lo, self.hi)
        if case["kind"] == "forest":
            self.boot = rng.integers(0, n, size=(case["T"], n)).astype(np.int32)


_ctx = None


def _context():
    """One context for the program, as a user has it."""
    global _ctx
    if _ctx is None:
        _ctx = S.Context(0)
    return _ctx


def prepare(case, seed):
    h, kind, ctx = _Inputs(case, seed), case["kind"], _context()
    st = {"kind": kind, "ctx": ctx, "h": h, "n": case["n"]}

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    if kind in ROUNDS:
        inp = RoundInputs(h.space, h.clauses, h.nodes, h.offsets, LEAF_SCALE, DELTA_NUM, DELTA_DEN, h.words, h.y, h.ls,
                          h.sf2, h.noise, h.ref, h.eps, "ehvi" if kind == "fantasy" else kind, case["q"],
                          kernel=case.get("kernel", 0), fantasy=kind == "fantasy", seed=seed, warp=h.warp)
        st["round"], st["N"] = ScoringRound(ctx, inp, case["N"]), case["N"]
        st["cand"] = _pool(case["d"], case["N"], seed)
    elif kind == "posterior":
        layout = S.scoot_gp_layout_init(h.space, case["n"], case["M"], case.get("kernel", 0))
        blob = (S.scoot_gp_prepare(h.space, h.words, h.y, h.ls, h.sf2, h.noise, layout) if h.warp is None else
                S.scoot_gp_prepare_warped(h.space, h.words, h.y, h.ls, h.sf2, h.noise, h.warp, layout))[0]
        st.update(layout=layout, blob=dev(blob), N=case["N"], cand=_pool(case["d"], case["N"], seed))
        st["mean"], st["var"] = (torch.empty((case["M"], case["N"]), device="cuda") for _ in range(2))
    else:
        st["obs"] = dev(h.words.view(np.int32))
        if kind == "forest":
            st.update(labels=dev(h.labels.astype(np.uint8)), boot=dev(h.boot), depth=case["depth"],
                      nodes=torch.zeros((case["T"], 2 * case["n"] - 1), dtype=torch.int64, device="cuda"),
                      counts=torch.zeros(case["T"], dtype=torch.int32, device="cuda"))
            return st
        st["y"] = dev(h.y)
        if kind == "mle":
            st["theta0"], st["kernel"] = dev(h.theta0), case.get("kernel", 0)
            st["theta"], st["grad"] = torch.zeros_like(st["theta0"]), torch.zeros_like(st["theta0"])
            st["lml"] = torch.zeros(h.theta0.shape[:2], dtype=torch.float64, device="cuda")
        else:
            layout = S.scoot_gp_layout_init(h.space, case["n"], case["M"], case.get("kernel", 0))
            st.update(layout=layout, ls=dev(h.ls), sf2=dev(h.sf2), noise=dev(h.noise),
                      warp=None if h.warp is None else dev(h.warp),
                      blob=torch.zeros(layout.bytes, dtype=torch.uint8, device="cuda"),
                      work=torch.empty(S.scoot_gp_device_work_bytes(layout), dtype=torch.uint8, device="cuda"))
    return st


def run(state):
    kind, ctx, h = state["kind"], state["ctx"], state["h"]
    if kind in ROUNDS:
        r = state["round"]
        idx, val, count = r.run(state["cand"], state["N"])
        out = {"mask": r.mask, "votes": r.votes, "idx": idx, "count": count, "n_known": r.n_known,
               "n_feasible": r.n_feasible}
        if kind == "mace":
            out["acq"] = r.acq3
        else:
            out["val"] = val
            if kind != "fantasy":
                out["acq"] = r.acq
        return out
    if kind == "posterior":
        S.scoot_gp_posterior(ctx, state["layout"], state["blob"], state["cand"], state["N"], state["mean"], state["var"])
        return {"mean": state["mean"], "var": state["var"]}
    if kind == "mle":
        S.scoot_gp_mle(ctx, h.space, state["obs"], state["n"], state["y"], state["theta0"], h.lo, h.hi,
                       (1 << state["theta0"].shape[2]) - 1, MLE_STEPS, MLE_LR, state["theta"], state["lml"],
                       state["grad"], kernel=state["kernel"])
        return {"theta": state["theta"], "lml": state["lml"], "grad": state["grad"]}
    if kind == "forest":
        S.scoot_rf_train(ctx, h.space, state["obs"], state["n"], state["labels"], state["boot"], state["depth"],
                         LEAF_SCALE, state["nodes"], state["counts"])
        return {"nodes": state["nodes"], "counts": state["counts"]}
    L = state["layout"]
    S.scoot_gp_prepare_device(ctx, h.space, L, state["obs"], state["y"], state["ls"], state["sf2"], state["noise"],
                              state["blob"], state["work"], warp=state["warp"])
    b = state["blob"]
    return {"alpha": b[L.off_alpha:L.off_alpha + 4 * L.n_obj * L.n].view(torch.float32),
            "linv": b[L.off_linv:L.off_linv + 4 * L.n_obj * L.n_tiles * 2048].view(torch.float32),
            "xs": b[L.off_xs:L.off_xs + 4 * L.n_obj * L.n * L.d].view(torch.float32)}


# ---------------------------------------------------------------------------------------------- what a pass needs

def work(case):
    """Each input read once and each output written once; a multiply-add is two operations.  About 0.4 of a pool is
    left after the constraints and the forest."""
    kind, d, n = case["kind"], case["d"], case["n"]
    M = case.get("M", 1)
    posterior = n * (3 * d + 12) + n * (n + 1) + 4 * n
    if kind == "mle":
        evals = (MLE_STEPS + 1) * case["starts"] * M
        return {"bytes": 4 * n * (d + M) + 8 * case["starts"] * M * (3 * d + 7),
                "flops": evals * (2 * (n ** 3 / 3 + n ** 3 / 6 + n * n) + n * (n + 1) / 2 * (6 * d + 60))}
    if kind == "forest":
        return {"bytes": 4 * n * d + case["T"] * (4 * n + 16 * n), "flops": case["T"] * d * n * 8 * 4}
    if kind == "gp-state":
        return {"bytes": 4 * M * (n * n + 2 * n * d), "flops": M * (n ** 3 / 3 * 2 + n * n / 2 * (3 * d + 12))}
    N = case["N"]
    if kind == "posterior":
        return {"bytes": N * (4 * d + 8 * M) + 4 * M * n * n, "flops": N * M * posterior}
    live = 0.4 * N
    rows = {"mace": 3, "fantasy": 0}.get(kind, 1)
    acq = {"ei": 30, "mace": 50, "ehvi-exact": 20 * 40}.get(kind, case["S"] * (2 * M + 16 * M))
    byts = N * (4 * d + 1 + 4 + 4 * rows) + 4 * M * n * n
    flops = live * (M * posterior + acq + 2 * case["T"] * 6)
    if kind == "fantasy":  # each further pick: one downdate of every objective and its acquisition
        flops += (case["q"] - 1) * live * (M * (2 * n + 3 * d + 12) + acq)
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["kind"] == "forest":
        return "exact"
    if case["kind"] == "mle":       # 64 bits throughout, 60 steps of an ascent (5e-13 measured against exact())
        return {"rel": 1e-11, "max": 1e-9}
    if case["kind"] == "gp-state":  # factorised in 64 bits, stored in 32 (3e-8 measured)
        return {"rel": 1.5e-7, "max": 1e-5}
    # 32-bit sums of up to a few hundred terms of size 15 to 100 each for a mean of size 1, and the improvement over
    # the front is a small difference of such means: up to 4e-6 measured for acquisitions, 7e-6 for moments
    return {"rel": 2e-5, "max": 1e-3}


# ---------------------------------------------------------------------------------------------- the same in 64 bits

def _features(words, d):
    """Covariance inputs [N][d] in 64 bits of words [d][N]."""
    out = torch.empty((words.shape[1], d), dtype=torch.float64, device=words.device)
    for i, (kind, lo, hi, _, _) in enumerate(PARAMS[:d]):
        v = words[i].view(torch.float32).double() if kind == S.CONTINUOUS else words[i].double()
        if kind == S.INT_LOG:
            v = (v.log() - math.log(lo)) / (math.log(hi) - math.log(lo))
        elif kind != S.CATEGORICAL:
            lo32, hi32 = float(np.float32(lo)), float(np.float32(hi))
            v = (v - lo32) / (hi32 - lo32)
        out[:, i] = v
    return out


def _matern(r2, kernel):
    r = r2.clamp_min(0).sqrt()
    if kernel == 1:
        a = math.sqrt(3.0) * r
        return (1 + a) * torch.exp(-a)
    a = math.sqrt(5.0) * r
    return (1 + a + a * a / 3) * torch.exp(-a)


class _GP:
    """One objective's GP in 64 bits."""

    def __init__(self, h, m, d, kernel):
        self.d, self.kernel = d, kernel
        self.ell, self.sf2, self.tau2 = h.ls[m].astype(np.float64), float(h.sf2[m]), float(h.noise[m])
        self.warp = None if h.warp is None else h.warp[m].astype(np.float64)
        self.u = self.inputs(_features(torch.from_numpy(h.words.view(np.int32)).cuda(), d))
        n = len(self.u)
        K = self.cov(self.u, self.u) + self.tau2 * torch.eye(n, dtype=torch.float64, device="cuda")
        self.L = torch.linalg.cholesky(K)
        self.alpha = torch.cholesky_solve(torch.from_numpy(h.y[m].astype(np.float64)).cuda()[:, None], self.L)[:, 0]

    def inputs(self, f):
        if self.warp is None:
            return f
        f = f.clone()
        for i in range(self.d):
            if PARAMS[i][0] != S.CATEGORICAL:
                x = f[:, i].clamp(0, 1)
                f[:, i] = -torch.expm1(self.warp[i, 1] * torch.log1p(-x ** self.warp[i, 0]))
        return f

    def cov(self, a, b):
        r2 = torch.zeros((len(a), len(b)), dtype=torch.float64, device="cuda")
        for i in range(self.d):
            t = a[:, i:i + 1] - b[:, i][None]
            r2 += (t != 0).double() / self.ell[i] ** 2 if PARAMS[i][0] == S.CATEGORICAL else (t / self.ell[i]) ** 2
        return self.sf2 * _matern(r2, self.kernel)

    def posterior(self, f, keep=False):
        """Mean and variance of features f; with keep the whitened rows too."""
        mean, var = (torch.empty(len(f), dtype=torch.float64, device="cuda") for _ in range(2))
        V = torch.empty((len(f), len(self.u)), dtype=torch.float64, device="cuda") if keep else None
        for s in range(0, len(f), 1 << 16):
            k = self.cov(self.inputs(f[s:s + (1 << 16)]), self.u)
            v = torch.linalg.solve_triangular(self.L, k.T, upper=False).T
            mean[s:s + (1 << 16)] = k @ self.alpha
            var[s:s + (1 << 16)] = (self.sf2 - v.square().sum(1)).clamp_min(0)
            if keep:
                V[s:s + (1 << 16)] = v
        return mean, var, V


def _live(case, h, words):
    """Whether each candidate satisfies the constraints and the forest's threshold."""
    N = case["N"]
    ok = torch.ones(N, dtype=torch.bool, device="cuda")
    for c in h.clauses:
        guard = torch.ones(N, dtype=torch.bool, device="cuda")
        for g in range(int(c["n_guard"])):
            guard &= words[int(c["guard_param"][g])] == int(c["guard_value"][g])
        total = sum(int(c["coef"][t]) * words[int(c["term_param"][t])].long() for t in range(int(c["n_term"])))
        ok &= ~guard | (total >= int(c["rhs"]))
    at = ok.nonzero()[:, 0]
    x = torch.stack([words[i, at].view(torch.float32) if PARAMS[i][0] == S.CONTINUOUS else words[i, at].float()
                     for i in range(case["d"])])
    val, left, feat, leaf = (torch.from_numpy(h.nodes[f].astype(t)).cuda()
                             for f, t in (("val", np.float32), ("left", np.int64), ("feat", np.int64), ("flags", np.bool_)))
    votes = torch.zeros(len(at), dtype=torch.float64, device="cuda")
    for t in range(case["T"]):
        root = int(h.offsets[t])
        node = torch.full((len(at),), root, dtype=torch.int64, device="cuda")
        for _ in range(case["depth"]):
            xv = x.gather(0, feat[node][None])[0]
            node = torch.where(leaf[node], node, root + left[node] + (xv > val[node]))
        votes += val[node]
    ok[at] = DELTA_DEN * votes >= DELTA_NUM * LEAF_SCALE * case["T"]
    return ok


def _boxes(points, ref):
    """Boxes (lo, hi) of the region above ref that no point dominates, open above on the last objective."""
    pts = {tuple(p) for p in points.tolist() if all(a > b for a, b in zip(p, ref))}
    pts = [p for p in pts if not any(o != p and all(a >= b for a, b in zip(o, p)) for o in pts)]
    if len(ref) == 1:
        return [((max([p[0] for p in pts], default=ref[0]),), (math.inf,))]
    edges = [ref[0]] + sorted({p[0] for p in pts}) + [math.inf]
    out = []
    for lo, hi in zip(edges[:-1], edges[1:]):
        rest = np.array([p[1:] for p in pts if p[0] >= hi]).reshape(-1, len(ref) - 1)
        out += [((lo,) + a, (hi,) + b) for a, b in _boxes(rest, ref[1:])]
    return out


def _ehvi(mean, sd, eps, boxes):
    """Mean over the base samples of the improvement summed over the boxes; mean, sd [M][L], eps [S][M]."""
    out = torch.empty(mean.shape[1], dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // len(eps))
    for s in range(0, len(out), step):
        y = [mean[m, s:s + step, None] + sd[m, s:s + step, None] * eps[None, :, m] for m in range(len(mean))]
        total = torch.zeros_like(y[0])
        for lo, hi in boxes:
            p = None
            for m in range(len(y)):
                w = (y[m].clamp(max=hi[m]) if hi[m] < math.inf else y[m]).sub(lo[m]).clamp_(min=0)
                p = w if p is None else p.mul_(w)
            total += p
        out[s:s + step] = total.mean(1)
    return out


def _phi(z):
    return torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)


def _cdf(z):
    return 0.5 * torch.erfc(-z / math.sqrt(2.0))


def _improvement(mean, sd, best):
    """E[max(0, Y - best)] of Y ~ N(mean, sd^2)."""
    a = mean - best
    z = a / sd.clamp_min(1e-300)
    return torch.where(sd > 0, a * _cdf(z) + sd * _phi(z), a.clamp_min(0))


def _fantasy_values(case, h, gps, feats):
    """The values of the q sequential picks: each the largest EHVI, then its mean joins the front and the variances
    take the rank-1 term of an observation there."""
    post = [g.posterior(feats, keep=True) for g in gps]
    mean, var, V = torch.stack([p[0] for p in post]), torch.stack([p[1] for p in post]), [p[2] for p in post]
    eps, ref = torch.from_numpy(h.eps.astype(np.float64)).cuda(), h.ref.astype(np.float64).tolist()
    points, past = h.y.T.astype(np.float64), [[] for _ in gps]
    picked, vals = [], []
    for j in range(min(case["q"], len(feats))):
        acq = _ehvi(mean, var.clamp_min(0).sqrt(), eps, _boxes(points, ref))
        if picked:
            acq[picked] = -math.inf
        p = int(acq.argmax())
        picked.append(p)
        vals.append(float(acq[p]))
        points = np.concatenate([points, mean[:, p].float().double().cpu().numpy()[None]])
        for m, g in enumerate(gps):
            c = g.cov(feats, feats[p:p + 1])[:, 0] - V[m] @ V[m][p]
            for f in past[m]:
                c -= f * f[p]
            f = c / (var[m, p] + g.tau2).sqrt()
            past[m].append(f)
            var[m] -= f * f
    return vals


def _exact_round(case, h, seed):
    kind, N, d = case["kind"], case["N"], case["d"]
    words = _pool(d, N, seed)[:, :N]
    at = _live(case, h, words).nonzero()[:, 0]
    feats = _features(words[:, at], d)
    gps = [_GP(h, m, d, case.get("kernel", 0)) for m in range(case["M"])]
    none = {"mask": None, "votes": None, "idx": None, "count": None, "n_known": None, "n_feasible": None}

    def top(v):
        out = torch.full((case["q"],), -math.inf, dtype=torch.float64, device="cuda")
        k = min(case["q"], len(v))
        out[:k] = v.topk(k)[0] if torch.is_tensor(v) else torch.tensor(v[:k], dtype=torch.float64)
        return out

    if kind == "fantasy":
        return {**none, "val": top(_fantasy_values(case, h, gps, feats))}
    post = [g.posterior(feats) for g in gps]
    mean, sd = torch.stack([p[0] for p in post]), torch.stack([p[1] for p in post]).sqrt()
    if kind in ("ei", "mace"):
        best, xi = float(h.y[0].max()), float(np.float32(1e-4))
        rows = [_improvement(mean[0], sd[0], best - xi)]
        if kind == "mace":
            t = case["n"]
            kappa = 2 * math.log(t * t * math.pi ** 2 / (6 / t ** 2))
            rows = [mean[0] + kappa * sd[0], _cdf((mean[0] - (best - xi)) / sd[0].clamp_min(1e-300))] + rows
    else:
        boxes = _boxes(h.y.T.astype(np.float64), h.ref.astype(np.float64).tolist())
        if kind == "ehvi":
            rows = [_ehvi(mean, sd, torch.from_numpy(h.eps.astype(np.float64)).cuda(), boxes)]
        else:
            total = torch.zeros_like(mean[0])
            for lo, hi in boxes:
                p = 1.0
                for m in range(len(mean)):
                    w = _improvement(mean[m], sd[m], lo[m])
                    p = p * (w if hi[m] == math.inf else w - _improvement(mean[m], sd[m], hi[m]))
                total += p
            rows = [total]
    acq = torch.full((len(rows), N), -math.inf, dtype=torch.float64, device="cuda")
    for r, v in enumerate(rows):
        acq[r, at] = v
    return {**none, "acq": acq} if kind == "mace" else {**none, "acq": acq[0], "val": top(rows[0])}


def _exact_mle(case, h):
    """The same projected ascent of the log marginal likelihood, every start and objective at once."""
    n, d, M, St = case["n"], case["d"], case["M"], case["starts"]
    f = _features(torch.from_numpy(h.words.view(np.int32)).cuda(), d)
    parts = [f[:, i][:, None] - f[:, i][None] for i in range(d)]
    parts = torch.stack([(t != 0).double() if PARAMS[i][0] == S.CATEGORICAL else t * t for i, t in enumerate(parts)])
    y = torch.from_numpy(h.y.astype(np.float64)).cuda()
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    lo, hi = torch.from_numpy(h.lo).cuda(), torch.from_numpy(h.hi).cuda()
    th = torch.from_numpy(h.theta0).cuda().clone()
    m1, m2 = torch.zeros_like(th), torch.zeros_like(th)

    def value(th):
        il2, sf2, tau2 = torch.exp(-2 * th[..., :d]), th[..., d].exp(), th[..., d + 1].exp()
        r2 = torch.einsum("smc,cij->smij", il2, parts)
        r = r2.sqrt()
        a = math.sqrt(3.0 if case.get("kernel", 0) == 1 else 5.0) * r
        if case.get("kernel", 0) == 1:
            k, dk = (1 + a) * torch.exp(-a), -1.5 * torch.exp(-a)
        else:
            k, dk = (1 + a + a * a / 3) * torch.exp(-a), -(5 / 6) * (1 + a) * torch.exp(-a)
        L = torch.linalg.cholesky(sf2[..., None, None] * k + tau2[..., None, None] * eye)
        Ki = torch.cholesky_solve(eye.expand_as(L), L)
        al = torch.einsum("smij,mj->smi", Ki, y)
        w = 0.5 * (al[..., :, None] * al[..., None, :] - Ki)
        g = torch.empty_like(th)
        g[..., :d] = -2 * sf2[..., None] * il2 * torch.einsum("smij,cij->smc", dk * w, parts)
        g[..., d] = sf2 * (w * k).sum((-1, -2))
        g[..., d + 1] = tau2 * torch.diagonal(w, dim1=-2, dim2=-1).sum(-1)
        logdet = 2 * torch.diagonal(L, dim1=-2, dim2=-1).log().sum(-1)
        return -0.5 * (al * y).sum(-1) - 0.5 * logdet - 0.5 * n * math.log(2 * math.pi), g

    for t in range(MLE_STEPS):
        _, g = value(th)
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        step = MLE_LR * (1 - t / MLE_STEPS)
        th = th + step * (m1 / (1 - 0.9 ** (t + 1))) / ((m2 / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
        th = torch.minimum(torch.maximum(th, lo), hi)
    lml, g = value(th)
    return {"theta": th, "lml": lml, "grad": g}


def _exact_state(case, h):
    n, d, M = case["n"], case["d"], case["M"]
    rb = (n + 63) // 64
    order = [i for i in range(d) if PARAMS[i][0] != S.CATEGORICAL] + [i for i in range(d) if PARAMS[i][0] == S.CATEGORICAL]
    alpha, linv, xs = [], [], []
    for m in range(M):
        g = _GP(h, m, d, case.get("kernel", 0))
        alpha.append(g.alpha)
        full = torch.zeros((64 * rb, 64 * rb), dtype=torch.float64, device="cuda")
        full[:n, :n] = torch.linalg.solve_triangular(g.L, torch.eye(n, dtype=torch.float64, device="cuda"), upper=False)
        for b in range(rb):  # 32 x 64 tiles, transposed, row block by row block
            for c in range(2 * (b + 1)):
                linv.append(full[64 * b:64 * b + 64, 32 * c:32 * c + 32].T.reshape(-1))
        xs.append(torch.stack([g.u[:, i] if PARAMS[i][0] == S.CATEGORICAL else g.u[:, i] / g.ell[i] for i in order], 1))
    return {"alpha": torch.cat(alpha), "linv": torch.cat(linv), "xs": torch.cat([x.reshape(-1) for x in xs])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "forest":
        return None
    h = _Inputs(case, seed)
    if kind in ROUNDS:
        return _exact_round(case, h, seed)
    if kind == "mle":
        return _exact_mle(case, h)
    if kind == "gp-state":
        return _exact_state(case, h)
    feats = _features(_pool(case["d"], case["N"], seed)[:, :case["N"]], case["d"])
    post = [_GP(h, m, case["d"], case.get("kernel", 0)).posterior(feats) for m in range(case["M"])]
    return {"mean": torch.stack([p[0] for p in post]), "var": torch.stack([p[1] for p in post])}
