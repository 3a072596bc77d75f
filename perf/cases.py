"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through `binding.Context` the way a program that selects kernels does:

  one        one GEMM against a prepared catalogue (a dispatcher that meets a shape for the first
             time): tree ensemble, result in host memory
  one_plain  the same without preparation, any model
  host       a short list of GEMMs from host buffers to host results
  batch      a list of GEMMs against the whole catalogue, tree ensemble
  segments   a list of GEMMs, each against its own subset of the catalogue, mixed element types
  mlp        a list of GEMMs against the whole catalogue, bf16 feed-forward ranker
  ridge      the same with the linear scorer
  featurize  feature rows of (problem, candidate) pairs for a training set, per-problem subsets
  score      a tree ensemble over given feature rows
  search     for each GEMM of a list: the valid part of the whole search space, ranked by a tree
             ensemble, answered with ids of the space

Sizes come from the repository's configurations (`workloads.CONFIGS`), its tests and benchmark.
The pools are the synthetic cross-product grids of those configurations or the valid part of the
enumerated search space ("valid"), which is what a deployment ranks.
"""
import functools

import numpy as np
import torch

from paper_2609_35587_b200 import binding as ks
from paper_2609_35587_b200 import workloads as wl

DEV = torch.device("cuda", 0)
WIDE = "1024,1024,512,256"  # hidden layers of the largest ranker preset


def listed():
    return [
        # a decode-time GEMM (M in 1..64) in a serving process, the latency stream's single call
        dict(name="one_decode", kind="one", problems="decode", pool="grid", C=60000, trees=500, depth=8,
             law="pernode", k=10),
        # one GEMM ranked by the feed-forward model with one-hot categorical inputs, no preparation
        dict(name="one_neural", kind="one_plain", problems="decode", pool="valid", C=61140, hidden="256,256",
             onehot=True, k=10),
        # a short list of GEMMs against a small pool, host buffers in and out: launches and copies count
        dict(name="tiny_host", kind="host", problems="plain", pool="small", P=64, C=2048, trees=100, depth=6,
             law="pernode", k=5),
        # the GEMMs of one transformer layer against all valid kernels
        dict(name="few_layers", kind="batch", problems="cross", pool="valid", P=7, C=61140, trees=500, depth=8,
             law="hist256", k=10),
        # the whole tuning table: 1,024 shapes x 60,000 kernels
        dict(name="full_space", kind="batch", problems="plain", pool="grid", P=1024, C=60000, trees=500, depth=8,
             law="pernode", k=10),
        # shapes of four operand types, each with its own candidate set, a larger ensemble
        dict(name="cross_precision", kind="segments", problems="cross", pool="grid", P=4096, C=62208, seg=16384,
             trees=1000, depth=8, law="pernode", k=10),
        # the tuning table by the small feed-forward ranker (tensor cores)
        dict(name="neural_ranker", kind="mlp", problems="plain", pool="grid", P=1024, C=60000, hidden="256,256",
             onehot=False, k=10),
        # a model's GEMMs by the ranker of the shipped size (1.76 M weights)
        dict(name="neural_wide", kind="mlp", problems="cross", pool="grid", P=16, C=60000, hidden=WIDE, onehot=False,
             k=10),
        # the tuning table by the linear baseline
        dict(name="ridge_table", kind="ridge", problems="plain", pool="grid", P=1024, C=60000, onehot=False, k=10),
        # feature rows of a training set: sampled candidates per problem, four operand types
        dict(name="training_rows", kind="featurize", problems="cross", pool="grid", P=300, C=62208, seg=7000),
        # scores of given feature rows (evaluating an ensemble on a held-out set)
        dict(name="score_rows", kind="score", problems="plain", pool="grid", rows=1000003, trees=500, depth=8,
             law="pernode"),
        # a few GEMMs with nothing prepared: the valid kernels out of 534,600, ranked
        dict(name="cold_search", kind="search", problems="cross", P=4, trees=500, depth=8, law="hist256", k=10,
             flags=ks.KS_VALID_COUPLED),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _ensemble(rng):
    return dict(trees=rng.choice([_log(rng, 50, 1000), 916, 500]), depth=rng.choice([6, 7, 8, 8]),
                law=rng.choice(wl.LAWS))


def draw(rng):
    """One more case: any kind, sizes over the whole range of the listed ones and between them."""
    kind = rng.choice(["one", "one_plain", "host", "batch", "batch", "segments", "mlp", "mlp", "ridge", "featurize",
                       "score", "search"])
    problems = rng.choice(["plain", "cross", "stream"])
    pool = rng.choice(["grid", "grid", "valid"])
    C, k = _log(rng, 500, 60000), rng.choice([1, 5, 10, 32])
    if kind == "one":
        return dict(kind=kind, problems=rng.choice(["decode", "stream"]), pool=pool, C=C, k=k, **_ensemble(rng))
    if kind == "one_plain":
        if rng.random() < 0.5:
            return dict(kind=kind, problems="decode", pool=pool, C=C, k=k, **_ensemble(rng))
        return dict(kind=kind, problems="decode", pool=pool, C=C, hidden=rng.choice(["256,256", "256", "128,64"]),
                    onehot=rng.random() < 0.5, k=k)
    if kind == "host":
        return dict(kind=kind, problems=problems, pool=rng.choice(["small", "grid"]), P=_log(rng, 8, 512),
                    C=_log(rng, 500, 5000), k=k, **_ensemble(rng))
    if kind == "batch":
        e = _ensemble(rng)
        # at most the pair walks of the largest batch
        P = min(_log(rng, 2, 1024), max(2, int(1024 * 60000 * 4000 / (C * e["trees"] * e["depth"]))))
        return dict(kind=kind, problems=problems, pool=pool, P=P, C=C, k=k, **e)
    if kind == "segments":
        return dict(kind=kind, problems=problems, pool=pool, P=_log(rng, 16, 1024), C=60000, seg=_log(rng, 300, 16384),
                    k=k, **_ensemble(rng))
    if kind == "mlp":
        hidden = rng.choice(["256,256", "128", "192,128", "512,256", "1024,512,256", WIDE])
        w = _flops_per_row(hidden, False)
        P = max(1, min(_log(rng, 1, 1024), int(3.3e12 / (w * C))))
        return dict(kind=kind, problems=problems, pool=pool, P=P, C=C, hidden=hidden, onehot=rng.random() < 0.3, k=k)
    if kind == "ridge":
        return dict(kind=kind, problems=problems, pool=pool, P=_log(rng, 2, 1024), C=C, onehot=rng.random() < 0.5, k=k)
    if kind == "featurize":
        if rng.random() < 0.3:  # every pair of a smaller set
            return dict(kind=kind, problems=problems, pool=pool, P=max(2, min(_log(rng, 2, 1024), 2000000 // C)), C=C)
        return dict(kind=kind, problems=problems, pool=pool, P=_log(rng, 2, 300), C=60000, seg=_log(rng, 100, 7000))
    if kind == "score":
        return dict(kind=kind, problems=problems, pool=pool, rows=_log(rng, 1000, 1000000), **_ensemble(rng))
    return dict(kind=kind, problems=problems, P=_log(rng, 1, 16), k=k, flags=rng.choice([1, 1, 5, 0]), **_ensemble(rng))


# ------------------------------------------------------------------------------------------


def _problems(how, seed, P):
    if how in ("plain", "cross"):
        return wl.problems_batch(seed, P, cross_precision=how == "cross")
    p = wl.problems_stream(seed, P)
    if how == "decode":
        p["m"] = wl._log_uniform_dim(seed, 1, np.arange(P), 1, 64, 1)
    return p


def _pool(ctx, how, seed, C):
    """The pool as device records and as host records."""
    if how == "valid":
        rec, _, n = ctx.valid_catalogue(wl.problems_batch(seed, 1), ks.KS_VALID_COUPLED)
        # all of it, or evenly spaced ones; the rows stay in the order of the search space
        return rec[torch.arange(min(C, n), device=DEV) * n // min(C, n)].contiguous(), None
    grid = wl.candidates_small_grid if how == "small" else wl.candidates_full_grid
    c = grid(seed, C)
    return ks.to_device(c, DEV), c


def _length(p, seg):
    """Candidates of problem p: seg or up to an eighth fewer."""
    return seg - p * 97 % max(1, seg // 8)


def _segments(seed, P, C, seg):
    """A random subset of pool indices for every problem, ascending."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    length = torch.tensor([_length(p, min(seg, C)) for p in range(P)], device=DEV)
    parts = []
    for lo in range(0, P, 256):
        n = length[lo:lo + 256, None]
        pick = torch.rand((len(n), C), device=DEV, generator=g).topk(min(seg, C), 1).indices.to(torch.int32)
        pick = torch.where(torch.arange(pick.shape[1], device=DEV) < n, pick, C).sort(1).values
        parts.append(pick[pick < C])
    off = torch.zeros(P + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(length, 0, out=off[1:])
    return off, torch.cat(parts).contiguous()


def _stats(problems):
    return wl.feature_stats("cfg2" if problems == "cross" else "cfg1")


def _trees(ctx, case, seed):
    off, nodes = wl.gbdt_complete(seed, case["trees"], case["depth"], _stats(case["problems"]), 0.1, case["law"])
    return ctx.model_create_gbdt(off, nodes, 0.0)


def _mlp(ctx, case, seed):
    st = _stats(case["problems"])
    hidden = [int(w) for w in case["hidden"].split(",")] if case.get("hidden") else []
    mu, sigma = wl.onehot_stats(st["mu"], st["sigma"]) if case["onehot"] else (st["mu"], st["sigma"])
    return ctx.model_create_mlp(wl.mlp_xavier(seed, [80 if case["onehot"] else 64] + hidden + [1], mu, sigma))


def prepare(case, seed):
    kind = case["kind"]
    ctx = ks.Context(wl.gpu_desc(), 0)
    st = dict(kind=kind, ctx=ctx, k=case.get("k"), neural="hidden" in case)
    P = case.get("P", 1)
    if kind == "search":
        prob = _problems(case["problems"], seed, P)
        return dict(st, problems=[(p, ks.to_device(p, DEV)) for p in np.split(prob, P)], flags=case["flags"],
                    model=_trees(ctx, case, seed))
    if kind == "score":
        per = -(-case["rows"] // 16)
        prob = _problems(case["problems"], seed, 16)
        rec, _ = _pool(ctx, case["pool"], seed, min(per, 60000))
        x = ctx.featurize(ks.to_device(prob, DEV), 16, rec, rec.shape[0])
        x = x.repeat(-(-case["rows"] // x.shape[0]), 1)[:case["rows"]].contiguous()
        return dict(st, x=x, model=_trees(ctx, case, seed))
    prob = _problems(case["problems"], seed, P)
    rec, host = _pool(ctx, case["pool"], seed, case["C"])
    st.update(P=P, C=rec.shape[0], d_p=ks.to_device(prob, DEV), d_c=rec)
    st.update(off=None, idx=None, pairs=P * rec.shape[0])
    if "seg" in case:
        st["off"], st["idx"] = _segments(seed, P, rec.shape[0], case["seg"])
        st["pairs"] = st["idx"].numel()
    if kind != "featurize":
        st["model"] = _trees(ctx, case, seed) if "trees" in case else _mlp(ctx, case, seed)
    if kind == "host":
        # pinned, as a program that feeds the GPU keeps its staging buffers
        pin = lambda a: torch.from_numpy(a.view(np.uint8).reshape(len(a), -1).copy()).pin_memory()
        st.update(h_p=pin(prob), h_c=pin(host))
    if kind in ("one", "one_plain"):
        cat = ctx.catalogue_prepare(rec, st["C"], st["model"]) if kind == "one" else None
        st["call"] = ctx.select_one_caller(rec, st["C"], st["model"], st["k"], catalogue=cat)
        st["problem"] = ks.problem_structs(prob)[0]
    return st


def _answer(st, idx, score):
    # The feed-forward rankers round every hidden unit to bf16: with the layers' sums in another
    # order up to 3 % of the positions of a top-10 list change places with a neighbour (scores 1e-4
    # apart), so their answer is compared by its scores.
    return {"score": score} if st["neural"] else {"index": idx, "score": score}


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind in ("one", "one_plain"):
        return _answer(st, *st["call"](st["problem"]))
    if kind == "host":
        return _answer(st, *ctx.select_host(st["h_p"], st["P"], st["h_c"], st["C"], st["model"], st["k"]))
    if kind == "featurize":
        return ctx.featurize(st["d_p"], st["P"], st["d_c"], st["C"], st["off"], st["idx"], st["pairs"])
    if kind == "score":
        return ctx.score(st["x"], st["model"])
    if kind == "search":
        answer = []
        for p, d_p in st["problems"]:
            rec, ids, n = ctx.valid_catalogue(p, st["flags"])
            idx, score = ctx.select(d_p, 1, rec[:n], n, st["model"], st["k"])
            answer.append((ctx.remap_indices(idx, ids, n), score, n))
        return answer
    return _answer(st, *ctx.select(st["d_p"], st["P"], st["d_c"], st["C"], st["model"], st["k"], st["off"], st["idx"],
                                   st["pairs"]))


@functools.lru_cache(None)
def _flops_per_row(hidden, onehot):
    w = [73 if onehot else 63] + ([int(v) for v in hidden.split(",")] if hidden else []) + [1]
    return 2 * sum(a * b for a, b in zip(w, w[1:]))


def work(case):
    """Bytes: every input once, every result once. Flops: for a tree one comparison a level and
    one addition, for a layer its multiplications and additions; about 60 operations for the
    columns of a pair that depend on both of its sides."""
    kind = case["kind"]
    if kind == "score":
        return {"bytes": case["rows"] * (256 + 4), "flops": case["rows"] * case["trees"] * (case["depth"] + 1)}
    P, C = case.get("P", 1), case.get("C", 61000)
    if kind == "search":  # the survivors of the space for every problem, with their ids
        C = {0: 137000, 1: 61000, 5: 61000}[case["flags"]]
    pairs = sum(_length(p, min(case["seg"], C)) for p in range(P)) if "seg" in case else P * C
    moved = 16 * (P + C) + (4 * pairs + 8 * P if "seg" in case else 0)
    if kind == "featurize":
        return {"bytes": moved + pairs * 256, "flops": 60 * pairs}
    per = case["trees"] * (case["depth"] + 1) if "trees" in case else _flops_per_row(case.get("hidden", ""),
                                                                                    case["onehot"])
    model = case["trees"] * (2 << case["depth"]) * 4 if "trees" in case else per
    if kind == "search":
        return {"bytes": P * (20 * C + 8 * case["k"]) + model, "flops": P * ks.KS_CATALOGUE_SIZE * 30 + pairs * (per + 60)}
    return {"bytes": moved + model + 8 * P * case["k"], "flops": pairs * (per + 60)}


def tolerance(case):
    if case["kind"] == "featurize":
        return "exact"
    if "hidden" in case:
        # against the same model in torch, sums in another order: rel 2.8e-4, max 3.6e-3
        return {"rel": 1.2e-3, "max": 1.5e-2}
    # fp32 sums of 50 to 1,000 leaves (63 terms for the linear scorer) against sums in 64 bits: rel
    # 2.8e-7, max 2.6e-6 (a score near zero); candidates that close may change places
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.005}
