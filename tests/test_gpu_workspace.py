"""Calls whose whole workspace cannot be had (a hook stands in for a full device): a batch for the walk of
whole classes goes to the candidates' own walks, a split walk of several rounds of blocks walks whole blocks, the linear
scorer ranks pair by pair, a wide ranker takes few rows at a time, and what cannot do with less is refused. The answers agree with those with all of the workspace, and with the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl
from tests.helpers import topk_accept

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()
MB = 1 << 20


@pytest.fixture(scope="module")
def ks():
    from paper_2609_35587_b200 import binding
    return binding


@pytest.fixture()
def ctx(ks):
    c = ks.Context(DESC, 0)
    yield c
    c.close()


def host(pair):
    return tuple(t.cpu().numpy() for t in pair)


def test_trees(ks, ctx):
    """300 problems: the class walk's programs and scores are 20 MB beside some 100 for the tables."""
    dev = torch.device("cuda", 0)
    base = wl.candidates_full_grid(1, None)
    cand = np.ascontiguousarray(base[(base["tile_m"] == 128) & (base["tile_k"] == 64)])
    prob = wl.problems_batch(3, 300, cross_precision=False)
    gbdt = (*wl.gbdt_complete(4, 30, 6, wl.feature_stats("cfg1"), 0.1), 0.0)
    model = ctx.model_create_gbdt(*gbdt)
    args = ks.to_device(prob, dev), 300, ks.to_device(cand, dev), len(cand), model, 10
    full = host(ctx.select(*args))
    assert ctx.debug_class_walks() == 1
    need = 4
    while True:  # the least that the call does with
        ctx.debug_limit_workspace(need * MB)
        try:
            got = host(ctx.select(*args))
            break
        except ks.KsError as e:
            assert e.status == ks.KS_ERR_OOM
            need += 4
    lean = ctx.debug_class_walks() == 1
    again = host(ctx.select(*args))  # (a size once refused is not asked for again)
    assert np.array_equal(got[0], again[0]) and np.array_equal(got[1], again[1])
    assert lean and ctx.debug_class_walks() == 1
    for idx, sc in (full, got):
        for p in (0, 150, 299):
            _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 10, gbdt=gbdt, want_scores=True)
            ok, msg = topk_accept(idx[p], sc[p], ref, np.arange(len(cand), dtype=np.int32), 10, 1e-5)
            assert ok, (p, msg)
    ctx.debug_limit_workspace(0)
    after = host(ctx.select(*args))
    assert ctx.debug_class_walks() == 2 and np.array_equal(after[1], full[1])


@pytest.mark.parametrize("P,C", [(9, 60000), (40, 25000)])
def test_split_walk(ks, ctx, P, C):
    """531 and 1,000 blocks: the tiles in front take some 30 MB, the rows of the candidates beside them or the class
    records of a few problems a fraction of that."""
    dev = torch.device("cuda", 0)
    prob, cand = wl.problems_batch(3, P, cross_precision=False), wl.candidates_full_grid(1, C)
    gbdt = (*wl.gbdt_complete(4, 60, 6, wl.feature_stats("cfg1"), 0.1, "slots128"), 0.0)
    model = ctx.model_create_gbdt(*gbdt)
    args = ks.to_device(prob, dev), P, ks.to_device(cand, dev), C, model, 10
    full = host(ctx.select(*args))
    assert ctx.debug_split_walks() == 1
    need = 2
    while True:  # the least that the call does with
        ctx.debug_limit_workspace(need * MB)
        try:
            got = host(ctx.select(*args))
            break
        except ks.KsError as e:
            assert e.status == ks.KS_ERR_OOM
            need += 2
    assert ctx.debug_split_walks() == 1
    for idx, sc in (full, got):
        for p in (0, P // 2, P - 1):
            _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 10, gbdt=gbdt, want_scores=True)
            ok, msg = topk_accept(idx[p], sc[p], ref, np.arange(C, dtype=np.int32), 10, 1e-5)
            assert ok, (p, msg)
    ctx.debug_limit_workspace(0)
    after = host(ctx.select(*args))
    assert ctx.debug_split_walks() == 2 and np.array_equal(after[1], full[1])


def test_linear_scorer(ks, ctx):
    """Ranked by classes the call takes some 40 MB, pair by pair 7; the answers are the same bits."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    model = ctx.model_create_mlp(wl.mlp_xavier(3, [64, 1], st["mu"], st["sigma"]))
    args = ks.to_device(wl.problems_batch(3, 40), dev), 40, ks.to_device(wl.candidates_full_grid(1, 50001), dev), 50001, model, 10
    full = host(ctx.select(*args))
    n = ctx.launch_count()
    ctx.debug_limit_workspace(16 * MB)
    less = host(ctx.select(*args))
    launches = ctx.launch_count() - n
    ctx.debug_limit_workspace(0)
    n = ctx.launch_count()
    again = host(ctx.select(*args))
    assert launches < ctx.launch_count() - n  # (tables of classes)
    for a, b, c in zip(full, less, again):
        assert np.array_equal(a, b) and np.array_equal(a, c)


@pytest.mark.parametrize("onehot", [False, True])
def test_wide_ranker(ks, ctx, onehot):
    """More pairs than are taken at a time (2,048) and, in the dense call, than are ranked in a round (1 M)."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    mu, sg = wl.onehot_stats(st["mu"], st["sigma"]) if onehot else (st["mu"], st["sigma"])
    model = ctx.model_create_mlp(wl.mlp_xavier(1, [80 if onehot else 64, 512, 128, 1], mu, sg))
    prob, cand = wl.problems_batch(2, 21), wl.candidates_full_grid(2, 50001)
    d_p, d_c = ks.to_device(prob, dev), ks.to_device(cand, dev)
    x = ctx.featurize(d_p, 1, d_c, 50001)[:5003].contiguous()
    records = lambda a: a.view(np.uint8).reshape(len(a), -1).copy()

    def answers():
        return [*host(ctx.select(d_p, 21, d_c, 50001, model, 7)), ctx.score(x, model).cpu().numpy(),
                *(t.numpy().copy() for t in ctx.select_one(prob[3:4], d_c, 50001, model, 7)),
                *(t.numpy().copy() for t in ctx.select_host(records(prob[:2]), 2, records(cand[:3000]), 3000, model, 7))]

    full = answers()
    ctx.debug_limit_workspace(20 * MB)
    for a, b in zip(full, answers()):
        assert np.array_equal(a, b)  # (a row's sums do not depend on the rows beside it)


def test_refused(ks, ctx):
    dev = torch.device("cuda", 0)
    cand, prob = wl.candidates_full_grid(1, 20000), wl.problems_batch(3, 40, cross_precision=False)
    model = ctx.model_create_gbdt(*wl.gbdt_complete(4, 30, 6, wl.feature_stats("cfg1"), 0.1), 0.0)
    ctx.debug_limit_workspace(MB)
    for _ in range(2):
        with pytest.raises(ks.KsError) as e:
            ctx.select(ks.to_device(prob, dev), 40, ks.to_device(cand, dev), 20000, model, 10)
        assert e.value.status == ks.KS_ERR_OOM
