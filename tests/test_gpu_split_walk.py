"""Walks whose trees the machine's CTAs share out: block counts at the edges of the split (one block, one CTA less
than blocks, whole rounds), chunk counts that do not divide, depths of every form, both geometries. Where a
block is cut depends on its place, a candidate's score must not: a pool that repeats the same candidates
gives every copy the same score, bit for bit, and the copies rank by index."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.fixture(scope="module")
def ks():
    from paper_2609_35587_b200 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(ks):
    return ks.Context(DESC, 0)


@pytest.mark.parametrize("C,P,trees,depth,law", [(1024, 1, 9, 8, "pernode"), (1025, 1, 33, 6, "slots128"),
                                                 (60001, 1, 61, 8, "pernode"), (3000, 19, 100, 6, "hist256"),
                                                 (150500, 1, 40, 7, "pernode"), (100500, 1, 130, 8, "hist256"), (2048, 73, 70, 3, "slots128"),
                                                 (1500, 148, 25, 8, "slots128"), (9000, 3, 17, 10, "hist256")])
def test_copies_of_candidates_tie(ks, ctx, C, P, trees, depth, law):
    dev, k, period = torch.device("cuda", 0), 32, 431
    off, nodes = wl.gbdt_complete(C + trees, trees, depth, wl.feature_stats("cfg1"), 0.1, law)
    model = ctx.model_create_gbdt(off, nodes, 0.25)
    base = wl.candidates_full_grid(7, period)
    cand = base[np.arange(C) % period]
    prob = wl.problems_batch(C, P)
    d_c, d_p = ks.to_device(cand, dev), ks.to_device(prob, dev)
    idx, sc = (t.cpu().numpy() for t in ctx.select(d_p, P, d_c, C, model, k))
    for p in sorted({0, P // 2, P - 1}):
        _, _, ref = oracle.select(prob[p:p + 1], base, DESC, 1, gbdt=(off, nodes, 0.25), want_scores=True)
        # the best k, and all copies of their candidates in index order
        got, every = idx[p], ref[np.arange(C) % period]
        best = -np.sort(-every)[:k]
        tol = 1e-5 * np.maximum(1, np.abs(best))
        assert np.all(np.abs(sc[p] - ref[got % period]) <= tol) and np.all(np.abs(sc[p] - best) <= tol)
        assert set(np.flatnonzero(every > best[-1] + 2 * tol[-1])) <= set(got)
        for c in set(got % period):
            mine = got[got % period == c]
            assert len(set(sc[p][got % period == c])) == 1
            assert np.array_equal(mine, np.arange(c, C, period)[:len(mine)])
    if P == 1:
        entries_agree(ks, ctx, model, prob, d_p, d_c, C, k, idx[0], sc[0], period)


def entries_agree(ks, ctx, model, prob, d_p, d_c, C, k, idx, sc, period):
    """The single calls and the scoring call give the answer of ks_select, and copies one score."""
    one_i, one_s = ctx.select_one(prob, d_c, C, model, k)
    assert np.array_equal(one_i.numpy(), idx) and np.array_equal(one_s.numpy(), sc)
    cat = ctx.catalogue_prepare(d_c, C, model)
    one_i, one_s = ctx.select_one_prepared(cat, prob, k)
    assert np.array_equal(one_i.numpy(), idx) and np.array_equal(one_s.numpy(), sc)
    rows = ctx.featurize(d_p, 1, d_c, C)
    score = ctx.score(rows, model).cpu().numpy()
    assert np.array_equal(score[idx], sc)
    for c in range(period):
        assert len(set(score[c::period])) == 1


@pytest.mark.parametrize("C,trees,depth,law,huge", [(60001, 250, 8, "pernode", ()), (60001, 250, 8, "pernode", (1e20, 1e16, 1e12, 1e9)),
                                                    (100500, 130, 8, "slots128", (3e37, 1e9)), (9000, 300, 6, "hist256", (1e12,))])
def test_copies_tie_whatever_the_leaves(ks, ctx, C, trees, depth, law, huge):
    """Leaves of one scale over ten binades, and huge ones that cancel over the trees, where every order of
    additions has a sum of its own: blocks that are cut at different places, and blocks that are cut alike."""
    dev, k, period = torch.device("cuda", 0), 32, 431
    off, nodes = wl.gbdt_complete(C + trees, trees, depth, wl.feature_stats("cfg1"), 0.1, law)
    rng = np.random.default_rng(trees)
    leaf = nodes["feat"] == 0xFFFF
    nodes["v"][leaf] *= np.exp2(rng.integers(-5, 6, int(leaf.sum()))).astype(np.float32)
    at = rng.permutation(trees)[:2 * len(huge)].reshape(-1, 2)
    for h, (up, down) in zip(huge, at):
        nodes["v"][off[up]:off[up + 1]][leaf[off[up]:off[up + 1]]] = h
        nodes["v"][off[down]:off[down + 1]][leaf[off[down]:off[down + 1]]] = -h
    model = ctx.model_create_gbdt(off, nodes, 0.25)
    cand = wl.candidates_full_grid(7, period)[np.arange(C) % period]
    prob = wl.problems_batch(C, 1)
    d_c, d_p = ks.to_device(cand, dev), ks.to_device(prob, dev)
    idx, sc = (t.cpu().numpy() for t in ctx.select(d_p, 1, d_c, C, model, k))
    assert np.all(np.diff(sc[0]) <= 0)
    entries_agree(ks, ctx, model, prob, d_p, d_c, C, k, idx[0], sc[0], period)


@pytest.mark.parametrize("trees", [129, 300, 500, 505, 509, 512, 513, 916])
@pytest.mark.parametrize("law", ["slots128", "hist256"])
def test_chunks_keep_the_unroll_and_the_top_levels(ks, ctx, trees, law):
    """A chunk's trees are a multiple of four a thread, and padding to whole chunks leaves the top levels of up to 512
    trees in the form that holds them twice as fast."""
    model = ctx.model_create_gbdt(*wl.gbdt_complete(trees, trees, 6, wl.feature_stats("cfg1"), 0.1, law), 0.0)
    told = dict(w.split("=") for w in model.describe().split()[1:])
    assert int(told["chunk_trees"]) % 4 == 0, told
    assert told["top_levels"] == ("3" if trees <= 512 else "3c"), told
