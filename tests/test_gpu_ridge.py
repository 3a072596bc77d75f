"""The linear scorer's kernels at the sizes where they can go wrong: dense batches ranked by classes (30 problems
and 600,000 pairs or more) and pair by pair, segments with the class tables, element types that change from problem
to problem, more classes than are staged (2,048) and more than there are slots (16,384), small
and ragged pools, k = 1, 10 and 32. The sums run in the same order as the oracle's problem, candidate and
pair parts do not, so scores agree to 1e-4 as in the other tests of this scorer."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl
from tests.helpers import topk_accept

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.fixture(scope="module")
def ks():
    from paper_2609_35587_b200 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(ks):
    return ks.Context(DESC, 0)


@pytest.mark.parametrize("P,C,k,valid,onehot", [(5, 1, 1, False, False), (31, 513, 32, False, True),
                                                (32, 4097, 10, False, False), (37, 20000, 32, True, False),
                                                (66, 61000, 10, True, True), (150, 3000, 1, False, False)])
def test_select_linear(ks, ctx, P, C, k, valid, onehot):
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    mu, sg = wl.onehot_stats(st["mu"], st["sigma"]) if onehot else (st["mu"], st["sigma"])
    mlp = wl.mlp_xavier(P, [80 if onehot else 64, 1], mu, sg)
    model = ctx.model_create_mlp(mlp)
    prob = wl.problems_batch(P, P, cross_precision=True)
    if valid:
        rec, _, n = ctx.valid_catalogue(prob[:1], ks.KS_VALID_COUPLED)
        d_c = rec[torch.arange(min(C, n), device=dev) * n // min(C, n)].contiguous()
        cand = d_c.cpu().numpy().view(wl.CANDIDATE_DT).reshape(-1)
    else:
        cand = wl.candidates_full_grid(3, C)
        d_c = ks.to_device(cand, dev)
    idx, sc = ctx.select(ks.to_device(prob, dev), P, d_c, len(cand), model, k)
    idx, sc = idx.cpu().numpy(), sc.cpu().numpy()
    pool = np.arange(len(cand), dtype=np.int32)
    for p in sorted({0, 1, 3, P // 2, P - 2, P - 1}):
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, k, mlp=mlp, want_scores=True)
        ok, msg = topk_accept(idx[p], sc[p], ref, pool, k, 1e-4)
        assert ok, (p, msg)


@pytest.mark.parametrize("P,n", [(1, 1480), (3, 40), (1200, 90), (1184, 300), (2, 5000)])
def test_merge_of_partial_lists(ks, ctx, P, n):
    """A block or a warp per problem, numbers of keys around their steps: the static score, whose
    ranking is exact, on pools that give n partial lists' worth of keys."""
    C = min(60000, max(1, n // 10 * 1024))
    model = ctx.model_create_static()
    prob, cand, _, _ = wl.make_inputs(3, P=P, C=C)
    dev = torch.device("cuda", 0)
    idx, sc = ctx.select(ks.to_device(prob, dev), P, ks.to_device(cand, dev), C, model, 10)
    some = sorted({0, P // 2, P - 1})
    ridx, rsc = oracle.select(prob[some], cand, DESC, 10, static=True)
    assert np.array_equal(idx.cpu().numpy()[some], ridx) and np.array_equal(sc.cpu().numpy()[some], rsc)


@pytest.mark.parametrize("P,C", [(8192, 300), (8193, 300), (8195, 70), (40, 0), (31, 0)])
def test_problems_beyond_the_class_tables(ks, ctx, P, C):
    """More problems than blocks, on pools small enough to be ranked pair by pair and on either side of 600,000
    pairs. An empty pool gives empty lists."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    mlp = wl.mlp_xavier(2, [64, 1], st["mu"], st["sigma"])
    prob, cand = wl.problems_batch(P, P, cross_precision=True), wl.candidates_full_grid(3, 300)[:C]
    idx = torch.full((P, 5), 7, dtype=torch.int32, device=dev)
    sc = torch.full((P, 5), 7.0, device=dev)
    ctx.select(ks.to_device(prob, dev), P, ks.to_device(cand, dev) if C else None, C, ctx.model_create_mlp(mlp), 5,
               out_idx=idx, out_score=sc)
    idx, sc = idx.cpu().numpy(), sc.cpu().numpy()
    if C == 0:
        assert (idx == -1).all() and np.isneginf(sc).all()
        return
    for p in (0, 1, P // 4, P // 4 + 1, P - 2, P - 1):
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 5, mlp=mlp, want_scores=True)
        ok, msg = topk_accept(idx[p], sc[p], ref, np.arange(C, dtype=np.int32), 5, 1e-4)
        assert ok, (p, msg)


@pytest.mark.parametrize("what,P,C,k", [("plain", 30, 60000, 10), ("plain", 1040, 600, 32), ("valid", 33, 61140, 7),
                                        ("no class", 40, 15001, 10), ("full", 32, 20000, 10), ("ties", 32, 18755, 32), ("not finite", 32, 19000, 10),
                                        ("many", 8200, 80, 3)])
def test_classes_against_pairs(ks, ctx, what, P, C, k):
    """A dense batch ranked by classes gives bit for bit what its pairs give one by one: the same pool as a
    segment of every problem takes the kernel that adds up each pair. Candidates without a class (a
    tile of 4,096 or more, or more classes than slots: there both kernels evaluate some in place, so the oracle is
    asked too), equal scores everywhere, scores that are not finite; more problems than blocks."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    mlp = wl.mlp_xavier(C, [64, 1], st["mu"], st["sigma"])
    w = mlp["weights"][0]  # bf16 bits
    if what == "ties":
        w[:] = 0
    if what == "not finite":
        w[0, 46] = 0x7F80  # +inf on a candidate column: inf, -inf or (0 inf) not a number
    model = ctx.model_create_mlp(mlp)
    prob = wl.problems_batch(C, P, cross_precision=True)
    if what == "valid":
        rec, _, n = ctx.valid_catalogue(prob[:1], ks.KS_VALID_COUPLED)
        C, d_c = min(C, n), rec[:min(C, n)].contiguous()
    else:
        cand = wl.candidates_full_grid(5, C)
        if what == "no class":
            cand["tile_m"][::50] = 4096
        if what == "full":  # 20,000 classes
            i = np.arange(C)
            cand["tile_m"], cand["tile_n"] = 16 * (1 + i % 16), 8 * (1 + i // 16 % 32)
            cand["tile_k"], cand["stages"] = 16 * (1 + i // 512 % 32), 2 + i // 16384
            cand["cluster_m"] = cand["cluster_n"] = 1
        d_c = ks.to_device(cand, dev)
    d_p = ks.to_device(prob, dev)
    idx, sc = ctx.select(d_p, P, d_c, C, model, k)
    off = torch.arange(P + 1, device=dev, dtype=torch.int64) * C
    every = torch.arange(C, device=dev, dtype=torch.int32).repeat(P)
    ridx, rsc = ctx.select(d_p, P, d_c, C, model, k, off, every, P * C)
    assert torch.equal(idx, ridx)
    assert torch.equal(sc.view(torch.int32), rsc.view(torch.int32))
    if what == "full":
        for p in (0, P - 1):
            _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, k, mlp=mlp, want_scores=True)
            ok, msg = topk_accept(idx[p].cpu().numpy(), sc[p].cpu().numpy(), ref, np.arange(C, dtype=np.int32), k, 1e-4)
            assert ok, (p, msg)


@pytest.mark.parametrize("P,C,classes", [(31, 58064, False), (31, 58065, True), (32, 18749, False), (32, 18750, True)])
def test_which_batches_go_by_classes(ks, ctx, P, C, classes):
    """Five kernels and the merge, or pair by pair three and the merge."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    model = ctx.model_create_mlp(wl.mlp_xavier(2, [64, 1], st["mu"], st["sigma"]))
    args = ks.to_device(wl.problems_batch(P, P), dev), P, ks.to_device(wl.candidates_full_grid(3, C), dev), C, model, 10
    n = ctx.launch_count()
    ctx.select(*args)
    assert ctx.launch_count() - n == (6 if classes else 4)


@pytest.mark.parametrize("P,length,onehot", [(40, 300, False), (33, 4096, True), (33, 4097, False), (64, 11000, False)])
def test_short_segments_of_many_classes(ks, ctx, P, length, onehot):
    """Segments shorter than the pool's classes are added up pair by pair, longer ones from the class sums: the bits of
    batches too small for class tables either way."""
    dev = torch.device("cuda", 0)
    st = wl.feature_stats("cfg2")
    mu, sg = wl.onehot_stats(st["mu"], st["sigma"]) if onehot else (st["mu"], st["sigma"])
    mlp = wl.mlp_xavier(P, [80 if onehot else 64, 1], mu, sg)
    model = ctx.model_create_mlp(mlp)
    prob = wl.problems_batch(P, P, cross_precision=True)
    rec, _, n = ctx.valid_catalogue(prob[:1], ks.KS_VALID_COUPLED)
    d_c = rec[:n].contiguous()
    rng = np.random.default_rng(P)
    si = np.concatenate([np.sort(rng.choice(n, length, replace=False)) for _ in range(P)]).astype(np.int32)

    def ranked(first, count):
        part = si[first * length:(first + count) * length]
        so = (np.arange(count + 1) * length).astype(np.int64)
        idx, sc = ctx.select(ks.to_device(prob[first:first + count], dev), count, d_c, n, model, 10,
                             ks.to_device(so, dev), ks.to_device(part, dev), len(part))
        return idx.cpu().numpy(), sc.cpu().numpy()

    idx, sc = ranked(0, P)
    for first, count in ((0, 31), (P - 5, 5)):
        some = ranked(first, count)
        assert np.array_equal(some[0], idx[first:first + count]) and np.array_equal(some[1], sc[first:first + count])
    cand = d_c.cpu().numpy().view(wl.CANDIDATE_DT).reshape(-1)
    for p in (0, P - 1):
        seg = si[p * length:(p + 1) * length]
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 10, mlp=mlp, want_scores=True,
                                  seg_off=np.array([0, length], np.int64), seg_idx=seg)
        ok, msg = topk_accept(idx[p], sc[p], ref, seg, 10, 1e-4)
        assert ok, (p, msg)
