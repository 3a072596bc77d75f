"""The walk of whole classes of candidates (ks_gbdt_classes.cu), which serves large batches against a
catalogue with many near-duplicates: the depths it compiles (5 to 8), ragged numbers of problems (a round
serves 128, 64 or 32 of them), one tree, odd tree counts, mixed element types, partition splits, per-problem
segments (one empty, one of a single candidate), k from 1 to 32, units of more than 64 candidates, and
duplicate candidates. Each test asks which walk served its calls; a few problems of each batch are compared
with the oracle, first and last among them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl
from tests.helpers import topk_accept

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()
TOL = 1e-5  # as everywhere for tree ensembles; the integer sums are off by at most 2^-31 of the sum of the largest leaves a tree


@pytest.fixture(scope="module")
def ks():
    from paper_2609_35587_b200 import binding
    return binding


@pytest.fixture(scope="module")
def ctx(ks):
    return ks.Context(DESC, 0)


def dev(ks, a):
    return ks.to_device(a, torch.device("cuda", 0))


def pool(tile_m, tile_k=None):
    c = wl.candidates_full_grid(1, None)
    keep = np.isin(c["tile_m"], tile_m)
    return np.ascontiguousarray(c[keep if tile_k is None else keep & (c["tile_k"] == tile_k)])


def check(prob, cand, gbdt, k, idx, sc, which, so=None, si=None):
    for p in which:
        seg = np.arange(len(cand), dtype=np.int32) if so is None else si[so[p]:so[p + 1]]
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, k, gbdt=gbdt, want_scores=True,
                                  seg_off=np.array([0, len(seg)], np.int64), seg_idx=seg)
        ok, msg = topk_accept(idx[p], sc[p], ref, seg, k, TOL)
        assert ok, (p, msg)


def served(ctx, call):
    """The call's answer, and whether the walk of whole classes gave it."""
    before = ctx.debug_class_walks()
    answer = call()
    return answer, ctx.debug_class_walks() - before == 1


@pytest.mark.parametrize("P,trees,depth,law,stats,k,partition", [
    (257, 37, 5, "pernode", "cfg1", 10, False), (320, 33, 6, "hist256", "cfg2", 32, True),
    (300, 1, 7, "slots128", "cfg1", 1, False), (513, 24, 8, "pernode", "cfg2", 10, True),
    (96, 50, 8, "hist256", "cfg1", 5, False)])
def test_dense_batches(ks, ctx, P, trees, depth, law, stats, k, partition):
    cand = pool([128, 192] if P < 128 else [128], None if P < 300 else 64)
    prob = wl.problems_batch(P, P, cross_precision=False) if stats == "cfg1" else wl.problems_batch(P, P)
    if P == 513:  # two element-type combinations, one of few problems
        prob["dtype_ab"][5:40], prob["dtype_d"][5:40] = 2, 1
    off, nodes = wl.gbdt_complete(depth, trees, depth, wl.feature_stats(stats), 0.1, law)
    if partition:
        nodes = wl.with_partition_splits(3, nodes)
    model = ctx.model_create_gbdt(off, nodes, 0.5)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), P, dev(ks, cand), len(cand), model, k))
    assert classes == (P != 96)  # (one round of problems does not pay for compiling units of 48)
    assert ctx.device_status() == ks.KS_OK
    check(prob, cand, (off, nodes, 0.5), k, idx.cpu().numpy(), sc.cpu().numpy(), [0, 1, 5, 39, P // 2, P - 1])


def test_segments(ks, ctx):
    cand = pool([128, 64])
    P = 330
    rng = np.random.default_rng(4)
    size = [0, 1, 30000] + [20000 + p for p in range(P - 3)]
    si = np.concatenate([np.sort(rng.permutation(len(cand))[:n]) for n in size]).astype(np.int32)
    so = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    prob = wl.problems_stream(6, P)
    off, nodes = wl.gbdt_complete(8, 20, 8, wl.feature_stats("cfg1"), 0.1)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), P, dev(ks, cand), len(cand), model, 10,
                                                        dev(ks, so), dev(ks, si), int(so[-1])))
    assert classes
    check(prob, cand, (off, nodes, 0.0), 10, idx.cpu().numpy(), sc.cpu().numpy(), [0, 1, 2, 3, 200, P - 1], so, si)


def test_large_units_and_duplicates(ks, ctx):
    """Runs of candidates that agree in the six knobs, longer than a unit (64): instruction shapes and
    schedules vary, and every candidate is there twice. Equal candidates have equal scores, so the copies
    come out in index order."""
    base = pool([256], 32)
    base = base[(base["stages"] == 4) & (base["cluster_m"] == 1) & (base["cluster_n"] == 1)]
    reps = []
    for i in range(40):
        c = base.copy()
        c["instr_k"] = 8 + 4 * (i % 5)
        c["instr_n"] = np.where(i % 2 == 0, c["tile_n"], c["tile_n"] // 4 * (1 + i % 3))
        c["tile_n"] = np.where(i % 4 == 3, 64, c["tile_n"])
        reps.append(c)
    cand = np.ascontiguousarray(np.concatenate(reps + reps))[:12000]
    cand = np.concatenate([cand, pool([64], 128)])
    prob = wl.problems_batch(9, 300)
    off, nodes = wl.gbdt_complete(2, 40, 7, wl.feature_stats("cfg1"), 0.1, "hist256")
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), 300, dev(ks, cand), len(cand), model, 32))
    assert classes
    assert ctx.device_status() == ks.KS_OK
    check(prob, cand, (off, nodes, 0.0), 32, idx.cpu().numpy(), sc.cpu().numpy(), [0, 17, 299])


def full_units(n):
    """n groups that agree in the six knobs, of 64 candidates each."""
    base = pool([64, 128, 192, 256])
    knobs = ["tile_m", "tile_n", "tile_k", "stages", "cluster_m", "cluster_n"]
    c = np.zeros((n, 64), wl.CANDIDATE_DT)
    for name in knobs:
        c[name] = np.unique(base[knobs])[:n][name][:, None]
    i = np.arange(64)
    c["kernel_sched"], c["epi_sched"], c["tile_sched"] = i % 4, i // 4 % 3, i % 2
    c["instr_m"], c["instr_n"], c["instr_k"] = 64, c["tile_n"] // (1 + i % 2), 8 + i // 4
    return np.ascontiguousarray(c.reshape(-1)[np.random.default_rng(n).permutation(64 * n)])


def test_one_round_of_problems(ks, ctx):
    """The fewest problems that are served: a single round of the slots."""
    cand, prob = full_units(80), wl.problems_batch(2, 120, cross_precision=False)
    off, nodes = wl.gbdt_complete(3, 30, 7, wl.feature_stats("cfg1"), 0.1)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), 120, dev(ks, cand), len(cand), model, 10))
    assert classes
    check(prob, cand, (off, nodes, 0.0), 10, idx.cpu().numpy(), sc.cpu().numpy(), [0, 1, 31, 32, 64, 119])


def test_classes_in_pieces(ks, ctx):
    """Units of two classes (schedules of another resident-block count) whose members alternate in the order
    of the catalogue, the larger of them too large to be compiled at once: 62 of 64 candidates, where an
    ensemble of so many tile rows leaves room for 59."""
    base = pool([64, 128, 192, 256])
    knobs = ["tile_m", "tile_n", "tile_k", "stages", "cluster_m", "cluster_n"]
    groups = np.unique(base[knobs])
    c = np.zeros((len(groups), 64), wl.CANDIDATE_DT)
    for name in knobs:
        c[name] = groups[name][:, None]
    c["kernel_sched"], c["epi_sched"] = [0] * 31 + [1] * 2 + [3] * 31, 1
    i = np.arange(64)
    c["instr_m"], c["instr_n"], c["instr_k"] = 64, c["tile_n"] // (1 + i % 2), 8 + i // 2
    prob = wl.problems_batch(4, 130)
    x = oracle.featurize(prob[:1], np.ascontiguousarray(c[:, [0, 31, 33]].reshape(-1)), DESC).reshape(-1, 3, 64)
    b = np.maximum(1, x[:, :, 55])
    cand = np.ascontiguousarray(c[(b[:, 0] == b[:, 2]) & (b[:, 0] != b[:, 1])][:70].reshape(-1))
    assert len(cand) == 70 * 64
    off, nodes = wl.gbdt_complete(5, 1000, 8, wl.feature_stats("cfg2"), 0.1)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), 130, dev(ks, cand), len(cand), model, 32))
    assert classes
    check(prob, cand, (off, nodes, 0.0), 32, idx.cpu().numpy(), sc.cpu().numpy(), range(0, 130, 6))


def test_several_planes_of_scores(ks, ctx):
    """More problems than a gigabyte of scores holds (4,224 with this pool, then the rest), and than are
    ordered by counting."""
    cand, P = wl.candidates_full_grid(1, None), 4300
    prob = wl.problems_batch(2, P, cross_precision=False)
    off, nodes = wl.gbdt_complete(3, 6, 5, wl.feature_stats("cfg1"), 0.1)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    (idx, sc), classes = served(ctx, lambda: ctx.select(dev(ks, prob), P, dev(ks, cand), len(cand), model, 10))
    assert classes
    check(prob, cand, (off, nodes, 0.0), 10, idx.cpu().numpy(), sc.cpu().numpy(), [0, 4223, 4224, 4290, P - 1])


@pytest.mark.parametrize("P,C,trees,depth,most", [(96, 20000, 500, 8, 200e6), (130, (1 << 21) + 1, 5, 5, 1.5e9)])
def test_batches_refused_on_the_host(ks, P, C, trees, depth, most):
    """Too few problems for any pool, and more candidates than a gigabyte holds the scores of 128 problems
    for: such a batch reserves no memory for this walk (240 MB of programs, 1.07 GB of scores). What it does
    reserve: 85 MB for 96 problems and half of it to grow; 16 x 2,097,153 records of 32 bytes, their classes and
    order, 1.4 GB with room."""
    ctx = ks.Context(DESC, 0)
    cand, prob = np.resize(wl.candidates_full_grid(1, None), C), wl.problems_batch(2, P, cross_precision=False)
    off, nodes = wl.gbdt_complete(3, trees, depth, wl.feature_stats("cfg1"), 0.1, "hist256")
    model, d_p, d_c = ctx.model_create_gbdt(off, nodes, 0.0), dev(ks, prob), dev(ks, cand)
    out = torch.empty((P, 3), dtype=torch.int32, device="cuda"), torch.empty((P, 3), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    _, classes = served(ctx, lambda: ctx.select(d_p, P, d_c, C, model, 3, out_idx=out[0], out_score=out[1]))
    assert not classes and free - torch.cuda.mem_get_info()[0] < most
    ctx.close()


def test_wait_runs_out(ks):
    """A chunk wait that the test hook lets run out is reported, and the next call is clean."""
    ctx = ks.Context(DESC, 0)
    cand, prob = pool([128], 64), wl.problems_batch(3, 320)
    off, nodes = wl.gbdt_complete(4, 20, 6, wl.feature_stats("cfg1"), 0.1)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    args = dev(ks, prob), 320, dev(ks, cand), len(cand), model, 10
    ctx.debug_set_wait(64, True)
    ctx.select(*args)
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT
    ctx.debug_set_wait(0, False)
    (idx, sc), classes = served(ctx, lambda: ctx.select(*args))
    assert classes and ctx.device_status() == ks.KS_OK
    check(prob, cand, (off, nodes, 0.0), 10, idx.cpu().numpy(), sc.cpu().numpy(), [0, 319])
    ctx.close()
