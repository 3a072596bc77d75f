"""Tree ensembles on batches too small to fill the machine, whose tiles are built in front of a walk that
splits the trees: both sides of the rule that splits them, one problem and many, ragged pools, mixed element
types, segments of unequal length (never split), depth 6. Scores agree to the tolerance of the other tests of tree ensembles."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl
from tests.helpers import topk_accept

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()
TOL = 1e-5


@pytest.mark.parametrize("P,C,trees,depth,k,segmented", [
    (1, 30011, 60, 8, 10, False), (2, 1025, 33, 7, 10, False), (7, 5011, 60, 6, 10, False), (31, 517, 400, 6, 32, False),
    (32, 517, 400, 5, 10, False), (64, 2048, 100, 6, 5, False),
    (40, 1024, 90, 6, 32, False), (300, 1000, 30, 6, 1, False), (40, 700, 30, 6, 10, True)])
def test_select(P, C, trees, depth, k, segmented):
    from paper_2609_35587_b200 import binding as ks
    dev = torch.device("cuda", 0)
    prob = wl.problems_batch(P, P, cross_precision=True)
    cand = wl.candidates_full_grid(1, None)[:C] if not segmented else wl.make_inputs(2, P=5, seg=1)[1]
    off, nodes = wl.gbdt_complete(depth, trees, depth, wl.feature_stats("cfg2"), 0.1, "pernode")
    ctx = ks.Context(DESC, 0)
    model = ctx.model_create_gbdt(off, nodes, 0.1)
    so = si = None
    if segmented:
        lens = np.full(P, C)
        lens[0] += 100
        so = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
        si = (np.arange(so[-1]) * 7 % len(cand)).astype(np.int32)
    args = () if so is None else (ks.to_device(so, dev), ks.to_device(si, dev), int(so[-1]))
    d_p, d_c = ks.to_device(prob, dev), ks.to_device(cand, dev)
    for _ in range(2):
        idx, sc = ctx.select(d_p, P, d_c, len(cand), model, k, *args)
        torch.cuda.synchronize()
    idx, sc = idx.cpu().numpy(), sc.cpu().numpy()
    for p in {0, P // 3, P // 2, P - 1}:
        seg = np.arange(len(cand), dtype=np.int32) if so is None else si[so[p]:so[p + 1]]
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, k, gbdt=(off, nodes, 0.1), want_scores=True,
                                  seg_off=np.array([0, len(seg)], np.int64), seg_idx=seg)
        ok, msg = topk_accept(idx[p], sc[p], ref, seg, k, TOL)
        assert ok, (p, msg)
    ctx.close()


@pytest.mark.parametrize("P,length,law", [(40, 300, "pernode"), (70, 4096, "hist256"), (33, 4097, "slots128"), (33, 700, "slots128")])
def test_short_segments_of_many_classes(P, length, law):
    """Segments shorter than the classes of the pool (more than 4,096 for a type combination), whose problems have no class
    records: the same bits as a batch too small for records, and the oracle's ranking."""
    from paper_2609_35587_b200 import binding as ks
    dev = torch.device("cuda", 0)
    ctx = ks.Context(DESC, 0)
    prob = wl.problems_batch(P, P, cross_precision=True)
    rec, _, n = ctx.valid_catalogue(prob[:1], ks.KS_VALID_COUPLED)
    d_c = rec[torch.arange(30000, device=dev) * n // 30000].contiguous()
    cand = d_c.cpu().numpy().view(wl.CANDIDATE_DT).reshape(-1)
    assert len(np.unique(cand[["tile_m", "tile_n", "tile_k", "stages", "cluster_m", "cluster_n"]])) > 4097
    gbdt = (*wl.gbdt_complete(3, 40, 7, wl.feature_stats("cfg2"), 0.1, law), 0.1)
    model = ctx.model_create_gbdt(*gbdt)
    rng = np.random.default_rng(P)
    si = np.concatenate([np.sort(rng.choice(len(cand), length, replace=False)) for _ in range(P)]).astype(np.int32)
    so = (np.arange(P + 1) * length).astype(np.int64)

    def ranked(first, count):
        part = si[first * length:(first + count) * length]
        idx, sc = ctx.select(ks.to_device(prob[first:first + count], dev), count, d_c, len(cand), model, 10,
                             ks.to_device(so[:count + 1], dev), ks.to_device(part, dev), len(part))
        return idx.cpu().numpy(), sc.cpu().numpy()

    idx, sc = ranked(0, P)
    for first, count in ((0, 3), (P - 20, 20)):  # (records: 32 problems or more)
        some = ranked(first, count)
        assert np.array_equal(some[0], idx[first:first + count]) and np.array_equal(some[1], sc[first:first + count])
    for p in (0, P - 1):
        seg = si[so[p]:so[p + 1]]
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 10, gbdt=gbdt, want_scores=True,
                                  seg_off=np.array([0, length], np.int64), seg_idx=seg)
        ok, msg = topk_accept(idx[p], sc[p], ref, seg, 10, TOL)
        assert ok, (p, msg)
    ctx.close()
