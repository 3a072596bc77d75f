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
