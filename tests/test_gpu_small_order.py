"""Batches of tree ensembles against small catalogues, which are ordered by counting (up to 8,192 candidates,
with many equal keys), and the first size that is sorted, each ranked by the candidates' own walks over whole blocks
(a split walk takes no order; the orders as the walk of whole classes uses them: test_gpu_classes.py). Scores agree to the tolerance of the other tests of tree ensembles."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl
from tests.helpers import topk_accept

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.mark.parametrize("P,C", [(520, 15), (520, 1000), (300, 4097), (150, 8191), (150, 8192), (150, 8193), (4097, 4200)])
def test_small_catalogue(P, C):
    from paper_2609_35587_b200 import binding as ks
    dev = torch.device("cuda", 0)
    prob = wl.problems_batch(P, P, cross_precision=False)
    base = wl.candidates_full_grid(1, None)
    cand = np.ascontiguousarray(base[np.random.default_rng(C).integers(0, min(len(base), 3 * C), C)])  # some twice
    off, nodes = wl.gbdt_complete(7, 20, 6, wl.feature_stats("cfg1"), 0.1, "hist256")
    ctx = ks.Context(DESC, 0)
    model = ctx.model_create_gbdt(off, nodes, 0.5)
    idx, sc = ctx.select(ks.to_device(prob, dev), P, ks.to_device(cand, dev), C, model, 10)
    assert ctx.debug_class_walks() == 0 and ctx.debug_split_walks() == 0
    idx, sc = idx.cpu().numpy(), sc.cpu().numpy()
    pool = np.arange(C, dtype=np.int32)
    for p in (0, P // 2, P - 1):
        _, _, ref = oracle.select(prob[p:p + 1], cand, DESC, 10, gbdt=(off, nodes, 0.5), want_scores=True,
                                  seg_off=np.array([0, C], np.int64), seg_idx=pool)
        ok, msg = topk_accept(idx[p], sc[p], ref, pool, 10, 1e-5)
        assert ok, (p, msg)
    ctx.close()
