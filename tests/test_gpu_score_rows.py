"""Scoring of given rows by ensembles with few thresholds and with nearly as many as the quantised walk takes
(40,000), at the edges of a group of 128 rows and over more groups than are resident: NaN and infinite
values, columns that no tree reads. Scores agree to the tolerance of the other tests of this model."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.mark.parametrize("trees,rows", [(3, 1), (40, 127), (180, 129), (40, 70001), (180, 8321)])
def test_rows(trees, rows):
    from paper_2609_35587_b200 import binding as ks
    device = torch.device("cuda", 0)
    w = wl.make_workload(1, P=24, C=3000, trees=trees, depth=8)
    off, nodes, base = w.gbdt
    # a threshold of its own for every numeric split, around the values the columns take
    rng = np.random.default_rng(trees)
    nodes = nodes.copy()
    x = oracle.featurize(w.problems, w.candidates, DESC)[:rows].copy()
    split = (nodes["feat"] != 0xFFFF) & (nodes["kind"] == 0)
    split &= ~np.isin(nodes["feat"], list(wl.CATEGORICAL_LEVELS))
    thr = nodes["v"][split]
    nodes["v"][split] = (thr * (1 + rng.uniform(-1e-3, 1e-3, thr.size))).astype(np.float32)
    numeric = np.array([c for c in range(63) if c not in wl.CATEGORICAL_LEVELS])
    for v in (np.nan, np.inf, -np.inf):
        x[rng.integers(0, rows, 60), numeric[rng.integers(0, len(numeric), 60)]] = v
    ctx = ks.Context(DESC, 0)
    model = ctx.model_create_gbdt(off, nodes, base)
    assert "select_fast_kernel" in model.describe()
    got = ctx.score(ks.to_device(x, device), model).cpu().numpy()
    ref = oracle.score_gbdt(x, off, nodes, base)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(1, np.abs(ref)))
    ctx.close()


def test_more_thresholds_than_are_staged(monkeypatch):
    """Small chunk buffers leave room for 408 rows of 127 thresholds, more than the kernel that builds tiles
    from rows can hold: such an ensemble (here 400 rows, 50,800 thresholds) takes the general kernel."""
    from paper_2609_35587_b200 import binding as ks
    monkeypatch.setenv("KS_FAST_GEOMETRY", "512,512,8")
    device = torch.device("cuda", 0)
    prob, cand, _, _ = wl.make_inputs(2, P=2, seg=1)
    x = oracle.featurize(prob, cand[:300], DESC)
    off, nodes = wl.gbdt_complete(3, 200, 8, wl.feature_stats("cfg2"), 0.1)
    nodes = nodes.copy()
    rng = np.random.default_rng(5)
    per = np.where(np.arange(63) < 41, 6 * 127, 7 * 127)
    feat = np.repeat(np.arange(63), per)
    lo, hi = x[:, :63].min(0), x[:, :63].max(0)
    thr = np.concatenate([np.linspace(lo[f], hi[f] + 1, n, dtype=np.float64) for f, n in enumerate(per)]).astype(np.float32)
    split = np.flatnonzero(nodes["feat"] != 0xFFFF)
    order = rng.permutation(len(split)) % len(feat)
    nodes["feat"][split], nodes["v"][split] = feat[order], thr[order]
    ctx = ks.Context(DESC, 0)
    model = ctx.model_create_gbdt(off, nodes, 0.0)
    assert "select_generic_kernel" in model.describe()
    got = ctx.score(ks.to_device(x, device), model).cpu().numpy()
    ref = oracle.score_gbdt(x, off, nodes, 0.0)
    assert np.all(np.abs(got - ref) <= 1e-5 * np.maximum(1, np.abs(ref)))
    ctx.close()
