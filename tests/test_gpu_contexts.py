"""Two contexts of one process whose calls overlap on the GPU: batches that the walk of whole classes serves on
one stream, and on another every other form of the tree kernel (a dense batch, segments, a batch whose trees
are split, single calls prepared and not, given rows) and the rankers. Each answer equals its own of a serial
run, bit for bit: what makes CTAs leave a launch belongs to a context."""
import numpy as np
import pytest
import torch

from paper_2609_35587_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.fixture(scope="module")
def ks():
    from paper_2609_35587_b200 import binding
    return binding


def trees(ctx, seed, n, depth, law="pernode"):
    return ctx.model_create_gbdt(*wl.gbdt_complete(seed, n, depth, wl.feature_stats("cfg1"), 0.1, law), 0.0)


def calls(ks, ctx):
    """What the second context is asked: name -> function that returns host arrays."""
    dev = torch.device("cuda", 0)
    put = lambda a: ks.to_device(a, dev)
    cand = wl.candidates_full_grid(2, 20000)
    prob = wl.problems_batch(5, 64, cross_precision=False)
    d_p, d_c = put(prob), put(cand)
    model = trees(ctx, 3, 60, 8)
    rows = ctx.featurize(d_p, 4, d_c, 3000, pairs=12000)
    so = torch.arange(0, 49, device=dev, dtype=torch.int64) * 5000
    si = torch.cat([torch.arange(p, 20000, 4, device=dev, dtype=torch.int32)[:5000] for p in range(4)] * 12).contiguous()
    st = wl.feature_stats("cfg1")
    narrow = ctx.model_create_mlp(wl.mlp_xavier(1, [64, 256, 256, 1], st["mu"], st["sigma"]))
    wide = ctx.model_create_mlp(wl.mlp_xavier(1, [64, 512, 256, 1], st["mu"], st["sigma"]))
    cat = ctx.catalogue_prepare(d_c, 20000, model)
    host = lambda pair: tuple(t.cpu().numpy().copy() for t in pair)
    return {
        "dense": lambda: host(ctx.select(d_p, 64, d_c, 20000, model, 10)),
        "segments": lambda: host(ctx.select(d_p, 48, d_c, 20000, model, 10, so, si, si.numel())),
        "split": lambda: host(ctx.select(d_p, 3, d_c, 20000, model, 10)),
        "one": lambda: host(ctx.select_one(prob[7:8], d_c, 20000, model, 10)),
        "prepared": lambda: host(ctx.select_one_prepared(cat, prob[9:10], 10)),
        "rows": lambda: (ctx.score(rows, model).cpu().numpy(),),
        "narrow": lambda: host(ctx.select(d_p, 2, d_c, 20000, narrow, 10)),
        "wide": lambda: host(ctx.select(d_p, 2, d_c, 20000, wide, 10)),
    }


def test_overlapping_contexts(ks):
    dev = torch.device("cuda", 0)
    a, b = ks.Context(DESC, 0), ks.Context(DESC, 0)
    cand, prob = wl.candidates_full_grid(1, 60000), wl.problems_batch(7, 512, cross_precision=False)
    d_p, d_c, model = ks.to_device(prob, dev), ks.to_device(cand, dev), trees(a, 1, 100, 8)
    alone = [t.clone() for t in a.select(d_p, 512, d_c, 60000, model, 10)]
    asked = calls(ks, b)
    serial, split = {}, set()
    for name, f in asked.items():
        before = b.debug_split_walks()
        serial[name] = f()
        if b.debug_split_walks() > before:
            split.add(name)
    assert split == {"split", "one", "prepared", "rows"}
    torch.cuda.synchronize()
    s_a, s_b = torch.cuda.Stream(), torch.cuda.Stream()
    n = 120
    with torch.cuda.stream(s_a):
        batches = [a.select(d_p, 512, d_c, 60000, model, 10) for _ in range(n)]  # queued, some tenths of a second
    rounds = 0
    with torch.cuda.stream(s_b):
        while True:
            for name, f in asked.items():
                for got, want in zip(f(), serial[name]):
                    assert np.array_equal(got, want), (rounds, name)
            rounds += 1
            if s_a.query():
                break
    s_a.synchronize()
    assert rounds >= 2  # (or nothing ran beside anything)
    for idx, score in batches:
        assert torch.equal(idx, alone[0]) and torch.equal(score, alone[1])
    assert a.device_status() == ks.KS_OK and b.device_status() == ks.KS_OK
