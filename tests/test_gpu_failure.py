"""The failure path of the bounded device-side waits, exercised on a healthy GPU: a test hook makes
a wait run out (the tree kernel arms its chunk barriers for more bytes than the copies bring, the
tensor-core kernel never copies its weights), with a probe budget of about a millisecond. The
kernels must set the status word and return, the call must report KS_ERR_TIMEOUT, nothing may
fault, and the next ordinary call on the same context must give the oracle's result."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.fixture()
def ks():
    from paper_2609_35587_b200 import binding
    return binding


def dev(ks, a):
    return ks.to_device(a, torch.device("cuda", 0))


def assert_matches_oracle(w, idx, sc, tol):
    ridx, rsc = oracle.select(w.problems, w.candidates, w.desc, w.k, gbdt=w.gbdt, mlp=w.mlp)
    if w.gbdt is not None:
        assert np.array_equal(idx, ridx)
    assert np.all(np.abs(sc - rsc) <= tol * np.maximum(1, np.abs(rsc)))


@pytest.mark.parametrize("law,starve", [("slots128", 1), ("pernode", 1), ("slots128", 3), ("pernode", 3)])
def test_tree_kernel_wait_runs_out(ks, law, starve):
    """With 1 the first chunk of every walk does not arrive, with 3 the tile of every split walk."""
    ctx = ks.Context(DESC, 0)
    w = wl.make_workload(1, P=3, C=2500, trees=60, law=law)
    model = ctx.model_create_gbdt(*w.gbdt)
    assert "select_fast_kernel" in model.describe()
    d_p, d_c = dev(ks, w.problems), dev(ks, w.candidates)
    cat = ctx.catalogue_prepare(d_c, 2500, model)
    ctx.debug_set_wait(2000, starve)
    # asynchronous batch call: the status word tells
    ctx.select(d_p, 3, d_c, 2500, model, w.k)
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT
    assert ctx.device_status() == ks.KS_OK          # reported once, then cleared
    # host-buffer call and single-problem calls report it themselves
    with pytest.raises(ks.KsError) as e:
        ctx.select_host(w.problems, 3, w.candidates, 2500, model, w.k)
    assert e.value.status == ks.KS_ERR_TIMEOUT
    with pytest.raises(ks.KsError) as e:
        ctx.select_one(w.problems[:1], d_c, 2500, model, w.k)
    assert e.value.status == ks.KS_ERR_TIMEOUT
    with pytest.raises(ks.KsError) as e:
        ctx.select_one_prepared(cat, w.problems[:1], w.k)
    assert e.value.status == ks.KS_ERR_TIMEOUT
    # scoring call on the same walk
    x = oracle.featurize(w.problems[:1], w.candidates, DESC)
    ctx.score(dev(ks, x), model)
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT
    # back to normal: same context, same model
    ctx.debug_set_wait(0, False)
    idx, sc = ctx.select(d_p, 3, d_c, 2500, model, w.k)
    assert ctx.device_status() == ks.KS_OK
    assert_matches_oracle(w, idx.cpu().numpy(), sc.cpu().numpy(), 1e-5)
    hi, hs = ctx.select_one(w.problems[1:2], d_c, 2500, model, w.k)
    assert np.array_equal(hi.numpy(), idx[1].cpu().numpy())
    hi, hs = ctx.select_one_prepared(cat, w.problems[1:2], w.k)
    assert np.array_equal(hi.numpy(), idx[1].cpu().numpy())
    s = ctx.score(dev(ks, x), model).cpu().numpy()
    rs = oracle.score_gbdt(x, *w.gbdt)
    assert np.all(np.abs(s - rs) <= 1e-5 * np.maximum(1, np.abs(rs)))
    ctx.close()


def test_short_probe_budget_alone_does_not_fail(ks):
    """The budget used above (2,000 probes) is ample for a healthy copy: without the hook the same
    call succeeds."""
    ctx = ks.Context(DESC, 0)
    w = wl.make_workload(1, P=3, C=2500, trees=60)
    model = ctx.model_create_gbdt(*w.gbdt)
    ctx.debug_set_wait(2000, False)
    idx, sc = ctx.select(dev(ks, w.problems), 3, dev(ks, w.candidates), 2500, model, w.k)
    assert ctx.device_status() == ks.KS_OK
    assert_matches_oracle(w, idx.cpu().numpy(), sc.cpu().numpy(), 1e-5)
    ctx.close()


def test_tensor_core_kernel_wait_runs_out(ks):
    ctx = ks.Context(DESC, 0)
    w = wl.make_workload(4, P=2, C=1500)
    model = ctx.model_create_mlp(w.mlp)
    assert "select_mlp_tc_kernel" in model.describe()
    d_p, d_c = dev(ks, w.problems), dev(ks, w.candidates)
    ctx.debug_set_wait(64, True)
    ctx.select(d_p, 2, d_c, 1500, model, w.k)
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT
    x = oracle.featurize(w.problems[:1], w.candidates, DESC)
    ctx.score(dev(ks, x), model)
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT
    ctx.debug_set_wait(0, False)
    idx, sc = ctx.select(d_p, 2, d_c, 1500, model, w.k)
    assert ctx.device_status() == ks.KS_OK
    _, _, allsc = oracle.select(w.problems, w.candidates, DESC, w.k, mlp=w.mlp, want_scores=True)
    got_i, got_s = idx.cpu().numpy(), sc.cpu().numpy()
    for i in range(2):
        ref = allsc[i * 1500:(i + 1) * 1500]
        assert np.all(np.abs(got_s[i] - ref[got_i[i]]) <= 2e-2 * np.maximum(1, np.abs(ref[got_i[i]])))
    ctx.close()


@pytest.mark.parametrize("C", [300, 20000])
def test_valid_catalogue_after_a_failed_walk(ks, C):
    """A split walk of which every other block's waits run out leaves arrival counters behind until the status
    is read. The count of valid candidates, which the last block of a pass tells the host, is its own all the same."""
    ctx = ks.Context(DESC, 0)
    w = wl.make_workload(1, P=1, C=1000, trees=200)
    model = ctx.model_create_gbdt(*w.gbdt)
    pool = dev(ks, oracle.enumerate_candidates(150000, C, wl.CANDIDATE_DT))
    want = {f: len(oracle.valid_catalogue(w.problems[:1], DESC, f, pool.cpu().numpy().view(wl.CANDIDATE_DT).reshape(-1),
                                          dtype=wl.CANDIDATE_DT)[0]) for f in (0, 1)}
    assert want[0] != want[1]
    assert ctx.valid_catalogue(w.problems[:1], 1, pool, C)[2] == want[1]
    ctx.debug_set_wait(2000, 2)
    ctx.select(dev(ks, w.problems), 1, dev(ks, w.candidates), 1000, model, w.k)
    ctx.debug_set_wait(0, 0)
    for f in (0, 1, 0):
        out, _, n = ctx.valid_catalogue(w.problems[:1], f, pool, C)
        assert n == want[f]
    assert ctx.device_status() == ks.KS_ERR_TIMEOUT  # (of the walk)
    hi, hs = ctx.select_one(w.problems[:1], dev(ks, w.candidates), 1000, model, w.k)
    assert_matches_oracle(w, hi.numpy()[None], hs.numpy()[None], 1e-5)
    ctx.close()


CHILD = """
import resource, numpy as np
from paper_2609_35587_b200 import binding as ks, workloads as wl
ctx = ks.Context(wl.gpu_desc(), 0)
st = wl.feature_stats("cfg1")
gbdt = wl.gbdt_complete(1, 4000, 8, st, 0.1, "slots128")  # 2 M nodes, 16 MB in the library's form
mlp = wl.mlp_xavier(1, [64, 1024, 1024, 1024, 1024, 1024, 1], st["mu"], st["sigma"])  # a weight image of 8.5 MB
small = wl.gbdt_complete(1, 3, 4, st, 0.1), wl.mlp_xavier(1, [64, 320, 1], st["mu"], st["sigma"])
ctx.model_create_gbdt(*small[0]).close(), ctx.model_create_mlp(small[1]).close()
soft, hard = resource.getrlimit(resource.RLIMIT_AS)
size = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (size + (3 << 20), hard))
got = []
for create, model in ((ctx.model_create_gbdt, gbdt), (ctx.model_create_mlp, (mlp,))):
    try:
        create(*model)
        got.append(ks.KS_OK)
    except ks.KsError as e:
        got.append(e.status)
resource.setrlimit(resource.RLIMIT_AS, (soft, hard))
ctx.model_create_gbdt(*small[0]).close(), ctx.model_create_mlp(small[1]).close()
print("statuses", got)
"""


def test_host_memory_runs_out(ks):
    """Creating a model where the host has no memory for its repacked form: a status, no exception across
    the C boundary (which would end the process)."""
    import os
    import subprocess
    import sys
    env = dict(os.environ, MALLOC_MMAP_THRESHOLD_="65536")  # large blocks are new mappings, not reused ones
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=120, env=env)
    assert r.returncode == 0, r.stderr[-2000:]
    assert f"statuses [{ks.KS_ERR_OOM}, {ks.KS_ERR_OOM}]" in r.stdout, r.stdout
