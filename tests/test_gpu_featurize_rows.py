"""The segmented feature kernel at the sizes where it can go wrong: empty segments, one row, the edges of a
warp's 32 rows and of a block's 256, segments that a block takes in several slabs, and an output that does
not start on an 8-byte boundary. Feature rows are equal bit by bit to the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_35587_b200 import workloads as wl

pytestmark = pytest.mark.gpu
DESC = wl.gpu_desc()


@pytest.mark.parametrize("P,longest", [(6, 300), (900, 2100)])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_segments(P, longest, shift):
    from paper_2609_35587_b200 import binding as ks
    device = torch.device("cuda", 0)
    prob = wl.problems_batch(P, P, cross_precision=True)
    cand = wl.make_inputs(2, P=5, seg=1)[1]
    lens = np.resize([0, 1, 31, 32, 33, 255, 256, 257], P)
    lens[P // 2] = longest
    so = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    si = (np.arange(so[-1]) * 7 % len(cand)).astype(np.int32)
    ctx = ks.Context(DESC, 0)
    flat = torch.full((int(so[-1]) * 64 + 4,), -1.0, device=device)
    out = flat[shift:shift + int(so[-1]) * 64].view(-1, 64)
    ctx.featurize(*(x for a in (prob, cand) for x in (ks.to_device(a, device), len(a))), ks.to_device(so, device),
                  ks.to_device(si, device), int(so[-1]), out=out)
    torch.cuda.synchronize()
    ref = oracle.featurize(prob, cand, DESC, so, si)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))
    edge = flat.cpu().numpy()
    assert (edge[:shift] == -1).all() and (edge[shift + ref.size:] == -1).all()
    ctx.close()


@pytest.mark.parametrize("sms", [1, 148, 65535, 65536, 200000])
def test_tile_counts_around_32_bits(sms):
    """Problems and tiles whose counts lie on both sides of 2^15 a side (up to 2^38 tiles), and
    descriptors on both sides of 2^16 SMs: the 32-bit and the 64-bit arithmetic give the oracle's bits."""
    from paper_2609_35587_b200 import binding as ks
    device = torch.device("cuda", 0)
    desc = DESC.copy()
    desc["num_sms"] = sms
    dims = np.array([1, 15, 4096, 32767, 32768, 32769, 65536, 524272, 524288], dtype=np.uint32)
    prob = wl.problems_batch(3, 81, cross_precision=True)
    prob["m"], prob["n"] = np.repeat(dims, 9), np.tile(dims, 9)
    prob["k"] = np.resize(dims[::-1], 81)
    cand = wl.candidates_full_grid(9, 40)
    cand["tile_m"] = np.resize([1, 16, 64, 256, 4095], 40)
    cand["tile_n"] = np.resize([1, 1, 16, 128, 512, 7], 40)
    cand["cluster_m"], cand["cluster_n"] = np.resize([1, 2, 3, 16], 40), np.resize([1, 4, 5], 40)
    ctx = ks.Context(desc, 0)
    out = ctx.featurize(ks.to_device(prob, device), 81, ks.to_device(cand, device), 40)
    ref = oracle.featurize(prob, cand, desc)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32).reshape(out.shape))
    ctx.close()
