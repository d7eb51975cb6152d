"""The selection of long grids, one warp per (token, head): S4-S7 against the
oracle on a sample of tokens, in both scoring forms, at the shapes where its
layout changes (k across 32 and odd, row pairs that do not split into 8
parts, m < k, ranks 1 to 4, vectors that do not split over the lanes, partial
segments of 64 keys, K beyond one round of masks), and where a warp leaves
its (token, head) to the block (long lists of ties, chunk scores that are
not finite)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_12364_gb300 import binding, workloads
from tests import parity

pytestmark = pytest.mark.gpu

B = 800   # 1600 (token, head)s
SAMPLE = np.array([0, 1, 7, 8, 63, 64, 300, 511, 640, 799])

CASES = [
    dict(topk=64, topm=64),
    dict(topk=63, topm=61),              # odd: a repeated second row
    dict(topk=33, topm=33),              # one column past a lane's first
    dict(topk=32, topm=32),
    dict(topk=24, topm=24, d_k=64),      # 12 row pairs in 8 parts
    dict(topk=5, topm=5),                # fewer row pairs than parts
    dict(topk=1, topm=1),
    dict(topk=48, topm=7),
    dict(topk=32, topm=32, rank=1),
    dict(topk=40, topm=40, rank=3, d_k=96),
    dict(topk=64, topm=64, rank=4),
    dict(topk=64, topm=64, d_k=256),     # 16 vectors a lane
    dict(topk=32, topm=32, d_k=24, rank=3),
    dict(topk=32, topm=32, rank=1, score_mode=1, act=1),
    dict(topk=64, topm=64, cores=2),
    dict(topk=64, topm=64, n=601),       # K = 1202: a partial segment (lists only)
    dict(topk=32, topm=32, n=2400),      # K = 4800: two rounds of masks
    dict(topk=32, topm=32, share_query=0),
]


def _forward(cfg, w, mode):
    x = workloads.make_tokens(cfg, B, device="cuda")
    t = parity.numpy_inputs(cfg, w, x)
    layer = binding.UltraMemLayer(
        cfg, dict(w, u=torch.from_numpy(t["u"]), t=torch.from_numpy(t["t"])), B)
    layer.candidates(mode)
    out, idx, wt = layer.forward(x, with_slots=True)
    torch.cuda.synchronize()
    assert layer.check() == 0
    layer.close()
    return t, out.float().cpu().numpy(), idx.cpu().numpy(), wt.cpu().numpy()


@pytest.mark.parametrize("mode", [0, 1], ids=["every_key", "lists"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_long_grid_selection(case, mode, gpu_lib):
    cfg = workloads.small_config(**dict(dict(dtype=1, n=600, d_k=128), **CASES[case]))
    w = workloads.make_weights(cfg, device="cuda")
    t, out, idx, wt = _forward(cfg, w, mode)
    o_out, o_idx, o_w = oracle.forward(cfg, t, B, tokens=SAMPLE)
    parity.compare(cfg, t, SAMPLE, out, idx, wt, o_out, o_idx, o_w)


@pytest.mark.parametrize("mode", [0, 1], ids=["every_key", "lists"])
@pytest.mark.parametrize("tied", [60, 500])
def test_tied_keys(tied, mode, gpu_lib):
    """Keys tied on both axes: within a warp's lists (60), and beyond them
    (500), where the block takes over; ties go to the smaller address."""
    cfg = workloads.small_config(dtype=1, n=600, d_k=128, topk=64, topm=64)
    w = workloads.make_weights(cfg, device="cuda")
    for name in ("k_row", "k_col"):
        w[name][:, 100:100 + tied] = w[name][:, :1]
    t, out, idx, wt = _forward(cfg, w, mode)
    o_out, o_idx, o_w = oracle.forward(cfg, t, B, tokens=SAMPLE)
    parity.compare(cfg, t, SAMPLE, out, idx, wt, o_out, o_idx, o_w)


def test_infinite_chunk_scores(gpu_lib):
    """A key with an infinite entry makes its axis score +-inf in every token
    of its head, so warps meet survivors that are not finite: the other
    head's selection is the one without that key's table entry changed."""
    cfg = workloads.small_config(dtype=1, n=600, d_k=128, topk=32, topm=32)
    w = workloads.make_weights(cfg, device="cuda")
    _, _, i0, w0 = _forward(cfg, w, 0)
    w["k_row"][0, 3, 0] = float("inf")
    _, _, i1, w1 = _forward(cfg, w, 0)
    assert np.array_equal(i0[:, 1], i1[:, 1]) and np.array_equal(w0[:, 1], w1[:, 1])
    K = workloads.keys_per_axis(cfg)
    assert ((i1 >= 0) & (i1 < K * K)).all()
    assert ((i1[:, 0] // K == 3).any(-1)).any()   # the key is selected where its score is +inf
