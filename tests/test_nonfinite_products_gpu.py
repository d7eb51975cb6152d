"""Infinite entries in W_p (lookup_reduce, shard_pool) and in the gradient
(dW_p of token counts that are not whole 16-byte rows) give what plain sums of
products give: an infinity, and a NaN only for 0 * inf or inf - inf.  The
pooled values are bf16 values, whose smaller terms are zero."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def _layer(B, d_out):
    cfg = workloads.small_config(dtype=1, expand_e=1, heads=1, topk=1, topm=1, n=24, d_v=256,
                                 d_out=d_out, shuffle_seed=0)
    w = workloads.make_weights(cfg, device="cuda")
    w["values"][:, 7] = 0
    w["values"][3] = 0
    gen = torch.Generator(device="cuda").manual_seed(2)
    idx = torch.randint(0, 24 * 24, (B, 1, 1), generator=gen, device="cuda")
    idx[0] = 3                                     # a pooled row of zeros
    return cfg, w, idx, torch.ones((B, 1, 1), device="cuda"), gen


def _same_kind(got, want):
    got = got.double()
    assert torch.equal(got.isnan(), want.isnan())
    assert torch.equal(got == float("inf"), want == float("inf"))
    assert torch.equal(got == -float("inf"), want == -float("inf"))


@pytest.mark.parametrize("B,d_out", [(5, 1024), (100, 1024), (127, 16384), (700, 1024),
                                     (2000, 2048)])
@pytest.mark.parametrize("shard", [False, True])
def test_infinite_projectors(B, d_out, shard, gpu_lib):
    cfg, w, idx, wt, _ = _layer(B, d_out)
    W = w["w_proj"][0]
    W[2, 5] = float("inf")
    W[9, 64] = -float("inf")
    W[7, 100] = float("inf")                       # meets pooled zeros only
    W[2, 300], W[3, 300] = float("inf"), float("-inf")
    W[4, 301] = float("nan")
    layer = binding.UltraMemLayer(cfg, w, B)
    if shard:
        counts, rows, pos = layer.shard_route(idx, 1, 24 * 24)
        out = layer.shard_pool(idx, wt, pos, layer.shard_lookup(rows))
    else:
        out = layer.lookup_reduce(idx, wt)
    assert layer.check() == binding.OK
    layer.close()
    acc = w["values"][idx.flatten()].double()
    want = (acc.unsqueeze(-1) * W[:, [0, 5, 64, 100, 300, 301]].double()).sum(1)
    _same_kind(out[:, [0, 5, 64, 100, 300, 301]], want)


@pytest.mark.parametrize("B", [513, 1001])
def test_infinite_gradients(B, gpu_lib):
    cfg, w, idx, wt, gen = _layer(B, 256)
    g = torch.randn((B, 256), generator=gen, device="cuda").bfloat16()
    g[5, 3] = float("inf")
    g[0, 9] = -float("inf")                        # meets the pooled row of zeros
    g[6, 20], g[7, 20] = float("inf"), -float("inf")
    g[11, 40] = float("nan")
    layer = binding.UltraMemLayer(cfg, w, B)
    dwp = layer.lookup_reduce_backward(idx, wt, g)[2][0]
    assert layer.check() == binding.OK
    layer.close()
    acc = w["values"][idx.flatten()].double()
    cols = [0, 3, 9, 20, 40]
    want = (acc.unsqueeze(-1) * g[:, None, cols].double()).sum(0)
    _same_kind(dwp[:, cols], want)
