"""fp32 storage: pooled rows and split sums of the projection whose partial
sums pass the largest fp32 value and come back, and products below 2^-102,
against fp64 sums rounded once."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

BIG = 3e38


def _pooling_layer(d_v, B, cores=0):
    cfg = workloads.small_config(dtype=0, expand_e=1, has_proj=0, d_v=d_v, d_out=d_v, heads=1,
                                 topm=16, topk=16, n=40, shuffle_seed=0, cores=cores)
    return cfg, workloads.make_weights(cfg, device="cuda")


@pytest.mark.parametrize("d_v,B,cores", [(64, 5, 0), (64, 310, 0), (256, 5, 0), (256, 310, 0),
                                         (256, 5, 4)])
def test_pooled_range(d_v, B, cores, gpu_lib):
    cfg, w = _pooling_layer(d_v, B, cores)
    gen = torch.Generator(device="cuda").manual_seed(3)
    V = w["values"]
    V[:4, 1] = torch.tensor([BIG, BIG, -BIG, -1e38])      # the sum passes FLT_MAX
    V[:16, 2] = 1e-20 * torch.randn(16, generator=gen, device="cuda")
    V[:16, 3] = 1e-25 * torch.randn(16, generator=gen, device="cuda")
    V[:16, 4] = 0
    V[:4, 5] = torch.tensor([BIG, BIG, BIG, 1.0])          # beyond fp32 at the end as well
    idx = torch.arange(16, device="cuda").expand(B, 1, 16).contiguous()
    wt = torch.ones((B, 1, 16) if not cores else (B, 1, 16, cores), device="cuda")
    small = torch.full_like(wt, 1e-18)
    layer = binding.UltraMemLayer(cfg, w, B)
    for weights in (wt, small):
        out = layer.lookup_reduce(idx, weights)
        w0 = weights[0, 0].double().reshape(16, -1)
        w0 = w0.repeat_interleave(d_v // w0.shape[1], 1)
        want = (V[:16].double() * w0).sum(0).float()
        # one rounding of an fp64 sum, whose order is not fixed: to the next fp32
        assert torch.equal(out.isinf(), want.isinf().expand_as(out))
        fin = want.isfinite()
        off = (out.view(torch.int32)[:, fin] - want.view(torch.int32)[fin]).abs()
        tiny = want[fin].abs() < 1e-3 * V[:16].abs().max(0).values[fin] * float(weights.max())
        assert int(off[:, ~tiny].max()) <= 1, off.max()
        for c in (1, 2, 3, 4):
            j = int(fin[:c].sum())
            assert fin[c] and int(off[:, j].max()) <= 1, (c, off[:, j].max())
    layer.close()


def test_split_projection_range(gpu_lib):
    """Partial sums of the projection's splits that pass FLT_MAX together."""
    cfg = workloads.small_config(dtype=0, expand_e=1, heads=1, topk=1, topm=1, n=24, d_v=1024,
                                 d_out=64, shuffle_seed=0)
    w = workloads.make_weights(cfg, device="cuda")
    w["values"][:] = 1.0
    W = w["w_proj"][0]
    W.zero_()
    W[0, :], W[128, :], W[256, :], W[700, :] = BIG, BIG, -BIG, -1e38    # 8 splits of 128
    layer = binding.UltraMemLayer(cfg, w, 3)
    out = layer.lookup_reduce(torch.zeros((3, 1, 1), dtype=torch.int64, device="cuda"),
                              torch.ones((3, 1, 1), device="cuda"))
    layer.close()
    assert torch.equal(out, W.double().sum(0).float().expand_as(out))
