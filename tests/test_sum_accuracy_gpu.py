"""The tensor-core sums of the lookup-reduce and its backward against a chain
of fp32 multiply-adds: their error against 64 bits is no larger than such a
chain's, at the sizes where the kernels split the sum differently (over CTAs,
over accumulators, over K blocks in the epilogue's registers).

One slot a token and no virtual expansion: the pooled row is a single product
w * v rounded to fp32, which the test works out itself, so that the sums are
all that can differ."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def _layer(B, d_v, d_out, seed=5):
    cfg = workloads.small_config(dtype=1, expand_e=1, heads=1, topk=1, topm=1, n=24, d_v=d_v,
                                 d_out=d_out, shuffle_seed=0)
    w = workloads.make_weights(cfg, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed)
    idx = torch.randint(0, 24 * 24, (B, 1, 1), generator=gen, device="cuda")
    wt = torch.randn((B, 1, 1), generator=gen, device="cuda") + 2.0
    acc = w["values"][idx.flatten()].float() * wt.view(B, 1)   # [B, d_v], one rounding
    return cfg, w, idx, wt, acc, gen


def _chain(a, b):
    """sum_k a[k, m] b[k, n] by fp32 multiply-adds in increasing k."""
    s = torch.zeros((a.shape[1], b.shape[1]), dtype=torch.float32, device="cuda")
    for k in range(a.shape[0]):
        # the product of an fp32 and a bf16 value is exact in fp64, and the sum of
        # it and s loses no bit that would turn the fp32 rounding (but for ties)
        s = torch.addr(s.double(), a[k].double(), b[k].double()).float()
    return s


@pytest.mark.parametrize("B,d_v,d_out", [
    (1, 4096, 1024),       # 8 splits
    (40, 4096, 1024),
    (64, 4096, 2048),
    (64, 1024, 2048),
    (100, 4096, 1024),     # 4 splits, 64-token tiles
    (300, 4096, 1024),     # 4 splits, 128-token tiles
    (127, 4096, 16384),    # below 128 tokens, unsplit
    (77, 1024, 16384),     # 80 columns: 96 a buffer, of 128
    (700, 4096, 1024),     # token rows, 128 outputs a tile, fewer tiles than SMs
    (2000, 4096, 2048),    # 256 outputs a tile
    (2000, 1024, 2048),
    (2000, 960, 2048),     # 15 K blocks
    (2000, 128, 2048),
])
def test_projection_sums(B, d_v, d_out, gpu_lib):
    """The share of outputs that are not the correctly rounded ones."""
    cfg, w, idx, wt, acc, _ = _layer(B, d_v, d_out)
    layer = binding.UltraMemLayer(cfg, w, B)
    out = layer.lookup_reduce(idx, wt)
    assert layer.check() == binding.OK
    layer.close()
    wp = w["w_proj"][0]
    right = (acc.double() @ wp.double()).bfloat16()
    chain = int((_chain(acc.T, wp).bfloat16() != right).sum())
    got = int((out != right).sum())
    # both counts are of rare independent events: three standard deviations
    assert got <= chain + 3 * (2 * chain) ** 0.5 + 3, (got, chain)


@pytest.mark.parametrize("B", [513, 1001, 2047, 4095])
def test_projector_gradient_sums(B, gpu_lib):
    """dW_p of token counts that are not whole 16-byte rows: rms error."""
    cfg, w, idx, wt, acc, gen = _layer(B, 256, 256)
    g = torch.randn((B, 256), generator=gen, device="cuda").bfloat16()
    layer = binding.UltraMemLayer(cfg, w, B)
    dwp = layer.lookup_reduce_backward(idx, wt, g)[2][0]
    assert layer.check() == binding.OK
    layer.close()
    right = acc.double().T @ g.double()
    rms = (dwp.double() - right).square().mean().sqrt()
    chain = (_chain(acc, g).double() - right).square().mean().sqrt()
    assert rms <= chain, (float(rms), float(chain))
