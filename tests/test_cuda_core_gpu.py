"""The CUDA-core path (fp32 storage, and bf16 layers whose rows TMA cannot
read) against the oracle where its tiling changes: 4-token and 16-token tiles,
slices of D_i that are not whole quads, the cluster's sum of the query's
splits, rank chunks with and without whole stages of 32, K and D'_v off the
quads, fp32 value rows of 33 to 64 vectors, and infinite values."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_12364_gb300 import binding, workloads
from tests import parity

pytestmark = pytest.mark.gpu

CASES = [
    # (overrides, tokens)
    (dict(), 3),
    (dict(d_in=1024, heads=4, d_k=128), 5),                # 8 splits, 4-token tiles
    (dict(d_in=1024, heads=4, d_k=128, n=100), 160),       # 16-token tiles
    (dict(d_in=1023, d_out=83), 21),                       # no quads
    (dict(d_in=600, d_k=96, rank=3), 33),                  # chunks of 32
    (dict(d_in=600, d_k=80, rank=2), 33),                  # chunks of 40
    (dict(n=25, expand_e=9, d_out=72), 17),                # K = 75
    (dict(d_v=256, d_out=260, heads=4), 33),               # two vectors a lane
    (dict(d_v=136, d_out=64), 310),                        # a partial second vector, 256 threads
    (dict(d_v=256, cores=4, d_out=64), 40),                # a slice within a vector pair
    (dict(d_v=264, d_out=64), 9),                          # wider rows: the general kernel
    (dict(expand_e=1, has_proj=0, d_v=256, d_out=256, n=50), 12),
    (dict(conv_k=3, query_ln=1, d_in=512), 9),             # the LayerNorm adds the splits
    (dict(share_query=0, d_in=512), 70),
    (dict(dtype=1, d_in=97), 40),                          # bf16 rows TMA cannot read
    (dict(dtype=1, d_in=1001, conv_k=2), 40),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_cuda_core_layers(case, gpu_lib):
    over, B = CASES[case]
    cfg = workloads.small_config(**dict(dict(dtype=0), **over))
    w = workloads.make_weights(cfg, device="cuda")
    x = workloads.make_tokens(cfg, B, device="cuda")
    t = parity.numpy_inputs(cfg, w, x)
    layer = binding.UltraMemLayer(
        cfg, dict(w, u=torch.from_numpy(t["u"]), t=torch.from_numpy(t["t"])), B)
    out, idx, wt = layer.forward(x, with_slots=True)
    torch.cuda.synchronize()
    assert layer.check() == 0
    o_out, o_idx, o_w = oracle.forward(cfg, t, B)
    parity.compare(cfg, t, np.arange(B), out.float().cpu().numpy(), idx.cpu().numpy(),
                   wt.cpu().numpy(), o_out, o_idx, o_w)
    layer.close()


@pytest.mark.parametrize("d_v", [64, 256])
def test_infinite_values_pool_to_infinity(d_v, gpu_lib):
    """Without a projector a pooled column that meets an infinite value is
    infinite (a NaN only where the plain sum is one), and no other is."""
    cfg = workloads.small_config(dtype=0, expand_e=1, has_proj=0, d_v=d_v, d_out=d_v, n=40,
                                 shuffle_seed=0)
    w = workloads.make_weights(cfg, device="cuda")
    w["values"][7, 5] = float("inf")
    idx = torch.arange(3 * 2 * 8).view(3, 2, 8).cuda()
    wt = torch.ones((3, 2, 8), device="cuda")
    layer = binding.UltraMemLayer(cfg, w, 3)
    out = layer.lookup_reduce(idx, wt)
    assert torch.isinf(out[0, 5]) and out[0, 5] > 0
    out[0, 5] = 0
    assert torch.isfinite(out).all()
    layer.close()
