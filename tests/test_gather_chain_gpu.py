"""The bf16 gather's sums of long batches at E = 9 and 16: a sum that begins
with 2^24 loses the ones that follow it in the same partial sum, so what is
missing shows how many terms a partial sum takes one after the other: at most
the 7 of a run of 8 slots."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [9, 16])
@pytest.mark.parametrize("m", [64, 61])
def test_partial_sums(E, m, gpu_lib):
    B = 400
    cfg = workloads.small_config(dtype=1, expand_e=E, heads=1, topk=m, topm=m, n=30, d_v=64,
                                 d_out=64, shuffle_seed=0)
    w = workloads.make_weights(cfg, device="cuda")
    w["values"][:] = 1.0
    w["w_proj"].zero_()
    for q in range(E):
        w["w_proj"][q].fill_diagonal_(1.0)       # out = the blocks' pooled rows, added up
    N = 900
    idx = (torch.arange(B, device="cuda") % E * N).view(B, 1, 1) + torch.arange(m, device="cuda")
    wt = torch.ones((B, 1, m), device="cuda")
    wt[:, :, 0] = 2.0 ** 24
    wt[:, :, m - 1] = -(2.0 ** 24)               # leaves the m - 2 ones, less those lost
    layer = binding.UltraMemLayer(cfg, w, B)
    out = layer.lookup_reduce(idx, wt).float()
    assert layer.check() == binding.OK
    layer.close()
    assert ((m - 2) - out).abs().max() <= 7, out.min()
