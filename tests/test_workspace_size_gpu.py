"""The tensor path's pooled rows take one array of three bf16 terms, which the
fp32 rows of the CUDA-core projection share."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


def test_pooled_rows_share_one_array(gpu_lib):
    B, d_v, E = 16384, 256, 16
    cfg = workloads.small_config(dtype=1, expand_e=E, d_v=d_v, d_out=64, heads=1, n=8, topk=8,
                                 topm=8)
    w = workloads.make_weights(cfg, device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    layer = binding.UltraMemLayer(cfg, w, B)
    used = free - torch.cuda.mem_get_info()[0]
    layer.close()
    values = B * E * d_v
    # per value: 6 bytes (three terms), 4 (the backward's dacc), 4 (its transposed
    # terms); the rest of the workspace is below 1 byte a value here
    assert used <= 15 * values, used / values
