"""The largest batches that a layer accepts on the CUDA-core path (2^20
tokens): every grid stays within the device's limits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_12364_gb300 import binding, workloads
from tests import parity

pytestmark = pytest.mark.gpu

SAMPLE = np.array([0, 15, 16, 1048544, 1048559, 1048560])


@pytest.mark.parametrize("dtype,d_in", [(0, 8), (1, 12)])
def test_largest_batch(dtype, d_in, gpu_lib):
    B = 1048561                       # 65536 tiles of 16 tokens
    cfg = workloads.small_config(dtype=dtype, d_in=d_in, d_k=8, heads=1, n=8, expand_e=1, d_v=8,
                                 d_out=8, topk=1, topm=1)
    w = workloads.make_weights(cfg, device="cuda")
    x = workloads.make_tokens(cfg, B, device="cuda")
    t = parity.numpy_inputs(cfg, w, x)
    layer = binding.UltraMemLayer(
        cfg, dict(w, u=torch.from_numpy(t["u"]), t=torch.from_numpy(t["t"])), 1 << 20)
    out, idx, wt = layer.forward(x, with_slots=True)
    again = layer.lookup_reduce(idx, wt)
    assert layer.check() == binding.OK
    layer.close()
    assert torch.equal(out, again)
    o_out, o_idx, o_w = oracle.forward(cfg, t, B, tokens=SAMPLE)
    parity.compare(cfg, t, SAMPLE, out.float().cpu().numpy(), idx.cpu().numpy(),
                   wt.cpu().numpy(), o_out, o_idx, o_w)
