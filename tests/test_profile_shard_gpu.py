"""A shard_pool on a layer that profiles leaves the stage times of the last
profiled call as they are."""
import time

import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


# the CUDA-core and the tensor-core projection
@pytest.mark.parametrize("d_v,d_out,B", [(64, 80, 20), (256, 1024, 40)])
def test_shard_pool_writes_no_stamps(d_v, d_out, B, gpu_lib):
    cfg = workloads.small_config(dtype=1, d_v=d_v, d_out=d_out, n=24)
    layer = binding.UltraMemLayer(cfg, workloads.make_weights(cfg, device="cuda"), B)
    x = workloads.make_tokens(cfg, B, device="cuda")
    _, idx, wt = layer.forward(x, with_slots=True)
    counts, rows, pos = layer.shard_route(idx, 1, 24 * 24)
    back = layer.shard_lookup(rows)
    layer.profile(True)
    layer.forward(x)
    torch.cuda.synchronize()
    before = layer.profile_read(gaps=True)
    time.sleep(0.01)
    layer.shard_pool(idx, wt, pos, back)
    torch.cuda.synchronize()
    assert layer.profile_read(gaps=True) == before
    layer.close()
