"""GPU parity of the lookup-reduce on given slots (S7-S9, Eq. 14-15) where its
dispatch changes: the gather that reads addresses (512 threads up to 304
tokens, above a warp per block or, with component cores, 256 threads; the
slots kernel for more slots than those serve) and the
tensor-core projection with the pooled rows as three bf16 terms (split over
its inner dimension at small batches, persistent at long ones)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_12364_gb300 import binding, workloads
from tests import parity

pytestmark = pytest.mark.gpu


def _slots(cfg, B, seed=3):
    gen = torch.Generator().manual_seed(seed)
    M = int(cfg["expand_e"]) * int(cfg["n"]) ** 2
    H, m, h = int(cfg["heads"]), int(cfg["topm"]), max(1, int(cfg.get("cores", 0)))
    idx = torch.randint(0, M, (B, H, m), generator=gen)
    w = torch.randn((B, H, m) if h == 1 else (B, H, m, h), generator=gen)
    return idx.cuda(), w.cuda()


CASES = [
    # (overrides, tokens, kernels launched)
    (dict(d_v=64, d_out=80), 25, 4),                           # below 2^19 multiply-adds
    (dict(d_v=64, d_out=80), 26, 2),                           # above: tensor cores
    (dict(d_v=256, d_out=1024, heads=1), 1, 2),                # one token, split
    (dict(d_v=256, d_out=1000), 37, 2),                        # ragged rows of W_p^T
    (dict(d_v=128, d_out=520, cores=2), 130, 2),               # two weights a slot
    (dict(d_v=128, d_out=523), 200, 2),                        # output rows off 16 bytes
    (dict(d_v=64, d_out=4096), 1000, 2),                       # 256-output tiles, one wave
    (dict(d_v=256, d_out=512, heads=4, topk=16, topm=128), 304, 2),   # 512 slots a token
    (dict(d_v=256, d_out=512, heads=4, topk=16, topm=64), 305, 2),    # 256 threads
    (dict(d_v=256, d_out=512, heads=4, topk=16, topm=65), 305, 3),    # 260 slots: slots kernel
    (dict(d_v=72, d_out=264, expand_e=9, n=11), 700, 2),       # a warp per block; ragged K blocks
    (dict(d_v=256, d_out=512, heads=2, topk=16, topm=70), 305, 2),    # 140 slots: two rounds
    (dict(d_v=128, d_out=512, cores=2, heads=4), 310, 2),      # cores: a CTA per token
    (dict(d_v=256, d_out=2048, topk=16, topm=16), 3000, 2),    # more tiles than SMs
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_lookup_reduce_dispatch(case, gpu_lib):
    over, B, launches = CASES[case]
    cfg = workloads.small_config(dtype=1, **over)
    w = workloads.make_weights(cfg, device="cuda")
    idx, wt = _slots(cfg, B)
    idx[B - 1, 0, 1] = -1                      # skipped and reported
    layer = binding.UltraMemLayer(cfg, w, B)
    out = layer.lookup_reduce(idx, wt)
    assert layer.last_launches() == launches
    assert layer.check() == binding.EDEVICE
    i, f = idx.cpu().numpy(), wt.cpu().numpy().astype(np.float64)
    i[B - 1, 0, 1], f[B - 1, 0, 1] = 0, 0.0
    t = {k: workloads.stored_numpy(v) for k, v in w.items() if k in ("values", "w_proj")}
    err, _ = parity.output_errors(out.float().cpu().numpy(), oracle.lookup_reduce(cfg, t, i, f))
    assert err.max() <= parity.out_tol(cfg), err.max()
    layer.close()


def test_infinite_and_nan_pooled_rows(gpu_lib):
    """A pooled value that is not finite reaches every output of its token as
    a plain product with W_p gives it, and no other token."""
    cfg = workloads.small_config(dtype=1, d_v=256, d_out=1024, topm=4)
    w = workloads.make_weights(cfg, device="cuda")
    w["w_proj"] = w["w_proj"].abs() + 1e-3     # no zeros: inf * w = inf
    idx, wt = _slots(cfg, 6)
    wt[1, 0, 0] = float("inf")
    wt[2, 1, 3] = float("nan")
    w["values"] = w["values"].abs() + 1e-3
    layer = binding.UltraMemLayer(cfg, w, 6)
    out = layer.lookup_reduce(idx, wt).float()
    assert torch.isinf(out[1]).all() and (out[1] > 0).all()
    assert torch.isnan(out[2]).all()
    assert torch.isfinite(out[[0, 3, 4, 5]]).all()
    layer.close()
