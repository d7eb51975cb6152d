"""The brute-force grid top-m (Eq. 5) where its kernel's layout changes: odd
and tiny grids (padded rows, fewer columns than threads), more columns than
the threads hold at once, ranks with and without 32-wide chunks, rows split
over several CTAs and merged, m up to 1024, and ties beyond the candidate
list (the radix select)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2411_12364_gb300 import binding, workloads
from tests.test_exact_gpu import _compare_exact, _layer

pytestmark = pytest.mark.gpu

CASES = [
    # (overrides, tokens)
    (dict(n=1, expand_e=4, topk=2, topm=3), 2),                    # a 2 x 2 grid
    (dict(n=37, expand_e=9, d_out=72), 3),                         # K = 111
    (dict(n=517, expand_e=1, has_proj=0, d_out=64, heads=1), 2),   # K = 517, 16 shares
    (dict(n=1100, heads=1), 1),                                    # K = 2200: two column blocks
    (dict(n=130, rank=4, d_k=128), 3),                             # 32-wide chunks
    (dict(n=130, rank=3, d_k=96), 3),                              # 3 chunks of the 4 held
    (dict(n=130, rank=5, d_k=40), 3),                              # 8-wide chunks
    (dict(n=100, topk=32, topm=1024), 3),                          # m = 1024
    (dict(n=100, topk=32, topm=64, heads=1), 1),                   # 3 shares of rows
    (dict(n=150, rank=1, score_mode=1, d_k=64), 3),                # product keys
    (dict(n=150, rank=1, d_k=64, dtype=0), 3),
    # 512 rows and more: rows that cannot hold a winner are dropped
    (dict(n=300, d_k=128, heads=4), 40),                           # 16-byte stages, two a chunk
    (dict(n=300, d_k=64, rank=1, score_mode=1, heads=4), 40),
    (dict(n=300, d_k=64, dtype=0, heads=4, topk=32, topm=500), 40),
    (dict(n=260, d_k=256, rank=4, heads=4), 40),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_exact_topm_layouts(case, gpu_lib):
    over, B = CASES[case]
    cfg = workloads.small_config(**dict(dict(dtype=1), **over))
    layer, w, x, t = _layer(cfg, B)
    g_idx, g_w = layer.retrieve_exact(x)
    torch.cuda.synchronize()
    assert layer.check() == 0
    tokens = np.unique(np.linspace(0, B - 1, min(B, 4)).astype(int))
    o_idx, o_w = oracle.exact_topm(cfg, t, B, tokens=tokens)
    _compare_exact(cfg, t, tokens, g_idx.cpu().numpy(), g_w.cpu().numpy(), o_idx, o_w)
    layer.close()


@pytest.mark.parametrize("B", [1, 90])
def test_ties_beyond_the_list(B, gpu_lib):
    """200 x 200 equal scores (40 000 > 2048 listed): the m smallest
    addresses, with the rows split over CTAs (1 token) and not (90)."""
    cfg = workloads.small_config(dtype=1, n=100, topm=40)
    w = workloads.make_weights(cfg, device="cuda")
    w["k_row"][:] = w["k_row"][:, :1]
    w["k_col"][:] = w["k_col"][:, :1]
    layer, w, x, t = _layer(cfg, B, w)
    g_idx, _ = layer.retrieve_exact(x)
    assert layer.check() == 0
    assert torch.equal(g_idx.cpu(), torch.arange(40).expand(B, cfg["heads"], 40))
    layer.close()


def test_equal_row_lengths_keep_every_row(gpu_lib):
    """Keys of +-1/8 entries: every R has nearly the same length, so no row can
    be dropped, and many scores tie."""
    cfg = workloads.small_config(dtype=1, n=300, d_k=64, heads=4, topm=20)
    w = workloads.make_weights(cfg, device="cuda")
    for name in ("k_row", "k_col"):
        w[name] = (w[name].float().sign() / 8).bfloat16()
    layer, w, x, t = _layer(cfg, 40, w)
    g_idx, g_w = layer.retrieve_exact(x)
    assert layer.check() == 0
    sample = np.array([0, 39])
    o_idx, o_w = oracle.exact_topm(cfg, t, 40, tokens=sample)
    _compare_exact(cfg, t, sample, g_idx.cpu().numpy(), g_w.cpu().numpy(), o_idx, o_w)
    layer.close()


def test_largest_grid_of_chunk_scores(gpu_lib):
    """The widest grid the chunk scores fit (K r + D_k = 27 868 words of
    shared memory beside the rest): the call still runs."""
    cfg = workloads.small_config(dtype=1, n=3475, expand_e=16, d_k=64, heads=1, shard_rows=16)
    K = 4 * cfg["n"]
    g = torch.Generator(device="cuda").manual_seed(1)
    w = {"w_q": torch.randn(64, cfg["d_in"], generator=g, device="cuda").bfloat16(),
         "k_row": torch.randn(1, K, 64, generator=g, device="cuda").bfloat16(),
         "k_col": torch.randn(1, K, 64, generator=g, device="cuda").bfloat16(),
         "core": torch.eye(2)[None] * torch.tensor([2.0, 1.0]),
         "values": torch.zeros(16, cfg["d_v"], dtype=torch.bfloat16, device="cuda"),
         "w_proj": torch.zeros(16, cfg["d_v"], cfg["d_out"], dtype=torch.bfloat16,
                               device="cuda")}
    layer = binding.UltraMemLayer(cfg, w, 1)
    x = torch.randn(1, cfg["d_in"], generator=g, device="cuda").bfloat16()
    idx, s = layer.retrieve_exact(x)
    assert layer.check() == 0
    q = x.float() @ w["w_q"].float().T
    sr = (w["k_row"][0].float() * q).view(K, 2, 32).sum(-1)
    sc = (w["k_col"][0].float() * q).view(K, 2, 32).sum(-1)
    top = ((sr * torch.tensor([2.0, 1.0], device="cuda")) @ sc.T).flatten().topk(cfg["topm"])
    assert np.allclose(s[0, 0].cpu(), top.values.cpu(), rtol=1e-4)
    layer.close()
