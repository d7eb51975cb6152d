"""Long grids of tokens whose scores tie (padding tokens of zeros): the ties go
to the smaller addresses, and such a batch is not many times slower than
another one."""
import pytest
import torch

from paper_2411_12364_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

B = 1000   # 2000 (token, head)s


@pytest.mark.parametrize("mode", [0, 1], ids=["every_key", "lists"])
@pytest.mark.parametrize("over", [
    dict(), dict(topk=63, topm=61), dict(topk=32, topm=32), dict(topk=5, topm=5),
    dict(topk=48, topm=7), dict(rank=1, score_mode=1, act=1), dict(rank=3, d_k=96),
    dict(rank=4), dict(cores=2), dict(n=2300, topk=40, topm=40)])
def test_zero_tokens(over, mode, gpu_lib):
    cfg = workloads.small_config(**dict(dict(dtype=1, n=600, d_k=128, topk=64, topm=64), **over))
    w = workloads.make_weights(cfg, device="cuda")
    x = workloads.make_tokens(cfg, B, device="cuda")
    x[5:700] = 0
    layer = binding.UltraMemLayer(cfg, w, B)
    layer.candidates(mode)
    idx, wt = layer.retrieve(x)
    assert layer.check() == binding.OK
    m = cfg["topm"]
    # row 0 with columns 0, 1, ...: m <= k of them
    assert (idx[5:700] == torch.arange(m, device="cuda")).all()
    assert (wt[5:700] == (1.0 / m if cfg["act"] else 0.0)).all()
    # the other tokens' as without the zeros
    other, wo = layer.retrieve(x[700:].contiguous())
    layer.close()
    assert torch.equal(idx[700:], other) and torch.equal(wt[700:], wo)


@pytest.mark.parametrize("mode", [0, 1], ids=["every_key", "lists"])
def test_partly_tied_keys(mode, gpu_lib):
    """Some keys above a tie of 900 on each axis: those first, then the tied ones
    by position; and the pairs of tied rows and columns by address."""
    cfg = workloads.small_config(dtype=1, n=600, d_k=128, topk=64, topm=64, share_query=1)
    w = workloads.make_weights(cfg, device="cuda")
    for name in ("k_row", "k_col"):
        w[name][:, 100:1000] = w[name][:, :1]
    x = workloads.make_tokens(cfg, B, device="cuda")
    layer = binding.UltraMemLayer(cfg, w, B)
    layer.candidates(mode)
    idx = layer.retrieve(x)[0]
    few = layer.retrieve(x[:64].contiguous())[0]         # a block per (token, head)
    assert layer.check() == binding.OK
    layer.close()
    assert torch.equal(idx[:64], few)


def test_zero_tokens_time(gpu_lib):
    """At most 4 times the time of Gaussian tokens (it is about as long; 9 times
    with a block after the other for each)."""
    cfg = workloads.small_config(dtype=1, n=1024, d_k=128, heads=2, topk=64, topm=64)
    w = workloads.make_weights(cfg, device="cuda")
    x = workloads.make_tokens(cfg, 1024, device="cuda")
    layer = binding.UltraMemLayer(cfg, w, 1024)

    def best(x):
        t = []
        for _ in range(20):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(5):
                layer.retrieve(x)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return min(t)

    gauss, zero = best(x), best(torch.zeros_like(x))
    layer.close()
    assert zero <= 4 * gauss, (zero, gauss)
