"""The lookup-reduce backward of long batches (512 tokens and more on the
tensor cores: dW_p from the gradient rows and the pooled rows as they are)
against the oracle: ragged token and column counts, one tile column to many,
component cores, and more slots than the address-reading gather takes."""
import pytest

from paper_2411_12364_gb300 import workloads
from tests.test_backward_gpu import _run

pytestmark = pytest.mark.gpu

CASES = [
    # (overrides, tokens, kernels launched)
    (dict(), 511, 5),                                      # below: 511 is not whole 16-byte rows
    (dict(), 512, 4),
    (dict(), 513, 4),                                      # a K block of one token
    (dict(d_out=264, d_v=72), 577, 4),                     # ragged rows and columns
    (dict(d_out=1024, d_v=256), 600, 4),                   # 64-column tiles
    (dict(d_out=2048, d_v=256, expand_e=16, n=7), 520, 4), # 256-column tiles
    (dict(cores=2), 640, 4),
    (dict(topk=16, topm=140), 520, 5),                     # 280 slots: the slots kernel
    (dict(d_out=84), 512, 4),                              # rows off 16 bytes: CUDA cores
    (dict(dtype=0), 512, 5),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_backward_long_batches(case, gpu_lib):
    over, B, launches = CASES[case]
    cfg = workloads.small_config(**dict(dict(dtype=1), **over))
    layer = _run(cfg, B)
    if over.get("d_out") != 84:
        assert layer.last_launches() == launches


def test_backward_long_bad_address(gpu_lib):
    _run(workloads.small_config(dtype=1), 530, bad=True)
