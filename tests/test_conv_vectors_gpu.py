"""Trick 4's convolution where it takes 8 channels of 1 or 4 tokens a thread
(bf16 rows of whole 16-byte vectors) and where it does not: sequence ends
inside a thread's tokens, a ragged last group, the state's rows."""
import pytest

from paper_2411_12364_gb300 import workloads
from tests.test_query_extras_gpu import _run_seq

pytestmark = pytest.mark.gpu

CASES = [
    # (overrides, n_seq, seq_len)
    (dict(d_in=1024, conv_k=4), 3, 407),    # 1221 tokens: four a thread
    (dict(d_in=1024, conv_k=6), 500, 3),    # sequences shorter than the taps' reach
    (dict(d_in=1024, conv_k=4), 1, 300),    # one token a thread
    (dict(d_in=104, conv_k=3), 5, 7),
    (dict(d_in=100, conv_k=3), 5, 7),       # no whole vectors
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_convolution_layouts(case, gpu_lib):
    over, n_seq, L = CASES[case]
    _run_seq(workloads.small_config(dtype=1, **over), n_seq, L, gpu_lib)
