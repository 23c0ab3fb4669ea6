"""A decode loop's parameters can be asked about before its first step."""
import pytest
import torch

import paper_2512_07503_b200 as sjd
from paper_2512_07503_b200.decode import DecodeLoop

pytestmark = pytest.mark.gpu


def test_parameters_of_a_new_loop():
    loop = DecodeLoop(batch=2, window=12, vocab=8192, n_total=40, logits_dtype=torch.bfloat16, top_k=300)
    assert (loop.params.stride_b, loop.params.stride_w) == (12 * 8192, 8192)
    assert sjd.sjd_row_kernel(loop.params) == 2 and sjd.sjd_row_path(loop.params) == 3
