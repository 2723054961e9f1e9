"""The batched verification's dense projections sum as exactly as the weight-streaming kernel's.

With draft_exit_k = n_layers the verification is the LM head alone: 32 rows (4 requests, gamma = 7) go through the
dense projections, the same hidden states (equal bit by bit) through the weight-streaming kernel in the greedy run.
Both carry the rows as the same hi and lo parts, so only the accumulation differs.  At K = 8192 the two kernels' logits
lie 1.8e-6 apart (2-norm) when both accumulate hi and lo products separately, 4.1e-6 when the dense kernel adds them
to one accumulator; 3e-6 is asked for.
"""
import pytest
import torch

import synth
from tests.gpu_util import make_model
from tests.test_gpu_batch import gpu_batch

pytestmark = pytest.mark.gpu


def test_verification_head_agrees_with_greedy_head():
    shape = synth.ModelShape(1, 8192, 2, 64, 64, 2000)
    base = synth.TINY.replace(shape=shape, draft_exit_k=1, in_kind=synth.IN_IDENTITY, n_vis=4, max_new=12)
    bw = synth.TINY_B4.replace(base=base)
    model, _, _ = make_model(base, gamma_max=7, max_seq=bw.max_seq() + 8, max_batch=4)
    try:
        ssd, greedy = gpu_batch(model, bw, 7), gpu_batch(model, bw, 0)
        for a, g in zip(ssd, greedy):
            assert a["tokens"] == g["tokens"]
            x, y = (torch.from_numpy(r["logits"]).double()[1:] for r in (a, g))  # row 0: the prefill's
            assert (x - y).norm() <= 3e-6 * y.norm()
    finally:
        model.close()
