"""A batched prefill gives a request the same bits whichever requests are prefilled with it.

The batches below hold 16 to 1008 rows (padded), so the dense projections take every tile width from 32 tokens up and,
were a tile's K steps shared for few rows, would add them in another order: K is 640, 768 and 4096 here, few weight
tiles each.  Request 0's K/V rows, first-token logits and token are compared with those of the request on its own.
"""
import pytest
import torch

import synth
from tests.gpu_util import make_model

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 150])
def test_request_does_not_depend_on_its_batch(n):
    shape = synth.ModelShape(2, 640, 12, 64, 4096, 1000)
    w = synth.TINY.replace(shape=shape, draft_exit_k=1, in_hidden=256, norm_gain="perturbed", gamma=1)
    model, _, _ = make_model(w, gamma_max=1, max_seq=600, max_batch=4)
    g = torch.Generator(device="cuda").manual_seed(11)
    prompt = torch.randint(0, shape.vocab, (4 * 600,), generator=g, device="cuda", dtype=torch.int32)
    try:
        ref = None
        for others in ([], [1], [40, 7], [90], [13, 200], [330, 17, 500]):
            B = 1 + len(others)
            lens = [n] + others
            logits = torch.full((B, 1, shape.vocab), float("nan"), device="cuda")
            first = torch.zeros(B, dtype=torch.int32, device="cuda")
            model.set_logits_capture(logits)
            model.prefill_batch(None, [0] * B, prompt[: sum(lens)], lens, first)
            model.sync()
            k, v, _ = model.kv()
            got = (k[:, 0, :, :n].clone(), v[:, 0, :, :n].clone(), logits[0].clone(), first[:1].clone())
            ref = ref or got
            assert all(torch.equal(a, b) for a, b in zip(got, ref)), others
    finally:
        model.set_logits_capture(None)
        model.close()
