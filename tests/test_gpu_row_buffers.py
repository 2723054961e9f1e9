"""The row buffers of a context for batched requests: not held where they are not used, smaller where memory ends.

A context holds the rows of one batched prefill pass (several prompts).  With SSD_OPT_PREFILL_ROWS no prefill uses
them; if they cannot be allocated, one prompt's rows take their place and a pass holds as many prompts as fit.
"""
import pytest
import torch

import paper_2510_22641_gb300 as lib
import synth
from tests.gpu_util import device_weights, make_model

pytestmark = pytest.mark.gpu

W = synth.TINY.replace(draft_exit_k=2, gamma=1)


def test_prefill_rows_holds_no_pass_buffers():
    """8192 rows of d = 256, 4 heads of 64 and d_ff = 1024 are 8 * 256 + 16 * 256 + 4 * 1024 bytes each: 84 MB."""
    dev = device_weights(synth.make_weights(W))
    used = {}
    for options in (0, lib.SSD_OPT_PREFILL_ROWS):
        free = torch.cuda.mem_get_info()[0]
        model, _, _ = make_model(W, {}, dev, gamma_max=1, max_seq=2048, max_batch=4, options=options)
        used[options] = free - torch.cuda.mem_get_info()[0]
        model.close()
    assert used[0] - used[lib.SSD_OPT_PREFILL_ROWS] >= 75e6, used


def test_batched_prefill_with_one_prompts_rows():
    """Every allocation of ssd_create fails once, in turn.  One of them, the pass's rows, has a smaller form: that
    context prefills the same batch in more passes to the same bits; all others report out of memory."""
    dev = device_weights(synth.make_weights(W))
    g = torch.Generator(device="cuda").manual_seed(4)
    lens = [100, 1, 64, 37]
    prompt = torch.randint(0, W.shape.vocab, (sum(lens),), generator=g, device="cuda", dtype=torch.int32)

    def prefill(model):
        logits = torch.full((4, 1, W.shape.vocab), float("nan"), device="cuda")
        model.set_logits_capture(logits)
        model.prefill_batch(None, [0] * 4, prompt, lens)
        model.sync()
        k, v, _ = model.kv()
        out = [logits] + [t[:, b, :, :n].clone() for t in (k, v) for b, n in enumerate(lens)]
        model.set_logits_capture(None)
        return out

    ref, whole = None, []  # countdowns at which ssd_create went on
    for n in range(1, 100):
        lib.set_fault_injection(lib.SSD_FAULT_ALLOC, n)
        try:
            model, _, _ = make_model(W, {}, dev, gamma_max=1, max_seq=112, max_batch=4)
        except lib.SSDError as e:
            assert e.status == 2, n  # SSD_ERR_OOM
            continue
        finally:
            lib.set_fault_injection(lib.SSD_FAULT_NONE, 0)
        got = prefill(model)
        model.close()
        ref = ref or got
        assert all(torch.equal(a, b) for a, b in zip(got, ref)), n
        whole.append(n)
        if len(whole) == 2:
            break
    assert whole[1] > whole[0] + 1, whole  # the first is the row buffers', the second past the last allocation
