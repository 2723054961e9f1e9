"""Batched requests on a wide model, whose decode rows all stream (K = 4160 is beyond the small-matrix kernel).

At 7B and 13B widths drafting and small verifications run through the weight-streaming kernel with batched rows:
positions, cache slots and strided draft rows per request.  d = d_ff = 4160 reaches that form of q/k/v (head_dim 64
and 128, with rotation), gate/up, down (whose draft rows lie gamma + 1 rows apart), the imitation network and the
head.  Three requests verify 6 to 15 rows; every request must match the oracle run on it alone.

Above 16 rows the dense projections share each tile's K steps: 65 steps and few weight tiles, so that q/k/v, gate/up,
down and the head run with two to four CTA pairs per tile at 32 to 128 rows, an owner with several 16-row chunks and,
at 70 rows, a last chunk of 6.  The reference is the greedy run of the same batch (at most 16 rows, streamed).
"""
import numpy as np
import pytest
import torch

import synth
from tests.gpu_util import make_model
from tests.test_gpu_batch import check_request, gpu_batch, oracle_runs, set_scale

pytestmark = pytest.mark.gpu


def wide(head_dim, batch=3, **kw):
    shape = synth.ModelShape(2, 4160, 1024 // head_dim, head_dim, 4160, 6000)
    base = synth.TINY.replace(shape=shape, draft_exit_k=1, in_hidden=192, norm_gain="perturbed", n_vis=4, max_new=6,
                              s=0.2, **kw)
    return synth.TINY_B4.replace(base=base, batch=batch, prompt_min=2, prompt_max=12)


@pytest.fixture(scope="module", params=[64, 128])
def bits(request):
    return request.param, synth.make_weights(wide(request.param).base)


def test_streamed_batch_matches_oracle(bits):
    head_dim, b = bits
    bw = wide(head_dim, gamma=4)
    model, _, _ = make_model(bw.base, b, gamma_max=4, max_seq=bw.max_seq(), max_batch=3)
    try:
        set_scale(model, bw.base)
        for r, ref in zip(gpu_batch(model, bw, 0), oracle_runs(bw, b, 0, greedy=True)):
            check_request(r, ref, 0)
        for gamma in (1, 4):
            for r, ref in zip(gpu_batch(model, bw, gamma), oracle_runs(bw, b, gamma)):
                check_request(r, ref, gamma)
    finally:
        model.close()


def close(a, ref):
    """Within 1e-4 of the rms: products of two bf16 parts (2^-17) behind at most 14 projections, sums in any order."""
    return (a - ref).double().pow(2).mean().sqrt() <= 1e-4 * ref.double().pow(2).mean().sqrt()


@pytest.mark.parametrize("batch,gamma", [(4, 7), (5, 13), (16, 6), (8, 15)])
def test_shared_k_steps_of_a_verification(bits, batch, gamma):
    head_dim, b = bits
    bw = wide(head_dim, batch, gamma=gamma)
    model, _, _ = make_model(bw.base, b, gamma_max=gamma, max_seq=bw.max_seq(), max_batch=batch)
    try:
        set_scale(model, bw.base)
        for a, g in zip(gpu_batch(model, bw, gamma), gpu_batch(model, bw, 0)):
            n = next((i for i, (x, y) in enumerate(zip(a["tokens"], g["tokens"])) if x != y), len(g["tokens"]))
            if n < len(g["tokens"]):  # only a near-tie may part them
                top = np.sort(g["logits"][n])
                assert top[-1] - top[-2] < 1e-3
            assert close(torch.from_numpy(a["logits"][: n + 1]), torch.from_numpy(g["logits"][: n + 1]))
    finally:
        model.close()


def test_shared_k_steps_of_a_prefill(bits):
    """One prompt's prefill shares K steps, a batched prefill of the same prompt does not."""
    head_dim, b = bits
    w = wide(head_dim).base
    model, _, _ = make_model(w, b, gamma_max=1, max_seq=320, max_batch=2)
    g = torch.Generator(device="cuda").manual_seed(2)
    prompt = torch.randint(0, w.shape.vocab, (300,), generator=g, device="cuda", dtype=torch.int32)
    try:
        set_scale(model, w)
        for n in (1, 17, 70, 112, 150, 300):
            out = []
            for batched in (False, True):
                logits = torch.full((2, 1, w.shape.vocab), float("nan"), device="cuda")
                model.set_logits_capture(logits)
                if batched:
                    model.prefill_batch(None, [0], prompt[:n], [n])
                else:
                    model.prefill(None, prompt[:n].clone())
                model.sync()
                k, v, _ = model.kv()
                out.append([t[:, 0, :, :n].clone() for t in (k, v)] + [logits[0]])
            assert all(close(a, r) for a, r in zip(*out)), n
    finally:
        model.set_logits_capture(None)
        model.close()
